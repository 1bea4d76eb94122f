"""The work that a user has this library do, as cases to measure.

run     lattice steps through lb_step_io with the whole trajectory recorded (each step's external forces read
        from and particle records written to page-locked memory), then a snapshot of velocity and density;
loop    the same, one step at a time: forces in, one step, records out and waited for (a controller in the loop);
run27   the D3Q27 lattice: lb_step, the records, a snapshot;
warm    the learned warm start of a box (warmstart.warm_start): network, particle velocities, steady flow, fluid;
train   Adam steps of the network on minibatches, then its parameters read back;
grad    loss and gradients of the network on one batch.

Records are FP64 numbers computed from an FP32 (or 16-bit) fluid and are kept as FP32; the snapshot and the
forces and velocities of a run with 16-bit storage are kept as BF16.
"""
import math
import os

import numpy as np
import torch

import paper_2403_05443_gb300 as pkg
from paper_2403_05443_gb300 import lbsph as L
from paper_2403_05443_gb300 import surrogate as SU
from paper_2403_05443_gb300 import warmstart as W

PREC = {"fp32": L.LB_FP32, "fp16": L.LB_FP16, "bf16": L.LB_BF16}
WEIGHTS = os.path.join(os.path.dirname(os.path.abspath(pkg.__file__)), "surrogate_config5.npy")
MOST_BYTES = 8 * (48**3 + 64**3 + 96**3 + 128**3) * 40 * 19 * 2 # populations moved by the largest listed case


# ---------------------------------------------------------------------------------------------------- the cases
def _run(name, **kw):
    c = dict(kind="run", boxes=1, edges="64", ny=0, nz=0, per_box=1, a=8.0, b=4.0, tau=0.8, drive="force", walls=0,
             precision="fp32", collision=0, steps=100)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a first run: one spheroid in a small box; the launch and the particle chain, not bandwidth
        _run("run_32", edges="32", a=4.0, b=2.0, tau=1.0, steps=200),
        # a controller that sees every step's records before it sets the next force
        _run("loop_64", kind="loop", steps=20),
        # the orientation sweep of the benchmark, default storage and the 16-bit one that meets its drag bound
        _run("sweep_fp32", boxes=8),
        _run("sweep_fp16", boxes=8, precision="fp16"),
        # a spheroid tumbling in a sheared channel (walls, a box that is no cube)
        _run("channel", edges="128", ny=64, nz=128, tau=1.0, drive="shear", walls=1),
        # the uneven batch of squirmers, the largest work, in the smallest storage
        _run("batch_bf16", boxes=32, edges="48,64,96,128", a=6.0, b=3.0, tau=1.0, drive="squirmer",
             precision="bf16", steps=40),
        # a suspension: many spheroids in one box
        _run("suspension", edges="128", per_box=16, a=5.5, b=2.75, tau=1.0),
        # the lattice comparison: the sweep on D3Q27
        _run("sweep_d3q27", kind="run27", boxes=8),
        # the warm start of the suspension, and of a box whose edge is no power of two
        dict(kind="warm", name="warm_128", n=128, ny=128, nz=128, per_box=16, a=8.0, b=4.0, tau=1.0),
        dict(kind="warm", name="warm_96", n=96, ny=96, nz=96, per_box=4, a=8.0, b=4.0, tau=0.8),
        # training at its usual minibatch, and one gradient of a large batch
        dict(kind="train", name="train_512", batch=512, steps=20, lr=1e-3),
        dict(kind="grad", name="grad_4096", batch=4096),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["run"] * 6 + ["loop", "run27", "run27", "warm", "warm", "train", "grad"])
    if kind == "train":
        return dict(kind="train", batch=int(_log(rng, 48, 1024)), steps=rng.randint(8, 24), lr=1e-3)
    if kind == "grad":
        return dict(kind="grad", batch=int(_log(rng, 16, 4096)))
    if kind == "warm":
        n, ny, nz = 4 * rng.randint(10, 32), rng.randint(40, 128), rng.randint(40, 128)
        if rng.random() < 0.5:
            n = ny = nz = rng.choice([48, 64, 80, 96, 128])
        b = round(rng.uniform(2.5, 4.0), 2)
        return dict(kind="warm", n=n, ny=ny, nz=nz, per_box=rng.randint(1, 4), a=round(b * rng.uniform(1.0, 2.0), 2),
                    b=b, tau=round(rng.uniform(0.7, 1.3), 3))
    prec = "fp32" if kind == "run27" else rng.choice(["fp32", "fp32", "fp16", "bf16"])
    steps = int(_log(rng, 8, 100 if kind == "loop" else 250))
    boxes = 1 if kind == "loop" else int(_log(rng, 1, 32))
    while boxes * steps > 1600:
        boxes = max(1, boxes // 2)
    edges = [8 * rng.randint(4, 16) for _ in range(rng.randint(1, 3))]
    while True:
        nodes = sum(edges[k % len(edges)] ** 3 for k in range(boxes))
        if nodes * steps * (27 * 4 if kind == "run27" else 19 * (4 if prec == "fp32" else 2)) <= 0.7 * MOST_BYTES:
            break
        edges = [max(32, e - 8) for e in edges]
        boxes, steps = max(1, boxes - 1), max(8, steps - 4)
    edges = edges[:boxes]
    c = _run(None, kind=kind, boxes=boxes, edges=",".join(map(str, edges)), precision=prec, steps=steps,
             tau=round(rng.uniform(0.65, 1.3), 3))
    c["collision"] = int(prec == "fp32" and rng.random() < 0.25)
    c["b"] = round(rng.uniform(2.0, 4.0), 2)
    c["a"] = round(min(c["b"] * rng.uniform(1.0, 2.5), 0.5 * min(edges) - 5.0, 9.0), 2)
    if kind == "run27":
        c["collision"] = rng.randint(0, 1)
        return c
    c["drive"] = rng.choice(["force", "squirmer"])
    if boxes == 1 and edges[0] >= 48:       # one box: odd extents, walls or several particles
        c["ny"], c["nz"] = rng.randint(40, edges[0]), rng.randint(40, edges[0])
        if rng.random() < 0.4:
            c["drive"], c["walls"] = "shear", 1
        elif edges[0] >= 96 and rng.random() < 0.5:
            c["drive"], c["per_box"], c["ny"], c["nz"], c["b"], c["a"] = "force", rng.randint(2, 4), 0, 0, 2.5, 4.5
    return c


# ---------------------------------------------------------------------------------------------------- inputs
def _dims(c):
    """The boxes' extents."""
    if c["kind"] == "warm":
        return [(c["n"], c["ny"], c["nz"])]
    e = [int(v) for v in c["edges"].split(",")]
    return [(e[k % len(e)], c["ny"] or e[k % len(e)], c["nz"] or e[k % len(e)]) for k in range(c["boxes"])]


def _quaternion(g):
    q = g.normal(size=4)
    q /= np.linalg.norm(q)
    return [float(v) for v in (q if q[0] >= 0 else -q)]


def _direction(g):
    v = g.normal(size=3)
    return v / np.linalg.norm(v)


def _scene(c, seed):
    """Boxes and particles: centres anywhere (several particles keep their bounding cubes apart), orientations
    uniform, forces of the size the library's workloads use."""
    g = np.random.default_rng(seed)
    boxes, parts = [], []
    drive = c.get("drive", "force")
    several = c["per_box"] > 1 or c["kind"] == "warm"
    for nx, ny, nz in _dims(c):
        box = dict(nx=nx, ny=ny, nz=nz, tau=c["tau"], rho0=1.0, counter_force=int(drive == "force"),
                   walls=c.get("walls", 0))
        if box["walls"]:
            box["wall_u_lo"], box["wall_u_hi"] = (-0.01, 0.0, 0.0), (0.01, 0.0, 0.0)
        side = 2 * (int(math.ceil(c["a"])) + 2) + 4
        ext = np.array([nx, ny, nz], float)
        centres = []
        while len(centres) < c["per_box"]:
            for _ in range(4000):
                x = g.uniform(0, 1, 3) * ext if several else 0.5 * (ext - [0, box["walls"], 0]) + g.uniform(-0.5, 0.5, 3)
                d = [np.abs(x - y) for y in centres]
                d = [np.minimum(v, ext - v) for v in d]
                strip = sum(v[1] < side + 12 and v[2] < side + 4 for v in d)    # a read-back serves four along a strip
                if strip < 4 and all((v >= side).any() for v in d):
                    centres.append(x)
                    break
            else:
                centres = []            # no room left: place them all again
        plist = []
        for x in centres:
            p = dict(semi=(c["a"], c["b"], c["b"]), x=[float(v) for v in x], q=_quaternion(g))
            if drive == "force":
                f = (2e-5 if several else 5e-4) * _direction(g)
                p["F_ext"] = [float(v) for v in f]
                p["T_ext"] = [float(v) for v in 2e-5 * _direction(g)]
            elif drive == "squirmer":
                p["B1"], p["B2"] = 1e-3, 1e-3 * float(g.choice([-2.0, 0.0, 2.0]))
            plist.append(p)
        boxes.append(box)
        parts.append(plist)
    return boxes, parts


def _couette(box):
    """The undisturbed flow of a sheared channel, the fluid such a run starts from."""
    y = torch.arange(box["ny"], dtype=torch.float64, device="cuda")
    u = torch.zeros(3, box["nz"], box["ny"], box["nx"], dtype=torch.float64, device="cuda")
    u[0] = (box["wall_u_lo"][0] + (box["wall_u_hi"][0] - box["wall_u_lo"][0]) * (y - 0.5) / (box["ny"] - 2))[None, :, None]
    return u.float()


def _external(parts):
    return np.array([list(p.get("F_ext", (0, 0, 0))) + list(p.get("T_ext", (0, 0, 0))) for pl in parts for p in pl])


def _samples(c, seed, n):
    """n spheroids (aspect ratio 1-4, short semi-axis 3-5, tau 0.6-1.5, edge 64): network inputs and resistance
    tensors of such bodies (stiffer across the long axis than along it, a small coupling)."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    r = lambda *s: torch.rand(*s, device="cuda", generator=gen, dtype=torch.float64)  # noqa: E731
    ratio, b, tau = 1 + 3 * r(n), 3 + 2 * r(n), 0.6 + 0.9 * r(n)
    e = torch.randn(n, 3, device="cuda", generator=gen, dtype=torch.float64)
    e = e / e.norm(dim=1, keepdim=True)
    e = torch.where(e[:, 2:] < 0, -e, e)
    x = torch.stack([ratio - 2, b - 3, 10 * ((tau - 0.5) / 3 - 1 / 6), 10 * b / 64 - 1, e[:, 0], e[:, 1], e[:, 2],
                     torch.ones_like(b)], 1)
    ee, eye = e[:, :, None] * e[:, None, :], torch.eye(3, device="cuda", dtype=torch.float64)[None]
    t = (1.1 + 0.25 * (ratio - 1))[:, None, None] * eye - (0.12 * (ratio - 1))[:, None, None] * ee
    w = (1.0 + 0.9 * (ratio - 1))[:, None, None] * eye - (0.5 * (ratio - 1))[:, None, None] * ee
    R = torch.zeros(n, 6, 6, device="cuda", dtype=torch.float64)
    R[:, :3, :3], R[:, 3:, 3:] = t, w
    n6 = 0.02 * torch.randn(n, 6, 6, device="cuda", generator=gen, dtype=torch.float64)
    R = R + n6 + n6.transpose(1, 2)
    return x.float().contiguous(), R.float().reshape(n, 36).contiguous()


OFF = {"W1": (0, (256, 16)), "b1": (4096, (256,)), "W2": (4352, (256, 256)), "b2": (69888, (256,)),
       "W3": (70144, (32, 256)), "b3": (78336, (32,))}


def _views(p):
    return {k: p[o:o + math.prod(s)].reshape(s) for k, (o, s) in OFF.items()}


def _params(seed):
    """Initial weights of a training run: He-style, the outputs near R = I."""
    g = np.random.default_rng(seed)
    p = np.zeros(SU.LB_MLP_NPARAM, np.float32)
    v = _views(p)
    v["W1"][:, :8] = g.normal(0, 0.5, (256, 8))
    v["W2"][:] = g.normal(0, math.sqrt(2.0 / 256), (256, 256))
    v["W3"][:21] = g.normal(0, 0.1 / 16, (21, 256))
    for i in range(6):
        v["b3"][i * (i + 1) // 2 + i] = 0.5413
    return p


# ---------------------------------------------------------------------------------------------------- prepare, run
def prepare(case, seed):
    if case["kind"] in ("train", "grad"):
        n, steps = case["batch"], case.get("steps", 1)
        x, R = _samples(case, seed, n * steps)
        net = SU.Surrogate(max_batch=n, params=_params(seed + 1))
        return dict(case=case, net=net, x=x, R=R, loss=torch.zeros(steps, device="cuda"),
                    grad=torch.zeros(SU.LB_MLP_NPARAM, device="cuda"))
    boxes, parts = _scene(case, seed)
    sim = L.Simulation(boxes, parts, precision=PREC[case.get("precision", "fp32")], max_semi=math.ceil(case["a"]),
                       collision=case.get("collision", 0), lattice=27 if case["kind"] == "run27" else 19)
    if case["kind"] == "warm":
        N = boxes[0]["nx"] * boxes[0]["ny"] * boxes[0]["nz"]
        return dict(case=case, sim=sim, net=W.load_params(WEIGHTS), df=torch.zeros(19 * N, device="cuda"))
    if boxes[0]["walls"]:
        u = _couette(boxes[0])
        L.lb_init_fluid(sim.ctx, 0, u.data_ptr(), u.numel() * 4, None, True)
    K, n = case["steps"], sum(len(p) for p in parts)
    ft = torch.from_numpy(np.tile(_external(parts), (K, 1, 1))).pin_memory()
    rec = torch.zeros(K, n, L.LB_RECORD_DOUBLES, dtype=torch.float64).pin_memory()
    new = lambda k: [torch.zeros((k, b["nz"], b["ny"], b["nx"]), device="cuda") for b in boxes]  # noqa: E731
    return dict(case=case, sim=sim, n=n, ft=ft, rec=rec, u=new(3), rho=new(1))


def _snapshot(s):
    for b, (u, rho) in enumerate(zip(s["u"], s["rho"])):
        L.lb_get_fields(s["sim"].ctx, b, L.LB_FIELD_U, u.data_ptr(), u.numel() * 4, True)
        L.lb_get_fields(s["sim"].ctx, b, L.LB_FIELD_RHO, rho.data_ptr(), rho.numel() * 4, True)


def _outputs(case, rec, u, rho):
    """A run's trajectory [steps][particles] and its snapshots, in the types they are kept in."""
    kept = torch.float32 if case["precision"] == "fp32" else torch.bfloat16
    if case["precision"] != "fp32":
        u, rho = [a.to(kept) for a in u], [a.to(kept) for a in rho]
    if len(u) > 8:                          # many boxes: one array each
        u, rho = [torch.cat([a.reshape(-1) for a in u])], [torch.cat([a.reshape(-1) for a in rho])]
    return dict(force=rec[..., :12].to(kept), velocity=rec[..., 12:18].to(kept), pose=rec[..., 18:].float(), u=u, rho=rho)


def run(state):
    s, c = state, state["case"]
    if c["kind"] == "grad":
        SU.lb_mlp_loss_grad(s["net"].h, s["x"].data_ptr(), s["R"].data_ptr(), c["batch"], s["loss"].data_ptr(),
                            s["grad"].data_ptr())
        return dict(loss=s["loss"], grad=s["grad"])
    if c["kind"] == "train":
        n = c["batch"]
        for t in range(c["steps"]):
            SU.lb_mlp_train_step(s["net"].h, s["x"].data_ptr() + t * n * 32, s["R"].data_ptr() + t * n * 144, n, c["lr"],
                                 s["loss"].data_ptr() + 4 * t)
        return dict(params=s["net"].params(), loss=s["loss"])
    sim = s["sim"]
    if c["kind"] == "warm":
        W.warm_start(sim, 0, s["net"])
        L.lb_get_fields(sim.ctx, 0, L.LB_FIELD_DF, s["df"].data_ptr(), s["df"].numel() * 4, True)
        vel = np.array([list(p["U"]) + list(p["Om"]) for p in sim.parts_of(0)], np.float32)
        return dict(velocity=vel, df=s["df"])
    if c["kind"] == "loop":
        for k in range(c["steps"]):
            L.lb_set_external(sim.ctx, -1, s["ft"][k].numpy())
            L.lb_step(sim.ctx, 1)
            L.lb_get_force_torque(sim.ctx, -1, s["n"], s["rec"][k].numpy())
        _snapshot(s)
        return _outputs(c, s["rec"], s["u"], s["rho"])
    if c["kind"] == "run27":
        L.lb_step(sim.ctx, c["steps"])
        L.lb_get_force_torque(sim.ctx, -1, s["n"], s["rec"][-1].numpy())
        _snapshot(s)
        return _outputs(c, s["rec"][-1:], s["u"], s["rho"])
    L.lb_step_io(sim.ctx, c["steps"], s["ft"].data_ptr(), s["rec"].data_ptr())
    _snapshot(s)                            # waits for the steps: the records are there too
    return _outputs(c, s["rec"], s["u"], s["rho"])


def work(case):
    if case["kind"] in ("train", "grad"):
        n, steps, P = case["batch"], case.get("steps", 1), 256 * 8 + 256 * 256 + 256 * 21
        state = 4 * SU.LB_MLP_NPARAM * (6 if case["kind"] == "train" else 2)    # p, m1, m2 in and out; p in, g out
        return dict(bytes=steps * (n * (8 + 36) * 4 + state), flops=steps * 6.0 * n * P)
    N = sum(a * b * c for a, b, c in _dims(case))
    if case["kind"] == "warm":              # the populations written, read and written out; seven transforms, N solves
        return dict(bytes=3 * 76.0 * N, flops=N * (35.0 * math.log2(N) + 1200.0))
    q, size = (27, 4) if case["kind"] == "run27" else (19, 4 if case["precision"] == "fp32" else 2)
    # a step reads and writes every population (no state of a listed sweep or batch fits the chip); the snapshot
    # reads them twice and writes four numbers per node
    return dict(bytes=N * (2.0 * q * size * case["steps"] + 2 * q * size + 32), flops=14.0 * q * N * case["steps"])


# ---------------------------------------------------------------------------------------------------- in 64 bits
def exact(case, seed):
    if case["kind"] in ("train", "grad"):
        return _exact_net(case, seed)
    boxes, parts = _scene(case, seed)
    if case["kind"] == "warm":
        return _exact_warm(case, boxes[0], parts[0])
    N = sum(a * b * c for a, b, c in _dims(case))
    if case["steps"] * (len(boxes) * 7e-3 + N * 6e-9) > 18.0:     # about its seconds
        return None
    got = [_Exact64(b, p, case).run(case["steps"]) for b, p in zip(boxes, parts)]
    rec = torch.from_numpy(np.concatenate([g[0] for g in got], 1))
    u, rho = [g[1] for g in got], [g[2] for g in got]
    if case["kind"] == "run27":
        rec = rec[-1:]
    if len(u) > 8:
        u, rho = [torch.cat([a.reshape(-1) for a in u])], [torch.cat([a.reshape(-1) for a in rho])]
    return dict(force=rec[..., :12], velocity=rec[..., 12:18], pose=rec[..., 18:], u=u, rho=rho)


def _head(y):
    Lm = torch.zeros(y.shape[0], 6, 6, dtype=y.dtype, device=y.device)
    i, j = torch.tril_indices(6, 6)
    Lm = Lm.index_put((torch.arange(y.shape[0], device=y.device)[:, None], i[None].to(y.device), j[None].to(y.device)),
                      torch.where((i == j).to(y.device), torch.nn.functional.softplus(y[:, :21]), y[:, :21]))
    return Lm @ Lm.transpose(1, 2)


def _forward(p, x):
    v = _views(p)
    h = torch.relu(x @ v["W1"][:, :8].T + v["b1"])
    h = torch.relu(h @ v["W2"].T + v["b2"])
    return _head(h @ v["W3"].T + v["b3"])


def _exact_net(case, seed):
    n, steps = case["batch"], case.get("steps", 1)
    x, R = (t.double() for t in _samples(case, seed, n * steps))
    p = torch.from_numpy(_params(seed + 1)).to(x).requires_grad_()
    keep = torch.ones_like(p, requires_grad=False)      # the padding of the parameter block stays zero
    v = _views(keep)
    v["W1"][:, 8:], v["W3"][21:], v["b3"][21:] = 0, 0, 0
    m1 = m2 = 0.0
    losses = []
    for t in range(steps):
        d = _forward(p, x[t * n:(t + 1) * n]) - R[t * n:(t + 1) * n].reshape(n, 6, 6)
        loss = d.square().mean()
        g = torch.autograd.grad(loss, p)[0] * keep
        losses.append(loss.detach())
        if case["kind"] == "grad":
            return dict(loss=torch.stack(losses), grad=g)
        m1, m2 = 0.9 * m1 + 0.1 * g, 0.999 * m2 + 0.001 * g * g
        a, b = m1 / (1 - 0.9 ** (t + 1)), m2 / (1 - 0.999 ** (t + 1))
        p = (p.detach() - case["lr"] * a / (b.sqrt() + 1e-8)).requires_grad_()
    return dict(params=p.detach(), loss=torch.stack(losses))


def _lattice(q):
    c = [(0, 0, 0)] + [(x, y, z) for x in (-1, 0, 1) for y in (-1, 0, 1) for z in (-1, 0, 1)
                       if 0 < x * x + y * y + z * z <= (2 if q == 19 else 3)]
    w = {19: [1 / 3, 1 / 18, 1 / 36], 27: [8 / 27, 2 / 27, 1 / 54, 1 / 216]}[q]
    return np.array(c), np.array([w[sum(v * v for v in k)] for k in c])


def _hamilton(a, b):
    return np.concatenate([[a[0] * b[0] - a[1:] @ b[1:]], a[0] * b[1:] + b[0] * a[1:] + np.cross(a[1:], b[1:])])


def _rotation(q):
    w, v = q[0], q[1:]
    K = np.array([[0, -v[2], v[1]], [v[2], 0, -v[0]], [-v[1], v[0], 0]])
    return (w * w - v @ v) * np.eye(3) + 2 * np.outer(v, v) + 2 * w * K


class _Body:
    def __init__(self, p):
        self.semi, self.x, self.q = np.array(p["semi"], float), np.array(p["x"], float), np.array(p["q"], float)
        self.q /= np.linalg.norm(self.q)
        self.U, self.W = np.zeros(3), np.zeros(3)
        self.F, self.T = np.array(p.get("F_ext", np.zeros(3)), float), np.array(p.get("T_ext", np.zeros(3)), float)
        self.B1, self.B2 = p.get("B1", 0.0), p.get("B2", 0.0)
        a, b, c = self.semi
        self.M = 4.0 / 3.0 * math.pi * a * b * c
        self.Ib = self.M * np.array([b * b + c * c, a * a + c * c, a * a + b * b]) / 5.0
        self.dP, self.dL, self.dm, self.back = np.zeros(3), np.zeros(3), 0.0, 0.0

    def shape(self):
        E = _rotation(self.q)
        return (E / self.semi**2) @ E.T


class _Exact64:
    """One box of the method in 64 bits, step by step as the paper's Appendix has it."""

    def __init__(self, box, parts, case):
        self.box, self.dev = box, torch.device("cuda")
        c, w = _lattice(27 if case["kind"] == "run27" else 19)
        self.c, self.w, self.Q = c, w, len(w)
        self.ct, self.wt = torch.tensor(c, dtype=torch.float64, device=self.dev), torch.tensor(w, device=self.dev)
        self.opp = [int(np.where((c == -k).all(1))[0][0]) for k in c]
        self.ghost, self.tau = case.get("collision", 0), box["tau"]
        self.ext = (box["nx"], box["ny"], box["nz"])
        self.per = (True, not box["walls"], True)
        self.dims = (box["nz"], box["ny"], box["nx"])
        self.body = [_Body(p) for p in parts]
        self.owner = self.solid()
        self.f = self.wt.reshape(-1, 1, 1, 1) * (self.owner == 0)[None]
        if box["walls"]:
            u = _couette(box).double()
            uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
            self.f = torch.stack([self.equilibrium(i, 1.0, u, uu)[0] for i in range(self.Q)]) * (self.owner == 0)
        self.links()

    def image(self, d, k):
        return d - self.ext[k] * torch.floor(d / self.ext[k] + 0.5) if self.per[k] else d

    def solid(self):
        o = torch.zeros(self.dims, dtype=torch.int32, device=self.dev)
        if self.box["walls"]:
            o[:, 0], o[:, -1] = -1, -1
        ax = [torch.arange(n, dtype=torch.float64, device=self.dev) for n in self.ext]
        for i, p in enumerate(self.body):
            A = p.shape()
            dx, dy, dz = (self.image(ax[k] - p.x[k], k) for k in range(3))
            dx, dy, dz = dx[None, None, :], dy[None, :, None], dz[:, None, None]
            v = (A[0, 0] * dx * dx + A[1, 1] * dy * dy + 2 * A[0, 1] * dx * dy) + A[2, 2] * dz * dz \
                + 2 * A[0, 2] * dx * dz + 2 * A[1, 2] * dy * dz
            o = torch.where(v <= 1.0, i + 1, o)
        return o

    def coords(self, idx):
        nx, ny, _ = self.ext
        return torch.stack([idx % nx, (idx // nx) % ny, idx // (nx * ny)], 1).double()

    def links(self):
        fluid = self.owner == 0
        self.fluid, self.nfluid = fluid.double(), int(fluid.sum())
        own, nx, ny = self.owner.reshape(-1), self.ext[0], self.ext[1]
        inner = (own > 0).nonzero()[:, 0]
        ext = torch.tensor(self.ext, device=self.dev)
        x = (self.coords(inner).long()[None] - self.ct.long()[:, None]) % ext       # [direction][solid node]: the other end
        node = (x[..., 2] * ny + x[..., 1]) * nx + x[..., 0]
        self.dir, k = (own[node] == 0).nonzero(as_tuple=True)
        self.node, self.who = node[self.dir, k], own[inner[k]].long() - 1
        self.lx, self.lc, self.lw = self.coords(self.node), self.ct[self.dir], self.wt[self.dir]
        self.lopp = torch.tensor(self.opp, device=self.dev)[self.dir]

    def force(self):
        g = np.array(self.box.get("body_force", (0.0, 0.0, 0.0)), float)
        return g - sum((p.F for p in self.body), np.zeros(3)) / self.nfluid if self.box["counter_force"] else g

    def equilibrium(self, i, rho, u, uu):
        cu = float(self.c[i][0]) * u[0] + float(self.c[i][1]) * u[1] + float(self.c[i][2]) * u[2]
        return self.w[i] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * uu), cu

    def moments(self):
        g = self.force()
        rho = self.f.sum(0)
        m = [sum(float(self.c[i][k]) * self.f[i] for i in range(self.Q) if self.c[i][k]) for k in range(3)]
        safe = torch.where(self.owner == 0, rho, 1.0)
        return rho, safe, [(m[k] + 0.5 * g[k]) / safe for k in range(3)], g

    def slip(self, r, particle):
        s = torch.zeros_like(r)
        p0 = self.body
        if all(p.B1 == 0 and p.B2 == 0 for p in p0):
            return s
        for i, p in enumerate(p0):
            m = particle == i
            e = torch.tensor(_rotation(p.q)[:, 0].copy(), device=self.dev)
            a, b = p.semi[0], p.semi[1]
            rr = r[m]
            zr = rr @ e
            rp = rr - zr[:, None] * e
            d = rp.norm(dim=1)
            z = zr.clamp(-a, a)
            e2 = max(0.0, 1 - b * b / (a * a))
            ec = math.sqrt(e2)
            den = (a * a - e2 * z * z).sqrt()
            se, sp = -(a * a - z * z).clamp(min=0).sqrt() / den, math.sqrt(1 - e2) * z / den
            zeta = zr / a if ec < 1e-8 else ((d * d + (zr + a * ec) ** 2).sqrt() - (d * d + (zr - a * ec) ** 2).sqrt()) / (2 * a * ec)
            amp = -(p.B1 + p.B2 * zeta) * se
            t = amp[:, None] * (se[:, None] * e + sp[:, None] * rp / d[:, None].clamp(min=1e-12))
            s[m] = torch.where(d[:, None] < 1e-12, 0.0, t)
        return s

    def step(self):
        box, n, tau = self.box, len(self.body), self.tau
        # collision
        eps = sum(p.back for p in self.body) / self.nfluid
        if eps:
            self.f += eps * self.wt.reshape(-1, 1, 1, 1) * self.fluid
        rho, safe, u, g = self.moments()
        uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
        ug = u[0] * g[0] + u[1] * g[1] + u[2] * g[2]
        post = torch.empty_like(self.f)
        P, j = {}, [0.0] * 3
        if self.ghost:
            for i in range(self.Q):
                d = self.f[i] - self.equilibrium(i, rho, u, uu)[0]
                for a in range(3):
                    ca = float(self.c[i][a])
                    j[a] = j[a] + ca * d
                    for b in range(a, 3):
                        P[a, b] = P.get((a, b), 0.0) + ca * float(self.c[i][b]) * d
        for i in range(self.Q):
            c = [float(v) for v in self.c[i]]
            eq, cu = self.equilibrium(i, rho, u, uu)
            cg = float(np.dot(c, g))
            S = (1 - 0.5 / tau) * self.w[i] * (3 * (cg - ug) + 9 * cu * cg)
            if self.ghost:
                h = sum((c[a] * c[b] - (1 / 3 if a == b else 0)) * (1 if a == b else 2) * P[a, b] for a, b in P)
                out = eq + (1 - 1 / tau) * self.w[i] * (3 * sum(c[a] * j[a] for a in range(3)) + 4.5 * h) + S
            else:
                out = self.f[i] - (self.f[i] - eq) / tau + S
            post[i] = out * self.fluid
        # forces of the links and the drag matrices, then the velocities
        x = torch.tensor(np.array([p.x for p in self.body]), device=self.dev)
        r = self.lx + 0.5 * self.lc - x[self.who]
        r = torch.stack([self.image(r[:, k], k) for k in range(3)], 1)
        fb = post.reshape(self.Q, -1)[self.dir, self.node]
        us = self.slip(r, self.who)
        v = torch.cat([self.lc, torch.linalg.cross(r, self.lc)], 1)
        amp = 2 * fb - 6 * self.lw * (us * self.lc).sum(1)
        sums = torch.zeros(n, 42, dtype=torch.float64, device=self.dev)
        sums.index_add_(0, self.who, torch.cat([amp[:, None] * v, (6 * self.lw[:, None, None] * v[:, :, None] * v[:, None, :]).reshape(-1, 36)], 1))
        records = []
        for p, s in zip(self.body, sums.cpu().numpy()):
            F0, Z = s[:6], s[6:].reshape(6, 6)
            E = _rotation(p.q)
            In = (E * p.Ib) @ E.T
            Om = np.array([[0, -p.W[2], p.W[1]], [p.W[2], 0, -p.W[0]], [-p.W[1], p.W[0], 0]])
            A = Z.copy()
            A[:3, :3] += p.M * np.eye(3)
            A[3:, 3:] += In + Om @ In - In @ Om
            new = np.linalg.solve(A, np.concatenate([p.M * p.U + p.F + p.dP, In @ p.W + p.T + p.dL]) + F0)
            mean = 0.5 * (np.concatenate([p.U, p.W]) + new)
            p.U, p.W = new[:3], new[3:]
            records.append([F0, F0 - Z @ new, new])
            p.mean = mean
        # streaming and bounce-back with the new velocities
        fn = torch.stack([torch.roll(post[i], tuple(int(k) for k in self.c[i][::-1]), (0, 1, 2)) for i in range(self.Q)]) * self.fluid
        if box["walls"]:
            for i in range(self.Q):
                if self.c[i][1] == 0:
                    continue
                y, uw = (1, box["wall_u_lo"]) if self.c[i][1] < 0 else (box["ny"] - 2, box["wall_u_hi"])
                fn[self.opp[i]][:, y] = (post[i][:, y] - 6 * self.w[i] * float(np.dot(uw, self.c[i]))) * self.fluid[:, y]
        U, Wv = (torch.tensor(np.array([getattr(p, k) for p in self.body]), device=self.dev) for k in ("U", "W"))
        ub = U[self.who] + torch.linalg.cross(Wv[self.who], r) + us
        fn.reshape(self.Q, -1)[self.lopp, self.node] = fb - 6 * self.lw * (ub * self.lc).sum(1)
        # pose, map, covered and uncovered nodes
        for p in self.body:
            p.x = p.x + p.mean[:3]
            w = p.mean[3:]
            k = np.linalg.norm(w)
            if k > 1e-300:
                p.q = _hamilton(np.concatenate([[math.cos(0.5 * k)], math.sin(0.5 * k) / k * w]), p.q)
            p.dP, p.dL, p.back, p.dm = np.zeros(3), np.zeros(3), p.dm, 0.0
        o = self.solid()
        moved = (o != self.owner).reshape(-1).nonzero()[:, 0]
        if len(moved):
            flat = fn.reshape(self.Q, -1)
            was, now, X = self.owner.reshape(-1)[moved].cpu().numpy(), o.reshape(-1)[moved].cpu().numpy(), self.coords(moved)
            for k, node in enumerate(moved.tolist()):
                p = self.body[int(max(was[k], now[k])) - 1]
                d = np.array([float(self.image(X[k, a] - p.x[a], a)) for a in range(3)])
                if now[k] > 0:
                    fv = flat[:, node].cpu().numpy()
                    jv, m = fv @ self.c, fv.sum()
                    flat[:, node] = 0.0
                else:
                    uv = p.U + np.cross(p.W, d)
                    cu = self.c @ uv
                    flat[:, node] = torch.tensor(self.w * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * uv @ uv), device=self.dev)
                    jv, m = -uv, -1.0
                p.dP, p.dL, p.dm = p.dP + jv, p.dL + np.cross(d, jv), p.dm + m
            self.owner = o
            self.links()
        self.f = fn
        return np.array([np.concatenate([F0, F, v, p.x, p.q]) for (F0, F, v), p in zip(records, self.body)])

    def run(self, steps):
        rec = np.array([self.step() for _ in range(steps)])
        rho, _, u, _ = self.moments()
        return rec, torch.stack(u) * self.fluid, ((rho - 1.0) * self.fluid)[None]


def _exact_warm(case, box, parts):
    """Network, velocities and the lattice fluid's steady state with its non-equilibrium part, in 64 bits."""
    e64 = _Exact64(box, parts, case)
    dev, N, Ld = e64.dev, math.prod(e64.dims), float(box["nx"] * box["ny"] * box["nz"]) ** (1 / 3)
    nu, om = (box["tau"] - 0.5) / 3, 1 / box["tau"]
    feats, D = [], []
    for p in e64.body:
        e = _rotation(p.q)[:, 0]
        e = -e if e[2] < 0 else e
        a, b = p.semi[0], p.semi[1]
        feats.append([a / b - 2, b - 3, 10 * (nu - 1 / 6), 10 * b / Ld - 1, *e, 1.0])
        D.append([math.sqrt(6 * math.pi * nu * b)] * 3 + [math.sqrt(8 * math.pi * nu * b**3)] * 3)
    R = _forward(torch.from_numpy(np.load(WEIGHTS).astype(np.float64)).to(dev), torch.tensor(feats, device=dev)).cpu().numpy()
    vel = np.array([np.linalg.solve(r, np.concatenate([p.F, p.T]) / d) / d for r, p, d in zip(R, e64.body, np.array(D))])
    # force density: on the fluid nodes next to a particle, the counter force on every fluid node
    fluid, own = e64.fluid, e64.owner
    near = torch.zeros_like(own)
    for ax in range(3):
        for s in (1, -1):
            o = torch.roll(own, s, ax)
            near = torch.where((own == 0) & (near == 0), o, near)
    g = torch.zeros((3,) + e64.dims, dtype=torch.float64, device=dev)
    for k in range(3):
        g[k] = fluid * e64.force()[k]
        for i, p in enumerate(e64.body):
            m = near == i + 1
            g[k] += m * (p.F[k] / int(m.sum()))
    gh = torch.fft.fftn(g.to(torch.complex128), dim=(1, 2, 3))
    ang = [2 * math.pi * torch.arange(n, dtype=torch.float64, device=dev) / n for n in e64.ext]
    zero = torch.zeros(e64.dims, dtype=torch.complex128, device=dev)
    H1, H2, D2, D0 = [zero.clone() for _ in range(3)], {}, {}, zero.clone()
    for i in range(1, e64.Q):
        c = [float(v) for v in e64.c[i]]
        th = c[0] * ang[0][None, None, :] + c[1] * ang[1][None, :, None] + c[2] * ang[2][:, None, None]
        ex = torch.polar(torch.ones_like(th), -th)
        one = torch.complex(2 * torch.sin(0.5 * th) ** 2, torch.sin(th))        # 1 - ex
        h, q = ex / (1 - (1 - om) * ex), one / (1 - (1 - om) * ex)
        D0 += e64.w[i] * q
        for a in range(3):
            if c[a]:
                H1[a] += e64.w[i] * c[a] * h
                for b in range(3):
                    if c[b]:
                        H2[a, b] = H2.get((a, b), 0) + e64.w[i] * c[a] * c[b] * h
                        D2[a, b] = D2.get((a, b), 0) + 3 * e64.w[i] * c[a] * c[b] * q
    M = torch.zeros(e64.dims + (4, 4), dtype=torch.complex128, device=dev)
    y = torch.zeros(e64.dims + (4,), dtype=torch.complex128, device=dev)
    fo = 3 * (1 - 0.5 * om)
    M[..., 0, 0] = D0
    for a in range(3):
        M[..., 0, 1 + a], M[..., 1 + a, 0] = -3 * om * H1[a], -om * H1[a]
        y[..., 0] += fo * H1[a] * gh[a]
        y[..., 1 + a] = 0.5 * gh[a] + fo * sum(H2[a, b] * gh[b] for b in range(3))
        for b in range(3):
            M[..., 1 + a, 1 + b] = D2[a, b]
    M[0, 0, 0], y[0, 0, 0] = torch.eye(4, dtype=torch.complex128, device=dev), 0
    sol = torch.linalg.solve(M.reshape(-1, 4, 4), y.reshape(-1, 4, 1)).reshape(e64.dims + (4,))
    sol = torch.fft.ifftn(sol.permute(3, 0, 1, 2), dim=(1, 2, 3)).real
    u, dr = sol[1:].contiguous(), sol[0] - (sol[0] * fluid).sum() / e64.nfluid
    P = sum(p.M * v[:3] for p, v in zip(e64.body, vel))
    for k in range(3):
        u[k] += fluid * ((-P[k] - (u[k] * fluid).sum()) / e64.nfluid)
    # populations: equilibrium of (1 + drho, u), and the first-order part of the velocity gradient
    du = [[0.5 * (torch.roll(u[b], -1, 2 - a) - torch.roll(u[b], 1, 2 - a)) for b in range(3)] for a in range(3)]
    div = (du[0][0] + du[1][1] + du[2][2]) / 3
    rho, uu = 1 + dr, u[0] ** 2 + u[1] ** 2 + u[2] ** 2
    cs, _ = L.lb_lattice()              # only the order in which the library lists its directions
    df = torch.zeros((19,) + e64.dims, dtype=torch.float64, device=dev)
    for k, c in enumerate(cs):
        w = float(e64.w[int(np.where((e64.c == c).all(1))[0][0])])
        cu = sum(float(c[a]) * u[a] for a in range(3))
        q = -div + sum(float(c[a] * c[b]) * du[a][b] for a in range(3) for b in range(3) if c[a] * c[b])
        df[k] = fluid * (w * (dr + rho * (3 * cu + 4.5 * cu * cu - 1.5 * uu)) - 3 * box["tau"] * rho * w * q)
    return dict(velocity=vel, df=df.reshape(-1))
