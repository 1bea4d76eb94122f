// Field read-back kernel (lb_get_fields): the pre-collision state of every
// node of one box at the start of iteration t, i.e. the second half of
// iteration t-1 of the paper's Appendix (step 2 streaming, step 6 bounce-back
// with U(t), Omega(t), the remap of step 8) without the collision, with
// density and velocity moments.  Every decision is taken per node from the
// occupancy maps.
//
// One launch, two kinds of blocks:
//   - plain blocks, one thread per 4 consecutive x nodes ("quad"), 256 quads per
//     block: each direction is one 16-byte load of the source row (8 bytes in
//     16-bit storage), the +-1 shift in x comes from the neighbouring lane by a
//     shuffle (a scalar load at warp and row ends, which also wraps x); solid
//     nodes are written as 0, the nodes of a particle's redo mask are left out;
//   - surface blocks (the first ones of the grid), one thread per node of a
//     particle's cube, which do the masked nodes: the pull, the node's own
//     populations for the links that end inside the old surface (Eq. fb, Eq. ub)
//     and the uncovered nodes.  A node in the masks of two particles is written
//     twice with the same value.
//
// Bound: the populations, read once (HBM) - so the plain blocks need as many loads
// in flight as fit.  With the surface code in every thread a block took 255 registers
// and an SM held 8 warps, each waiting at the block's list of particles; apart, the
// plain code fits 128 (two blocks per SM; three would spill 250-480 bytes per thread), and the
// surface nodes cost few warps.  Measured per call, u or rho: a 64^3 box with one
// particle 17 -> 7.5 us (FP16), the 32 squirmer boxes of 48^3 to 128^3 nodes in BF16
// 57 -> 16.6 on average, 128^3 nodes with 16 particles in FP32 88 -> 56; all populations
// of 128^3 nodes before the first step 72 -> 54, the owner field 9.5 -> 7.1.
#include "bulk_tile.cuh"

namespace lbsph {

// The 6 nodes x = X0-1 .. X0+4 of a cube row as bits 0..5: its word shifted by the window's
// offset d in the cube, and by what of the window lies beyond the periodic end.
__device__ __forceinline__ unsigned window6(uint64_t word, int S, int d, int nx)
{
    unsigned m = d < S ? (unsigned)(word >> d) : 0u;
    if (d + 6 > nx) m |= (unsigned)(word << (nx - d));
    return m & 0x3fu;
}

// Does the range [lo, hi] (lo >= -1) of a periodic axis of length L meet [ow, ow+S-1] (mod L)?
__device__ __forceinline__ bool hits(int lo, int hi, int ow, int S, int L)
{
    if (hi - lo + 1 >= L) return true;
    int d = lo - ow;
    if (d < 0) d += L;
    if (d >= L) d -= L;
    return d < S || hi - lo >= L - d;
}

// ---------------------------------------------------------------------------
enum { FK_F = 0, FK_MOMENTS = 1, FK_SOLID = 2 };

constexpr int FIELD_BLOCKS = 2;             // blocks per SM the registers are held to

// Density deviation and momentum of one node's populations, in this order of additions.
__device__ __forceinline__ void node_moments(const float (&f)[Q], float rho0, const float* g, float& drho, float& ux,
                                             float& uy, float& uz)
{
    drho = 0.f;
#pragma unroll
    for (int i = 0; i < Q; ++i) drho += f[i];
    const float jx = (f[1] - f[2]) + (f[7] - f[8]) + (f[9] - f[10]) + (f[11] - f[12]) + (f[13] - f[14]);
    const float jy = (f[3] - f[4]) + (f[7] - f[8]) - (f[9] - f[10]) + (f[15] - f[16]) + (f[17] - f[18]);
    const float jz = (f[5] - f[6]) + (f[11] - f[12]) - (f[13] - f[14]) + (f[15] - f[16]) - (f[17] - f[18]);
    const float ir = 1.0f / (rho0 + drho);
    ux = (jx + 0.5f * g[0]) * ir;
    uy = (jy + 0.5f * g[1]) * ir;
    uz = (jz + 0.5f * g[2]) * ir;
}

// The box's uniform force, by one warp: body force and the counter force over the fluid nodes.
__device__ __forceinline__ void box_force(const KParams& P, const BoxDev& B, int lane, float* g_out)
{
    double fx = 0.0, fy = 0.0, fz = 0.0;
    int nsol = 0;                           // at most N < 2^31 / 19
    for (int j = lane; j < B.pcnt; j += 32) {
        const PartK& k = P.pk[B.pbeg + j];
        fx += k.Fext[0]; fy += k.Fext[1]; fz += k.Fext[2];
        nsol += k.nsolid;
    }
    for (int o = B.pcnt > 1 ? 16 : 0; o > 0; o >>= 1) {
        fx += __shfl_xor_sync(0xffffffffu, fx, o);
        fy += __shfl_xor_sync(0xffffffffu, fy, o);
        fz += __shfl_xor_sync(0xffffffffu, fz, o);
        nsol += __shfl_xor_sync(0xffffffffu, nsol, o);
    }
    if (lane == 0) {
        const double nf = (double)(B.N - B.nwall - nsol);
        double g[3] = {B.body[0], B.body[1], B.body[2]};
        if (B.counter && nf > 0) { g[0] -= fx / nf; g[1] -= fy / nf; g[2] -= fz / nf; }
        g_out[0] = (float)g[0]; g_out[1] = (float)g[1]; g_out[2] = (float)g[2];
    }
}

// A 256-quad tile may meet at most MAXC particles (grown by one node; old and new cubes): else ST_CAPACITY.  One warp.
// The blocks here would do with any number; callers have always been refused beyond MAXC, and still are.
__device__ __forceinline__ void tile_capacity(const KParams& P, const BoxDev& B, int q0, int lane)
{
    const int ny = B.ny, nz = B.nz;
    const int qlast = min(q0 + KBLOCK, (int)B.nq) - 1;
    const int r0 = div_magic(q0, B.dq_m, B.dq_s), r1 = div_magic(qlast, B.dq_m, B.dq_s);
    const int z0 = div_magic(r0, B.dy_m, B.dy_s), z1 = div_magic(r1, B.dy_m, B.dy_s);
    const int y0 = r0 - z0 * ny, y1 = r1 - z1 * ny;
    const int ylo = z0 == z1 ? y0 - 1 : -1, yhi = z0 == z1 ? y1 + 1 : ny;
    int nc = 0;
    for (int base = 0; base < B.pcnt; base += 32) {
        bool hit = false;
        if (base + lane < B.pcnt) {
            const PartK& k = P.pk[B.pbeg + base + lane];
            const int S = k.S;
            hit = (hits(ylo, yhi, k.ow_old[1], S, ny) && hits(z0 - 1, z1 + 1, k.ow_old[2], S, nz)) ||
                  (hits(ylo, yhi, k.ow_new[1], S, ny) && hits(z0 - 1, z1 + 1, k.ow_new[2], S, nz));
        }
        nc += __popc(__ballot_sync(0xffffffffu, hit));
    }
    if (lane == 0 && nc > MAXC) atomicOr(P.status, ST_CAPACITY);
}

// Node l of particle p's cube, if its redo mask holds it and no particle covers it now.
template <class St, int WHAT>
__device__ __forceinline__ void surface_node(const KParams& P, const BoxDev& B, int p, int l, const float* s_g)
{
    using T = typename St::T;
    const int nx = B.nx, ny = B.ny, nz = B.nz, N = (int)B.N;
    const NeedHdr h = P.need_hdr[p];
    const int S = h.S;
    const int r = l / S, mz = r / S;            // cube row r = mz S + my
    bool on = mz < S;
    if (on) on = (P.need[(size_t)p * (MAXS * MAXS) + r] >> (l - r * S)) & 1ull;
    const int X = wrapd(h.ow[0] + (l - r * S), nx), y = wrapd(h.ow[1] + (r - mz * S), ny), z = on ? wrapd(h.ow[2] + mz, nz) : 0;
    if (B.walls && (y == 0 || y == ny - 1)) on = false;
    const float rho0 = B.rho0f, inv = B.inv_scale;
    const unsigned long long pol = l2_evict_normal();
    const T* A = reinterpret_cast<const T*>(P.src) + B.off;
    const int own = (z * ny + y) * nx + X;
    float f[Q], o[Q];
    if (on) {
        const int xx[3] = {X == 0 ? nx - 1 : X - 1, X, X == nx - 1 ? 0 : X + 1};
        const int yy[3] = {y == 0 ? ny - 1 : y - 1, y, y == ny - 1 ? 0 : y + 1};
        const int zz[3] = {z == 0 ? nz - 1 : z - 1, z, z == nz - 1 ? 0 : z + 1};
#pragma unroll
        for (int i = 0; i < Q; ++i)
            f[i] = St::ld1(A + (i * N + (zz[1 - cz_of(i)] * ny + yy[1 - cy_of(i)]) * nx + xx[1 - cx_of(i)]), inv, pol);
        // the node's own populations, wanted by the links that end in a surface: all of them at once, so that one
        // latency covers them
#pragma unroll
        for (int i = 1; i < Q; ++i) o[i] = St::ld1(A + (i * N + own), inv, pol);
        const int wall_cy = !B.walls ? 0 : (y == 1 ? 1 : (y == ny - 2 ? -1 : 0));     // directions from a wall
        if (wall_cy != 0) {
            const float* uw = y == 1 ? B.uw_lo : B.uw_hi;
#pragma unroll
            for (int i = 1; i < Q; ++i)
                if (cy_of(i) != 0 && cy_of(i) == wall_cy)
                    f[i] = o[opp_of(i)] + 6.0f * w_of(i) * rho0 * (cx_of(i) * uw[0] + cy_of(i) * uw[1] + cz_of(i) * uw[2]);
        }
        int c0 = -1;                            // the particle whose old map holds the node
        for (int c = B.pbeg; c < B.pbeg + B.pcnt; ++c) {
            const PartK& C = P.pk[c];
            const int Sc = C.S;
            const int ax = wrapd(X - C.ow_new[0], nx), ay = wrapd(y - C.ow_new[1], ny), az = wrapd(z - C.ow_new[2], nz);
            if (ax < Sc && ay < Sc && az < Sc && ((C.rows_new[az * Sc + ay] >> ax) & 1ull)) on = false;
            const int oo[3] = {C.ow_old[0], C.ow_old[1], C.ow_old[2]};
            if (!(hits(X - 1, X + 1, oo[0], Sc, nx) && hits(y - 1, y + 1, oo[1], Sc, ny) && hits(z - 1, z + 1, oo[2], Sc, nz)))
                continue;
            // occupancy of x - 1, x, x + 1 (bits 0..2) in the 9 rows (y + dy, z + dz) of the old map
            const int d = wrapd(wrapd(X - 1, nx) - oo[0], nx);
            int my3[3], mz3[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                my3[a] = wrapd(yy[a] - oo[1], ny);
                mz3[a] = wrapd(zz[a] - oo[2], nz);
            }
            unsigned w[3][3], any = 0u;
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int b = 0; b < 3; ++b) {
                    w[a][b] = 0u;
                    if (my3[a] < Sc && mz3[b] < Sc) w[a][b] = window6(C.rows_old[mz3[b] * Sc + my3[a]], Sc, d, nx);
                    any |= w[a][b];
                }
            if ((any & 7u) == 0u) continue;
            if (c0 < 0 && ((w[1][1] >> 1) & 1u)) c0 = c;
            const float ro[3] = {C.ro_old[0], C.ro_old[1], C.ro_old[2]}, U[3] = {C.U[0], C.U[1], C.U[2]},
                        W[3] = {C.W[0], C.W[1], C.W[2]};
            const int squirmer = C.squirmer;
#pragma unroll
            for (int i = 1; i < Q; ++i) {
                if (!((w[1 - cy_of(i)][1 - cz_of(i)] >> (1 - cx_of(i))) & 1u)) continue;
                if (cy_of(i) != 0 && cy_of(i) == wall_cy) continue;
                int sx = d + 1 - cx_of(i);
                if (sx >= nx) sx -= nx;
                const float rx = ro[0] + sx + 0.5f * cx_of(i);
                const float ry = ro[1] + my3[1 - cy_of(i)] + 0.5f * cy_of(i);
                const float rz = ro[2] + mz3[1 - cz_of(i)] + 0.5f * cz_of(i);
                float ux = U[0] + (W[1] * rz - W[2] * ry);
                float uy = U[1] + (W[2] * rx - W[0] * rz);
                float uz = U[2] + (W[0] * ry - W[1] * rx);
                if (squirmer) {
                    float qx, qy, qz;
                    squirmer_slip(C.e_old, C.a, C.eps2, C.B1, C.B2, rx, ry, rz, qx, qy, qz);
                    ux += qx; uy += qy; uz += qz;
                }
                const float ubc = cx_of(i) * ux + cy_of(i) * uy + cz_of(i) * uz;
                f[i] = o[opp_of(i)] + 6.0f * w_of(i) * rho0 * ubc;
            }
        }
        if (on && c0 >= 0) {
            // uncovered: f = f_eq(rho0, U + Omega x r) (remap, step 8)
            const PartK& c = P.pk[c0];
            const int ax = wrapd(X - c.ow_new[0], nx), ay = wrapd(y - c.ow_new[1], ny), az = wrapd(z - c.ow_new[2], nz);
            const float rx = c.ro_new[0] + ax, ry = c.ro_new[1] + ay, rz = c.ro_new[2] + az;
            const float ux = c.U[0] + (c.W[1] * rz - c.W[2] * ry);
            const float uy = c.U[1] + (c.W[2] * rx - c.W[0] * rz);
            const float uz = c.U[2] + (c.W[0] * ry - c.W[1] * rx);
            const float uu = ux * ux + uy * uy + uz * uz;
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                const float cu = cx_of(i) * ux + cy_of(i) * uy + cz_of(i) * uz;
                f[i] = w_of(i) * rho0 * (3.0f * cu + 4.5f * cu * cu - 1.5f * uu);
            }
        }
    }
    if (WHAT == FK_MOMENTS) __syncthreads();    // the box force
    if (!on) return;
    if (WHAT == FK_F) {
#pragma unroll
        for (int i = 0; i < Q; ++i) P.out_f[i * N + own] = P.out_dev ? f[i] : f[i] + w_of(i) * rho0;
    } else {
        float drho, u[3];
        node_moments(f, rho0, s_g, drho, u[0], u[1], u[2]);
        if (P.out_rho) P.out_rho[own] = drho;
        if (P.out_u)
            for (int a = 0; a < 3; ++a) P.out_u[a * N + own] = u[a];
    }
}

template <class St, int WHAT>
__global__ void __launch_bounds__(KBLOCK, FIELD_BLOCKS) fields_kernel(const __grid_constant__ KParams P)
{
    using T = typename St::T;
    __shared__ float s_g[3];
    const BoxDev& B = P.boxes[P.only_box];
    const int lane = threadIdx.x & 31;
    if (WHAT != FK_SOLID && (int)blockIdx.x < P.surf_blocks) {
        if (WHAT == FK_MOMENTS && threadIdx.x < 32) box_force(P, B, lane, s_g);
        surface_node<St, WHAT>(P, B, B.pbeg + blockIdx.x / P.surf_per, (blockIdx.x % P.surf_per) * KBLOCK + threadIdx.x, s_g);
        return;
    }
    // ---- this thread's quad
    const int nx = B.nx, ny = B.ny, nz = B.nz, nxq = B.nxq;
    const int N = (int)B.N;                     // 19 N < 2^31
    const int q0 = ((int)blockIdx.x - P.surf_blocks) * KBLOCK;
    int q = q0 + (int)threadIdx.x;
    const bool valid = q < (int)B.nq;
    if (!valid) q = (int)B.nq - 1;
    const int row = div_magic(q, B.dq_m, B.dq_s);
    const int xq = q - row * nxq;
    const int z = div_magic(row, B.dy_m, B.dy_s);
    const int y = row - z * ny;
    const T* A = reinterpret_cast<const T*>(P.src) + B.off;
    const float inv = B.inv_scale, rho0 = B.rho0f;
    const unsigned long long pol = l2_evict_normal();
    const int own = row * nx + 4 * xq;
    const bool first = P.nopull != 0;
    const int pcnt = B.pcnt;
    NeedHdr hd;                                 // the cube of one particle per lane, on its way while the populations load
    hd.ow[0] = hd.ow[1] = hd.ow[2] = hd.S = 0;
    if (lane < pcnt) hd = P.need_hdr[B.pbeg + lane];

    // ---- pull (stream): v[i] = f*_i(x - c_i) for the 4 nodes
    float4 v[Q];
    if (WHAT != FK_SOLID) {
        if (first) {
            // before the first collision: the initial distributions in place
#pragma unroll
            for (int i = 0; i < Q; ++i) v[i] = St::ld4(A + (i * N + own), inv, pol);
        } else {
            int rofs[3][3];  // element offset of source rows (y + dy, z + dz), wrapped
            {
                const int yy[3] = {y == 0 ? ny - 1 : y - 1, y, y == ny - 1 ? 0 : y + 1};
                const int zz[3] = {z == 0 ? nz - 1 : z - 1, z, z == nz - 1 ? 0 : z + 1};
#pragma unroll
                for (int a = 0; a < 3; ++a)
#pragma unroll
                    for (int b = 0; b < 3; ++b) rofs[a][b] = (zz[b] * ny + yy[a]) * nx;
            }
            const bool left_ld = (lane == 0) || (xq == 0);
            const bool right_ld = (lane == 31) || (xq == nxq - 1);
#pragma unroll
            for (int i = 0; i < Q; ++i) v[i] = St::ld4(A + (i * N + rofs[1 - cy_of(i)][1 - cz_of(i)]) + 4 * xq, inv, pol);
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                const T* rp = A + (i * N + rofs[1 - cy_of(i)][1 - cz_of(i)]);
                const float4 t = v[i];
                if (cx_of(i) == 1) {           // source x - 1
                    float e = __shfl_up_sync(0xffffffffu, t.w, 1);
                    if (left_ld) e = St::ld1(rp + (xq == 0 ? nx - 1 : 4 * xq - 1), inv, pol);
                    v[i] = make_float4(e, t.x, t.y, t.z);
                } else if (cx_of(i) == -1) {   // source x + 1
                    float e = __shfl_down_sync(0xffffffffu, t.x, 1);
                    if (right_ld) e = St::ld1(rp + (xq == nxq - 1 ? 0 : 4 * xq + 4), inv, pol);
                    v[i] = make_float4(t.y, t.z, t.w, e);
                }
            }
        }
    }
    if (threadIdx.x < 32) {
        if (pcnt > MAXC) tile_capacity(P, B, q0, lane);
    } else if (WHAT == FK_MOMENTS && threadIdx.x < 64) {
        box_force(P, B, lane, s_g);
    }
    if (WHAT == FK_MOMENTS) __syncthreads();

    // ---- walls: link bounce-back (Eq. fb with u_b = u_w) of the rows next to them
    const bool wallrow = B.walls && (y == 0 || y == ny - 1);
    if (WHAT != FK_SOLID && B.walls && !first && (y == 1 || y == ny - 2)) {
        const int wall_cy = y == 1 ? 1 : -1;    // directions from the wall
        const float* uw = y == 1 ? B.uw_lo : B.uw_hi;
#pragma unroll
        for (int i = 1; i < Q; ++i) {
            if (cy_of(i) == 0 || cy_of(i) != wall_cy) continue;
            const float4 o = St::ld4(A + (opp_of(i) * N + own), inv, pol);
            const float ubc = cx_of(i) * uw[0] + cy_of(i) * uw[1] + cz_of(i) * uw[2];
#pragma unroll
            for (int k = 0; k < 4; ++k) set_comp(v[i], k, comp(o, k) + 6.0f * w_of(i) * rho0 * ubc);
        }
    }
    // ---- nodes solid now (zero; owner: the lowest particle), and nodes of the surface blocks (skip)
    unsigned zero = wallrow ? 0xfu : 0u, skip = 0u;
    int owner[4];
    if (WHAT == FK_SOLID)
        for (int k = 0; k < 4; ++k) owner[k] = wallrow ? -1 : 0;
    for (int j0 = 0; j0 < pcnt; j0 += 32) {
        if (j0 > 0) {
            hd.S = 0;
            if (j0 + lane < pcnt) hd = P.need_hdr[B.pbeg + j0 + lane];
        }
        for (unsigned m = cubes_near(hd, row, B); m != 0; m &= m - 1) {
            const int j = j0 + __ffs((int)m) - 1;
            const NeedHdr c = P.need_hdr[B.pbeg + j];
            int dz = z - c.ow[2];
            if (dz < 0) dz += nz;
            int dy = y - c.ow[1];
            if (dy < 0) dy += ny;
            int dx = 4 * xq - c.ow[0];
            if (dx < 0) dx += nx;
            if (dz >= c.S || dy >= c.S || wallrow) continue;
            if (dx >= c.S && dx + 3 < nx) continue;
            const uint64_t w = P.pk[B.pbeg + j].rows_new[dz * c.S + dy];
            const uint64_t nd = WHAT == FK_SOLID || first ? 0ull : P.need[(size_t)(B.pbeg + j) * (MAXS * MAXS) + dz * c.S + dy];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int mx = dx + k < nx ? dx + k : dx + k - nx;
                if (mx >= c.S) continue;
                if ((w >> mx) & 1ull) {
                    if (WHAT == FK_SOLID && !((zero >> k) & 1u)) owner[k] = j + 1;
                    zero |= 1u << k;
                }
                if ((nd >> mx) & 1ull) skip |= 1u << k;
            }
        }
    }
    if (!valid) return;
    if (WHAT == FK_SOLID) {
        *reinterpret_cast<int4*>(P.out_solid + own) = make_int4(owner[0], owner[1], owner[2], owner[3]);
        return;
    }
    skip &= ~zero;
    if (WHAT == FK_F) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                const float f = comp(v[i], k);
                set_comp(v[i], k, ((zero >> k) & 1u) ? 0.0f : (P.out_dev ? f : f + w_of(i) * rho0));
            }
        if (skip == 0u) {
#pragma unroll
            for (int i = 0; i < Q; ++i) *reinterpret_cast<float4*>(P.out_f + (i * N + own)) = v[i];
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if ((skip >> k) & 1u) continue;
#pragma unroll
                for (int i = 0; i < Q; ++i) P.out_f[i * N + own + k] = comp(v[i], k);
            }
        }
        return;
    }
    float4 out[4];                              // rho, u_x, u_y, u_z of the four nodes
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        float f[Q], a[4];
#pragma unroll
        for (int i = 0; i < Q; ++i) f[i] = comp(v[i], k);
        node_moments(f, rho0, s_g, a[0], a[1], a[2], a[3]);
#pragma unroll
        for (int e = 0; e < 4; ++e) set_comp(out[e], k, ((zero >> k) & 1u) ? 0.0f : a[e]);
    }
    float* dst[4] = {P.out_rho, P.out_u, P.out_u ? P.out_u + N : nullptr, P.out_u ? P.out_u + 2 * N : nullptr};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        if (!dst[e]) continue;
        if (skip == 0u) {
            *reinterpret_cast<float4*>(dst[e] + own) = out[e];
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (!((skip >> k) & 1u)) dst[e][own + k] = comp(out[e], k);
        }
    }
}

// ---------------------------------------------------------------------------
// blocks: 256-quad tiles of the box; p.surf_blocks more for the nodes next to a surface
template <class St>
static cudaError_t launch_mode(KParams p, int blocks, cudaStream_t s)
{
    if (p.out_solid) p.surf_blocks = 0;
    const int g = blocks + p.surf_blocks;
    if (p.out_f) fields_kernel<St, FK_F><<<g, KBLOCK, 0, s>>>(p);
    else if (p.out_solid) fields_kernel<St, FK_SOLID><<<g, KBLOCK, 0, s>>>(p);
    else fields_kernel<St, FK_MOMENTS><<<g, KBLOCK, 0, s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_fields(const KParams& p, int precision, int blocks, cudaStream_t s)
{
    if (precision == 1) return launch_mode<StF16>(p, blocks, s);
    if (precision == 2) return launch_mode<StBF16>(p, blocks, s);
    return launch_mode<StF32>(p, blocks, s);
}

}  // namespace lbsph
