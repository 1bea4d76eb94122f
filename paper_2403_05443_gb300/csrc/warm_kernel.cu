// Warm start of a run (lb_init_fluid, lb_stokes_field): an initial fluid at
// the local equilibrium of given velocity and density fields (optionally with
// the viscous stress of the velocity field in its non-equilibrium part), and
// the periodic steady flow (with its density) that the particles' external
// forces drive in the lattice fluid, as those fields.
//
// The force density g puts F_ext of each particle uniformly on the fluid nodes
// next to it, and the box's uniform counter force and body force on the fluid
// nodes; the mean of g (if the forces do not balance) is dropped.  The flow is
// the exact steady state of the linear lattice dynamics itself (D3Q19 BGK with
// Guo forcing, lattice_steady_kernel), not of a discretised Stokes operator:
// at the scales of a few nodes the lattice's viscous and pressure operators
// differ from any fixed stencil by several per cent, and a start that differs
// from the lattice's own steady state by that much relaxes on the flow's slow
// time scales.  The mean flow is then set so that the fluid and particle
// momenta add up to zero (rho0 sum_fluid u = -sum_p M_p U_p, with the
// particles' initial velocities), as they do in a run from rest with a
// balancing counter force.  The transforms are separable mixed-radix FFTs along x, y
// and z in FP32, two real fields to a complex one; the per-mode solve carries twice
// FP32's digits.
#include <cmath>

#include "lattice_common.cuh"

namespace lbsph {

// f = f_eq(rho0 + drho, u) - w rho0 on fluid nodes (deviation storage), 0
// elsewhere; drho may be null (uniform density).  stress: plus the first-order
// non-equilibrium part -3 tau rho w_i (c_ia c_ib - delta_ab / 3) d_a u_b with
// d_a the periodic central difference (u is read on every node, solid or not)
template <class St>
__global__ void init_fluid_kernel(const BoxDev B, void* fbuf, const float* u, const float* drho, const int* owner,
                                  float tau, int stress)
{
    using T = typename St::T;
    const long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (n >= B.N) return;
    T* f = reinterpret_cast<T*>(fbuf) + B.off;
    const bool fluid = owner[n] == 0;
    const float ux = fluid ? u[n] : 0.0f, uy = fluid ? u[B.N + n] : 0.0f, uz = fluid ? u[2 * B.N + n] : 0.0f;
    const float uu = ux * ux + uy * uy + uz * uz;
    const float dr = (fluid && drho) ? drho[n] : 0.0f;
    const float rho = B.rho0f + dr;
    float du[3][3] = {{0.0f, 0.0f, 0.0f}, {0.0f, 0.0f, 0.0f}, {0.0f, 0.0f, 0.0f}};   // du[a][b] = d_a u_b
    if (stress && fluid) {
        const int nx = B.nx, ny = B.ny, nz = B.nz, m = (int)n, row = nx * ny;           // 19 N < 2^31
        const int r = (int)((unsigned)m / (unsigned)nx), x = m - r * nx, z = div_magic(r, B.dy_m, B.dy_s), y = r - z * ny;
        const int nb[3][2] = {{x == nx - 1 ? m + 1 - nx : m + 1, x == 0 ? m + nx - 1 : m - 1},
                              {y == ny - 1 ? m + nx - row : m + nx, y == 0 ? m + row - nx : m - nx},
                              {z == nz - 1 ? m - (nz - 1) * row : m + row, z == 0 ? m + (nz - 1) * row : m - row}};
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) du[a][b] = 0.5f * (u[b * B.N + nb[a][0]] - u[b * B.N + nb[a][1]]);
    }
    const float dv = (du[0][0] + du[1][1] + du[2][2]) * (1.0f / 3.0f);
    const unsigned long long pol = l2_evict_normal();
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const float cu = cx_of(i) * ux + cy_of(i) * uy + cz_of(i) * uz;
        float d = w_of(i) * (dr + rho * (3.0f * cu + 4.5f * cu * cu - 1.5f * uu));
        if (stress) {
            const int c[3] = {cx_of(i), cy_of(i), cz_of(i)};
            float q = -dv;
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int b = 0; b < 3; ++b)
                    if (c[a] * c[b] != 0) q += (float)(c[a] * c[b]) * du[a][b];
            d += -3.0f * tau * rho * w_of(i) * q;
        }
        St::st1(f + (long long)i * B.N + n, fluid ? d : 0.0f, B.scale, pol);
    }
}

// shell owner of a fluid node: the particle (p + 1) owning one of its six face
// neighbours, 0 if none (periodic; the first one found if several)
__device__ __forceinline__ int shell_owner(const int* owner, unsigned nx, unsigned ny, unsigned nz, unsigned n)
{
    const unsigned r = n / nx, x = n - r * nx, z = r / ny, y = r - z * ny, row = nx * ny;       // 19 N < 2^31
    const int v[6] = {owner[n - x + (x == 0 ? nx - 1 : x - 1)], owner[(y == 0 ? n + row - nx : n - nx)],
                      owner[(z == 0 ? n + (nz - 1) * row : n - row)], owner[n - x + (x == nx - 1 ? 0 : x + 1)],
                      owner[(y == ny - 1 ? n + nx - row : n + nx)], owner[(z == nz - 1 ? n - (nz - 1) * row : n + row)]};
    int o = 0;
#pragma unroll
    for (int k = 0; k < 6; ++k)
        if (o == 0 && v[k] > 0) o = v[k];
    return o;
}

// ---- lb_stokes_field: buffers and constants of one call
struct Stokes {
    int nx, ny, nz, np, counter;
    long long N;
    double body[3], rho0, omega;
    float kappa;                        // power of two by which the density travels with the velocity's z component
    const int* owner;
    const PartDev* pd;
    int* shell;                         // [N] -1 not fluid, 0 fluid, p + 1 fluid next to particle p
    int* counts;                        // [np + 1] fluid nodes, shell nodes per particle
    float* table;                       // [np + 1][3] force density of a fluid node by its shell entry
    double* sum;                        // [4] sums of u and drho over the fluid nodes
    float* shift;                       // [4]
    unsigned* done;                     // [2] blocks done
    float2* z;                          // [2][N] gx + i gy and gz; in Fourier space, then ux + i uy and uz + i kappa drho
    float* u;                           // [3][N]
    float* drho;                        // [N] or null
};

// Shell entries, node counts, and (the last block) the force density's values: F_ext / nshell
// on the fluid nodes next to a particle (a uniform traction just outside its surface, under
// which a sphere's interior moves rigidly at its Stokes velocity), plus the body force and
// (counter) -sum F_ext / N_fluid on every fluid node.  The values are formed once per
// particle: forming them in FP64 at every node (a sum over the particles and two divisions)
// took 1,590 us at 128^3 nodes and 16 particles, one atomic per fluid node another 50.
__global__ void __launch_bounds__(256) shell_kernel(const Stokes S)
{
    __shared__ int s_n;
    __shared__ bool s_last;
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    int fluid = 0;
    // a fixed number of blocks: with one per 256 nodes their counter atomics took 30 us at 128^3
    for (long long n = blockIdx.x * 256ll + threadIdx.x; n < S.N; n += gridDim.x * 256ll) {
        int e = -1;
        if (S.owner[n] == 0) {
            const int o = shell_owner(S.owner, S.nx, S.ny, S.nz, (unsigned)n);
            e = o > 0 && o <= S.np ? o : 0;
            ++fluid;
        }
        S.shell[n] = e;
        if (e > 0) atomicAdd(S.counts + e, 1);
    }
    fluid = __reduce_add_sync(0xffffffffu, fluid);
    if ((threadIdx.x & 31) == 0) atomicAdd(&s_n, fluid);
    __syncthreads();
    if (threadIdx.x == 0) {
        atomicAdd(S.counts, s_n);
        __threadfence();
        s_last = atomicAdd(S.done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const int nf = __ldcg(S.counts);
    for (int t = threadIdx.x; t < 3 * (S.np + 1); t += 256) {
        const int p = t / 3, k = t % 3;
        double f = S.body[k];
        if (S.counter && nf > 0)
            for (int q = 0; q < S.np; ++q) f -= S.pd[q].Fext[k] / (double)nf;
        if (p > 0) f += S.pd[p - 1].Fext[k] * (1.0 / (double)__ldcg(S.counts + p));
        S.table[t] = (float)f;
    }
}

// ---- Transforms.  Lines of any length n = r0 r1 ... (radices 8, 4, 2, 3, 5 as written-out
// butterflies, any other prime by its definition) in shared memory, Stockham order: stage s
// with ns = r0 ... r_(s-1) takes x[b + m n/r] for butterfly b, multiplies by w^(k m) with
// k = b mod ns, w = exp(sign 2 pi i / (ns r)), and writes X[(b / ns) ns r + k + m ns].  A
// block takes L neighbouring lines (16 consecutive x for the axes y and z, so that global
// accesses are 128-byte runs; one line at a time along y and z touched 8 bytes of every
// sector), in place; the two fields of real data travel as real and imaginary part of one
// complex field.  Traffic (16 bytes in, 16 out per node and pass, within L2 up to 128^3) and
// the stages' shared-memory accesses bound a pass.  Measured at 128^3: seven passes of one
// line per block over 3 + 4 complex fields took 1,270 us, the six passes here 158
// (fft_kernel: 21 forward and 23 us each, 45 for the last with its sums).
constexpr int FFT_T = 256, FFT_ST = 12;
struct FftPlan {
    int n, ns_, L, lp;                  // stages, lines per block, padded pitch of a row of lines
    float sign;
    int radix[FFT_ST], ns[FFT_ST], nb[FFT_ST];          // nb = n / radix
    unsigned nm[FFT_ST];                // division by ns (magic_div)
    int nsft[FFT_ST];
};

template <int R>
__device__ __forceinline__ void dft(float2 (&v)[R], float sign);
__device__ __forceinline__ float2 cadd2(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub2(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul2(float2 a, float2 b) { return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
__device__ __forceinline__ float2 rot(float2 a, float s) { return make_float2(-s * a.y, s * a.x); }      // i s a
template <>
__device__ __forceinline__ void dft<2>(float2 (&v)[2], float)
{
    const float2 a = v[0];
    v[0] = cadd2(a, v[1]);
    v[1] = csub2(a, v[1]);
}
template <>
__device__ __forceinline__ void dft<3>(float2 (&v)[3], float s)
{
    const float2 t = cadd2(v[1], v[2]), d = csub2(v[1], v[2]);
    const float2 m = make_float2(v[0].x - 0.5f * t.x, v[0].y - 0.5f * t.y), q = rot(d, s * 0.866025403784438647f);
    v[0] = cadd2(v[0], t);
    v[1] = cadd2(m, q);
    v[2] = csub2(m, q);
}
template <>
__device__ __forceinline__ void dft<4>(float2 (&v)[4], float s)
{
    const float2 a = cadd2(v[0], v[2]), b = csub2(v[0], v[2]), c = cadd2(v[1], v[3]), d = rot(csub2(v[1], v[3]), s);
    v[0] = cadd2(a, c);
    v[1] = cadd2(b, d);
    v[2] = csub2(a, c);
    v[3] = csub2(b, d);
}
template <>
__device__ __forceinline__ void dft<5>(float2 (&v)[5], float s)
{
    const float c1 = 0.309016994374947424f, c2 = -0.809016994374947424f, s1 = s * 0.951056516295153572f, s2 = s * 0.587785252292473129f;
    const float2 a = cadd2(v[1], v[4]), b = cadd2(v[2], v[3]), d = csub2(v[1], v[4]), e = csub2(v[2], v[3]);
    const float2 m1 = make_float2(v[0].x + c1 * a.x + c2 * b.x, v[0].y + c1 * a.y + c2 * b.y);
    const float2 m2 = make_float2(v[0].x + c2 * a.x + c1 * b.x, v[0].y + c2 * a.y + c1 * b.y);
    const float2 q1 = rot(make_float2(s1 * d.x + s2 * e.x, s1 * d.y + s2 * e.y), 1.0f);
    const float2 q2 = rot(make_float2(s2 * d.x - s1 * e.x, s2 * d.y - s1 * e.y), 1.0f);
    v[0] = cadd2(v[0], cadd2(a, b));
    v[1] = cadd2(m1, q1);
    v[2] = cadd2(m2, q2);
    v[3] = csub2(m2, q2);
    v[4] = csub2(m1, q1);
}
template <>
__device__ __forceinline__ void dft<8>(float2 (&v)[8], float s)
{
    float2 e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
    dft<4>(e, s);
    dft<4>(o, s);
    const float h = 0.707106781186547524f;
    o[1] = make_float2(h * (o[1].x - s * o[1].y), h * (o[1].y + s * o[1].x));
    o[2] = rot(o[2], s);
    o[3] = make_float2(h * (-o[3].x - s * o[3].y), h * (s * o[3].x - o[3].y));
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        v[k] = cadd2(e[k], o[k]);
        v[k + 4] = csub2(e[k], o[k]);
    }
}

// one stage of radix R over the block's lines: a -> b; lines fastest (shift lb = log2 L)
template <int R>
__device__ __forceinline__ void fft_stage(const FftPlan& P, int st, int lb, const float2* a, float2* b, const float2* tw)
{
    const int nb = P.nb[st], ns = P.ns[st], step = nb / ns, L = 1 << lb;      // w^(k m) = tw[k m step]
    for (int t = threadIdx.x; t < nb << lb; t += FFT_T) {
        const int l = t & (L - 1), j = t >> lb;
        const int q = div_magic(j, P.nm[st], P.nsft[st]), k = j - q * ns;
        float2 v[R];
#pragma unroll
        for (int m = 0; m < R; ++m) v[m] = a[(j + m * nb) * P.lp + l];
#pragma unroll
        for (int m = 1; m < R; ++m) v[m] = cmul2(v[m], tw[k * m * step]);
        dft<R>(v, P.sign);
        const int o = q * ns * R + k;
#pragma unroll
        for (int m = 0; m < R; ++m) b[(o + m * ns) * P.lp + l] = v[m];
    }
}
// a stage of any radix by its definition, one output per thread
__device__ __forceinline__ void fft_stage_any(const FftPlan& P, int st, int lb, const float2* a, float2* b, const float2* tw)
{
    const int nb = P.nb[st], ns = P.ns[st], r = P.radix[st], step = nb / ns, L = 1 << lb;
    for (int t = threadIdx.x; t < P.n << lb; t += FFT_T) {
        const int l = t & (L - 1), jm = t >> lb, mo = jm / nb, j = jm - mo * nb;
        const int q = div_magic(j, P.nm[st], P.nsft[st]), k = j - q * ns;
        // angle of input m: m (k step + mo nb), modulo n
        int inc = k * step + mo * nb, at = 0;
        if (inc >= P.n) inc -= P.n;
        float2 s = make_float2(0.0f, 0.0f);
        for (int m = 0; m < r; ++m) {
            s = cadd2(s, cmul2(a[(j + m * nb) * P.lp + l], tw[at]));
            at += inc;
            if (at >= P.n) at -= P.n;
        }
        b[(q * ns * r + k + mo * ns) * P.lp + l] = s;
    }
}

enum { FFT_INPLACE = 0, FFT_FIRST = 1, FFT_LAST = 2 };

// Lines along axis (0 x, 1 y, 2 z) of field blockIdx.y.  FFT_FIRST (axis x) takes the force
// density from the shell entries; FFT_LAST (axis x) writes the real fields, sums them over the
// fluid nodes, and its last block forms the shifts: a uniform velocity so that fluid and
// particle momentum add up to zero (rho0 sum_fluid u + sum_p M_p U_p = 0) and no net mass.
template <int MODE>
__global__ void __launch_bounds__(FFT_T) fft_kernel(const __grid_constant__ Stokes S, const __grid_constant__ FftPlan P, int axis, int lb)
{
    extern __shared__ float2 fsm[];
    float2* a = fsm;
    float2* b = a + P.n * P.lp;
    float2* tw = b + P.n * P.lp;
    const int n = P.n, L = 1 << lb, comp = blockIdx.y;
    for (int j = threadIdx.x; j < n; j += FFT_T) {
        float sn, cs;
        sincospif(2.0f * (float)j / (float)n, &sn, &cs);
        tw[j] = make_float2(cs, P.sign * sn);
    }
    float2* z = S.z + comp * S.N;
    // first element, line pitch, element stride and number of lines of this block
    long long base, ls, es;
    int nl;
    if (axis == 0) {
        const long long rows = (long long)S.ny * S.nz, r0 = (long long)blockIdx.x << lb;
        base = r0 * S.nx; ls = S.nx; es = 1;
        nl = (int)min((long long)L, rows - r0);
    } else {
        const int tiles = (S.nx + L - 1) >> lb, pl = blockIdx.x / tiles, x0 = (blockIdx.x - pl * tiles) << lb;
        const long long row = (long long)S.nx * S.ny;
        base = (axis == 1 ? pl * row : (long long)pl * S.nx) + x0; ls = 1; es = axis == 1 ? S.nx : row;
        nl = min(L, S.nx - x0);
    }
    // along x consecutive threads take consecutive elements of a line, else consecutive lines
    if (axis == 0) {
        for (int l = threadIdx.x >> 5; l < nl; l += FFT_T / 32)
            for (int j = threadIdx.x & 31; j < n; j += 32) {
                if (MODE == FFT_FIRST) {
                    const int e = S.shell[base + l * ls + j];
                    float2 v = make_float2(0.0f, 0.0f);
                    if (e >= 0) v = comp == 0 ? make_float2(S.table[3 * e], S.table[3 * e + 1]) : make_float2(S.table[3 * e + 2], 0.0f);
                    a[j * P.lp + l] = v;
                } else {
                    a[j * P.lp + l] = z[base + l * ls + j];
                }
            }
    } else {
        for (int t = threadIdx.x; t < n << lb; t += FFT_T) {
            const int l = t & (L - 1), j = t >> lb;
            if (l < nl) a[j * P.lp + l] = z[base + l + j * es];
        }
    }
    __syncthreads();
    for (int st = 0; st < P.ns_; ++st) {
        switch (P.radix[st]) {
        case 8: fft_stage<8>(P, st, lb, a, b, tw); break;
        case 5: fft_stage<5>(P, st, lb, a, b, tw); break;
        case 4: fft_stage<4>(P, st, lb, a, b, tw); break;
        case 3: fft_stage<3>(P, st, lb, a, b, tw); break;
        case 2: fft_stage<2>(P, st, lb, a, b, tw); break;
        default: fft_stage_any(P, st, lb, a, b, tw);
        }
        __syncthreads();
        float2* t = a;
        a = b;
        b = t;
    }
    if (MODE != FFT_LAST) {
        if (axis == 0) {
            for (int l = threadIdx.x >> 5; l < nl; l += FFT_T / 32)
                for (int j = threadIdx.x & 31; j < n; j += 32) z[base + l * ls + j] = a[j * P.lp + l];
        } else {
            for (int t = threadIdx.x; t < n << lb; t += FFT_T) {
                const int l = t & (L - 1), j = t >> lb;
                if (l < nl) z[base + l + j * es] = a[j * P.lp + l];
            }
        }
        return;
    }
    // real fields and their sums over the fluid nodes (per thread as a sum and its rounding errors)
    float hi[2] = {0.0f, 0.0f}, lo[2] = {0.0f, 0.0f};
    const float ik = 1.0f / S.kappa;
    for (int l = threadIdx.x >> 5; l < nl; l += FFT_T / 32)
        for (int j = threadIdx.x & 31; j < n; j += 32) {
            const long long at = base + l * ls + j;
            const float2 v = a[j * P.lp + l];
            const float w[2] = {v.x, comp == 0 ? v.y : v.y * ik};
            S.u[(comp == 0 ? 0 : 2) * S.N + at] = w[0];
            if (comp == 0) S.u[S.N + at] = w[1];
            else if (S.drho) S.drho[at] = w[1];
            if (S.shell[at] >= 0) {
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const float t = hi[c] + w[c], d = t - hi[c];
                    lo[c] += (hi[c] - (t - d)) + (w[c] - d);
                    hi[c] = t;
                }
            }
        }
    __shared__ double s_sum[FFT_T / 32][2];
    __shared__ bool s_last;
    double v[2] = {(double)hi[0] + (double)lo[0], (double)hi[1] + (double)lo[1]};
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        for (int o = 16; o > 0; o >>= 1) v[c] += __shfl_xor_sync(0xffffffffu, v[c], o);
        if ((threadIdx.x & 31) == 0) s_sum[threadIdx.x >> 5][c] = v[c];
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        double t = 0.0;
        for (int w = 0; w < FFT_T / 32; ++w) t += s_sum[w][threadIdx.x];
        atomicAdd(S.sum + 2 * comp + threadIdx.x, t);
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(S.done + 1, 1u) == gridDim.x * gridDim.y - 1;
    __syncthreads();
    if (!s_last || threadIdx.x >= 4) return;
    __threadfence();
    const int k = threadIdx.x, nf = __ldcg(S.counts);
    double Pk = 0.0;
    if (k < 3)
        for (int p = 0; p < S.np; ++p) Pk += S.pd[p].M * S.pd[p].U[k];
    S.shift[k] = nf > 0 ? (float)((-Pk / S.rho0 - __ldcg(S.sum + k)) / (double)nf) : 0.0f;
}

// the shifts, on the fluid nodes
__global__ void __launch_bounds__(256) shift_kernel(const Stokes S)
{
    const float s[4] = {S.shift[0], S.shift[1], S.shift[2], S.shift[3]};
    for (long long n = blockIdx.x * 256ll + threadIdx.x; n < S.N; n += gridDim.x * 256ll) {
        if (S.shell[n] < 0) continue;
#pragma unroll
        for (int k = 0; k < 3; ++k) S.u[k * S.N + n] += s[k];
        if (S.drho) S.drho[n] += s[3];
    }
}

// Steady state of the linear lattice fluid itself (D3Q19 BGK, omega = 1/tau,
// Guo forcing, about rho0) under the force density g, mode by mode (k = 2 pi
// (x/nx, y/ny, z/nz) for the DFT index (x, y, z)).  The steady pre-collision
// populations are the post-collision ones streamed, f^_i = e_i f^*_i with
// e_i = exp(-i k.c_i), hence f^_i = h_i (omega f^eq_i + (1 - omega/2) F^_i),
// h_i = e_i / (1 - (1 - omega) e_i), F_i = 3 w_i c_i.g, and their moments
// (drho, u = j + g/2) solve
//   D0 drho - 3 rho0 omega H1 . u = 3 (1 - omega/2) H1 . g
//   -omega H1 drho + rho0 D2 u     = g/2 + 3 (1 - omega/2) H2 g
// with H1 = sum w_i c_i h_i, H2 = sum w_i c_i c_i^T h_i,
// D0 = sum w_i (1 - e_i) q_i and D2 = sum 3 w_i c_i c_i^T (1 - e_i) q_i,
// q_i = 1 / (1 - (1 - omega) e_i).  The terms of c and -c are complex conjugates, so H1 = i a
// with a real and H2, D0, D2 are real: over the nine pairs of directions
//   a = sum 2 w c Im h,  H2 = sum 2 w c c^T Re h,  D0 = sum 2 w r,  D2 = sum 6 w c c^T r,
//   r = Re (1 - e) q = (1 + (1 - omega)) 2 sin^2(th/2) / |1 - (1 - omega) e|^2 >= 0,
// without cancellation (D0 and D2 vanish like k^2).  With drho = i s and b = g/2 + fo H2 g
// (fo = 3 (1 - omega/2)) the equations are real, for the real and the imaginary part of g alike:
//   rho0 D2 u = b - omega a s,   (D0 + 3 omega^2 a.D2^-1 a) s = fo a.g + 3 omega a.D2^-1 b,
// D2 symmetric positive definite, inverted by cofactors, and a scalar equation whose terms on
// the left have one sign.  (One 3 x 3 system with the pressure eliminated is stiff along a by 1 / (nu k^2),
// and its determinant loses the square of that.)  The terms of one direction are FP32; sums and
// solve are carried to twice FP32's digits (ff below).
// One thread takes a mode and its conjugate: the fields are real, so the transforms of two of
// them come as one, Z(k) = X(k) + i Y(k), X(k) = (Z(k) + conj Z(-k)) / 2, and go back the
// same way.  The k = 0 mode (mean flow and mass, set afterwards) and numerically singular
// modes are zero; the 1/N of the inverse DFT is folded in.
// Numbers as the unevaluated sum of two FP32 (Dekker, "A floating-point technique for
// extending the available precision", 1971; Knuth's two-sum): 48 bits of significand from FP32
// instructions, which this part issues 64 times as often as FP64 ones.  In u = D2^-1 (b - omega a s)
// the longitudinal part cancels down to about nu k^2 of its terms (1e-4 at an edge of 64 and
// tau = 0.52): 2^-46 over that stays far below the FP32 rounding of the directions' terms.
struct ff {
    float h, l;
};
__device__ __forceinline__ ff two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b), d = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, d)), __fsub_rn(b, d))};
}
__device__ __forceinline__ ff quick(float a, float b)       // |a| >= |b|
{
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ ff operator+(ff a, ff b)
{
    const ff s = two_sum(a.h, b.h);
    return quick(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ ff operator-(ff a, ff b) { return a + ff{-b.h, -b.l}; }
__device__ __forceinline__ ff operator+(ff a, float b)
{
    const ff s = two_sum(a.h, b);
    return quick(s.h, __fadd_rn(s.l, a.l));
}
__device__ __forceinline__ ff operator*(ff a, ff b)
{
    const float p = __fmul_rn(a.h, b.h);
    return quick(p, __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.h, -p))));
}
__device__ __forceinline__ ff operator*(ff a, float b)
{
    const float p = __fmul_rn(a.h, b);
    return quick(p, __fmaf_rn(a.l, b, __fmaf_rn(a.h, b, -p)));
}
__device__ __forceinline__ ff recip(ff a)
{
    const float x = 1.0f / a.h;
    const float e = __fmaf_rn(-a.l, x, __fmaf_rn(-a.h, x, 1.0f));      // 1 - a x
    return quick(x, __fmul_rn(x, e));
}

struct SteadyConst {
    ff fo, fo18, om2, om18, om_18;          // fo, fo / 18, omega^2, 18 omega, omega / 18
    ff six_rho_n, inv_n;                    // 6 / (rho0 N), 1 / N
    float om, om1, opm;                     // omega, 1 - omega, 2 - omega
};

// One thread per mode of the planes z <= nz / 2 that comes no later than its conjugate.
// Sums in units of 1/18: D0 = D0' / 18, a = a' / 18, H2 = H2' / 18, D2 = D2' / 6.
// Measured at 128^3: 4,207 us as a complex 4 x 4 FP64 elimination with pivoting per mode,
// 102 us like this.
__global__ void __launch_bounds__(128) steady_kernel(const Stokes S, const SteadyConst K)
{
    const int nx = S.nx, ny = S.ny, nz = S.nz;
    const int r = (int)(blockIdx.x * 128u + threadIdx.x);           // 19 N < 2^31
    const int plane = nx * ny;
    if (r >= (nz / 2 + 1) * plane) return;
    const int z = r / plane, y = (r - z * plane) / nx, x = r - z * plane - y * nx;
    const int r2 = ((z == 0 ? 0 : nz - z) * ny + (y == 0 ? 0 : ny - y)) * nx + (x == 0 ? 0 : nx - x);
    if (r2 < r) return;
    const float2 z1 = S.z[r], z1c = S.z[r2], z2 = S.z[S.N + r];
    // from the index nearer to zero, so that the small angles of both ends keep their digits
    const float fx = (float)(2 * x > nx ? x - nx : x) / nx, fy = (float)(2 * y > ny ? y - ny : y) / ny, fz = (float)z / nz;
    const ff zero = {0.0f, 0.0f};
    ff a[3] = {zero, zero, zero}, D0 = zero;
    ff H[6] = {zero, zero, zero, zero, zero, zero}, D[6] = {zero, zero, zero, zero, zero, zero};      // xx yy zz xy xz yz
#pragma unroll
    for (int m = 0; m < 9; ++m) {
        const int i = 2 * m + 1, cx = cx_of(i), cy = cy_of(i), cz = cz_of(i);
        // theta / pi, reduced to [-1, 1) so that the half angle stays in the accurate range
        float tp = 2.0f * (fx * cx + fy * cy + fz * cz);
        tp -= 2.0f * floorf(0.5f * tp + 0.5f);
        float sh, ch;
        sincospif(0.5f * tp, &sh, &ch);
        const float s2 = sh * sh, c2 = ch * ch;
        // |1 - (1 - omega) e|^2 as a sum of terms of one sign, cos th - (1 - omega) from the half angle that is
        // small where it cancels
        const float dd = K.om1 >= 0.0f ? K.om * K.om + 4.0f * K.om1 * s2 : K.opm * K.opm - 4.0f * K.om1 * c2;
        const float hn = K.om1 >= 0.0f ? K.om - 2.0f * s2 : 2.0f * c2 - K.opm;
        const float wt = m < 3 ? 2.0f : 1.0f;                       // 36 w
        const float id = wt / dd;
        const float hre = hn * id, him = -2.0f * sh * ch * id, rr = K.opm * (2.0f * s2) * id;
        D0 = D0 + rr;
        if (cx) { a[0] = a[0] + (float)cx * him; H[0] = H[0] + hre; D[0] = D[0] + rr; }
        if (cy) { a[1] = a[1] + (float)cy * him; H[1] = H[1] + hre; D[1] = D[1] + rr; }
        if (cz) { a[2] = a[2] + (float)cz * him; H[2] = H[2] + hre; D[2] = D[2] + rr; }
        if (cx * cy) { H[3] = H[3] + (float)(cx * cy) * hre; D[3] = D[3] + (float)(cx * cy) * rr; }
        if (cx * cz) { H[4] = H[4] + (float)(cx * cz) * hre; D[4] = D[4] + (float)(cx * cz) * rr; }
        if (cy * cz) { H[5] = H[5] + (float)(cy * cz) * hre; D[5] = D[5] + (float)(cy * cz) * rr; }
    }
    // [part][component] of g: real, imaginary
    const float g[2][3] = {{0.5f * (z1.x + z1c.x), 0.5f * (z1.y + z1c.y), z2.x}, {0.5f * (z1.y - z1c.y), 0.5f * (z1c.x - z1.x), z2.y}};
    float u[2][3] = {}, sd[2] = {};
    // E = D2'^-1 by cofactors (its eigenvalues lie close together), E a, and the pressure's factor
    const ff Cxx = D[1] * D[2] - D[5] * D[5], Cxy = D[4] * D[5] - D[3] * D[2], Cxz = D[3] * D[5] - D[4] * D[1];
    const ff Cyy = D[0] * D[2] - D[4] * D[4], Cyz = D[3] * D[4] - D[0] * D[5], Czz = D[0] * D[1] - D[3] * D[3];
    const ff det = D[0] * Cxx + D[3] * Cxy + D[4] * Cxz;
    // numerically singular: a determinant below 1e-13 of the product of the diagonal
    if (r != 0 && D0.h > 0.0f && det.h > 1e-13f * D[0].h * D[1].h * D[2].h) {
        const ff idet = recip(det);
        const ff ea[3] = {(Cxx * a[0] + Cxy * a[1] + Cxz * a[2]) * idet, (Cxy * a[0] + Cyy * a[1] + Cyz * a[2]) * idet,
                          (Cxz * a[0] + Cyz * a[1] + Czz * a[2]) * idet};
        const ff is = recip(D0 + K.om2 * (a[0] * ea[0] + a[1] * ea[1] + a[2] * ea[2]));
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const ff ag = a[0] * g[c][0] + a[1] * g[c][1] + a[2] * g[c][2];
            const ff bx = K.fo18 * (H[0] * g[c][0] + H[3] * g[c][1] + H[4] * g[c][2]) + 0.5f * g[c][0];
            const ff by = K.fo18 * (H[3] * g[c][0] + H[1] * g[c][1] + H[5] * g[c][2]) + 0.5f * g[c][1];
            const ff bz = K.fo18 * (H[4] * g[c][0] + H[5] * g[c][1] + H[2] * g[c][2]) + 0.5f * g[c][2];
            const ff x0 = (Cxx * bx + Cxy * by + Cxz * bz) * idet, x1 = (Cxy * bx + Cyy * by + Cyz * bz) * idet,
                     x2 = (Cxz * bx + Cyz * by + Czz * bz) * idet;
            const ff s = (K.fo * ag + K.om18 * (a[0] * x0 + a[1] * x1 + a[2] * x2)) * is;
            const ff q = K.om_18 * s;
            const ff ux = (x0 - q * ea[0]) * K.six_rho_n, uy = (x1 - q * ea[1]) * K.six_rho_n, uz = (x2 - q * ea[2]) * K.six_rho_n;
            const ff sn = s * K.inv_n;
            u[c][0] = ux.h + ux.l; u[c][1] = uy.h + uy.l; u[c][2] = uz.h + uz.l;
            sd[c] = sn.h + sn.l;
        }
    }
    // drho = i s: real part -Im s, imaginary part Re s
    const float dre = -sd[1] * S.kappa, dim = sd[0] * S.kappa;
    S.z[r] = make_float2(u[0][0] - u[1][1], u[1][0] + u[0][1]);
    S.z[S.N + r] = make_float2(u[0][2] - dim, u[1][2] + dre);
    if (r2 != r) {
        S.z[r2] = make_float2(u[0][0] + u[1][1], u[0][1] - u[1][0]);
        S.z[S.N + r2] = make_float2(u[0][2] + dim, dre - u[1][2]);
    }
}
static unsigned nblk(long long n, int t) { return (unsigned)((n + t - 1) / t); }

cudaError_t launch_init_fluid(const BoxDev& B, int precision, void* fbuf, const float* u, const float* drho,
                              const int* owner, float tau, int stress, cudaStream_t s)
{
    const unsigned g = nblk(B.N, 256);
    if (precision == 1) init_fluid_kernel<StF16><<<g, 256, 0, s>>>(B, fbuf, u, drho, owner, tau, stress);
    else if (precision == 2) init_fluid_kernel<StBF16><<<g, 256, 0, s>>>(B, fbuf, u, drho, owner, tau, stress);
    else init_fluid_kernel<StF32><<<g, 256, 0, s>>>(B, fbuf, u, drho, owner, tau, stress);
    return cudaGetLastError();
}

// radices of a line of length n: 8, 4, 2, then 3, 5, then whatever primes are left
static FftPlan fft_plan(int n, float sign)
{
    FftPlan P{};
    P.n = n;
    P.sign = sign;
    int left = n, ns = 1;
    auto take = [&](int r) {
        P.radix[P.ns_] = r;
        P.ns[P.ns_] = ns;
        P.nb[P.ns_] = n / r;
        magic_div((unsigned)ns, P.nm[P.ns_], P.nsft[P.ns_]);
        ++P.ns_;
        ns *= r;
        left /= r;
    };
    while (left % 8 == 0 && left != 16) take(8);        // 16 = 4 x 4
    for (int r : {4, 2, 3, 5})
        while (left % r == 0) take(r);
    for (int r = 7; left > 1; r += 2) {
        if (r * r > left) r = left;
        while (left % r == 0) take(r);
    }
    return P;
}

// z: 2 N float2; shell: N ints; counts: np + 1 ints; table: 3 (np + 1) floats; sum: 4 doubles,
// shift: 4 floats, done: 2 counters; u [3][N], drho [N] or null: the result
cudaError_t launch_stokes(const BoxDev& B, const int* owner, const PartDev* pd, int np, int counter_on,
                          const double body[3], float2* z, int* shell, int* counts, float* table, double* sum, float* u,
                          float* drho, double tau, cudaStream_t s)
{
    cudaError_t e;
    Stokes S{};
    S.nx = B.nx; S.ny = B.ny; S.nz = B.nz; S.np = np; S.counter = counter_on; S.N = B.N;
    for (int k = 0; k < 3; ++k) S.body[k] = body[k];
    S.rho0 = B.rho0; S.omega = 1.0 / tau;        // in FP64: at tau = 0.52 an FP32 omega is worth 1e-6 of the viscosity
    // drho is of the order of mu u / r a few nodes from a particle: scaled so that neither of
    // the two fields that share a transform loses digits to the other
    int ex = 0;
    std::frexp(0.5 / (B.rho0 * (1.0 / S.omega - 0.5) / 3.0), &ex);
    S.kappa = (float)std::ldexp(1.0, ex);
    S.owner = owner; S.pd = pd; S.shell = shell; S.counts = counts; S.table = table; S.sum = sum;
    S.shift = reinterpret_cast<float*>(sum + 4);
    S.done = reinterpret_cast<unsigned*>(S.shift + 4);
    S.z = z; S.u = u; S.drho = drho;
    if ((e = cudaMemsetAsync(counts, 0, sizeof(int) * (np + 1), s)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(sum, 0, 4 * sizeof(double) + 4 * sizeof(float) + 2 * sizeof(unsigned), s)) != cudaSuccess) return e;
    const unsigned g = nblk(S.N, 256) < 1216 ? nblk(S.N, 256) : 1216;
    shell_kernel<<<g, 256, 0, s>>>(S);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    auto pass = [&](int mode, int ax, float sign) {
        FftPlan P = fft_plan(ax == 0 ? B.nx : (ax == 1 ? B.ny : B.nz), sign);
        // 16 lines (128-byte runs along x) while two buffers of them take at most 72 KiB of shared memory
        int lb = 4;
        while (lb > 0 && 2ll * P.n * ((1 << lb) + 1) * 8 > 72 * 1024) --lb;
        P.lp = (1 << lb) + 1;
        const size_t sm = sizeof(float2) * (2ull * P.n * P.lp + P.n);
        const long long lines = ax == 0 ? ((long long)B.ny * B.nz + (1 << lb) - 1) >> lb
                                        : (long long)(ax == 1 ? B.nz : B.ny) * ((B.nx + (1 << lb) - 1) >> lb);
        const dim3 grid((unsigned)lines, 2);
        auto go = [&](auto* k) {
            if (sm > 48 * 1024) {
                const cudaError_t r = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
                if (r != cudaSuccess) return r;
            }
            k<<<grid, FFT_T, sm, s>>>(S, P, ax, lb);
            return cudaGetLastError();
        };
        return mode == FFT_FIRST ? go(fft_kernel<FFT_FIRST>) : (mode == FFT_LAST ? go(fft_kernel<FFT_LAST>) : go(fft_kernel<FFT_INPLACE>));
    };
    if ((e = pass(FFT_FIRST, 0, -1.0f)) != cudaSuccess) return e;
    for (int ax = 1; ax < 3; ++ax)
        if ((e = pass(FFT_INPLACE, ax, -1.0f)) != cudaSuccess) return e;
    SteadyConst K;
    const double om = S.omega, fo = 3.0 * (1.0 - 0.5 * om);
    auto split = [](double v) { const float h = (float)v; return ff{h, (float)(v - (double)h)}; };
    K.fo = split(fo); K.fo18 = split(fo / 18.0); K.om2 = split(om * om); K.om18 = split(18.0 * om); K.om_18 = split(om / 18.0);
    K.six_rho_n = split(6.0 / (S.rho0 * (double)S.N)); K.inv_n = split(1.0 / (double)S.N);
    K.om = (float)om; K.om1 = (float)(1.0 - om); K.opm = (float)(2.0 - om);
    steady_kernel<<<nblk((long long)(B.nz / 2 + 1) * B.nx * B.ny, 128), 128, 0, s>>>(S, K);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    for (int ax = 2; ax > 0; --ax)
        if ((e = pass(FFT_INPLACE, ax, 1.0f)) != cudaSuccess) return e;
    if ((e = pass(FFT_LAST, 0, 1.0f)) != cudaSuccess) return e;
    shift_kernel<<<g, 256, 0, s>>>(S);
    return cudaGetLastError();
}

}  // namespace lbsph
