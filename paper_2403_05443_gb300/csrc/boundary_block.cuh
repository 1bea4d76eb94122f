// Boundary block (see boundary_kernel.cu for the method), shared by the
// boundary kernel and the persistent step kernel.
#pragma once

#include <type_traits>

#include "lattice_common.cuh"

namespace lbsph {

// round(f * 2^46) toward zero, from the IEEE 754 fields with integer
// instructions (exact for |f| >= 2^-23, off by less than 2^-46 below; 64-bit
// float-to-integer conversions run at the slow FP64 rate on this part)
__device__ __forceinline__ long long fixq(float f)
{
    const unsigned u = __float_as_uint(f);
    const int ex = (int)((u >> 23) & 0xffu);
    const long long m = (long long)((u & 0x7fffffu) | 0x800000u);
    const int sh = ex - 104;                    // f * 2^46 = m * 2^(ex - 127 - 23 + 46)
    long long v;
    if (ex == 0 || sh <= -24) v = 0;            // zero, subnormal, or |f| < 2^-46
    else if (sh >= 0) v = m << (sh > 38 ? 38 : sh);   // saturates for |f| >= 2^16 (no deviation is)
    else v = m >> (-sh);
    return (u >> 31) ? -v : v;
}

// a b - c d with one rounding less; written out, like the bounce-back terms, so that a
// node's rounding does not depend on which products the compiler finds in common
__device__ __forceinline__ float cross_term(float a, float b, float c, float d)
{
    return __fmaf_rn(a, b, -__fmul_rn(c, d));
}

__device__ __forceinline__ long long warp_sum(long long v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += (long long)__shfl_xor_sync(0xffffffffu, (unsigned long long)v, o);
    return v;
}

// block c (of P.gx) of particle p; BBLOCK threads.  A function of its own, as the
// critical and the auxiliary block are: inlined into the step kernel they cost the bulk
// loop registers (spilled ones, in some builds; us per step, with and without inlining:
// 8 boxes of 64^3 in FP32 56.3 / 55.0 and in FP16 39.1 / 37.0, the 32 squirmer boxes in
// BF16 404 / 380).  The parameters are copied once at its start: read through the
// reference each is a load on the particle's chain (channel 33.6 / 32.1 us in that comparison).
template <class St, bool FIRST>
__device__ __noinline__ void boundary_block(const BndParams& kernel_params, int p, int c)
{
    const BndParams P = kernel_params;
    using T = typename St::T;
    constexpr int NW = BBLOCK / 32;
    const int gx = P.gx;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cap = P.list_cap, smax = P.smax;

    extern __shared__ uint64_t s_bits[];            // ring slots 0 and 1 (smax*smax rows each), then the node list
    unsigned* s_list = reinterpret_cast<unsigned*>(s_bits + 2 * smax * smax);
    __shared__ PartK K;
    __shared__ long long s_red[NW][ACC_COV];        // per-warp link sums
    __shared__ long long s_rare[NACC - ACC_COV];    // covered / uncovered nodes (rare: shared atomics)
    __shared__ int s_wsum[NW];
    __shared__ PartK s_pk[MAXNB];                   // partners' snapshots (particles whose cubes reach this one's)
    __shared__ NeedHdr s_ph[MAXNB];

    // ---- one round of independent loads
    const BoxDyn dyn = ldcg_dyn(P.pdyn + p);
    const int rrow = c + gx * tid;                  // this thread's cube row
    uint64_t need = rrow < smax * smax ? __ldcg(P.need + (size_t)p * (MAXS * MAXS) + rrow) : 0ull;
    {
        ldcg_copy(&K, P.pk + p, tid, BBLOCK);
        if (tid < NACC - ACC_COV) s_rare[tid] = 0;
        const uint64_t* r0 = P.rows + (size_t)p * 2 * (MAXS * MAXS);
        const int n = smax * smax;
#pragma unroll 4
        for (int r = tid; r < n; r += BBLOCK) {
            s_bits[r] = __ldcg(r0 + r);
            s_bits[n + r] = __ldcg(r0 + MAXS * MAXS + r);
        }
    }
    __syncthreads();

    // partners: their snapshots and redo-mask cubes (the critical blocks of a
    // partner run only after this block: the cluster's items come first)
    const int nnb = min(K.nnb, MAXNB);
    if (nnb > 0) {
        for (int j = 0; j < nnb; ++j) ldcg_copy(&s_pk[j], P.pk + K.nb[j], tid, BBLOCK);
        if (tid < nnb) s_ph[tid] = ldcg_hdr(P.need_hdr + K.nb[tid]);
        __syncthreads();
    }
    const int S = K.S;
    const uint64_t* slot1 = P.rows + ((size_t)p * 2 + 1) * (MAXS * MAXS);
    const uint64_t* s_new = s_bits + (K.rows_new == slot1 ? smax * smax : 0);
    const uint64_t* s_old = s_bits + (K.rows_old == slot1 ? smax * smax : 0);
    const int nx = K.nx, ny = K.ny, nz = K.nz;
    const bool walls = K.walls != 0;
    int dsh[3];                                     // o_new - o_old: old-local = new-local + dsh
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int L = k == 0 ? nx : (k == 1 ? ny : nz);
        int v = K.ow_new[k] - K.ow_old[k];
        if (v > L / 2) v -= L;
        if (v < -L / 2) v += L;
        dsh[k] = FIRST ? 0 : v;
    }
    auto bit_new = [&](int ax, int ay, int az) -> bool {
        if (ax < 0 || ax >= S || ay < 0 || ay >= S || az < 0 || az >= S) return false;
        return (s_new[az * S + ay] >> ax) & 1ull;
    };
    auto bit_old = [&](int ax, int ay, int az) -> bool {
        ax += dsh[0]; ay += dsh[1]; az += dsh[2];
        if (ax < 0 || ax >= S || ay < 0 || ay >= S || az < 0 || az >= S) return false;
        return (s_old[az * S + ay] >> ax) & 1ull;
    };
    // the nodes ax - 1, ax, ax + 1 of row (ay, az) of a map (0 <= x < S inside) as bits 0..2
    auto row3 = [&](const uint64_t* map, int ax, int ay, int az) -> unsigned {
        if (ax < -1 || ax > S || ay < 0 || ay >= S || az < 0 || az >= S) return 0u;
        const uint64_t w = map[az * S + ay];
        return (unsigned)(ax >= 1 ? w >> (ax - 1) : w << (1 - ax)) & 7u;
    };
    // a node (X, Y, Z in the box) in partner j's new or old cube: its local coordinates
    auto ploc = [&](int j, bool nw, int X_, int Y_, int Z_, int& lx, int& ly, int& lz) -> bool {
        const int* ow = nw ? s_pk[j].ow_new : s_pk[j].ow_old;
        lx = X_ - ow[0]; if (lx < 0) lx += nx;
        ly = Y_ - ow[1]; if (ly < 0) ly += ny;
        lz = Z_ - ow[2]; if (lz < 0) lz += nz;
        const int Sq = s_pk[j].S;
        return lx < Sq && ly < Sq && lz < Sq;
    };
    auto pbit = [&](int j, bool nw, int X_, int Y_, int Z_) -> bool {
        int lx, ly, lz;
        if (!ploc(j, nw, X_, Y_, Z_, lx, ly, lz)) return false;
        const uint64_t* rw = nw ? s_pk[j].rows_new : s_pk[j].rows_old;
        return (__ldcg(rw + lz * s_pk[j].S + ly) >> lx) & 1ull;
    };
    // integer sums that belong to partner j (global atomics: rare)
    auto padd = [&](int j, int e, long long v) {
        if (v != 0) atomicAdd(reinterpret_cast<unsigned long long*>(P.acc + (size_t)K.nb[j] * NACC + e),
                              static_cast<unsigned long long>(v));
    };
    // ---- this block's rows: the nodes to redo, compacted into shared memory
    {
        if (rrow >= S * S) need = 0;
        // block-wide exclusive scan of the row counts
        const int cnt = __popcll(need);
        int inc = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += v;
        }
        if (lane == 31) s_wsum[warp] = inc;
        __syncthreads();
        int base = inc - cnt;
        for (int w = 0; w < warp; ++w) base += s_wsum[w];
        const int my = rrow % S, mz = rrow / S;
        for (int k = 0; need; ++k) {
            const int mx = __ffsll((long long)need) - 1;
            need &= need - 1;
            if (base + k < cap) s_list[base + k] = (unsigned)((mz << 16) | (my << 8) | mx);
        }
    }
    __syncthreads();
    int total = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) total += s_wsum[w];
    if (tid == 0 && total > cap) atomicOr(P.status, ST_CAPACITY);
    const int count = min(total, cap);

    const int N = (int)K.N;
    const T* A = reinterpret_cast<const T*>(P.src) + K.off;
    const float inv = K.inv_scale, rho0 = K.rho0f, scale = K.scale;
    const unsigned long long pol = l2_evict_normal();
    T* D = reinterpret_cast<T*>(P.dst) + K.off;

    // ---- this block's nodes, two warps per node: the even warp of a pair takes
    // the rest population and the directions 1..10, the odd warp 11..18 (each
    // warp's path stays uniform and each thread's dependent chain is about half
    // as long); the node's moments (and, for the ghost-mode collision, its second
    // moments) are added up through shared memory, in one order on both warps, so
    // that both take identical decisions and values.  Per-thread link sums.
    long long aF[3] = {0, 0, 0}, aT[3] = {0, 0, 0};
    auto rare_add = [&](int j, long long v) {
        if (v != 0) atomicAdd(reinterpret_cast<unsigned long long*>(&s_rare[j - ACC_COV]), (unsigned long long)v);
    };
    constexpr int NX = St::GHOST ? 10 : 4;         // exchanged partial moments per node
    __shared__ float s_xch[NW / 2][2][NX][32];
    const int wpair = warp >> 1;
    const int rounds = (count + (BBLOCK / 2) - 1) / (BBLOCK / 2);

    auto node_round = [&](auto Hc, int rnd) {
        constexpr int H = decltype(Hc)::value;
        auto mine = [](int i) { return H == 0 ? i <= 10 : i >= 11; };
        const int e = rnd * (BBLOCK / 2) + wpair * 32 + lane;
        bool act = e < count;
        int mx = 0, my = 0, mz = 0, X = 0, Y = 0, Z = 0;
        int own = 0;                                // offsets within a box fit 32 bits: 19 N < 2^31
        bool wallrow = false, sol_new = false, sol_old = false;
        int pn = -1, po = -1;
        if (act) {
            const unsigned code = s_list[e];
            mx = code & 0xff; my = (code >> 8) & 0xff; mz = (code >> 16) & 0xff;
            X = wrapd(K.ow_new[0] + mx, nx); Y = wrapd(K.ow_new[1] + my, ny); Z = wrapd(K.ow_new[2] + mz, nz);
            own = (Z * ny + Y) * nx + X;
            wallrow = walls && (Y == 0 || Y == ny - 1);
            sol_new = bit_new(mx, my, mz);
            sol_old = !FIRST && bit_old(mx, my, mz);
            // partners: a node in the redo masks of two particles is done once, by
            // the one of lower index; a partner may hold it now (pn) or before (po)
            if (nnb > 0) {
                bool dup = false;
                for (int j = 0; j < nnb; ++j) {
                    if (K.nb[j] < p) {
                        const NeedHdr& h = s_ph[j];
                        int lx = X - h.ow[0], ly = Y - h.ow[1], lz = Z - h.ow[2];
                        if (lx < 0) lx += nx;
                        if (ly < 0) ly += ny;
                        if (lz < 0) lz += nz;
                        if (lx < h.S && ly < h.S && lz < h.S &&
                            ((__ldcg(P.need + (size_t)K.nb[j] * (MAXS * MAXS) + lz * h.S + ly) >> lx) & 1ull))
                            dup = true;
                    }
                    if (pbit(j, true, X, Y, Z)) pn = j;
                    if (!FIRST && pbit(j, false, X, Y, Z)) po = j;
                }
                if (dup) act = false;
            }
        }
        const bool solN = sol_new || pn >= 0, solO = sol_old || po >= 0;
        // 0 nothing, 1 solid before and after (untouched), 2 uncovered, 3 first
        // collision, 4 fluid before (pull with bounce-back; covered if solid now)
        const int kind = !act ? 0 : ((wallrow || (solN && (solO || FIRST))) ? 1 : (solO ? 2 : (FIRST ? 3 : 4)));
        float f[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) f[i] = 0.0f;
        if (kind == 2) {
            // uncovered: f = f_eq(rho0, U + Omega x r) with r = x - x_c(t+1) of the
            // body that held it, whose sums get its cube coordinates m
            int m0 = mx, m1 = my, m2 = mz;
            const PartK& Ko = sol_old ? K : s_pk[po];
            if (!sol_old) ploc(po, true, X, Y, Z, m0, m1, m2);
            const float rx = Ko.ro_new[0] + m0, ry = Ko.ro_new[1] + m1, rz = Ko.ro_new[2] + m2;
            const float ux = Ko.U[0] + (Ko.W[1] * rz - Ko.W[2] * ry);
            const float uy = Ko.U[1] + (Ko.W[2] * rx - Ko.W[0] * rz);
            const float uz = Ko.U[2] + (Ko.W[0] * ry - Ko.W[1] * rx);
            const float uu = ux * ux + uy * uy + uz * uz;
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                if (!mine(i)) continue;
                const float cu = cx_of(i) * ux + cy_of(i) * uy + cz_of(i) * uz;
                f[i] = w_of(i) * rho0 * (3.0f * cu + 4.5f * cu * cu - 1.5f * uu);
            }
            if (H == 0) {
                const long long uv[10] = {1, m0, m1, m2, m0 * m0, m0 * m1, m0 * m2, m1 * m1, m1 * m2, m2 * m2};
                for (int e2 = 0; e2 < 10; ++e2) {
                    if (sol_old) rare_add(ACC_UNC + e2, uv[e2]);
                    else padd(po, ACC_UNC + e2, uv[e2]);
                }
            }
        } else if (kind == 3) {
            // first collision: the node's initial distributions, no streaming
#pragma unroll
            for (int i = 0; i < Q; ++i)
                if (mine(i)) f[i] = St::ld1(A + (i * N + own), inv, pol);
        } else if (kind == 4) {
            // fluid at t-1: decide every source first, then issue the loads together
            unsigned bb = 0, wl = 0, pb = 0;        // own, wall and partner bounce-back
            unsigned ro[3][3];                      // the old map around the node, rows (y + a - 1, z + b - 1)
            int zy[3][3];
            const int xs[3] = {wrapd(X - 1, nx), X, wrapd(X + 1, nx)};
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int b = 0; b < 3; ++b) {
                    ro[a][b] = row3(s_old, mx + dsh[0], my + dsh[1] + a - 1, mz + dsh[2] + b - 1);
                    zy[a][b] = (wrapd(Z + b - 1, nz) * ny + wrapd(Y + a - 1, ny)) * nx;
                }
#pragma unroll
            for (int i = 1; i < Q; ++i) {
                if (!mine(i)) continue;
                const int Ys = Y - cy_of(i);
                if (walls && (Ys == 0 || Ys == ny - 1)) wl |= 1u << i;
                else bb |= ((ro[1 - cy_of(i)][1 - cz_of(i)] >> (1 - cx_of(i))) & 1u) << i;
            }
            if (nnb > 0) {
                for (int i = 1; i < Q; ++i) {
                    if (!mine(i) || (((bb | wl) >> i) & 1u)) continue;
                    const int Xs = wrapd(X - cx_of(i), nx), Ys = wrapd(Y - cy_of(i), ny), Zs = wrapd(Z - cz_of(i), nz);
                    for (int j = 0; j < nnb; ++j)
                        if (pbit(j, false, Xs, Ys, Zs)) pb |= 1u << i;
                }
            }
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                if (!mine(i)) continue;
                const bool back = ((bb | wl | pb) >> i) & 1u;
                f[i] = St::ld1(A + (back ? opp_of(i) * N + own : i * N + zy[1 - cy_of(i)][1 - cz_of(i)] + xs[1 - cx_of(i)]), inv, pol);
            }
            // mid-link bounce-back terms: + 6 w_i rho0 (u_b . c_i) (Eq. fb, Eq. ub, Eq. ubsquirmer).  Walls and a passive
            // body's own links without a branch per direction; a squirmer's apart; partners' in one loop over the links,
            // so that code which most nodes skip stays small: with all of it once per direction the warps
            // waited for instructions (an item's nodes 6.3 us after its list, of 23.7 per iteration of a 32^3 box; now 20.1,
            // and 36.1 -> 32.3 for a channel of 128 x 64 x 128 nodes)
            if (walls) {
#pragma unroll
                for (int i = 1; i < Q; ++i) {
                    if (!mine(i) || cy_of(i) == 0) continue;
                    const float* uw = (Y - cy_of(i) == 0) ? K.uw_lo : K.uw_hi;
                    const float ubc = cx_of(i) * uw[0] + cy_of(i) * uw[1] + cz_of(i) * uw[2];
                    f[i] = (wl >> i) & 1u ? __fmaf_rn(6.0f * w_of(i) * rho0, ubc, f[i]) : f[i];
                }
            }
            const bool squirmer = K.squirmer != 0;
            // r_b = x - c_i/2 - x_c(t-1) = ro_old + dsh + m - c_i/2
            const float p0 = K.ro_old[0] + (float)(dsh[0] + mx), p1 = K.ro_old[1] + (float)(dsh[1] + my),
                        p2 = K.ro_old[2] + (float)(dsh[2] + mz);
            if (!squirmer) {
#pragma unroll
                for (int i = 1; i < Q; ++i) {
                    if (!mine(i)) continue;
                    const float px = p0 - 0.5f * cx_of(i), py = p1 - 0.5f * cy_of(i), pz = p2 - 0.5f * cz_of(i);
                    const float ux = K.U[0] + cross_term(K.W[1], pz, K.W[2], py);
                    const float uy = K.U[1] + cross_term(K.W[2], px, K.W[0], pz);
                    const float uz = K.U[2] + cross_term(K.W[0], py, K.W[1], px);
                    const float ubc = cx_of(i) * ux + cy_of(i) * uy + cz_of(i) * uz;
                    f[i] = (bb >> i) & 1u ? __fmaf_rn(6.0f * w_of(i) * rho0, ubc, f[i]) : f[i];
                }
            }
            if (squirmer) {
                // its own links one by one: the slip is long, and a link is taken by few lanes
                const float ex[3] = {K.e_old[0], K.e_old[1], K.e_old[2]};
#pragma unroll
                for (int i = 1; i < Q; ++i) {
                    if (!mine(i) || !((bb >> i) & 1u)) continue;
                    const float px = K.ro_old[0] + (float)(dsh[0] + mx) - 0.5f * cx_of(i);
                    const float py = K.ro_old[1] + (float)(dsh[1] + my) - 0.5f * cy_of(i);
                    const float pz = K.ro_old[2] + (float)(dsh[2] + mz) - 0.5f * cz_of(i);
                    float ux = K.U[0] + (K.W[1] * pz - K.W[2] * py);
                    float uy = K.U[1] + (K.W[2] * px - K.W[0] * pz);
                    float uz = K.U[2] + (K.W[0] * py - K.W[1] * px);
                    float qx, qy, qz;
                    squirmer_slip(ex, K.a, K.eps2, K.B1, K.B2, px, py, pz, qx, qy, qz);
                    ux += qx; uy += qy; uz += qz;
                    const float ubc = cx_of(i) * ux + cy_of(i) * uy + cz_of(i) * uz;
                    f[i] += 6.0f * w_of(i) * rho0 * ubc;
                }
            }
#pragma unroll 1
            for (unsigned m = pb; m != 0; m &= m - 1) {
                const int i = __ffs((int)m) - 1;
                const int cx = c_of(pack_c(0), i), cy = c_of(pack_c(1), i), cz = c_of(pack_c(2), i);
                // a partner's surface: its velocity at r_b = x - c_i/2 - x_c(t) of that body
                const int Xs = wrapd(X - cx, nx), Ys = wrapd(Y - cy, ny), Zs = wrapd(Z - cz, nz);
                int j = 0;
                while (j < nnb - 1 && !pbit(j, false, Xs, Ys, Zs)) ++j;
                const PartK* Kq = &s_pk[j];
                int l0, l1, l2;
                ploc(j, false, X, Y, Z, l0, l1, l2);
                const float px = Kq->ro_old[0] + (float)l0 - 0.5f * cx;
                const float py = Kq->ro_old[1] + (float)l1 - 0.5f * cy;
                const float pz = Kq->ro_old[2] + (float)l2 - 0.5f * cz;
                float ux = Kq->U[0] + cross_term(Kq->W[1], pz, Kq->W[2], py);
                float uy = Kq->U[1] + cross_term(Kq->W[2], px, Kq->W[0], pz);
                float uz = Kq->U[2] + cross_term(Kq->W[0], py, Kq->W[1], px);
                if (Kq->squirmer) {
                    float qx, qy, qz;
                    squirmer_slip(Kq->e_old, Kq->a, Kq->eps2, Kq->B1, Kq->B2, px, py, pz, qx, qy, qz);
                    ux += qx; uy += qy; uz += qz;
                }
                const float ubc = cx * ux + cy * uy + cz * uz;
                const float c6 = 6.0f * w_of(i) * rho0;
#pragma unroll
                for (int k = 1; k < Q; ++k)
                    if (mine(k)) f[k] = k == i ? __fmaf_rn(c6, ubc, f[k]) : f[k];
            }
        }
        // ---- the node's moments: this warp's part and the partner warp's
        float tot[NX];
        {
            float part[NX];
#pragma unroll
            for (int k = 0; k < NX; ++k) part[k] = 0.0f;
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                if (!mine(i)) continue;
                const int cx = cx_of(i), cy = cy_of(i), cz = cz_of(i);
                part[0] += f[i];
                if (cx) part[1] += cx * f[i];
                if (cy) part[2] += cy * f[i];
                if (cz) part[3] += cz * f[i];
                if constexpr (NX > 4) {
                    if (cx) part[4] += f[i];
                    if (cy) part[5] += f[i];
                    if (cz) part[6] += f[i];
                    if (cx * cy) part[7] += (cx * cy) * f[i];
                    if (cx * cz) part[8] += (cx * cz) * f[i];
                    if (cy * cz) part[9] += (cy * cz) * f[i];
                }
            }
#pragma unroll
            for (int k = 0; k < NX; ++k) s_xch[wpair][H][k][lane] = part[k];
            asm volatile("bar.sync %0, %1;" ::"r"(1 + wpair), "r"(64) : "memory");
#pragma unroll
            for (int k = 0; k < NX; ++k) tot[k] = s_xch[wpair][0][k][lane] + s_xch[wpair][1][k][lane];
            asm volatile("bar.sync %0, %1;" ::"r"(1 + wpair), "r"(64) : "memory");
        }
        bool write = kind == 2 || kind == 3 || (kind == 4 && !solN);
        if (kind == 4 && solN && H == 0) {
            // covered: mass and momentum go to the next solve of the body that
            // holds the node now
            const long long Jx = fixq(tot[1]), Jy = fixq(tot[2]), Jz = fixq(tot[3]);
            int m0 = mx, m1 = my, m2 = mz;
            if (!sol_new) ploc(pn, true, X, Y, Z, m0, m1, m2);
            const long long cv[8] = {1, fixq(tot[0]), Jx, Jy, Jz, m1 * Jz - m2 * Jy, m2 * Jx - m0 * Jz,
                                     m0 * Jy - m1 * Jx};
            for (int e2 = 0; e2 < 8; ++e2) {
                if (sol_new) rare_add(ACC_COV + e2, cv[e2]);
                else padd(pn, ACC_COV + e2, cv[e2]);
            }
        }
        if (write) {
            collide_half<St::GHOST, H>(f, tot, K.omega, rho0, dyn.g[0], dyn.g[1], dyn.g[2], dyn.eps);
#pragma unroll
            for (int i = 0; i < Q; ++i)
                if (mine(i)) St::st1(D + (i * N + own), f[i], scale, pol);
            // momentum-exchange sums of the new links (x, b), with f*(t)
            unsigned rn[3][3], lk = 0u;             // the new map around the node; the links into it
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int b = 0; b < 3; ++b) rn[a][b] = row3(s_new, mx, my + a - 1, mz + b - 1);
#pragma unroll
            for (int b = 1; b < Q; ++b)
                if (mine(b)) lk |= ((rn[1 + cy_of(b)][1 + cz_of(b)] >> (1 + cx_of(b))) & 1u) << b;
            if (lk) {
                long long fx = 0, fy = 0, fz = 0;
#pragma unroll
                for (int b = 1; b < Q; ++b) {
                    if (!mine(b)) continue;
                    const long long d = fixq((lk >> b) & 1u ? f[b] : 0.0f);
                    if (cx_of(b) == 1) fx += d; else if (cx_of(b) == -1) fx -= d;
                    if (cy_of(b) == 1) fy += d; else if (cy_of(b) == -1) fy -= d;
                    if (cz_of(b) == 1) fz += d; else if (cz_of(b) == -1) fz -= d;
                }
                aF[0] += fx; aF[1] += fy; aF[2] += fz;
                aT[0] += my * fz - mz * fy;
                aT[1] += mz * fx - mx * fz;
                aT[2] += mx * fy - my * fx;
            }
            // links to partners' surfaces: their sums, about their cube origins
            if (nnb > 0) {
                for (int b = 1; b < Q; ++b) {
                    if (!mine(b)) continue;
                    const int Xb = wrapd(X + cx_of(b), nx), Yb = wrapd(Y + cy_of(b), ny), Zb = wrapd(Z + cz_of(b), nz);
                    for (int j = 0; j < nnb; ++j) {
                        if (!pbit(j, true, Xb, Yb, Zb)) continue;
                        int l0, l1, l2;
                        ploc(j, true, X, Y, Z, l0, l1, l2);
                        const long long d = fixq(f[b]);
                        const long long gx_ = cx_of(b) * d, gy_ = cy_of(b) * d, gz_ = cz_of(b) * d;
                        padd(j, ACC_F, gx_); padd(j, ACC_F + 1, gy_); padd(j, ACC_F + 2, gz_);
                        padd(j, ACC_T, l1 * gz_ - l2 * gy_);
                        padd(j, ACC_T + 1, l2 * gx_ - l0 * gz_);
                        padd(j, ACC_T + 2, l0 * gy_ - l1 * gx_);
                    }
                }
            }
        } else if (act && solN && !wallrow) {
            // solid now: zero it (never read as a source)
#pragma unroll
            for (int i = 0; i < Q; ++i)
                if (mine(i)) St::st1(D + (i * N + own), 0.0f, scale, pol);
        }
    };
    for (int rnd = 0; rnd < rounds; ++rnd) {
        if (warp & 1) node_round(std::integral_constant<int, 1>{}, rnd);
        else node_round(std::integral_constant<int, 0>{}, rnd);
    }

    // ---- per-warp link sums into shared memory, then one atomic per nonzero sum
    if (__any_sync(0xffffffffu, (aF[0] | aF[1] | aF[2] | aT[0] | aT[1] | aT[2]) != 0)) {
#pragma unroll
        for (int k = 0; k < 3; ++k) { aF[k] = warp_sum(aF[k]); aT[k] = warp_sum(aT[k]); }
    }
    if (lane == 0) {
#pragma unroll
        for (int k = 0; k < 3; ++k) { s_red[warp][ACC_F + k] = aF[k]; s_red[warp][ACC_T + k] = aT[k]; }
    }
    __syncthreads();
    if (tid < NACC) {
        long long v = 0;
        if (tid < ACC_COV) {
#pragma unroll
            for (int w = 0; w < NW; ++w) v += s_red[w][tid];
        } else {
            v = s_rare[tid - ACC_COV];
        }
        if (v != 0) atomicAdd(reinterpret_cast<unsigned long long*>(P.acc + (size_t)p * NACC + tid), static_cast<unsigned long long>(v));
    }
}

}  // namespace lbsph
