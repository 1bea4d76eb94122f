// Field read-back kernel (lb_get_fields): the pre-collision state of every
// node of one box at the start of iteration t, i.e. the second half of
// iteration t-1 of the paper's Appendix (step 2 streaming, step 6 bounce-back
// with U(t), Omega(t), the remap of step 8) without the collision, with
// density and velocity moments.  Every decision is taken per node from the
// occupancy maps, in a layout independent of the bulk + boundary kernels that
// advance the simulation, so the read-back also cross-checks them.
//
// Thread mapping: one thread per 4 consecutive x nodes ("quad"), 256 threads
// per block, blocks in x-fastest order over the box.  Each direction is read
// with one 16-byte load of the source row; the +-1 shift in x comes from the
// neighbouring lane by a warp shuffle (a scalar load at warp and row ends,
// which also wraps x periodically).  Threads whose nodes (grown by one) touch
// a particle's bounding cube or a wall test them against the occupancy
// bitmaps (old map for the streaming sources, new map for the node itself).
//
// Away from the particles the kernel is bound by the populations it reads; near
// them by the latency of what each thread looks up, so a tile keeps only the indices of
// the particles it meets (their state is read through L1 where it is needed), a
// neighbourhood row is one load and two shifts, the box's uniform force is summed by one
// warp while the others load, and the owner field reads no populations.  Measured, FP32:
// u or rho of a 64^3 box with one particle 48.6 -> 18.4 us, of 128 x 64 x 128 nodes between
// walls 52 -> 39, of 128^3 nodes with 16 particles 321 -> 90 (13, 27 and 57 without the
// bounce-back); the owner field of 128^3 nodes 118 -> 11.
#include "lattice_common.cuh"

namespace lbsph {

// Is lattice node (X, Y, Z) (wrapped into the box) a solid node of one of the
// tile's particles?  old selects map t-1 (streaming sources) or map t.
__device__ __forceinline__ const PartK* lookup(const PartK* pk, const int* cs, int nc, bool old, int X, int Y, int Z, int nx,
                                               int ny, int nz, int& mx, int& my, int& mz)
{
    for (int c = 0; c < nc; ++c) {
        const PartK& K = pk[cs[c]];
        const int* ow = old ? K.ow_old : K.ow_new;
        const int S = K.S;
        const int ax = wrapd(X - ow[0], nx);
        if (ax >= S) continue;
        const int ay = wrapd(Y - ow[1], ny);
        if (ay >= S) continue;
        const int az = wrapd(Z - ow[2], nz);
        if (az >= S) continue;
        const uint64_t* rows = old ? K.rows_old : K.rows_new;
        if ((rows[az * S + ay] >> ax) & 1ull) {
            mx = ax; my = ay; mz = az;
            return &K;
        }
    }
    return nullptr;
}

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

template <class St, int WHAT>
__global__ void __launch_bounds__(KBLOCK, 1) fields_kernel(const KParams P)
{
    using T = typename St::T;
    __shared__ int s_c[MAXC];
    __shared__ int s_nc;
    __shared__ float s_g[3];

    // ---- box of this block
    const BoxDev& B = P.boxes[P.only_box];
    const int nx = B.nx, ny = B.ny, nz = B.nz, nxq = B.nxq;
    const int N = (int)B.N;                     // 19 N < 2^31
    // the blocks walk the box's tiles, so that the box force is summed once per block
    for (int tile = blockIdx.x; tile < B.nblocks; tile += gridDim.x) {
    if (tile != (int)blockIdx.x) __syncthreads();        // the last tile's list has been read
    const int q0 = tile * KBLOCK;
    const int qlast = min(q0 + KBLOCK, (int)B.nq) - 1;

    // ---- this thread's quad
    int q = q0 + (int)threadIdx.x;
    const bool valid = q < (int)B.nq;
    if (!valid) q = (int)B.nq - 1;
    const int row = div_magic(q, B.dq_m, B.dq_s);
    const int xq = q - row * nxq;
    const int z = div_magic(row, B.dy_m, B.dy_s);
    const int y = row - z * ny;
    const int lane = threadIdx.x & 31;
    const T* A = reinterpret_cast<const T*>(P.src) + B.off;
    const float inv = B.inv_scale;
    const unsigned long long pol = l2_evict_normal();
    const int own = row * nx + 4 * xq;
    const bool first = P.nopull != 0;

    // ---- pull (stream): v[i] = f*_i(x - c_i) for the 4 nodes
    float4 v[Q];
    if (WHAT != FK_SOLID) {
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
        if (first) {
            // before the first collision: the initial distributions in place
#pragma unroll
            for (int i = 0; i < Q; ++i) v[i] = St::ld4(A + (i * N + own), inv, pol);
        } else {
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                const T* rp = A + (i * N + rofs[1 - cy_of(i)][1 - cz_of(i)]);
                float4 t = St::ld4(rp + 4 * xq, inv, pol);
                if (cx_of(i) == 1) {           // source x - 1
                    float l = __shfl_up_sync(0xffffffffu, t.w, 1);
                    if (left_ld) l = St::ld1(rp + (xq == 0 ? nx - 1 : 4 * xq - 1), inv, pol);
                    t = make_float4(l, t.x, t.y, t.z);
                } else if (cx_of(i) == -1) {   // source x + 1
                    float r = __shfl_down_sync(0xffffffffu, t.x, 1);
                    if (right_ld) r = St::ld1(rp + (xq == nxq - 1 ? 0 : 4 * xq + 4), inv, pol);
                    t = make_float4(t.y, t.z, t.w, r);
                }
                v[i] = t;
            }
        }
    }

    // ---- particles near the tile (first warp), box force (second warp)
    if (threadIdx.x < 32) {
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
            const unsigned m = __ballot_sync(0xffffffffu, hit);
            const int at = nc + __popc(m & ((1u << lane) - 1u));
            if (hit && at < MAXC) s_c[at] = B.pbeg + base + lane;
            nc += __popc(m);
        }
        if (lane == 0) {
            if (nc > MAXC) atomicOr(P.status, ST_CAPACITY);
            s_nc = nc < MAXC ? nc : MAXC;
        }
    } else if (WHAT == FK_MOMENTS && threadIdx.x < 64 && tile == (int)blockIdx.x) {
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
            s_g[0] = (float)g[0]; s_g[1] = (float)g[1]; s_g[2] = (float)g[2];
        }
    }
    __syncthreads();
    const int nc = s_nc;

    // ---- walls: link bounce-back (Eq. fb with u_b = u_w) of the rows next to them
    const bool wallrow = B.walls && (y == 0 || y == ny - 1);
    const float rho0 = B.rho0f;
    const int wall_cy = !B.walls || first ? 0 : (y == 1 ? 1 : (y == ny - 2 ? -1 : 0));     // directions from a wall
    if (WHAT != FK_SOLID && wall_cy != 0) {
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
    // ---- particles whose cubes the thread's nodes (grown by one) touch: the neighbourhood's occupancy as 6-bit
    // windows of the 9 rows (y + dy, z + dz), and bounce-back (Eq. fb, Eq. ub) where the source was inside
    unsigned so = 0u, sn = 0u;                  // this row's windows of all particles, old and new map
    for (int c = 0; c < nc; ++c) {
        const PartK& C = P.pk[s_c[c]];
        const int S = C.S;
        const int on[3] = {C.ow_new[0], C.ow_new[1], C.ow_new[2]}, oo[3] = {C.ow_old[0], C.ow_old[1], C.ow_old[2]};
        if (hits(y, y, on[1], S, ny) && hits(z, z, on[2], S, nz) && hits(4 * xq - 1, 4 * xq + 4, on[0], S, nx))
            sn |= window6(C.rows_new[wrapd(z - on[2], nz) * S + wrapd(y - on[1], ny)], S,
                          wrapd(wrapd(4 * xq - 1, nx) - on[0], nx), nx);
        if (WHAT == FK_SOLID || first || wallrow) continue;
        if (!(hits(y - 1, y + 1, oo[1], S, ny) && hits(z - 1, z + 1, oo[2], S, nz) && hits(4 * xq - 1, 4 * xq + 4, oo[0], S, nx))) continue;
        const uint64_t* rows = C.rows_old;
        const int d = wrapd(wrapd(4 * xq - 1, nx) - oo[0], nx);
        int my[3], mz[3];                       // cube rows of y - 1, y, y + 1 and z - 1, z, z + 1
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            my[a] = wrapd(wrapd(y + a - 1, ny) - oo[1], ny);
            mz[a] = wrapd(wrapd(z + a - 1, nz) - oo[2], nz);
        }
        unsigned w[3][3], any = 0u;
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                w[a][b] = 0u;
                if (my[a] < S && mz[b] < S) w[a][b] = window6(rows[mz[b] * S + my[a]], S, d, nx);
                any |= w[a][b];
            }
        so |= w[1][1];
        if (any == 0u) continue;
        const float ro[3] = {C.ro_old[0], C.ro_old[1], C.ro_old[2]}, U[3] = {C.U[0], C.U[1], C.U[2]},
                    W[3] = {C.W[0], C.W[1], C.W[2]};
        const int squirmer = C.squirmer;
        // six directions at a time, so that their loads (the nodes' own populations of the opposite direction) overlap
#pragma unroll
        for (int i0 = 1; i0 < Q; i0 += 6) {
            float4 o[6];
            unsigned lm[6];
#pragma unroll
            for (int e = 0; e < 6; ++e) {
                const int i = i0 + e;
                lm[e] = (w[1 - cy_of(i)][1 - cz_of(i)] >> (1 - cx_of(i))) & 0xfu;
                if (cy_of(i) != 0 && cy_of(i) == wall_cy) lm[e] = 0u;
                if (lm[e]) o[e] = St::ld4(A + (opp_of(i) * N + own), inv, pol);
            }
#pragma unroll
            for (int e = 0; e < 6; ++e) {
                const int i = i0 + e;
                if (lm[e] == 0u) continue;
                const float ry = ro[1] + my[1 - cy_of(i)] + 0.5f * cy_of(i);
                const float rz = ro[2] + mz[1 - cz_of(i)] + 0.5f * cz_of(i);
#pragma unroll 1
                for (int k = 0; k < 4; ++k) {
                    if (!((lm[e] >> k) & 1u)) continue;
                    int sx = d + k + 1 - cx_of(i);
                    if (sx >= nx) sx -= nx;
                    const float rx = ro[0] + sx + 0.5f * cx_of(i);
                    float ux = U[0] + (W[1] * rz - W[2] * ry);
                    float uy = U[1] + (W[2] * rx - W[0] * rz);
                    float uz = U[2] + (W[0] * ry - W[1] * rx);
                    if (squirmer) {
                        float qx, qy, qz;
                        squirmer_slip(C.e_old, C.a, C.eps2, C.B1, C.B2, rx, ry, rz, qx, qy, qz);
                        ux += qx; uy += qy; uz += qz;
                    }
                    const float ubc = cx_of(i) * ux + cy_of(i) * uy + cz_of(i) * uz;
                    const float fb = comp(o[e], k) + 6.0f * w_of(i) * rho0 * ubc;
                    v[i].x = k == 0 ? fb : v[i].x;
                    v[i].y = k == 1 ? fb : v[i].y;
                    v[i].z = k == 2 ? fb : v[i].z;
                    v[i].w = k == 3 ? fb : v[i].w;
                }
            }
        }
    }
    if (WHAT == FK_SOLID) {
        int solid_out[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            solid_out[k] = wallrow ? -1 : 0;
            if (wallrow || !((sn >> (k + 1)) & 1u)) continue;
            int mx, my, mz;
            const PartK* c = lookup(P.pk, s_c, nc, false, 4 * xq + k, y, z, nx, ny, nz, mx, my, mz);
            if (c) solid_out[k] = (int)(c - P.pk) - B.pbeg + 1;
        }
        if (valid) *reinterpret_cast<int4*>(P.out_solid + own) = make_int4(solid_out[0], solid_out[1], solid_out[2], solid_out[3]);
        continue;
    }
    const float gx = s_g[0], gy = s_g[1], gz = s_g[2];
    float rho_out[4], u_out[4][3];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int X = 4 * xq + k;
        bool skip = !valid;
        rho_out[k] = 0.f; u_out[k][0] = u_out[k][1] = u_out[k][2] = 0.f;
        float f[Q];
        const bool sol_old = !wallrow && ((so >> (k + 1)) & 1u);
        const bool sol_new = !wallrow && ((sn >> (k + 1)) & 1u);
        int mx, my, mz;
        if (wallrow || sol_new) {
            // a wall, solid before and after, or covered: its mass and momentum go to the particle (remap, step 8)
            skip = true;
        } else if (sol_old) {
            // uncovered: f = f_eq(rho0, U + Omega x r) (remap, step 8)
            const PartK* c0 = lookup(P.pk, s_c, nc, true, X, y, z, nx, ny, nz, mx, my, mz);
            const PartK& c = c0 ? *c0 : P.pk[s_c[0]];
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
        } else {
            // fluid at t-1: pulled populations, bounced back where the source was solid
#pragma unroll
            for (int i = 0; i < Q; ++i) f[i] = comp(v[i], k);
        }
        if (skip) {
#pragma unroll
            for (int i = 0; i < Q; ++i) set_comp(v[i], k, 0.0f);
            continue;
        }
        if (WHAT == FK_MOMENTS) {
            float drho = 0.f;
#pragma unroll
            for (int i = 0; i < Q; ++i) drho += f[i];
            const float jx = (f[1] - f[2]) + (f[7] - f[8]) + (f[9] - f[10]) + (f[11] - f[12]) + (f[13] - f[14]);
            const float jy = (f[3] - f[4]) + (f[7] - f[8]) - (f[9] - f[10]) + (f[15] - f[16]) + (f[17] - f[18]);
            const float jz = (f[5] - f[6]) + (f[11] - f[12]) - (f[13] - f[14]) + (f[15] - f[16]) - (f[17] - f[18]);
            const float ir = 1.0f / (rho0 + drho);
            rho_out[k] = drho;
            u_out[k][0] = (jx + 0.5f * gx) * ir;
            u_out[k][1] = (jy + 0.5f * gy) * ir;
            u_out[k][2] = (jz + 0.5f * gz) * ir;
        } else {
#pragma unroll
            for (int i = 0; i < Q; ++i) set_comp(v[i], k, P.out_dev ? f[i] : f[i] + w_of(i) * rho0);
        }
    }

    if (!valid) continue;
    if (WHAT == FK_F) {
#pragma unroll
        for (int i = 0; i < Q; ++i) *reinterpret_cast<float4*>(P.out_f + (i * N + own)) = v[i];
    } else {
        if (P.out_rho) *reinterpret_cast<float4*>(P.out_rho + own) = make_float4(rho_out[0], rho_out[1], rho_out[2], rho_out[3]);
        if (P.out_u) {
#pragma unroll
            for (int a = 0; a < 3; ++a)
                *reinterpret_cast<float4*>(P.out_u + (a * N + own)) = make_float4(u_out[0][a], u_out[1][a], u_out[2][a], u_out[3][a]);
        }
    }
    }
}

// ---------------------------------------------------------------------------
// Field read-back: pre-collision populations at the start of iteration t
// (streaming, bounce-back and remap fix-ups of t-1 without a collision), every
// tile tested against the particles' occupancy maps.
template <class St>
static cudaError_t launch_mode(const KParams& p, int blocks, cudaStream_t s)
{
    int dev = 0, nsm = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    const int g = blocks < nsm ? blocks : nsm;          // one block of this many registers per SM
    if (p.out_f) fields_kernel<St, FK_F><<<g, KBLOCK, 0, s>>>(p);
    else if (p.out_solid) fields_kernel<St, FK_SOLID><<<blocks, KBLOCK, 0, s>>>(p);
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
