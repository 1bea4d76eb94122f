// Resistance-tensor surrogate: tensor-core GEMM (tcgen05), the network's
// loss / backward / Adam kernels and small SPD solves, behind
// include/lbsurrogate.h.
//
// GEMM (C = A B^T, BF16 operands, FP32 accumulation): one CTA of one
// warpgroup (128 threads) per 128 x N tile (N <= 256).  For each K chunk of 64
// the threads stage A (128 x 64) and B (N x 64) into shared memory in the
// canonical no-swizzle K-major layout of 8-row x 16-byte core matrices (core
// (g, c) of rows 8g.. and K columns 8c.. at byte (8g + c) * 128, so adjacent
// core matrices are 128 bytes apart along K and 1024 bytes apart along the
// rows); one elected thread issues four tcgen05.mma (M = 128, K = 16 each)
// accumulating in tensor memory and commits them to an mbarrier that every
// thread waits on (bounded).  Two stages: while the products of chunk c run,
// the threads stage chunk c + 1 into the other stage (whose products, those of
// chunk c - 1, were waited for).  The staging loads are coalesced for either
// operand layout: 16-byte loads of 8 consecutive K (K-major operands) or of 8
// consecutive rows (transposed operands) where strides and alignment allow,
// else one element per thread with consecutive threads on the contiguous
// index.  The
// epilogue: warp w reads TMEM lanes 32w..32w+31 (one output row per lane) with
// tcgen05.ld, adds the bias, applies ReLU and writes FP32 and/or BF16.
// This form serves any strides (lb_gemm_bf16); the network has kernels of its own, see
// net_kernel and grad_kernel below.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "../../include/lbsurrogate.h"

namespace lbsur {

constexpr int GM = 128;                 // tile rows: one TMEM lane per row
constexpr int GN = 256;                 // widest tile (one MMA, N <= 256)
constexpr int GK = 64;                  // K chunk per staging round
constexpr int GTHREADS = 128;           // one warpgroup
constexpr int SMEM_A = GM * GK * 2;     // 16 KiB
constexpr int SMEM_B = GN * GK * 2;     // 32 KiB
constexpr int GEMM_STAGE = SMEM_A + SMEM_B;
constexpr int GEMM_SMEM = 2 * GEMM_STAGE; // two stages, 96 KiB
constexpr long long SPIN_LIMIT = 1ll << 24;

struct GemmArgs {
    const __nv_bfloat16* A;
    long long a_sm, a_sk;
    const __nv_bfloat16* B;
    long long b_sn, b_sk;
    int M, N, K;
    const float* bias;
    int relu;
    float* C32;
    __nv_bfloat16* C16;
    long long c_sm, c_sn;
};

__device__ unsigned g_gemm_status;      // bit 0: a completion wait gave up

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor: no swizzle, K-major, byte offsets between
// core matrices along K (lbo) and along the rows (sbo); bits 46-48 = 0b001
__device__ __forceinline__ unsigned long long sdesc(unsigned addr, unsigned lbo, unsigned sbo)
{
    return (unsigned long long)((addr & 0x3FFFFu) >> 4) | ((unsigned long long)((lbo >> 4) & 0x3FFFu) << 16) |
           ((unsigned long long)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// instruction descriptor of kind::f16: D FP32, A and B BF16, both K-major
__host__ __device__ constexpr unsigned idesc_bf16(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(N >> 3) << 17) | ((unsigned)(M >> 4) << 24);
}

__device__ __forceinline__ bool mbar_wait(unsigned long long* b, unsigned parity)
{
    for (long long n = 0; n < SPIN_LIMIT; ++n) {
        unsigned ok;
        asm volatile("{\n\t.reg .pred p;\n\t"
                     "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok) : "r"(smem_u32(b)), "r"(parity) : "memory");
        if (ok) return true;
    }
    return false;
}

// byte offset of element (r, k) of a staged 64-wide K chunk
__device__ __forceinline__ int core_off(int r, int k) { return (((r >> 3) * 8 + (k >> 3)) << 7) + ((r & 7) << 4) + ((k & 7) << 1); }

// Rows [r0, r0 + rows) x K columns [k0, k0 + 64) of X (element (r, k) at
// X[r s_r + k s_k]) into a stage in the core-matrix layout; rows at or beyond
// nrow and columns at or beyond K are zero.  rows is a multiple of 8, r0 and k0
// of 64.
__device__ __forceinline__ void stage_operand(const __nv_bfloat16* X, long long s_r, long long s_k, int r0, int rows,
                                              int nrow, int k0, int K, unsigned char* dst, int tid)
{
    const __nv_bfloat16 zero = __float2bfloat16(0.0f);
    const bool al = (reinterpret_cast<uintptr_t>(X) & 15u) == 0;
    if (s_k == 1 && al && (s_r & 7) == 0) {
        // K-major: 8 consecutive K per thread, one 16-byte load and store
        for (int idx = tid; idx < rows * (GK / 8); idx += GTHREADS) {
            const int r = idx / (GK / 8), kc = (idx % (GK / 8)) * 8;
            const int m = r0 + r, kk = k0 + kc;
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (m < nrow) {
                if (kk + 8 <= K) {
                    v = __ldg(reinterpret_cast<const uint4*>(X + m * s_r + kk));
                } else {
                    unsigned w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (kk + j < K)
                            w[j >> 1] |= (unsigned)__bfloat16_as_ushort(X[m * s_r + kk + j]) << (16 * (j & 1));
                    v = make_uint4(w[0], w[1], w[2], w[3]);
                }
            }
            *reinterpret_cast<uint4*>(dst + core_off(r, kc)) = v;
        }
    } else if (s_r == 1 && al && (s_k & 7) == 0) {
        // transposed: 8 consecutive rows per thread, one 16-byte load, eight
        // 2-byte stores (the rows of a core matrix are 16 bytes apart)
        for (int idx = tid; idx < (rows / 8) * GK; idx += GTHREADS) {
            const int rc = (idx % (rows / 8)) * 8, k = idx / (rows / 8);
            const int m = r0 + rc, kk = k0 + k;
            unsigned w[4] = {0u, 0u, 0u, 0u};
            if (kk < K && m + 8 <= nrow) {
                const uint4 v = __ldg(reinterpret_cast<const uint4*>(X + m + kk * s_k));
                w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (kk < K && m + j < nrow)
                        w[j >> 1] |= (unsigned)__bfloat16_as_ushort(X[m + j + kk * s_k]) << (16 * (j & 1));
            }
#pragma unroll
            for (int j = 0; j < 8; ++j)
                *reinterpret_cast<unsigned short*>(dst + core_off(rc + j, k)) = (unsigned short)(w[j >> 1] >> (16 * (j & 1)));
        }
    } else if (s_r == 1) {
        // transposed, unaligned: consecutive threads on consecutive rows
        for (int idx = tid; idx < rows * GK; idx += GTHREADS) {
            const int r = idx % rows, k = idx / rows;
            const int m = r0 + r, kk = k0 + k;
            *reinterpret_cast<__nv_bfloat16*>(dst + core_off(r, k)) = (m < nrow && kk < K) ? X[m + kk * s_k] : zero;
        }
    } else {
        for (int idx = tid; idx < rows * GK; idx += GTHREADS) {
            const int r = idx / GK, k = idx % GK;
            const int m = r0 + r, kk = k0 + k;
            *reinterpret_cast<__nv_bfloat16*>(dst + core_off(r, k)) =
                (m < nrow && kk < K) ? X[m * s_r + kk * s_k] : zero;
        }
    }
}

__global__ void __launch_bounds__(GTHREADS) gemm_kernel(const GemmArgs g)
{
    extern __shared__ __align__(128) unsigned char sm[];
    __shared__ unsigned long long bar;
    __shared__ unsigned s_tmem;
    // stage b: A at sm + b GEMM_STAGE, B SMEM_A after it
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int m0 = blockIdx.x * GM, n0 = blockIdx.y * GN;
    const int nrem = g.N - n0;
    const int nt = ((nrem < GN ? nrem : GN) + 15) & ~15;      // MMA N: multiple of 16
    const unsigned ncols = nt <= 32 ? 32u : (nt <= 64 ? 64u : (nt <= 128 ? 128u : 256u));
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(ncols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&bar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const unsigned tmem = s_tmem;
    const unsigned idesc = idesc_bf16(GM, nt);
    unsigned phase = 0;
    bool ok = true;
    const int nchunk = (g.K + GK - 1) / GK;
    stage_operand(g.A, g.a_sm, g.a_sk, m0, GM, g.M, 0, g.K, sm, tid);
    stage_operand(g.B, g.b_sn, g.b_sk, n0, nt, g.N, 0, g.K, sm + SMEM_A, tid);
    // generic-proxy writes of the stage before the tensor core reads them
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    for (int c = 0; c < nchunk; ++c) {
        unsigned char* sa = sm + (c & 1) * GEMM_STAGE;
        unsigned char* sb = sa + SMEM_A;
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
            for (int kk = 0; kk < GK / 16; ++kk) {
                const unsigned long long ad = sdesc(smem_u32(sa) + kk * 256u, 128u, 1024u);
                const unsigned long long bd = sdesc(smem_u32(sb) + kk * 256u, 128u, 1024u);
                const unsigned acc = (c > 0 || kk > 0) ? 1u : 0u;
                asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                             "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
                             "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
                             : "memory");
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             smem_u32(&bar))
                         : "memory");
        }
        if (c + 1 < nchunk) {
            // the next chunk into the other stage while these products run
            unsigned char* na = sm + ((c + 1) & 1) * GEMM_STAGE;
            stage_operand(g.A, g.a_sm, g.a_sk, m0, GM, g.M, (c + 1) * GK, g.K, na, tid);
            stage_operand(g.B, g.b_sn, g.b_sk, n0, nt, g.N, (c + 1) * GK, g.K, na + SMEM_A, tid);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        }
        const bool got = mbar_wait(&bar, phase);
        phase ^= 1u;
        if (__syncthreads_or(!got)) {
            ok = false;
            break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    }
    if (!ok) {
        // give the issued products a second bounded wait before freeing TMEM
        if (tid == 0) atomicOr(&g_gemm_status, 1u);
        (void)mbar_wait(&bar, phase ^ 1u);
    } else {
        const int m = m0 + warp * 32 + lane;
        for (int c0 = 0; c0 < nt; c0 += 16) {
            unsigned r[16];
            const unsigned ta = tmem + ((unsigned)(warp * 32) << 16) + (unsigned)c0;
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                         : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
                           "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
                           "=r"(r[14]), "=r"(r[15])
                         : "r"(ta));
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            if (m < g.M) {
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const int n = n0 + c0 + j;
                    if (n >= g.N) continue;
                    float v = __uint_as_float(r[j]);
                    if (g.bias) v += g.bias[n];
                    if (g.relu) v = fmaxf(v, 0.0f);
                    const long long o = m * g.c_sm + n * g.c_sn;
                    if (g.C32) g.C32[o] = v;
                    if (g.C16) g.C16[o] = __float2bfloat16(v);
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
}

cudaError_t launch_gemm(const GemmArgs& g, cudaStream_t s)
{
    // the opt-in to 96 KiB of dynamic shared memory is per device: set it on
    // every launch (a cheap call) rather than once per process
    const cudaError_t e = cudaFuncSetAttribute(gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, GEMM_SMEM);
    if (e != cudaSuccess) return e;
    const dim3 grid((g.M + GM - 1) / GM, (g.N + GN - 1) / GN);
    gemm_kernel<<<grid, GTHREADS, GEMM_SMEM, s>>>(g);
    return cudaGetLastError();
}

}  // namespace lbsur

using namespace lbsur;

extern "C" lb_status lb_gemm_bf16(const uint16_t* A, int64_t a_sm, int64_t a_sk, const uint16_t* B, int64_t b_sn,
                                  int64_t b_sk, int32_t M, int32_t N, int32_t K, const float* bias, int32_t relu,
                                  float* C32, uint16_t* C16, int64_t c_sm, int64_t c_sn, void* stream)
{
    if (!A || !B || M < 1 || N < 1 || K < 1 || (!C32 && !C16)) return LB_EINVAL;
    GemmArgs g{};
    g.A = reinterpret_cast<const __nv_bfloat16*>(A);
    g.a_sm = a_sm; g.a_sk = a_sk;
    g.B = reinterpret_cast<const __nv_bfloat16*>(B);
    g.b_sn = b_sn; g.b_sk = b_sk;
    g.M = M; g.N = N; g.K = K;
    g.bias = bias; g.relu = relu;
    g.C32 = C32; g.C16 = reinterpret_cast<__nv_bfloat16*>(C16);
    g.c_sm = c_sm; g.c_sn = c_sn;
    return launch_gemm(g, static_cast<cudaStream_t>(stream)) == cudaSuccess ? LB_OK : LB_ECUDA;
}

extern "C" lb_status lb_gemm_status(void)
{
    if (cudaDeviceSynchronize() != cudaSuccess) return LB_ECUDA;
    unsigned v = 0, z = 0;
    if (cudaMemcpyFromSymbol(&v, g_gemm_status, sizeof(v)) != cudaSuccess) return LB_ECUDA;
    if (v && cudaMemcpyToSymbol(g_gemm_status, &z, sizeof(z)) != cudaSuccess) return LB_ECUDA;
    return v ? LB_ETIMEOUT : LB_OK;
}

// ---------------------------------------------------------------------------
// The network: parameters, activations and its two kernels.
namespace lbsur {

constexpr int NIN = LB_MLP_IN, NINP = LB_MLP_IN_PAD, NH = LB_MLP_HID, NOUT = LB_MLP_OUT, NOUTP = LB_MLP_OUT_PAD;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + NH * NINP, OFF_W2 = OFF_B1 + NH, OFF_B2 = OFF_W2 + NH * NH,
              OFF_W3 = OFF_B2 + NH, OFF_B3 = OFF_W3 + NOUTP * NH, NPARAM = OFF_B3 + NOUTP;
static_assert(NPARAM == LB_MLP_NPARAM, "parameter layout");

// A BF16 matrix X(r, k) kept as 8 x 8 core matrices (8 rows of 16 bytes), the
// cores of one column group k / 8 together: element (r, k) at byte
// (k / 8) * cs + (r / 8) * 128 + (r % 8) * 16 + (k % 8) * 2.  The tensor core reads
// the same bytes as a K-major operand over k (row groups 128 bytes apart, K groups
// cs apart) and as an MN-major operand over r (groups of k cs apart, K groups of 8
// rows 128 apart), so one copy of the weights serves the forward and the backward
// products and one copy of the activations serves the products over the samples;
// nothing is transposed.  A row group times one column group is 128 contiguous
// bytes, so 8 threads holding 8 consecutive rows store them without conflicts.
__host__ __device__ constexpr int core_at(int cs, int r, int k) { return (k >> 3) * cs + (r >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2; }

// the weights' BF16 copy: W1 (256 x 16), W2 (256 x 256), W3 (32 x 256), as above
constexpr int CS_W12 = NH / 8 * 128, CS_W3 = NOUTP / 8 * 128;
constexpr int PK_W1 = 0, PK_W2 = PK_W1 + NH * NINP * 2, PK_W3 = PK_W2 + NH * NH * 2, PK_BYTES = PK_W3 + NOUTP * NH * 2;

// activations and their gradients in global memory, samples as rows: `cs` bytes
// per group of 8 features, 128-sample tiles of 16 row groups (2 KiB) within it
struct Acts {
    unsigned char *X, *H1, *H2, *dY, *dH2, *dH1;
    long long cs;
    float* loss_part;                   // [tiles]
    float* d32;                         // up to SPLIT_MIN tiles: FP32 dH1, dH2, dY, [2 * 256 + 32][ns] by column
    float* b_part;                      // more tiles: their column sums, [4 tiles][2 * 256 + 32], per 32 samples
    int ns;                             // samples a column of d32 holds
    unsigned* count;                    // tiles done (zero between launches)
};
constexpr int TILE = 128;               // samples per tile: one TMEM lane each
constexpr int NSUM = 2 * NH + NOUTP;
constexpr int SPLIT_MIN = 8;            // tiles up to which every sum over the samples runs in their order

__global__ void pack_kernel(const float* p, unsigned char* w)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    int base, cs, r, k;
    if (i < NH * NINP) { base = PK_W1; cs = CS_W12; r = i / NINP; k = i % NINP; }
    else if (i >= OFF_W2 && i < OFF_W2 + NH * NH) { base = PK_W2; cs = CS_W12; r = (i - OFF_W2) / NH; k = (i - OFF_W2) % NH; }
    else if (i >= OFF_W3 && i < OFF_W3 + NOUTP * NH) { base = PK_W3; cs = CS_W3; r = (i - OFF_W3) / NH; k = (i - OFF_W3) % NH; }
    else return;
    *reinterpret_cast<__nv_bfloat16*>(w + base + core_at(cs, r, k)) = __float2bfloat16(p[i]);
}

// lower-triangular index t of (i, j), j <= i: t = i (i + 1) / 2 + j
__host__ __device__ constexpr int tri(int i, int j) { return i * (i + 1) / 2 + j; }

__device__ __forceinline__ float softplus(float y) { return y > 20.0f ? y : log1pf(expf(y)); }
__device__ __forceinline__ float sigmoid(float y) { return 1.0f / (1.0f + expf(-y)); }

// ---- PTX helpers
// programmatic dependent launch: wait for the kernels before this one; let the next one start its prologue.
// A kernel launched like that may be running while the one before it still writes, so what that one writes is
// read by plain (or .cg) loads after the wait and never by non-coherent ones (__ldg), which ask for data that
// nobody writes while the reading kernel runs; a caller's inputs may be the outputs of the call before.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void mbar_init(unsigned long long* b)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(b)) : "memory");
}
__device__ __forceinline__ void mbar_expect(unsigned long long* b, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_load(void* dst, const void* src, unsigned bytes, unsigned long long* bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void fence_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void mma_bf16(unsigned d, unsigned long long a, unsigned long long b, unsigned idesc, bool acc)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d), "l"(a), "l"(b), "r"(idesc),
                 "r"(acc ? 1u : 0u)
                 : "memory");
}
__device__ __forceinline__ void mma_commit(unsigned long long* bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// n products of K = 16 into accumulator d, operand descriptors advancing by da and db
// (in 16-byte units) per product
__device__ __forceinline__ void mma_chain(unsigned d, unsigned long long a, unsigned da, unsigned long long b, unsigned db,
                                          unsigned idesc, int n, bool acc)
{
    for (int k = 0; k < n; ++k) {
        mma_bf16(d, a, b, idesc, acc || k > 0);
        a += da;
        b += db;
    }
}

// 16 (8) accumulator columns of this warp's 32 lanes; the values are there after tmem_wait
__device__ __forceinline__ void tmem_ld16(unsigned addr, unsigned (&r)[16])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(addr));
}
__device__ __forceinline__ void tmem_ld8(unsigned addr, unsigned (&r)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(addr));
}
__device__ __forceinline__ void tmem_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ unsigned pack2(float a, float b)
{
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const unsigned*>(&h);
}

// ---- Forward pass, head and (BWD) the activations' gradients of one 128-sample
// tile per block, everything between the inputs and the weight products in one
// kernel.  All three weight matrices (152 KiB) and one 128 x 256 activation tile
// live in shared memory, the accumulators in tensor memory, the ReLU masks in
// registers (one bit per element); the activations go to global memory only for
// the products over the samples (grad_kernel).  Five products per tile, each issued
// by one thread and followed by an epilogue of 512 threads (thread = sample x a quarter of
// the columns): the chain of five waits and epilogues bounds the kernel at every batch
// size up to 152 tiles, so nothing is split further.
// In cycles at 512 samples: set-up and inputs 2,800, the three 256-wide products 2,500
// each (16 x 132, the tensor core's rate), hidden epilogues 2,900, head 6,000, gradient
// epilogues 6,400 with the FP32 copy; times of both kernels at grad_kernel.
struct NetArgs {
    const float* x;
    const float* p;                     // biases
    const unsigned char* w;             // packed weights
    const float* Rt;
    float* y_out;
    float* R_out;
    float* loss;                        // !BWD: the loss is summed here by the last tile
    Acts act;
    int n;
};

constexpr int NS_W2 = 0, NS_W3 = NS_W2 + NH * NH * 2, NS_H = NS_W3 + NOUTP * NH * 2, NS_BIAS = NS_H + TILE * NH * 2,
              NS_W1 = NS_BIAS + (2 * NH + NOUTP) * 4, NS_X = NS_W1 + NH * NINP * 2, NS_TAB = NS_W1,
              NET_SMEM = NS_TAB + 29 * TILE * 4;      // the head's tables take the place of W1 and X
constexpr int CS_T = TILE / 8 * 128;    // column-group stride of a 128-row tile in shared memory
constexpr int NTHREADS = 512;           // four threads per sample, 64 columns each
static_assert(NET_SMEM <= 227 * 1024 - 256, "shared memory of the network kernel");
static_assert(NS_X + TILE * NINP * 2 <= NET_SMEM && NS_W1 % 128 == 0, "W1 and X fit the tables' place");

// Epilogues of one thread's 64 columns.  out: its place in global memory (a group of 8
// columns every cs bytes; plain 16-byte stores, 512 contiguous bytes a warp: a bulk store of
// the tile held the next epilogue back by the 3,000 cycles it took to read the tile).
// Hidden layer: relu(acc + b) as BF16 into the tile and, per group of 8 columns, which are
// above zero (one byte each of the result).
template <bool OUT>
__device__ __forceinline__ unsigned long long hidden(unsigned acc, const float* b, unsigned char* tile, unsigned char* out,
                                                     long long cs, bool live)
{
    unsigned long long m = 0;
    unsigned r[4][16];
#pragma unroll
    for (int q = 0; q < 4; ++q) tmem_ld16(acc + q * 16u, r[q]);
    tmem_wait();
#pragma unroll
    for (int c = 0; c < 64; c += 8) {
        const unsigned(&u)[16] = r[c >> 4];
        const int o = c & 8;
        const float4 b0 = *reinterpret_cast<const float4*>(b + c), b1 = *reinterpret_cast<const float4*>(b + c + 4);
        unsigned h[4];
        h[0] = pack2(fmaxf(__uint_as_float(u[o]) + b0.x, 0.0f), fmaxf(__uint_as_float(u[o + 1]) + b0.y, 0.0f));
        h[1] = pack2(fmaxf(__uint_as_float(u[o + 2]) + b0.z, 0.0f), fmaxf(__uint_as_float(u[o + 3]) + b0.w, 0.0f));
        h[2] = pack2(fmaxf(__uint_as_float(u[o + 4]) + b1.x, 0.0f), fmaxf(__uint_as_float(u[o + 5]) + b1.y, 0.0f));
        h[3] = pack2(fmaxf(__uint_as_float(u[o + 6]) + b1.z, 0.0f), fmaxf(__uint_as_float(u[o + 7]) + b1.w, 0.0f));
        unsigned bits = 0;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            if (!live) h[t] = 0u;
            // both halves' 15 magnitude bits carry into the bit above when any is set
            const unsigned nz = ((h[t] & 0x7fff7fffu) + 0x7fff7fffu) & 0x80008000u;
            bits |= (nz >> (15 - t)) | (nz >> (27 - t));
        }
        const uint4 v = make_uint4(h[0], h[1], h[2], h[3]);
        *reinterpret_cast<uint4*>(tile + (c >> 3) * CS_T) = v;
        if (OUT) *reinterpret_cast<uint4*>(out + (c >> 3) * cs) = v;
        m |= (unsigned long long)(bits & 0xffu) << c;
    }
    return m;
}

// Gradient: masked, BF16 into the tile; the FP32 values (d32, by column), or above
// SPLIT_MIN tiles their sums over the warp (part), for the bias gradients
__device__ __forceinline__ void masked(unsigned acc, unsigned long long m, unsigned char* tile, unsigned char* out, long long cs,
                                       float* d32, int ns, float* part, int lane)
{
    unsigned r[4][16];
#pragma unroll
    for (int q = 0; q < 4; ++q) tmem_ld16(acc + q * 16u, r[q]);
    tmem_wait();
#pragma unroll
    for (int c = 0; c < 64; c += 8) {
        float v[8];
        const unsigned bits = (unsigned)(m >> c);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            v[2 * t] = (bits & (1u << t)) ? __uint_as_float(r[c >> 4][(c & 8) + 2 * t]) : 0.0f;
            v[2 * t + 1] = (bits & (16u << t)) ? __uint_as_float(r[c >> 4][(c & 8) + 2 * t + 1]) : 0.0f;
        }
        const uint4 h = make_uint4(pack2(v[0], v[1]), pack2(v[2], v[3]), pack2(v[4], v[5]), pack2(v[6], v[7]));
        *reinterpret_cast<uint4*>(tile + (c >> 3) * CS_T) = h;
        *reinterpret_cast<uint4*>(out + (c >> 3) * cs) = h;
        if (d32) {
#pragma unroll
            for (int j = 0; j < 8; ++j) d32[(c + j) * ns] = v[j];
        } else {
            // columns by lane bits 4, 3, 2 (each step sends half of what is left), then the sums of the 4 lanes
#pragma unroll
            for (int o = 16, n = 4; o >= 4; o >>= 1, n >>= 1) {
                const bool up = (lane & o) != 0;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (k >= n) break;
                    const float send = up ? v[k] : v[k + n], keep = up ? v[k + n] : v[k];
                    v[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                }
            }
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
            if ((lane & 3) == 0) part[c + (lane >> 2)] = v[0];
        }
    }
}

// Output head: L from the 21 outputs (diagonal through softplus), R^ = L L^T; with
// targets, the loss (1/(36 n)) sum (R^ - Rt)^2 and its gradient with respect to the
// outputs: dR = 2 (R^ - Rt) / (36 n), dL = 2 dR L (dR symmetric), dy = dL (off the
// diagonal), dL_ii sigmoid(y_ii).  One row i of one sample per call, from the sample's
// table T (L's lower triangle, then the sigmoids; dy, or y, in its place afterwards): with
// consecutive threads on consecutive rows the targets are read in whole lines (36
// floats per sample read by its own thread cost 32 line accesses per load, 4,800 cycles a
// tile).  Returns the row's squared errors.
constexpr int TS = 29;                  // floats a sample's table takes (27, odd for the banks)
__device__ __forceinline__ float head_row(const float* T, int i, const float* rt, float* R_out, float c, float (&dy)[6])
{
    float err = 0.0f, Li[6], dR[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) Li[k] = k <= i ? T[i * (i + 1) / 2 + k] : 0.0f;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        float a = 0.0f;
#pragma unroll
        for (int k = 0; k < 6; ++k) a += Li[k] * (k <= j ? T[tri(j, k)] : 0.0f);
        if (R_out) R_out[j] = a;
        dR[j] = 0.0f;
        if (rt) {
            const float d = a - rt[j];
            err += d * d;
            dR[j] = c * d;
        }
    }
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        float a = 0.0f;
#pragma unroll
        for (int k = 0; k < 6; ++k) a += dR[k] * (j <= k ? T[tri(k, j)] : 0.0f);
        a *= 2.0f;
        dy[j] = j == i ? a * T[NOUT + i] : a;
    }
    return err;
}

template <bool BWD>
__global__ void __launch_bounds__(NTHREADS, 1) net_kernel(const NetArgs A)
{
    extern __shared__ __align__(128) unsigned char sm[];
    __shared__ unsigned long long bar[3];           // W1; W2 and W3; products
    __shared__ unsigned s_tmem;
    __shared__ float s_red[NTHREADS / 32];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, wq = warp & 3, part = warp >> 2;
    const int tile = blockIdx.x, row = wq * 32 + lane, s = tile * TILE + row;
    const bool live = s < A.n;
    const long long out0 = (long long)tile * CS_T;      // this tile within a column group
    unsigned char* sH = sm + NS_H;
    unsigned char* sdY = sH;            // dY takes the tile's place between H2 and dH2
    float* sb = reinterpret_cast<float*>(sm + NS_BIAS);
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&s_tmem)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int k = 0; k < 3; ++k) mbar_init(bar + k);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // the inputs and the weights may come from the kernels just before; once they are
    // done, grad_kernel may set itself up beside this kernel (it waits in turn)
    pdl_wait();
    pdl_trigger();
    if (tid == 0) {
        mbar_expect(bar, NH * NINP * 2);
        bulk_load(sm + NS_W1, A.w + PK_W1, NH * NINP * 2, bar);
        mbar_expect(bar + 1, NH * NH * 2 + NOUTP * NH * 2);
        bulk_load(sm + NS_W2, A.w + PK_W2, NH * NH * 2 + NOUTP * NH * 2, bar + 1);   // W3 follows W2 in both
    }
    if (tid < TILE) {
        // the sample's 8 features, the padding columns zero
        float f[NIN];
        const float* xs = A.x + (long long)s * NIN;
        if (live && (reinterpret_cast<uintptr_t>(A.x) & 15u) == 0) {
            const float4 u = *reinterpret_cast<const float4*>(xs), v = *(reinterpret_cast<const float4*>(xs) + 1);
            f[0] = u.x; f[1] = u.y; f[2] = u.z; f[3] = u.w; f[4] = v.x; f[5] = v.y; f[6] = v.z; f[7] = v.w;
        } else {
#pragma unroll
            for (int k = 0; k < NIN; ++k) f[k] = live ? xs[k] : 0.0f;
        }
        const uint4 c0 = make_uint4(pack2(f[0], f[1]), pack2(f[2], f[3]), pack2(f[4], f[5]), pack2(f[6], f[7]));
        const uint4 c1 = make_uint4(0u, 0u, 0u, 0u);
        *reinterpret_cast<uint4*>(sm + NS_X + core_at(CS_T, row, 0)) = c0;
        *reinterpret_cast<uint4*>(sm + NS_X + core_at(CS_T, row, 8)) = c1;
        if (BWD) {
            *reinterpret_cast<uint4*>(A.act.X + out0 + core_at(0, row, 0)) = c0;
            *reinterpret_cast<uint4*>(A.act.X + A.act.cs + out0 + core_at(0, row, 0)) = c1;
        }
    }
    for (int k = tid; k < 2 * NH + NOUTP; k += NTHREADS)
        sb[k] = A.p[k < NH ? OFF_B1 + k : (k < 2 * NH ? OFF_B2 + k - NH : OFF_B3 + k - 2 * NH)];
    fence_async();
    tc_before();
    __syncthreads();
    tc_after();
    const unsigned tmem = s_tmem, tlane = tmem + ((unsigned)(wq * 32) << 16);
    unsigned phase = 0;
    bool ok = true;
    constexpr unsigned ID256 = idesc_bf16(TILE, NH), ID32 = idesc_bf16(TILE, NOUTP), BMN = 1u << 16;   // B MN-major
    const unsigned aH = smem_u32(sH);
    // waits for a barrier; one thread polls and the others park at the block barrier (16 warps
    // polling took the issuing thread's slots: 150 cycles per product instead of 50)
    auto wait_all = [&](unsigned long long* b, unsigned parity) {
        const bool got = tid > 0 || mbar_wait(b, parity);
        if (__syncthreads_or(!got)) ok = false;
        tc_after();
        return ok;
    };
    auto product_done = [&]() {
        phase ^= 1u;
        return wait_all(bar + 2, phase ^ 1u);
    };
    // end of an epilogue: the tile is in shared memory for the tensor core and the bulk stores
    auto settled = [&]() {
        fence_async();
        tc_before();
        __syncthreads();
        tc_after();
    };
    unsigned long long m1 = 0, m2 = 0;
    const int col = part * 64;
    unsigned char* mine = sH + core_at(CS_T, row, col);
    const long long to = (long long)(col >> 3) * A.act.cs + out0 + core_at(0, row, 0);
    const bool keep = gridDim.x <= SPLIT_MIN;       // FP32 gradients for sums in the samples' order
    bool pending = true;                            // W2 and W3 still on their way
    do {
        // ---- layer 1
        if (!wait_all(bar, 0u)) break;
        if (tid == 0) {
            mma_chain(tmem, sdesc(smem_u32(sm + NS_X), CS_T, 128u), 0u, sdesc(smem_u32(sm + NS_W1), CS_W12, 128u), 0u, ID256, 1, false);
            mma_commit(bar + 2);
        }
        if (!product_done()) break;
        m1 = hidden<BWD>(tlane + (unsigned)col, sb + col, mine, A.act.H1 + to, A.act.cs, live);
        settled();
        // ---- layer 2
        if (!wait_all(bar + 1, 0u)) break;
        pending = false;
        if (tid == 0) {
            mma_chain(tmem + NH, sdesc(aH, CS_T, 128u), 2 * CS_T / 16, sdesc(smem_u32(sm + NS_W2), CS_W12, 128u), 2 * CS_W12 / 16, ID256, NH / 16, false);
            mma_commit(bar + 2);
        }
        if (!product_done()) break;
        m2 = hidden<BWD>(tlane + NH + (unsigned)col, sb + NH + col, mine, A.act.H2 + to, A.act.cs, live);
        settled();
        // ---- output layer
        if (tid == 0) {
            mma_chain(tmem, sdesc(aH, CS_T, 128u), 2 * CS_T / 16, sdesc(smem_u32(sm + NS_W3), CS_W3, 128u), 2 * CS_W3 / 16, ID32, NH / 16, false);
            mma_commit(bar + 2);
        }
        if (!product_done()) break;
        // ---- head: the outputs into the samples' tables, the diagonals through softplus and sigmoid, the rows
        {
            float* T = reinterpret_cast<float*>(sm + NS_TAB);
            unsigned v[8];
            tmem_ld8(tlane + part * 8, v);
            tmem_wait();
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int t = part * 8 + k;
                if (t < NOUT) T[row * TS + t] = __uint_as_float(v[k]) + sb[2 * NH + t];
            }
            __syncthreads();
            if (A.y_out) {
                for (int k = tid; k < min(A.n - tile * TILE, TILE) * NOUT; k += NTHREADS)
                    A.y_out[(long long)tile * TILE * NOUT + k] = T[k / NOUT * TS + k % NOUT];
                __syncthreads();
            }
#pragma unroll 1
            for (int k = tid; k < 6 * TILE; k += NTHREADS) {
                const int r = k / 6, i = k - r * 6, t = i * (i + 3) / 2;
                const float y = T[r * TS + t];
                T[r * TS + NOUT + i] = sigmoid(y);
                T[r * TS + t] = softplus(y);
            }
            __syncthreads();
            float err = 0.0f, dy[2][6] = {};
#pragma unroll 1
            for (int q = 0; q < 2; ++q) {
                const int k = tid + q * NTHREADS, r = k / 6, i = k - r * 6;
                const long long sr = (long long)tile * TILE + r;
                if (k < 6 * TILE && sr < A.n) {
                    float d[6];
                    err += head_row(T + r * TS, i, A.Rt ? A.Rt + sr * 36 + i * 6 : nullptr, A.R_out ? A.R_out + sr * 36 + i * 6 : nullptr,
                                    2.0f / (36.0f * (float)A.n), d);
#pragma unroll
                    for (int j = 0; j < 6; ++j) {
                        dy[0][j] = q == 0 ? d[j] : dy[0][j];
                        dy[1][j] = q == 1 ? d[j] : dy[1][j];
                    }
                }
            }
            for (int o = 16; o > 0; o >>= 1) err += __shfl_xor_sync(0xffffffffu, err, o);
            if (lane == 0) s_red[warp] = err;
            if (BWD) {
                __syncthreads();
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int k = tid + q * NTHREADS, r = k / 6, i = k - r * 6;
#pragma unroll
                    for (int j = 0; j < 6; ++j)
                        if (k < 6 * TILE && j <= i) T[r * TS + i * (i + 1) / 2 + j] = dy[q][j];
                }
                __syncthreads();
                // dY: 8 columns per thread as BF16 into the tile and to global memory, FP32 or warp sums for db3
                float w[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) w[k] = live && part * 8 + k < NOUT ? T[row * TS + part * 8 + k] : 0.0f;
                const uint4 h = make_uint4(pack2(w[0], w[1]), pack2(w[2], w[3]), pack2(w[4], w[5]), pack2(w[6], w[7]));
                *reinterpret_cast<uint4*>(sdY + core_at(CS_T, row, part * 8)) = h;
                *reinterpret_cast<uint4*>(A.act.dY + part * A.act.cs + (long long)tile * CS_T + core_at(0, row, 0)) = h;
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int c = 2 * NH + part * 8 + k;
                    if (keep) {
                        A.act.d32[c * A.act.ns + s] = w[k];
                    } else {
                        for (int o = 16; o > 0; o >>= 1) w[k] += __shfl_xor_sync(0xffffffffu, w[k], o);
                        if (lane == 0) A.act.b_part[(long long)(tile * 4 + wq) * NSUM + c] = w[k];
                    }
                }
            }
        }
        settled();
        if (warp == 0 && A.Rt) {
            float err = lane < NTHREADS / 32 ? s_red[lane] : 0.0f;
            for (int o = 16; o > 0; o >>= 1) err += __shfl_xor_sync(0xffffffffu, err, o);
            if (lane == 0) A.act.loss_part[tile] = err / (36.0f * (float)A.n);
        }
        if (!BWD) break;
        // ---- dH2 = (dY W3) * [H2 > 0]
        if (tid == 0) {
            mma_chain(tmem + NH, sdesc(smem_u32(sdY), CS_T, 128u), 2 * CS_T / 16, sdesc(smem_u32(sm + NS_W3), 128u, CS_W3), 256 / 16, ID256 | BMN, NOUTP / 16, false);
            mma_commit(bar + 2);
        }
        if (!product_done()) break;
        masked(tlane + NH + (unsigned)col, m2, mine, A.act.dH2 + to, A.act.cs, keep ? A.act.d32 + (long long)(NH + col) * A.act.ns + s : nullptr, A.act.ns,
               A.act.b_part + (long long)(tile * 4 + wq) * NSUM + NH + col, lane);
        settled();
        // ---- dH1 = (dH2 W2) * [H1 > 0]
        if (tid == 0) {
            mma_chain(tmem, sdesc(aH, CS_T, 128u), 2 * CS_T / 16, sdesc(smem_u32(sm + NS_W2), 128u, CS_W12), 256 / 16, ID256 | BMN, NH / 16, false);
            mma_commit(bar + 2);
        }
        if (!product_done()) break;
        masked(tlane + (unsigned)col, m1, mine, A.act.dH1 + to, A.act.cs, keep ? A.act.d32 + (long long)col * A.act.ns + s : nullptr, A.act.ns,
               A.act.b_part + (long long)(tile * 4 + wq) * NSUM + col, lane);
    } while (false);
    if (!ok) {
        // a completion never came: give what is in flight a second bounded wait before leaving
        if (tid == 0) atomicOr(&g_gemm_status, 1u);
        (void)mbar_wait(bar, 0u);
        if (pending) (void)mbar_wait(bar + 1, 0u);
        (void)mbar_wait(bar + 2, phase ^ 1u);
    }
    if (!BWD && A.loss) {
        // the last tile adds the tiles' losses, in order
        __shared__ bool s_last;
        if (tid == 0) {
            __threadfence();
            s_last = atomicAdd(A.act.count, 1u) == gridDim.x - 1;
            if (s_last) {
                __threadfence();
                float v = 0.0f;
                for (unsigned t = 0; t < gridDim.x; ++t) v += __ldcg(A.act.loss_part + t);
                *A.loss = v;
                *A.act.count = 0;
            }
        }
    }
    tc_before();
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
}

// ---- Products over the samples (weight gradients), column sums of the biases, the
// loss, and with ADAM the update of every parameter and of its BF16 copy in place.
// One block per 128 x 32 tile of a gradient: dW2 = dH2^T H1 (16 tiles), dW3^T = H2^T dY
// (2), dW1 = dH1^T X (2, 16 columns), and one per 32 biases.  Both operands are
// MN-major: the tiles that net_kernel wrote come in by 2 KiB bulk copies, 128 samples a
// stage, GST stages in flight.  Narrow tiles give the chip 20 blocks where a single
// 256-wide tile per half gave 2; the order of the sum over the samples stays that of one
// accumulator up to SPLIT_MIN tiles (an Adam step turns the last bit of a gradient near
// zero into the sign of the update), and is split over a cluster above it, whose first
// block adds the parts in rank order.
// Measured: an Adam step on 512 samples, both kernels, 28.8 us (net_kernel 18, this one
// 12, overlapped by programmatic launch) against 760 us before, when five products, three
// one-block column sums, the head and Adam were 13 kernels and each product staged its
// operands with one load in flight; loss and gradients of 4,096 samples 28.3 us against
// 2,805.  At 512 samples the 160 KiB of operands a block takes in set its time.
struct GradArgs {
    Acts act;
    int n, tiles;
    float* grad;                        // !ADAM
    float *p, *m1, *m2;                 // ADAM
    unsigned char* w;
    float lr, c1, c2;
    float* loss;
};

constexpr int GST = 5, GS_A = 16 * CS_T, GS_B = 4 * CS_T, GRAD_SMEM = GST * (GS_A + GS_B);
constexpr int GTHREADS_N = 18 * 32;     // sixteen warps for the result, one for the loads, one for the products
constexpr int GEMM_JOBS = 20, BIAS_JOBS = NSUM / 32, SPLIT = 4;
static_assert(32 * (SPLIT_MIN * TILE * 4 + 16) <= GRAD_SMEM, "32 columns of the samples fit the stages");
constexpr int GS_TILE = (SPLIT - 1) * TILE * 32 * 4;    // the result's tile, after the other blocks' parts
static_assert(GS_TILE + TILE * 33 * 4 <= GRAD_SMEM, "parts and tile fit the stages");

__device__ __forceinline__ void adam(float& p, float& m1, float& m2, float gi, float lr, float c1, float c2)
{
    const float a = 0.9f * m1 + 0.1f * gi;
    const float b = 0.999f * m2 + 0.001f * gi * gi;
    m1 = a;
    m2 = b;
    p -= lr * (a * c1) / (sqrtf(b * c2) + 1e-8f);
}

template <bool ADAM>
__global__ void __launch_bounds__(GTHREADS_N, 1) grad_kernel(const GradArgs G)
{
    extern __shared__ __align__(128) unsigned char sm[];
    __shared__ unsigned long long full[GST], empty[GST], done;
    __shared__ unsigned s_tmem;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    unsigned rank, nrank;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(nrank));
    const int job = blockIdx.x / (int)nrank;
    if (job >= GEMM_JOBS) {
        // biases: 32 columns, summed in the samples' order by one lane each; the loss
        const int c0 = (job - GEMM_JOBS) * 32;
        if (rank > 0) return;
        pdl_wait();
        float v = 0.0f;
        bool ok = true;
        if (G.tiles <= SPLIT_MIN) {
            // the columns by one bulk copy each, 16 bytes apart modulo 128 so that the lanes read without conflicts
            const int bytes = G.tiles * TILE * 4;
            if (tid == 0) {
                mbar_init(full);
                asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
                mbar_expect(full, 32u * (unsigned)bytes);
            }
            __syncthreads();
            if (warp > 0) return;
            bulk_load(sm + lane * (bytes + 16), G.act.d32 + (long long)(c0 + lane) * G.act.ns, (unsigned)bytes, full);
            ok = __all_sync(0xffffffffu, mbar_wait(full, 0u));
            const float4* d = reinterpret_cast<const float4*>(sm + lane * (bytes + 16));
#pragma unroll 8
            for (int t = 0; t < G.tiles * TILE / 4; ++t) {
                const float4 u = d[t];
                v += u.x;
                v += u.y;
                v += u.z;
                v += u.w;
            }
        } else {
            if (warp > 0) return;
#pragma unroll 8
            for (int t = 0; t < 4 * G.tiles; ++t) v += __ldcg(G.act.b_part + (long long)t * NSUM + c0 + lane);
        }
        if (!ok) {
            // a second bounded wait for the copies in flight before leaving
            (void)mbar_wait(full, 0u);
            if (lane == 0) atomicOr(&g_gemm_status, 1u);
            return;
        }
        if (c0 + lane >= 2 * NH + NOUT) v = 0.0f;     // padding
        const int c = c0 + lane, i = c < NH ? OFF_B1 + c : (c < 2 * NH ? OFF_B2 + c - NH : OFF_B3 + c - 2 * NH);
        if (ADAM) adam(G.p[i], G.m1[i], G.m2[i], v, G.lr, G.c1, G.c2);
        else G.grad[i] = v;
        if (c == NSUM - 1 && G.loss) {
            float l = 0.0f;
            for (int t = 0; t < G.tiles; ++t) l += G.act.loss_part[t];
            *G.loss = l;
        }
        return;
    }
    // ---- operands and place of this tile
    const bool w3 = job >= 16 && job < 18, w1 = job >= 18;
    const int ih = job < 16 ? job >> 3 : job & 1, jt = job < 16 ? job & 7 : 0, ncol = w1 ? 16 : 32;
    const unsigned char* a = (w1 ? G.act.dH1 : (w3 ? G.act.H2 : G.act.dH2)) + (long long)ih * 16 * G.act.cs;
    const unsigned char* b = (w1 ? G.act.X : (w3 ? G.act.dY : G.act.H1)) + (long long)jt * 4 * G.act.cs;
    const int t0 = (int)((long long)G.tiles * rank / nrank), t1 = (int)((long long)G.tiles * (rank + 1) / nrank);
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 32;" ::"r"(smem_u32(&s_tmem)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int k = 0; k < GST; ++k) { mbar_init(full + k); mbar_init(empty + k); }
        mbar_init(&done);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_before();
    __syncthreads();
    tc_after();
    // ---- parameters of this thread's row, last written by the kernel before net_kernel, which that one
    // waited for before it let this one start
    // The result comes out of tensor memory one row per thread and goes through a shared-memory tile: a warp's
    // accesses to the parameters are whole 128-byte lines, and an Adam step's square root and division (a chain of
    // some 300 cycles that the compiler does not interleave) run eight deep on sixteen warps instead of 32 deep on
    // four (17,900 cycles then).  Value j of a thread is element (tr + trs j, tc + tcs j) of the tile.
    const int nval = w1 ? 4 : 8;
    const int tr = w1 ? warp * 8 + (lane >> 4) : (w3 ? (warp & 3) * 32 + lane : warp * 8), trs = w1 ? 2 : (w3 ? 0 : 1);
    const int tc = w1 ? lane & 15 : (w3 ? (warp >> 2) * 8 : lane), tcs = w3 ? 1 : 0;
    const int stp = w1 ? 2 * NINP : NH;
    const int o0 = w1 ? OFF_W1 + (ih * 128 + tr) * NINP + tc
                      : (w3 ? OFF_W3 + tc * NH + ih * 128 + tr : OFF_W2 + (ih * 128 + tr) * NH + jt * 32 + tc);
    float pv[8], q1[8], q2[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const bool mine = ADAM && rank == 0 && warp < 16 && j < nval;
        pv[j] = mine ? G.p[o0 + j * stp] : 0.0f;
        q1[j] = mine ? G.m1[o0 + j * stp] : 0.0f;
        q2[j] = mine ? G.m2[o0 + j * stp] : 0.0f;
    }
    pdl_wait();
    const unsigned tmem = s_tmem;
    bool ok = true;
    int issued = 0;                             // stages this thread has loaded, or passed to the tensor core
    if (warp == 16) {
        // loads: one column group (2 KiB of a tile) per lane
        const int ng = 16 + ncol / 8;
        for (int t = t0; t < t1; ++t) {
            const int st = (t - t0) % GST, use = (t - t0) / GST;
            // one decision per warp: lanes whose waits ended differently would part at the barrier below
            if (!__all_sync(0xffffffffu, use == 0 || mbar_wait(empty + st, (unsigned)(use - 1) & 1u))) { ok = false; break; }
            unsigned char* d = sm + st * (GS_A + GS_B);
            if (lane == 0) mbar_expect(full + st, (unsigned)(ng * CS_T));
            __syncwarp();
            if (lane < 16) bulk_load(d + lane * CS_T, a + lane * G.act.cs + (long long)t * CS_T, CS_T, full + st);
            else if (lane < ng) bulk_load(d + GS_A + (lane - 16) * CS_T, b + (lane - 16) * G.act.cs + (long long)t * CS_T, CS_T, full + st);
            ++issued;
        }
    } else if (tid == 17 * 32) {
        const unsigned idesc = idesc_bf16(TILE, ncol) | (1u << 15) | (1u << 16);     // both MN-major
        for (int t = t0; t < t1; ++t) {
            const int st = (t - t0) % GST, use = (t - t0) / GST;
            if (!mbar_wait(full + st, (unsigned)use & 1u)) { ok = false; break; }
            tc_after();
            const unsigned ad = smem_u32(sm + st * (GS_A + GS_B)), bd = ad + GS_A;
            mma_chain(tmem, sdesc(ad, 128u, CS_T), 256 / 16, sdesc(bd, 128u, CS_T), 256 / 16, idesc, TILE / 16, t > t0);
            mma_commit(empty + st);
            ++issued;
        }
        if (ok) {
            mma_commit(&done);
            ok = mbar_wait(&done, 0u);          // the other warps park at the block barrier below
        }
    }
    const bool fail = __syncthreads_or(!ok);
    tc_after();
    unsigned acc[2][16] = {};
    if (!fail && warp < 4) {
        tmem_ld16(tmem + ((unsigned)(warp * 32) << 16), acc[0]);
        tmem_ld16(tmem + ((unsigned)(warp * 32) << 16) + 16u, acc[1]);      // not used for dW1
        tmem_wait();
    }
    float v[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(acc[j >> 4][j & 15]);
    if (fail) {
        if (tid == 0) atomicOr(&g_gemm_status, 1u);
        // a second bounded wait for what is in flight: the last copies into every stage, and the products (which
        // complete in order, so the last one's arrival covers them all)
        if (warp == 16)
            for (int k = max(0, issued - GST); k < issued; ++k) (void)mbar_wait(full + k % GST, (unsigned)(k / GST) & 1u);
        else if (tid == 17 * 32 && issued > 0)
            (void)mbar_wait(empty + (issued - 1) % GST, (unsigned)((issued - 1) / GST) & 1u);
        __syncthreads();
    }
    if (nrank > 1) {
        // the other blocks' parts into the first one's stages: column j of row m at (j * 128 + m) floats
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
        if (rank > 0 && warp < 4) {
            const unsigned local = smem_u32(sm) + ((rank - 1) * TILE * 32 + (unsigned)tid) * 4u;
            unsigned remote;
            asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(remote) : "r"(local));
#pragma unroll
            for (int j = 0; j < 32; ++j)
                asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(remote + j * TILE * 4), "f"(fail ? 0.0f : v[j]) : "memory");
        }
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
        if (rank == 0 && warp < 4) {
            const float* part = reinterpret_cast<const float*>(sm) + tid;
            for (unsigned r = 0; r + 1 < nrank; ++r)
#pragma unroll
                for (int j = 0; j < 32; ++j) v[j] += part[(r * 32 + j) * TILE];
        }
    }
    if (rank == 0) {
        float* T = reinterpret_cast<float*>(sm + GS_TILE);
        if (warp < 4) {
#pragma unroll
            for (int j = 0; j < 32; ++j)
                if (j < ncol) T[tid * 33 + j] = v[j];
        }
        __syncthreads();
        if (!fail && warp < 16) {
            unsigned char* w = G.w + (w1 ? PK_W1 : (w3 ? PK_W3 : PK_W2));
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                if (j >= nval) break;
                const int r = tr + trs * j, c = tc + tcs * j, o = o0 + j * stp;
                const float g = T[r * 33 + c];
                if (ADAM) {
                    adam(pv[j], q1[j], q2[j], g, G.lr, G.c1, G.c2);
                    G.p[o] = pv[j];
                    G.m1[o] = q1[j];
                    G.m2[o] = q2[j];
                    const int at = w3 ? core_at(CS_W3, c, ih * 128 + r) : core_at(CS_W12, ih * 128 + r, jt * 32 + c);
                    *reinterpret_cast<__nv_bfloat16*>(w + at) = __float2bfloat16(pv[j]);
                } else {
                    G.grad[o] = g;
                }
            }
        }
    }
    tc_before();
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 32;" ::"r"(tmem) : "memory");
}

// Cholesky solve of A u = f for one symmetric positive definite 6x6 A (FP64,
// A overwritten)
__device__ void chol_solve6(double (&A)[6][6], const double* f, double* u)
{
    double y[6];
    for (int j = 0; j < 6; ++j) {                      // A = C C^T, C lower, in place
        double d = A[j][j];
        for (int k = 0; k < j; ++k) d -= A[j][k] * A[j][k];
        d = d > 0.0 ? sqrt(d) : 0.0;
        A[j][j] = d;
        for (int i = j + 1; i < 6; ++i) {
            double a = A[i][j];
            for (int k = 0; k < j; ++k) a -= A[i][k] * A[j][k];
            A[i][j] = d > 0.0 ? a / d : 0.0;
        }
    }
    for (int i = 0; i < 6; ++i) {
        double a = f[i];
        for (int k = 0; k < i; ++k) a -= A[i][k] * y[k];
        y[i] = A[i][i] > 0.0 ? a / A[i][i] : 0.0;
    }
    for (int i = 5; i >= 0; --i) {
        double a = y[i];
        for (int k = i + 1; k < 6; ++k) a -= A[k][i] * u[k];
        u[i] = A[i][i] > 0.0 ? a / A[i][i] : 0.0;
    }
}

// Cholesky solve of R u = f per sample, FP64 (R read as FP32, symmetrised)
__global__ void spd_solve_kernel(const float* R, const double* f, double* u, int n)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    double A[6][6];
    for (int i = 0; i < 6; ++i)
        for (int j = 0; j < 6; ++j) A[i][j] = 0.5 * ((double)R[s * 36 + i * 6 + j] + (double)R[s * 36 + j * 6 + i]);
    chol_solve6(A, f + s * 6, u + s * 6);
}

// inverse of a 6x6 matrix M (Gauss-Jordan with partial pivoting, FP64),
// symmetrised, into out
__device__ void invert6_sym(const double* M, double* out)
{
    double A[6][12];
    for (int i = 0; i < 6; ++i)
        for (int j = 0; j < 12; ++j) A[i][j] = j < 6 ? M[i * 6 + j] : (j - 6 == i ? 1.0 : 0.0);
    for (int c = 0; c < 6; ++c) {
        int piv = c;
        for (int r = c + 1; r < 6; ++r)
            if (fabs(A[r][c]) > fabs(A[piv][c])) piv = r;
        if (piv != c)
            for (int j = 0; j < 12; ++j) { const double t = A[c][j]; A[c][j] = A[piv][j]; A[piv][j] = t; }
        const double d = A[c][c];
        const double id = d != 0.0 ? 1.0 / d : 0.0;
        for (int j = 0; j < 12; ++j) A[c][j] *= id;
        for (int r = 0; r < 6; ++r) {
            if (r == c) continue;
            const double fct = A[r][c];
            for (int j = 0; j < 12; ++j) A[r][j] -= fct * A[c][j];
        }
    }
    for (int i = 0; i < 6; ++i)
        for (int j = 0; j < 6; ++j) out[i * 6 + j] = 0.5 * (A[i][j + 6] + A[j][i + 6]);
}

__global__ void spd_invert_kernel(double* M, int n)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    double t[36];
    invert6_sym(M + s * 36, t);
    for (int k = 0; k < 36; ++k) M[s * 36 + k] = t[k];
}

// ---- features and scaling of the resistance tensor.  geom per sample:
// (a, b, nu, L, e_x, e_y, e_z, rho0): semi-axes a (along the unit long axis e)
// and b, kinematic viscosity, box edge (or the edge of the volume per
// particle), fluid density.  D = diag(s_t I3, s_r I3) with s_t^2 = 6 pi mu b and
// s_r^2 = 8 pi mu b^3 (mu = rho0 nu): the radius-b sphere's Stokes resistances,
// so that R^ = D^-1 R D^-1 is the identity for that sphere in free space.
__device__ __forceinline__ void scales(const double* g, double& st, double& sr)
{
    const double mu = g[7] * g[2], b = g[1];
    st = sqrt(6.0 * M_PI * mu * b);
    sr = sqrt(8.0 * M_PI * mu * b * b * b);
}

__global__ void features_geom_kernel(const double* geom, int n, float* x)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    const double* g = geom + s * 8;
    const double sg = g[6] < 0.0 ? -1.0 : 1.0;       // head-tail symmetry: e and -e are the same spheroid
    x[s * 8 + 0] = (float)(g[0] / g[1] - 2.0);
    x[s * 8 + 1] = (float)(g[1] - 3.0);
    x[s * 8 + 2] = (float)((g[2] - 1.0 / 6.0) * 10.0);
    x[s * 8 + 3] = (float)(g[1] / g[3] * 10.0 - 1.0);
    x[s * 8 + 4] = (float)(sg * g[4]);
    x[s * 8 + 5] = (float)(sg * g[5]);
    x[s * 8 + 6] = (float)(sg * g[6]);
    x[s * 8 + 7] = 1.0f;
}

// measured mobility M (6x6, FP64) -> R^ = (D M D)^-1 (FP32)
__global__ void targets_kernel(const double* M, const double* geom, int n, float* Rhat)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    double st, sr;
    scales(geom + s * 8, st, sr);
    double A[36], t[36];
    for (int i = 0; i < 6; ++i)
        for (int j = 0; j < 6; ++j) A[i * 6 + j] = (i < 3 ? st : sr) * M[s * 36 + i * 6 + j] * (j < 3 ? st : sr);
    invert6_sym(A, t);
    for (int k = 0; k < 36; ++k) Rhat[s * 36 + k] = (float)t[k];
}

// (U, Omega) = R^-1 (F, T) = D^-1 R^^-1 D^-1 (F, T)
__global__ void warm_velocities_kernel(const float* Rhat, const double* geom, const double* FT, int n, double* UW)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    double st, sr;
    scales(geom + s * 8, st, sr);
    double A[6][6], f[6], u[6];
    for (int i = 0; i < 6; ++i) {
        f[i] = FT[s * 6 + i] / (i < 3 ? st : sr);
        for (int j = 0; j < 6; ++j)
            A[i][j] = 0.5 * ((double)Rhat[s * 36 + i * 6 + j] + (double)Rhat[s * 36 + j * 6 + i]);
    }
    chol_solve6(A, f, u);
    for (int i = 0; i < 6; ++i) UW[s * 6 + i] = u[i] / (i < 3 ? st : sr);
}

}  // namespace lbsur

struct lb_mlp {
    int device = 0;
    int max_batch = 0;
    long long step = 0;
    float* p = nullptr;                 // FP32 master parameters
    float* m1 = nullptr;                // Adam moments
    float* m2 = nullptr;
    float* loss = nullptr;              // scratch loss for train_step without output
    unsigned char* w = nullptr;         // BF16 copy of the weights, packed (PK_*)
    Acts act{};
    std::vector<void*> allocs;
};

namespace {

template <class T>
bool mlp_alloc(lb_mlp* m, T** p, size_t count)
{
    void* q = nullptr;
    if (cudaMalloc(&q, count * sizeof(T)) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    m->allocs.push_back(q);
    *p = static_cast<T*>(q);
    return true;
}

void mlp_free(lb_mlp* m)
{
    for (void* q : m->allocs) cudaFree(q);
    m->allocs.clear();
}

inline unsigned blocks(long long n, int t) { return (unsigned)((n + t - 1) / t); }

// forward pass, head and (BWD) the activations' gradients of n samples
template <bool BWD>
cudaError_t launch_net(lb_mlp* m, const float* x, int n, const float* Rt, float* y, float* R, float* loss, cudaStream_t s)
{
    NetArgs A{};
    A.x = x; A.p = m->p; A.w = m->w; A.Rt = Rt; A.y_out = y; A.R_out = R; A.loss = loss; A.act = m->act; A.n = n;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(blocks(n, TILE));
    cfg.blockDim = dim3(NTHREADS);
    cfg.dynamicSmemBytes = NET_SMEM;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, net_kernel<BWD>, A);
}

// weight and bias gradients into grad, or (ADAM) the step with learning rate lr
template <bool ADAM>
cudaError_t launch_grad(lb_mlp* m, int n, float* grad, float lr, float c1, float c2, float* loss, cudaStream_t s)
{
    GradArgs G{};
    G.act = m->act; G.n = n; G.tiles = (int)blocks(n, TILE); G.grad = grad;
    G.p = m->p; G.m1 = m->m1; G.m2 = m->m2; G.w = m->w; G.lr = lr; G.c1 = c1; G.c2 = c2; G.loss = loss;
    // above SPLIT_MIN tiles (1,024 samples) each gradient tile is a cluster of SPLIT blocks
    const int nr = G.tiles > SPLIT_MIN ? SPLIT : 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((GEMM_JOBS + BIAS_JOBS) * nr);
    cfg.blockDim = dim3(GTHREADS_N);
    cfg.dynamicSmemBytes = GRAD_SMEM;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)nr;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, grad_kernel<ADAM>, G);
}

}  // namespace

extern "C" lb_status lb_mlp_create(int32_t device, int32_t max_batch, lb_mlp** out)
{
    if (!out || max_batch < 1 || max_batch > LB_MLP_MAX_BATCH) return LB_EINVAL;
    *out = nullptr;
    if (cudaSetDevice(device) != cudaSuccess) return LB_ECUDA;
    lb_mlp* m = new (std::nothrow) lb_mlp;
    if (!m) return LB_ENOMEM;
    m->device = device;
    m->max_batch = max_batch;
    const size_t T = blocks(max_batch, TILE), B = T * TILE;      // whole tiles
    Acts& a = m->act;
    a.cs = (long long)T * CS_T;
    a.ns = (int)std::min<size_t>(T, SPLIT_MIN) * TILE;
    bool ok = mlp_alloc(m, &m->p, NPARAM) && mlp_alloc(m, &m->m1, NPARAM) && mlp_alloc(m, &m->m2, NPARAM) &&
              mlp_alloc(m, &m->loss, 1) && mlp_alloc(m, &m->w, PK_BYTES) && mlp_alloc(m, &a.X, B * NINP * 2) &&
              mlp_alloc(m, &a.H1, B * NH * 2) && mlp_alloc(m, &a.H2, B * NH * 2) && mlp_alloc(m, &a.dY, B * NOUTP * 2) &&
              mlp_alloc(m, &a.dH2, B * NH * 2) && mlp_alloc(m, &a.dH1, B * NH * 2) && mlp_alloc(m, &a.loss_part, T) &&
              mlp_alloc(m, &a.d32, (size_t)a.ns * NSUM) &&
              mlp_alloc(m, &a.b_part, 4 * T * NSUM) && mlp_alloc(m, &a.count, 1);
    if (ok) {
        for (void* q : {(void*)m->p, (void*)m->m1, (void*)m->m2})
            ok = ok && cudaMemset(q, 0, NPARAM * sizeof(float)) == cudaSuccess;
        ok = ok && cudaMemset(m->w, 0, PK_BYTES) == cudaSuccess && cudaMemset(a.count, 0, sizeof(unsigned)) == cudaSuccess;
        // the kernels' shared memory on this device
        const cudaFuncAttribute ds = cudaFuncAttributeMaxDynamicSharedMemorySize;
        ok = ok && cudaFuncSetAttribute(net_kernel<false>, ds, NET_SMEM) == cudaSuccess &&
             cudaFuncSetAttribute(net_kernel<true>, ds, NET_SMEM) == cudaSuccess &&
             cudaFuncSetAttribute(grad_kernel<false>, ds, GRAD_SMEM) == cudaSuccess &&
             cudaFuncSetAttribute(grad_kernel<true>, ds, GRAD_SMEM) == cudaSuccess;
        ok = ok && cudaDeviceSynchronize() == cudaSuccess;
    }
    if (!ok) {
        mlp_free(m);
        delete m;
        return LB_ENOMEM;
    }
    *out = m;
    return LB_OK;
}

extern "C" lb_status lb_mlp_destroy(lb_mlp* m)
{
    if (!m) return LB_EINVAL;
    cudaSetDevice(m->device);
    cudaDeviceSynchronize();
    mlp_free(m);
    delete m;
    return LB_OK;
}

extern "C" lb_status lb_mlp_set_params(lb_mlp* m, const float* host)
{
    if (!m || !host) return LB_EINVAL;
    if (cudaSetDevice(m->device) != cudaSuccess) return LB_ECUDA;
    std::vector<float> h(host, host + NPARAM);
    // padding stays zero: W1 columns 8..15, W3 rows and b3 entries 21..31
    for (int r = 0; r < NH; ++r)
        for (int c = NIN; c < NINP; ++c) h[OFF_W1 + r * NINP + c] = 0.0f;
    for (int r = NOUT; r < NOUTP; ++r) {
        for (int c = 0; c < NH; ++c) h[OFF_W3 + r * NH + c] = 0.0f;
        h[OFF_B3 + r] = 0.0f;
    }
    if (cudaMemcpy(m->p, h.data(), NPARAM * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(m->m1, 0, NPARAM * sizeof(float)) != cudaSuccess ||
        cudaMemset(m->m2, 0, NPARAM * sizeof(float)) != cudaSuccess)
        return LB_ECUDA;
    pack_kernel<<<blocks(NPARAM, 256), 256>>>(m->p, m->w);
    if (cudaGetLastError() != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess) return LB_ECUDA;
    m->step = 0;
    return LB_OK;
}

extern "C" lb_status lb_mlp_get_params(lb_mlp* m, float* host)
{
    if (!m || !host) return LB_EINVAL;
    if (cudaSetDevice(m->device) != cudaSuccess) return LB_ECUDA;
    if (cudaDeviceSynchronize() != cudaSuccess ||
        cudaMemcpy(host, m->p, NPARAM * sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess)
        return LB_ECUDA;
    return LB_OK;
}

extern "C" lb_status lb_mlp_forward(lb_mlp* m, const float* x_dev, int32_t n, float* y_dev, float* R_dev, void* stream)
{
    if (!m || !x_dev || n < 1 || n > m->max_batch) return LB_EINVAL;
    if (cudaSetDevice(m->device) != cudaSuccess ||
        launch_net<false>(m, x_dev, n, nullptr, y_dev, R_dev, nullptr, static_cast<cudaStream_t>(stream)) != cudaSuccess)
        return LB_ECUDA;
    return LB_OK;
}

extern "C" lb_status lb_mlp_loss_grad(lb_mlp* m, const float* x_dev, const float* Rt_dev, int32_t n, float* loss_dev,
                                      float* grad_dev, void* stream)
{
    if (!m || !x_dev || !Rt_dev || !loss_dev || n < 1 || n > m->max_batch) return LB_EINVAL;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (cudaSetDevice(m->device) != cudaSuccess) return LB_ECUDA;
    if (!grad_dev)                      // the loss alone
        return launch_net<false>(m, x_dev, n, Rt_dev, nullptr, nullptr, loss_dev, s) == cudaSuccess ? LB_OK : LB_ECUDA;
    if (launch_net<true>(m, x_dev, n, Rt_dev, nullptr, nullptr, nullptr, s) != cudaSuccess ||
        launch_grad<false>(m, n, grad_dev, 0.0f, 0.0f, 0.0f, loss_dev, s) != cudaSuccess)
        return LB_ECUDA;
    return LB_OK;
}

extern "C" lb_status lb_mlp_train_step(lb_mlp* m, const float* x_dev, const float* Rt_dev, int32_t n, float lr,
                                       float* loss_dev, void* stream)
{
    if (!m || !x_dev || !Rt_dev || n < 1 || n > m->max_batch || !(lr > 0.0f)) return LB_EINVAL;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (cudaSetDevice(m->device) != cudaSuccess ||
        launch_net<true>(m, x_dev, n, Rt_dev, nullptr, nullptr, nullptr, s) != cudaSuccess)
        return LB_ECUDA;
    m->step += 1;
    const float c1 = (float)(1.0 / (1.0 - std::pow(0.9, (double)m->step)));
    const float c2 = (float)(1.0 / (1.0 - std::pow(0.999, (double)m->step)));
    return launch_grad<true>(m, n, nullptr, lr, c1, c2, loss_dev ? loss_dev : m->loss, s) == cudaSuccess ? LB_OK : LB_ECUDA;
}

extern "C" lb_status lb_spd_solve6(const float* R_dev, const double* f_dev, double* u_dev, int32_t n, void* stream)
{
    if (!R_dev || !f_dev || !u_dev || n < 1) return LB_EINVAL;
    spd_solve_kernel<<<blocks(n, 64), 64, 0, static_cast<cudaStream_t>(stream)>>>(R_dev, f_dev, u_dev, n);
    return cudaGetLastError() == cudaSuccess ? LB_OK : LB_ECUDA;
}

extern "C" lb_status lb_spd_invert6(double* M_dev, int32_t n, void* stream)
{
    if (!M_dev || n < 1) return LB_EINVAL;
    spd_invert_kernel<<<blocks(n, 64), 64, 0, static_cast<cudaStream_t>(stream)>>>(M_dev, n);
    return cudaGetLastError() == cudaSuccess ? LB_OK : LB_ECUDA;
}

extern "C" lb_status lb_mlp_features(const double* geom_dev, int32_t n, float* x_dev, void* stream)
{
    if (!geom_dev || !x_dev || n < 1) return LB_EINVAL;
    features_geom_kernel<<<blocks(n, 64), 64, 0, static_cast<cudaStream_t>(stream)>>>(geom_dev, n, x_dev);
    return cudaGetLastError() == cudaSuccess ? LB_OK : LB_ECUDA;
}

extern "C" lb_status lb_resistance_targets(const double* M_dev, const double* geom_dev, int32_t n, float* Rhat_dev,
                                           void* stream)
{
    if (!M_dev || !geom_dev || !Rhat_dev || n < 1) return LB_EINVAL;
    targets_kernel<<<blocks(n, 64), 64, 0, static_cast<cudaStream_t>(stream)>>>(M_dev, geom_dev, n, Rhat_dev);
    return cudaGetLastError() == cudaSuccess ? LB_OK : LB_ECUDA;
}

extern "C" lb_status lb_warm_velocities(const float* Rhat_dev, const double* geom_dev, const double* FT_dev, int32_t n,
                                        double* UW_dev, void* stream)
{
    if (!Rhat_dev || !geom_dev || !FT_dev || !UW_dev || n < 1) return LB_EINVAL;
    warm_velocities_kernel<<<blocks(n, 64), 64, 0, static_cast<cudaStream_t>(stream)>>>(Rhat_dev, geom_dev, FT_dev, n,
                                                                                         UW_dev);
    return cudaGetLastError() == cudaSuccess ? LB_OK : LB_ECUDA;
}
