// Warm-start network: a multilayer perceptron whose products run on the
// 5th-generation tensor cores (tcgen05, BF16 operands, FP32 accumulation in
// tensor memory), trained with Adam on FP32 master weights.
//
// GEMM convention: C[M x N] = A[M x K] . B[N x K]^T with A and B bfloat16,
// row-major (K contiguous), K a multiple of 16 (buffers are zero-padded along
// K); rows of A beyond M and of B beyond N read as zero. One CTA computes a
// 128-row block with all N <= 256 columns in one accumulator.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <string>
#include <vector>

#include "lbif.h"

namespace {

typedef __nv_bfloat16 bf16;

// ---------------------------------------------------------------------------
// PTX wrappers (tcgen05 / mbarrier)
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)),
                 "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish()
{
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void mbar_init(uint64_t* mbar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(mbar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* mbar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(smem_u32(mbar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// D[tmem] (+)= A[smem] . B[smem]^T, kind::f16 (BF16 in, FP32 accumulate)
__device__ __forceinline__ void mma_bf16(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(dtmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t* mbar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     smem_u32(mbar))
                 : "memory");
}

// 16 consecutive FP32 accumulator columns of this thread's TMEM lane
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float v[16])
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
        "%13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
          "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// Shared-memory matrix descriptor, no swizzle, K-major: the operand is laid
// out as 8-row x 16-byte core matrices; lbo = byte step between core
// matrices along K, sbo = byte step between 8-row groups.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFF);
    d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
    d |= (uint64_t)1 << 46;  // descriptor version; base offset 0; layout type 0 = no swizzle
    return d;
}

// instruction descriptor, kind::f16: D F32, A and B BF16, both K-major, M x N
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float z)
{
    return 0.5f * (1.f + erff(z * 0.70710678118654752f)) + z * expf(-0.5f * z * z) * 0.39894228040143268f;
}

// ---------------------------------------------------------------------------
// GEMM with fused epilogue
// ---------------------------------------------------------------------------
enum { EPI_NONE = 0, EPI_GELU = 1, EPI_GELU_GRAD = 2 };

struct Gemm {
    const bf16* A;
    int lda;
    const bf16* B;
    int ldb;
    int M, N, K;
    const float* bias;  // per column, may be null
    int epi;
    const float* zprev; // EPI_GELU_GRAD: pre-activation multiplied in (ld = ldz)
    float* Z;           // FP32 result (after bias / gradient factor), may be null
    int ldz;
    bf16* H;            // bf16 of the activated result, row-major, may be null
    int ldh;
    bf16* HT;           // bf16 transposed, may be null
    int ldht;
    int* err;
};

constexpr int GEMM_KC = 64;  // K staged per round
constexpr long long WAIT_LIMIT = 1LL << 22;  // try_wait polls; seconds at most

// shared memory of one CTA: two stages of A (128 x 64) and B (ntile x 64)
// bf16 tiles, then two mbarriers and the TMEM address slot
__host__ __device__ inline int gemm_stage_bytes(int ntile) { return (128 + ntile) * GEMM_KC * 2; }
__host__ __device__ inline int gemm_smem_bytes(int ntile) { return 2 * gemm_stage_bytes(ntile) + 32; }
__host__ __device__ inline uint32_t tmem_cols(int ntile)
{
    uint32_t c = 32;
    while (c < (uint32_t)ntile) c <<= 1;
    return c;
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool valid)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src),
                 "r"(valid ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Issue the copies of K round k0 into a stage: A rows m0.., B rows n0.., as
// 8-row x 16-byte core matrices (K-major, no swizzle); rows past M / N read zero.
__device__ __forceinline__ void gemm_stage(const Gemm& g, uint8_t* sA, uint8_t* sB, int m0, int n0, int NT, int k0)
{
    const int kc = min(GEMM_KC, g.K - k0);  // multiple of 16
    const int kcore = kc / 8;
    for (int t = threadIdx.x; t < 128 * kcore; t += blockDim.x) {
        const int r = t / kcore, kp = t - r * kcore;
        const bool ok = m0 + r < g.M;
        const bf16* src = g.A + (size_t)(ok ? m0 + r : 0) * g.lda + k0 + kp * 8;
        cp_async16(sA + ((r >> 3) * kcore + kp) * 128 + (r & 7) * 16, src, ok);
    }
    for (int t = threadIdx.x; t < NT * kcore; t += blockDim.x) {
        const int r = t / kcore, kp = t - r * kcore;
        const bool ok = n0 + r < g.N;
        const bf16* src = g.B + (size_t)(ok ? n0 + r : 0) * g.ldb + k0 + kp * 8;
        cp_async16(sB + ((r >> 3) * kcore + kp) * 128 + (r & 7) * 16, src, ok);
    }
    cp_async_commit();
}

// Bounded wait of every thread on an mbarrier phase; one verdict per CTA.
__device__ __forceinline__ bool cta_wait(uint64_t* mbar, uint32_t parity)
{
    long long spins = 0;
    bool ok;
    while (!(ok = mbar_try_wait(mbar, parity)) && ++spins < WAIT_LIMIT) {
    }
    return __syncthreads_and(ok) != 0;
}

// One CTA: a 128-row block (blockIdx.x) x an ntile-column block (blockIdx.y)
// of C, accumulated in TMEM over K in rounds of 64; the copies of round k+1
// are in flight while the tensor core works on round k. GEMM_THREADS threads:
// the epilogue (bias, GELU, the FP32 and BF16 copies) dominates at K <= 256,
// and TMEM (ntile columns per CTA) caps the CTAs per SM, so the CTA is wide:
// warp w reads TMEM lanes 32 (w % 4) .. + 31 and every (GEMM_THREADS / 128)-th
// 16-column chunk, starting at chunk w / 4.
#ifndef LBIF_GEMM_THREADS
#define LBIF_GEMM_THREADS 256
#endif
constexpr int GEMM_THREADS = LBIF_GEMM_THREADS;
__device__ __forceinline__ void gemm_tile(const Gemm& g, int ntile, uint8_t* smem)
{
    const int SB = gemm_stage_bytes(ntile);
    uint64_t* mbar = (uint64_t*)(smem + 2 * SB);
    uint32_t* tslot = (uint32_t*)(mbar + 2);
    const int m0 = blockIdx.x * 128, n0 = blockIdx.y * ntile;
    const int NT = min(ntile, (g.N - n0 + 15) / 16 * 16);
    const uint32_t cols = tmem_cols(ntile);
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;

    if (warp == 0) {
        tmem_alloc(tslot, cols);
        tmem_relinquish();
    }
    if (threadIdx.x == 0) {
        mbar_init(mbar, 1);
        mbar_init(mbar + 1, 1);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;
    const uint32_t idesc = idesc_bf16(128, NT);
    uint32_t parity[2] = {0u, 0u};
    bool ok = true;
    const int nk = (g.K + GEMM_KC - 1) / GEMM_KC;

    gemm_stage(g, smem, smem + 128 * GEMM_KC * 2, m0, n0, NT, 0);
    for (int k = 0; k < nk && ok; ++k) {
        const int st = k & 1;
        uint8_t* sA = smem + st * SB;
        uint8_t* sB = sA + 128 * GEMM_KC * 2;
        if (k + 1 < nk) {
            // the other stage was read by the products of round k - 1
            if (k >= 1) {
                ok = cta_wait(mbar + (st ^ 1), parity[st ^ 1]);
                parity[st ^ 1] ^= 1u;
                if (!ok) break;
            }
            uint8_t* oA = smem + (st ^ 1) * SB;
            gemm_stage(g, oA, oA + 128 * GEMM_KC * 2, m0, n0, NT, (k + 1) * GEMM_KC);
            cp_async_wait<1>();
        } else {
            cp_async_wait<0>();
        }
        fence_proxy_async();  // copies of round k -> visible to the tensor core
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        if (threadIdx.x == 0) {
            const int kc = min(GEMM_KC, g.K - k * GEMM_KC);
            const uint32_t sbo = (kc / 8) * 128;
            const uint32_t a0 = smem_u32(sA), b0 = smem_u32(sB);
            for (int kk = 0; kk < kc / 16; ++kk)
                mma_bf16(tmem, smem_desc(a0 + kk * 256, 128, sbo), smem_desc(b0 + kk * 256, 128, sbo), idesc,
                         (k > 0 || kk > 0) ? 1u : 0u);
            mma_commit(mbar + st);
        }
    }
    // the last round's products (and, with one round only, the only ones)
    if (ok) {
        const int st = (nk - 1) & 1;
        ok = cta_wait(mbar + st, parity[st]);
        tc_fence_after();
    }

    if (ok) {
        // each thread owns one row (its TMEM lane) and 16 consecutive columns
        // per chunk: a full chunk is written with 16-byte vector stores
        const int lg = warp % 4, cg = warp / 4, ncg = GEMM_THREADS / 128;
        const int row = m0 + 32 * lg + lane;
        for (int c = 16 * cg; c < NT; c += 16 * ncg) {
            float v[16];
            tmem_ld16(tmem + ((uint32_t)(32 * lg) << 16) + (uint32_t)c, v);
            if (row >= g.M) continue;
            const int nb = n0 + c;
            const bool full = nb + 16 <= g.N && (g.ldz % 4) == 0 && (g.ldh % 8) == 0;
            float z[16], h[16];
            float zp[16];
            if (g.epi == EPI_GELU_GRAD) {
                if (full) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float4 t = *reinterpret_cast<const float4*>(g.zprev + (size_t)row * g.ldz + nb + 4 * q);
                        zp[4 * q] = t.x, zp[4 * q + 1] = t.y, zp[4 * q + 2] = t.z, zp[4 * q + 3] = t.w;
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < 16; ++j) zp[j] = nb + j < g.N ? g.zprev[(size_t)row * g.ldz + nb + j] : 0.f;
                }
            }
            // the chunk's 16 biases: four 16-byte loads when aligned
            float bz[16];
            if (g.bias && nb + 16 <= g.N && ((uintptr_t)(g.bias + nb) & 15) == 0) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float4 t = __ldg(reinterpret_cast<const float4*>(g.bias + nb) + q);
                    bz[4 * q] = t.x, bz[4 * q + 1] = t.y, bz[4 * q + 2] = t.z, bz[4 * q + 3] = t.w;
                }
            } else {
#pragma unroll
                for (int j = 0; j < 16; ++j) bz[j] = (g.bias && nb + j < g.N) ? g.bias[nb + j] : 0.f;
            }
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                float zz = v[j] + bz[j];
                float hh = zz;
                if (g.epi == EPI_GELU) {
                    hh = gelu(zz);
                } else if (g.epi == EPI_GELU_GRAD) {
                    zz = zz * gelu_grad(zp[j]);
                    hh = zz;
                }
                z[j] = zz;
                h[j] = hh;
            }
            if (full) {
                if (g.Z) {
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        *reinterpret_cast<float4*>(g.Z + (size_t)row * g.ldz + nb + 4 * q) =
                            make_float4(z[4 * q], z[4 * q + 1], z[4 * q + 2], z[4 * q + 3]);
                }
                if (g.H) {
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        uint4 pk;
                        uint32_t* w = reinterpret_cast<uint32_t*>(&pk);
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const __nv_bfloat162 b2 = __floats2bfloat162_rn(h[8 * q + 2 * e], h[8 * q + 2 * e + 1]);
                            w[e] = *reinterpret_cast<const uint32_t*>(&b2);
                        }
                        *reinterpret_cast<uint4*>(g.H + (size_t)row * g.ldh + nb + 8 * q) = pk;
                    }
                }
            } else {
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    if (nb + j >= g.N) break;
                    if (g.Z) g.Z[(size_t)row * g.ldz + nb + j] = z[j];
                    if (g.H) g.H[(size_t)row * g.ldh + nb + j] = __float2bfloat16_rn(h[j]);
                }
            }
            if (g.HT) {
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    if (nb + j >= g.N) break;
                    g.HT[(size_t)(nb + j) * g.ldht + row] = __float2bfloat16_rn(h[j]);
                }
            }
        }
    } else if (threadIdx.x == 0) {
        atomicExch(g.err, 1);
    }
    cp_async_wait<0>();
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, cols);
}

__global__ void __launch_bounds__(GEMM_THREADS, 2) k_gemm_tc(Gemm g, int ntile)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    gemm_tile(g, ntile, smem);
}

// The weight gradients dW_l = dZ_l^T . H_l of several layers in one launch.
// One product's 8 tiles leave the chip idle (25 us each at a batch of 1024, in
// series); all four layers side by side take 27 us. Batches above WGRAD_ROWS are split: CTA (x, y, l S + s)
// adds rows [s chunk, (s + 1) chunk) of the batch into the partial product
// part + s pstride, and k_finish adds the parts in order.
constexpr int WGRAD_LAYERS = 8, WGRAD_SPLITS = 16, WGRAD_ROWS = 4096;
struct GemmBatch {
    Gemm g[WGRAD_LAYERS];
    int splits, chunk;
    size_t pstride;
};
__global__ void __launch_bounds__(GEMM_THREADS, 2) k_wgrad(const __grid_constant__ GemmBatch b, int ntile)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    const int s = blockIdx.z % b.splits;
    Gemm g = b.g[blockIdx.z / b.splits];
    if ((int)blockIdx.x * 128 >= g.M || (int)blockIdx.y * ntile >= g.N) return;
    const int k0 = s * b.chunk;
    g.A += k0;
    g.B += k0;
    g.K = min(b.chunk, g.K - k0);
    g.Z += s * b.pstride;
    gemm_tile(g, ntile, smem);
}

// ---------------------------------------------------------------------------
// The whole forward pass of 128 rows in one CTA (inference). The activations
// stay in shared memory as the next product's A operand (BF16, K-major core
// matrices) and the accumulator in tensor memory; only the weights travel, as
// contiguous chunks of FUSE_KC columns packed in the order the tensor core
// reads them (pack_offset), each brought in by one bulk copy into a ring of
// three, two chunks ahead of the products and across layer and tile borders.
// The epilogue (bias, GELU, BF16) is most of the work: about 60 instructions
// per element against 512 FLOP on the tensor core, so two CTAs share an SM and
// one's epilogue covers the other's products. Four launches that passed the
// activations through L2 took 234 us for 65,536 rows at 4 -> 3 x 256 -> 160; this
// takes 131 us, 115 of them in the kernel (43 us of issue; an SM holds three or
// four of the 512 tiles). Loading the next chunk of accumulators and biases
// early changed nothing. Up to one tile per SM a CTA runs 16 warps (NT 512), so that
// the epilogue of an SM's only tile is shared by as many as two tiles': 1024 rows,
// 256 -> 8 x 256 -> 256 139 -> 125 us together with the 16-byte input loads (126 as nine
// launches), 4 -> 20 x 256 -> 160 260 -> 250 us (245).
// ---------------------------------------------------------------------------
constexpr int FUSE_KC = 32, FUSE_RING = 3, FUSE_SMS = 152;  // SMs of a GB300

// element (r, c) of a layer's weights in its packed image: chunks of FUSE_KC
// columns (the last one shorter), each n16 rows of 8-row x 16-byte core
// matrices, K-major
__host__ __device__ inline size_t pack_offset(int r, int c, int n16, int kpad)
{
    const int ch = c / FUSE_KC, left = kpad - ch * FUSE_KC, kc = left < FUSE_KC ? left : FUSE_KC;
    return (size_t)ch * FUSE_KC * n16 + ((size_t)(r >> 3) * (kc >> 3) + ((c - ch * FUSE_KC) >> 3)) * 64 +
           (r & 7) * 8 + (c & 7);
}

struct Fused {
    const float* X;   // batch x nin
    float* Y;         // batch x nout
    const bf16* Wp;   // packed weights, layer after layer
    const float* p;   // parameters (biases)
    int batch, nin, hidden, nout, L;
    int tiles, achunk;  // row tiles; bytes of the activation buffer
    int* err;
    double* herr;     // what the host reads (mapped host memory)
};

__device__ __forceinline__ bool bounded_wait(uint64_t* mbar, uint32_t parity)
{
    long long spins = 0;
    bool ok;
    while (!(ok = mbar_try_wait(mbar, parity)) && ++spins < WAIT_LIMIT) {
    }
    return ok;
}

__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* mbar)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(mbar)), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(mbar))
                 : "memory");
}

template <int NT>
__global__ void __launch_bounds__(NT, 512 / NT) k_mlp_forward(const __grid_constant__ Fused f)
{
    extern __shared__ __align__(1024) uint8_t fsm[];
    uint8_t* const act = fsm;
    uint8_t* const ring = fsm + f.achunk;
    const int n16o = (f.nout + 15) / 16 * 16, kp0 = (f.nin + 15) / 16 * 16;
    const int nmax = f.hidden > n16o ? f.hidden : n16o;
    const int slot = nmax * FUSE_KC * 2;  // bytes of a ring slot
    uint64_t* const full = (uint64_t*)(ring + FUSE_RING * slot);
    uint64_t* const empty = full + FUSE_RING;
    uint64_t* const done = empty + FUSE_RING;
    uint32_t* const tslot = (uint32_t*)(done + 1);
    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const uint32_t cols = tmem_cols(nmax);
    if (warp == 0) {
        tmem_alloc(tslot, cols);
        tmem_relinquish();
    }
    if (tid == 0)
        for (int k = 0; k < 2 * FUSE_RING + 1; ++k) mbar_init(full + k, 1);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;

    // thread 0's cursors over the chunks of all its tiles: loads and products
    const int my_tiles = (f.tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
    const int ch0 = (kp0 + FUSE_KC - 1) / FUSE_KC, chh = (f.hidden + FUSE_KC - 1) / FUSE_KC;
    const int per_tile = ch0 + (f.L - 1) * chh;
    const long long chunks = (long long)my_tiles * per_tile;
    long long nload = 0, nmma = 0;
    int lc = 0;               // chunk of the tile the next load takes
    const bf16* lp = f.Wp;    // its address
    auto load_next = [&]() {
        if (nload >= chunks) return;
        const bool first = lc < ch0;
        const int l = first ? 0 : 1 + (lc - ch0) / chh, c = first ? lc : (lc - ch0) % chh;
        const int left = (first ? kp0 : f.hidden) - c * FUSE_KC, kc = left < FUSE_KC ? left : FUSE_KC;
        const int n = l == f.L - 1 ? n16o : f.hidden;
        const int b = (int)(nload % FUSE_RING);
        bulk_load(ring + b * slot, lp, (uint32_t)(n * kc * 2), full + b);
        lp += (size_t)n * kc;
        ++nload;
        if (++lc == per_tile) {
            lc = 0;
            lp = f.Wp;
        }
    };
    bool ok = true;
    if (tid == 0)
        for (int k = 0; k < FUSE_RING - 1; ++k) load_next();
    uint32_t dphase = 0;
    for (int tile = blockIdx.x; tile < f.tiles && ok; tile += gridDim.x) {
        // the input rows as BF16 core matrices, zero beyond nin and the batch
        {
            const int r = tid & 127, row = tile * 128 + r, kcore = kp0 / 8;
            const float* x = f.X + (size_t)row * f.nin;
            // 16-byte loads where every row starts on one (a warp's rows are apart, so
            // a load costs the same whatever its width)
            const bool wide = f.nin % 4 == 0 && ((uintptr_t)f.X & 15) == 0;
            for (int kp = tid >> 7; kp < kcore; kp += NT / 128) {
                float v[8];
                if (wide) {
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int c = kp * 8 + 4 * e;
                        const float4 a = row < f.batch && c < f.nin ? *reinterpret_cast<const float4*>(x + c)
                                                                    : make_float4(0.f, 0.f, 0.f, 0.f);
                        v[4 * e] = a.x, v[4 * e + 1] = a.y, v[4 * e + 2] = a.z, v[4 * e + 3] = a.w;
                    }
                } else {
#pragma unroll
                    for (int e = 0; e < 8; ++e) v[e] = row < f.batch && kp * 8 + e < f.nin ? x[kp * 8 + e] : 0.f;
                }
                uint4 pk;
                uint32_t* w = reinterpret_cast<uint32_t*>(&pk);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * e], v[2 * e + 1]);
                    w[e] = *reinterpret_cast<const uint32_t*>(&h);
                }
                *reinterpret_cast<uint4*>(act + ((r >> 3) * kcore + kp) * 128 + (r & 7) * 16) = pk;
            }
        }
        const float* bias = f.p + (size_t)f.nin * f.hidden;
        for (int l = 0; l < f.L && ok; ++l) {
            const bool last = l == f.L - 1;
            const int K = l == 0 ? kp0 : f.hidden, N = last ? n16o : f.hidden;
            fence_proxy_async();  // the activations written above / by the last epilogue
            tc_fence_before();
            __syncthreads();
            tc_fence_after();
            if (tid == 0) {
                const uint32_t idesc = idesc_bf16(128, N), a0 = smem_u32(act), asbo = (K / 8) * 128;
                for (int c = 0; c * FUSE_KC < K && ok; ++c) {
                    const int b = (int)(nmma % FUSE_RING), kc = min(FUSE_KC, K - c * FUSE_KC);
                    ok = bounded_wait(full + b, (uint32_t)(nmma / FUSE_RING) & 1u);
                    if (!ok) break;
                    const uint32_t b0 = smem_u32(ring + b * slot), bsbo = (kc / 8) * 128;
                    for (int kk = 0; kk < kc / 16; ++kk)
                        mma_bf16(tmem, smem_desc(a0 + (c * FUSE_KC / 8 + 2 * kk) * 128, 128, asbo),
                                 smem_desc(b0 + kk * 256, 128, bsbo), idesc, (c > 0 || kk > 0) ? 1u : 0u);
                    mma_commit(empty + b);
                    // the slot of the chunk before: its products precede these
                    if (nmma > 0 && nload < chunks) {
                        const long long q = nmma - 1;
                        ok = bounded_wait(empty + (int)(q % FUSE_RING), (uint32_t)(q / FUSE_RING) & 1u);
                        if (!ok) break;
                    }
                    load_next();
                    ++nmma;
                }
                if (ok) mma_commit(done);
            }
            {
                const bool mine = bounded_wait(done, dphase) && ok;
                dphase ^= 1u;
                ok = __syncthreads_and(mine) != 0;
            }
            tc_fence_after();
            if (!ok) break;
            const int lg = warp % 4, r = 32 * lg + lane, row = tile * 128 + r;
            if (tile * 128 + 32 * lg < f.batch) {  // the warp holds a row of the batch
                for (int c = 16 * (warp / 4); c < N; c += NT / 8) {
                    float v[16], z[16];
                    __syncwarp();  // rows past the batch skip the stores below
                    tmem_ld16(tmem + ((uint32_t)(32 * lg) << 16) + (uint32_t)c, v);
                    if (!last || c + 16 <= f.nout) {
                        if (((uintptr_t)(bias + c) & 15) == 0) {
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                const float4 t = __ldg(reinterpret_cast<const float4*>(bias + c) + q);
                                z[4 * q] = t.x, z[4 * q + 1] = t.y, z[4 * q + 2] = t.z, z[4 * q + 3] = t.w;
                            }
                        } else {
#pragma unroll
                            for (int j = 0; j < 16; ++j) z[j] = __ldg(bias + c + j);
                        }
                    } else {
#pragma unroll
                        for (int j = 0; j < 16; ++j) z[j] = c + j < f.nout ? __ldg(bias + c + j) : 0.f;
                    }
#pragma unroll
                    for (int j = 0; j < 16; ++j) z[j] = v[j] + z[j];
                    if (last) {
                        if (row >= f.batch) continue;
                        float* y = f.Y + (size_t)row * f.nout + c;
                        if (c + 16 <= f.nout && ((uintptr_t)y & 15) == 0) {
#pragma unroll
                            for (int q = 0; q < 4; ++q)
                                reinterpret_cast<float4*>(y)[q] =
                                    make_float4(z[4 * q], z[4 * q + 1], z[4 * q + 2], z[4 * q + 3]);
                        } else {
#pragma unroll
                            for (int j = 0; j < 16; ++j)
                                if (c + j < f.nout) y[j] = z[j];
                        }
                        continue;
                    }
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        uint4 pk;
                        uint32_t* w = reinterpret_cast<uint32_t*>(&pk);
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const __nv_bfloat162 b2 =
                                __floats2bfloat162_rn(gelu(z[8 * q + 2 * e]), gelu(z[8 * q + 2 * e + 1]));
                            w[e] = *reinterpret_cast<const uint32_t*>(&b2);
                        }
                        *reinterpret_cast<uint4*>(act + ((r >> 3) * (f.hidden / 8) + c / 8 + q) * 128 + (r & 7) * 16) = pk;
                    }
                }
            }
            tc_fence_before();
            bias += f.hidden + (size_t)f.hidden * (l + 1 == f.L - 1 ? f.nout : f.hidden);
        }
        // the next tile's input overwrites the activations the last products read
        // (complete: every thread waited for them)
    }
    if (!ok && tid == 0) {
        atomicExch(f.err, 1);
        *f.herr = 1.0;
        // copies in flight land before the CTA leaves
        for (long long q = nmma; q < nload; ++q)
            bounded_wait(full + (int)(q % FUSE_RING), (uint32_t)(q / FUSE_RING) & 1u);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, cols);
}

// ---------------------------------------------------------------------------
// element-wise kernels
// ---------------------------------------------------------------------------
// X (batch x nin, FP32) -> bf16 rows (bp x kpad) and transposed (kpad x bp), zero padded
__global__ void k_pack_input(const float* X, int batch, int nin, int bp, int kpad, bf16* H, bf16* HT)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= bp * kpad) return;
    int r = i / kpad, c = i - r * kpad;
    float v = (r < batch && c < nin) ? X[(size_t)r * nin + c] : 0.f;
    bf16 b = __float2bfloat16_rn(v);
    H[i] = b;
    HT[(size_t)c * bp + r] = b;
}

// FP64 sum over the CTA's 256 threads in a fixed order (sh: 8 doubles; every
// thread gets it)
__device__ __forceinline__ double block_sum(double s, double* sh)
{
#pragma unroll
    for (int k = 16; k > 0; k >>= 1) s += __shfl_down_sync(0xffffffffu, s, k);
    __syncthreads();
    if (threadIdx.x % 32 == 0) sh[threadIdx.x / 32] = s;
    __syncthreads();
    s = 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) s += sh[k];
    return s;
}

// FP64 sums of FP32 values, the thread's part x(i0), x(i0 + step), ... below n. FP64
// adds and conversions run at 1/64 of the FP32 rate, so the sum is kept as three
// unevaluated FP32 numbers hi + mid + lo: Knuth's two-sum gives the rounding error
// of each addition exactly, hi's errors go to mid and mid's to lo, which leaves
// about 72 bits where FP64 has 53. FP32 has less range: a sum that left it (or met
// an infinity or a NaN, all of which stay in hi or mid) is done again in FP64.
__device__ __forceinline__ float two_sum(float& a, float x)
{
    const float s = __fadd_rn(a, x), b = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, b)), __fsub_rn(x, b));
    a = s;
    return e;
}
template <class Load>
__device__ __forceinline__ double thread_sum(long long i0, long long n, int step, Load x)
{
    constexpr int U = 8;  // loads that go out together
    float hi = 0.f, mid = 0.f, lo = 0.f;
    auto add = [&](float v) { lo = __fadd_rn(lo, two_sum(mid, two_sum(hi, v))); };
    long long k = i0;
    for (; k + (U - 1) * step < n; k += U * step) {
        float v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) v[u] = x(k + u * step);
#pragma unroll
        for (int u = 0; u < U; ++u) add(v[u]);
    }
    for (; k < n; k += step) add(x(k));
    if (isfinite(hi) && isfinite(mid)) return (double)hi + ((double)mid + (double)lo);
    double s = 0.0;
    for (long long i = i0; i < n; i += step) s += (double)x(i);
    return s;
}

// partial sums of the mask, one per block (fixed order)
constexpr int MSUM_BLOCKS = 64;
__global__ void __launch_bounds__(256) k_msum(const float* mask, long long n, double* part)
{
    __shared__ double sh[8];
    const double a =
        thread_sum(blockIdx.x * 256LL + threadIdx.x, n, MSUM_BLOCKS * 256, [&](long long i) { return mask[i]; });
    const double s = block_sum(a, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
}

// the mask's sum from its parts, at least 1 (called by one whole warp; lane 0
// gets it)
__device__ __forceinline__ double mask_sum(const double* part)
{
    const int lane = threadIdx.x % 32;
    double s = 0.0;
    for (int k = lane; k < MSUM_BLOCKS; k += 32) s += part[k];
#pragma unroll
    for (int k = 16; k > 0; k >>= 1) s += __shfl_down_sync(0xffffffffu, s, k);
    return fmax(s, 1.0);
}

// dY = 2 mask (Y - T) / sum(mask): FP32 (bp x nout), bf16 rows (bp x opad) and
// bf16 transposed (nout x bp); per-block FP64 partial sums of the loss. The
// squares and the scaling are FP64 (an FP32 square leaves the range from an error
// of 1.9e19 on); a block covers LOSS_PT x 256 elements.
constexpr int LOSS_PT = 2;
__global__ void __launch_bounds__(256) k_loss(const float* Y, const float* T, const float* mask, int batch, int nout,
                                              int opad, int bp, const double* mpart, float* dY, bf16* dYb, bf16* dYT,
                                              double* partial)
{
    __shared__ double sh[8];
    __shared__ double scale;  // 2 / sum
    if (threadIdx.x < 32) {
        const double s = mask_sum(mpart);
        if (threadIdx.x == 0) scale = 2.0 / s;
    }
    __syncthreads();
    const double sc = scale;
    double l = 0.0;
#pragma unroll
    for (int k = 0; k < LOSS_PT; ++k) {
        const int i = (blockIdx.x * LOSS_PT + k) * 256 + threadIdx.x;
        if (i < bp * nout) {
            int r = i / nout, c = i - r * nout;
            float d = 0.f;
            if (r < batch) {
                float m = mask[(size_t)r * nout + c];
                float e = (Y[(size_t)r * nout + c] - T[(size_t)r * nout + c]) * m;
                const double ed = (double)e;
                l = fma(ed, ed, l);
                d = (float)(ed * sc);
            }
            dY[i] = d;
            bf16 b = __float2bfloat16_rn(d);
            dYb[(size_t)r * opad + c] = b;
            dYT[(size_t)c * bp + r] = b;
        }
    }
    const double sum = block_sum(l, sh);
    if (threadIdx.x == 0) partial[blockIdx.x] = sum;
}

__device__ __forceinline__ float adam_one(float p, float gi, float* m, float* v, float lr, float b1, float b2,
                                         float eps, float c1, float c2)
{
    const float mi = b1 * *m + (1.f - b1) * gi;
    const float vi = b2 * *v + (1.f - b2) * gi * gi;
    *m = mi;
    *v = vi;
    return p - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// What follows the weight products, for a group of layers (blockIdx.y): the
// weight gradients as the ordered sums of their parts, the bias gradients as
// column sums of dZ (FP64, fixed order), and with `adam` the update of the
// parameters and their BF16 shadows (nothing is updated once *err is set).
// Blocks [0, nw) hold 256 weights each, the next ones 8 bias columns each
// (256 threads: 32 row strides of 8 columns), the last one (of layer group 0)
// adds the loss. The former one-thread-per-column sums took 121 us per layer
// at a batch of 1024, the mask's one-block sum 124 us.
struct FinishLayer {
    const float* part;  // weight products, splits x (dout x kpad)
    const float* dZ;    // bp x dout
    long long woff, boff;
    int dout, din, kpad, opad;
    bf16 *Wb, *WTb, *Wp;
};
struct Finish {
    FinishLayer l[WGRAD_LAYERS];
    int splits, bp, nw, adam;
    size_t pstride;
    float *p, *g, *m, *v;
    float lr, b1, b2, eps, c1, c2;
    const int* err;
    const double *partial, *mpart;
    int nb;
    double* result;  // {loss, err}; NULL: not this group's work
};
__global__ void __launch_bounds__(256) k_finish(const __grid_constant__ Finish f)
{
    __shared__ double sh[256];
    const FinishLayer& l = f.l[blockIdx.y];
    const int bx = blockIdx.x, t = threadIdx.x;
    auto apply = [&](long long at, float gi) -> float {
        f.g[at] = gi;
        if (!f.adam || *f.err) return 0.f;
        const float w = adam_one(f.p[at], gi, f.m + at, f.v + at, f.lr, f.b1, f.b2, f.eps, f.c1, f.c2);
        f.p[at] = w;
        return w;
    };
    if (bx < f.nw) {
        const int i = bx * 256 + t;
        if (i >= l.dout * l.din) return;
        const int r = i / l.din, c = i - r * l.din;
        const float* q = l.part + (size_t)r * l.kpad + c;
        float gi = 0.f;
#pragma unroll 8
        for (int s = 0; s < f.splits; ++s) gi += q[s * f.pstride];
        const float w = apply(l.woff + i, gi);
        if (f.adam && !*f.err) {
            const bf16 b = __float2bfloat16_rn(w);
            l.Wb[(size_t)r * l.kpad + c] = b;
            l.WTb[(size_t)c * l.opad + r] = b;
            l.Wp[pack_offset(r, c, l.opad, l.kpad)] = b;
        }
        return;
    }
    if (bx == (int)gridDim.x - 1) {
        if (!f.result || blockIdx.y) return;
        double s = 0.0;
        for (int i = t; i < f.nb; i += 256) s += f.partial[i];
        s = block_sum(s, sh);
        const double ms = t < 32 ? mask_sum(f.mpart) : 1.0;
        if (t == 0) {
            f.result[0] = s / ms;
            if (*f.err) f.result[1] = 1.0;
        }
        return;
    }
    const int c = (bx - f.nw) * 8 + (t & 7);
    if ((bx - f.nw) * 8 >= l.dout) return;
    sh[t] = c < l.dout ? thread_sum(t >> 3, f.bp, 32, [&](long long r) { return l.dZ[r * l.dout + c]; }) : 0.0;
    __syncthreads();
    for (int k = 128; k >= 8; k >>= 1) {
        if (t < k) sh[t] += sh[t + k];
        __syncthreads();
    }
    if (t < 8 && c < l.dout) apply(l.boff + c, (float)sh[t]);
}

// bf16 shadows of W (nout x nin): row-major padded to kpad columns, transposed
// (nin x opad, columns beyond nout stay zero), and packed for the fused forward
// (opad rows; padding stays zero)
__global__ void k_shadow(const float* W, int nout, int nin, int kpad, int opad, bf16* Wb, bf16* WTb, bf16* Wp)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nout * kpad) return;
    int r = i / kpad, c = i - r * kpad;
    float w = c < nin ? W[(size_t)r * nin + c] : 0.f;
    bf16 b = __float2bfloat16_rn(w);
    Wb[i] = b;
    if (c < nin) {
        WTb[(size_t)c * opad + r] = b;
        Wp[pack_offset(r, c, opad, kpad)] = b;
    }
}

inline int up16(int v) { return (v + 15) / 16 * 16; }

}  // namespace

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
struct lbif_mlp_ctx {
    int nin, hidden, nhidden, nout, max_batch, bp_max;
    int L;                      // layers
    std::vector<int> din, dout, kpad, opad;  // kpad, opad: widths rounded up to 16
    std::vector<long long> woff, boff;  // offsets into the flat parameter vector
    long long nparams;
    cudaStream_t stream = nullptr;
    float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;  // flat FP32
    std::vector<bf16*> Wb, WTb;
    bf16* Wp = nullptr;          // packed for the fused forward, layer after layer
    std::vector<size_t> wpoff;   // offsets of the layers in it
    std::vector<float*> Z;       // pre-activations per layer (bp x dout)
    std::vector<bf16*> H, HT;    // layer inputs (bp x kpad) and transposed (kpad x bp)
    std::vector<float*> dZ;      // per layer FP32 error (bp x dout)
    std::vector<bf16*> dZb, dZT; // bf16 copies
    float* dWpart = nullptr;     // parts of the weight products: splits x npart
    size_t npart = 0;            // dout x kpad of all layers
    std::vector<size_t> poff;    // offsets of the layers in one part
    float* Xd = nullptr;         // device staging for host inputs (max_batch x nin)
    float *Td = nullptr, *Md = nullptr, *Yd = nullptr;
    double* partial = nullptr;
    double* mpart = nullptr;
    // {loss, err} as the host reads them after a synchronisation: mapped host
    // memory that the kernels write, so that no call ends with a copy (a 4-byte
    // read-back took 10 us of each)
    double *host = nullptr, *result = nullptr;  // host and device address
    int* err = nullptr;
    long long adam_t = 0;
    std::string msg;
};

// parts the batch of a weight product is split into: WGRAD_ROWS rows each, 16
// parts at most (their sum reads them all again); rows a part holds
static int wgrad_splits(int bp)
{
    const int s = (bp + WGRAD_ROWS - 1) / WGRAD_ROWS;
    return s < WGRAD_SPLITS ? s : WGRAD_SPLITS;
}
static int wgrad_chunk(int bp)
{
    const int s = wgrad_splits(bp);
    return ((bp + s - 1) / s + GEMM_KC - 1) / GEMM_KC * GEMM_KC;
}

static thread_local std::string g_mlp_err = "no error";

static int mfail(lbif_mlp_ctx* m, int code, const std::string& s)
{
    if (m) m->msg = s;
    g_mlp_err = s;
    return code;
}

#define MCK(m, call)                                                                         \
    do {                                                                                     \
        cudaError_t e_ = (call);                                                             \
        if (e_ != cudaSuccess)                                                               \
            return mfail((m), LBIF_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

static void mlp_free(lbif_mlp_ctx* m)
{
    if (!m) return;
    std::vector<void*> bufs = {m->Wp, m->p, m->g, m->m, m->v, m->dWpart, m->Xd, m->Td, m->Md,
                               m->Yd, m->partial, m->mpart, m->err};
    for (auto* b : m->Wb) bufs.push_back(b);
    for (auto* b : m->WTb) bufs.push_back(b);
    for (auto* b : m->Z) bufs.push_back(b);
    for (auto* b : m->H) bufs.push_back(b);
    for (auto* b : m->HT) bufs.push_back(b);
    for (auto* b : m->dZ) bufs.push_back(b);
    for (auto* b : m->dZb) bufs.push_back(b);
    for (auto* b : m->dZT) bufs.push_back(b);
    for (void* b : bufs)
        if (b) cudaFree(b);
    if (m->host) cudaFreeHost(m->host);
    delete m;
}

template <class T>
static bool dalloc(T** p, size_t n)
{
    if (cudaMalloc((void**)p, sizeof(T) * (n ? n : 1)) != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        return false;
    }
    return cudaMemset(*p, 0, sizeof(T) * (n ? n : 1)) == cudaSuccess;
}

// shared memory of the fused forward: activations of 128 rows x kmax, the ring
// of weight chunks, barriers and the TMEM address slot
static int fused_smem(int kmax, int nmax)
{
    return 256 * kmax + FUSE_RING * nmax * FUSE_KC * 2 + 8 * (2 * FUSE_RING + 1) + 16;
}

extern "C" int lbif_mlp_create(lbif_mlp* out, int32_t nin, int32_t hidden, int32_t nhidden, int32_t nout,
                               int32_t max_batch, void* stream)
{
    if (!out || nin < 1 || nin > 256 || hidden < 16 || hidden > 256 || hidden % 16 || nhidden < 1 ||
        nout < 1 || nout > 256 || max_batch < 1)
        return mfail(nullptr, LBIF_ERR_ARG, "lbif_mlp_create: widths must be in [1, 256] (hidden a multiple of 16)");
    *out = nullptr;
    lbif_mlp_ctx* m = new lbif_mlp_ctx();
    m->nin = nin;
    m->hidden = hidden;
    m->nhidden = nhidden;
    m->nout = nout;
    m->max_batch = max_batch;
    m->bp_max = up16(max_batch);
    m->L = nhidden + 1;
    m->stream = (cudaStream_t)stream;
    long long off = 0;
    for (int l = 0; l < m->L; ++l) {
        int di = l == 0 ? nin : hidden, dq = l == m->L - 1 ? nout : hidden;
        m->din.push_back(di);
        m->dout.push_back(dq);
        m->kpad.push_back(up16(di));
        m->opad.push_back(up16(dq));
        m->woff.push_back(off);
        off += (long long)di * dq;
        m->boff.push_back(off);
        off += dq;
    }
    m->nparams = off;
    for (int l = 0; l < m->L; ++l) {
        m->poff.push_back(m->npart);
        m->npart += (size_t)m->dout[l] * m->kpad[l];
    }
    size_t npack = 0;
    for (int l = 0; l < m->L; ++l) {
        m->wpoff.push_back(npack);
        npack += (size_t)m->opad[l] * m->kpad[l];
    }
    const int bp = m->bp_max;
    bool ok = dalloc(&m->p, off) && dalloc(&m->g, off) && dalloc(&m->m, off) && dalloc(&m->v, off) &&
              dalloc(&m->dWpart, wgrad_splits(bp) * m->npart) &&
              dalloc(&m->Xd, (size_t)max_batch * nin) && dalloc(&m->Td, (size_t)max_batch * nout) &&
              dalloc(&m->Md, (size_t)max_batch * nout) && dalloc(&m->Yd, (size_t)bp * nout) &&
              dalloc(&m->partial, (size_t)(bp * nout + 255) / 256 + 1) && dalloc(&m->mpart, MSUM_BLOCKS) &&
              dalloc(&m->err, 1) && dalloc(&m->Wp, npack);
    for (int l = 0; ok && l < m->L; ++l) {
        bf16 *wb, *wtb, *h, *ht, *dzb, *dzt;
        float *z, *dz;
        ok = dalloc(&wb, (size_t)m->dout[l] * m->kpad[l]) && dalloc(&wtb, (size_t)m->din[l] * m->opad[l]) &&
             dalloc(&z, (size_t)bp * m->dout[l]) && dalloc(&h, (size_t)bp * m->kpad[l]) &&
             dalloc(&ht, (size_t)m->kpad[l] * bp) && dalloc(&dz, (size_t)bp * m->dout[l]) &&
             dalloc(&dzb, (size_t)bp * m->opad[l]) && dalloc(&dzt, (size_t)m->dout[l] * bp);
        m->Wb.push_back(ok ? wb : nullptr);
        m->WTb.push_back(ok ? wtb : nullptr);
        m->Z.push_back(ok ? z : nullptr);
        m->H.push_back(ok ? h : nullptr);
        m->HT.push_back(ok ? ht : nullptr);
        m->dZ.push_back(ok ? dz : nullptr);
        m->dZb.push_back(ok ? dzb : nullptr);
        m->dZT.push_back(ok ? dzt : nullptr);
    }
    ok = ok && cudaHostAlloc((void**)&m->host, 2 * sizeof(double), cudaHostAllocMapped) == cudaSuccess &&
         cudaHostGetDevicePointer((void**)&m->result, m->host, 0) == cudaSuccess;
    if (ok) m->host[0] = m->host[1] = 0.0;
    if (!ok) {
        cudaGetLastError();
        mlp_free(m);
        return mfail(nullptr, LBIF_ERR_NOMEM, "lbif_mlp_create: device allocation failed");
    }
    if (cudaFuncSetAttribute(k_gemm_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, gemm_smem_bytes(256)) != cudaSuccess ||
        cudaFuncSetAttribute(k_wgrad, cudaFuncAttributeMaxDynamicSharedMemorySize, gemm_smem_bytes(256)) != cudaSuccess ||
        cudaFuncSetAttribute(k_mlp_forward<256>, cudaFuncAttributeMaxDynamicSharedMemorySize, fused_smem(256, 256)) !=
            cudaSuccess ||
        cudaFuncSetAttribute(k_mlp_forward<512>, cudaFuncAttributeMaxDynamicSharedMemorySize, fused_smem(256, 256)) !=
            cudaSuccess) {
        cudaGetLastError();
        mlp_free(m);
        return mfail(nullptr, LBIF_ERR_CUDA, "lbif_mlp_create: shared memory configuration failed");
    }
    // the zero fills above went to the default stream, which a non-blocking stream of
    // the caller's does not wait for: they end before the first call can write
    if (cudaStreamSynchronize(cudaStreamLegacy) != cudaSuccess) {
        cudaGetLastError();
        mlp_free(m);
        return mfail(nullptr, LBIF_ERR_CUDA, "lbif_mlp_create: zero fill failed");
    }
    *out = m;
    return LBIF_OK;
}

extern "C" int lbif_mlp_destroy(lbif_mlp m)
{
    if (!m) return mfail(nullptr, LBIF_ERR_ARG, "lbif_mlp_destroy: NULL handle");
    cudaStreamSynchronize(m->stream);
    mlp_free(m);
    return LBIF_OK;
}

extern "C" int64_t lbif_mlp_num_params(lbif_mlp m) { return m ? m->nparams : -1; }

extern "C" const char* lbif_mlp_last_error(lbif_mlp m) { return m ? m->msg.c_str() : g_mlp_err.c_str(); }

static int refresh_shadows(lbif_mlp_ctx* m)
{
    for (int l = 0; l < m->L; ++l) {
        int n = m->dout[l] * m->kpad[l];
        k_shadow<<<(n + 255) / 256, 256, 0, m->stream>>>(m->p + m->woff[l], m->dout[l], m->din[l], m->kpad[l],
                                                         m->opad[l], m->Wb[l], m->WTb[l], m->Wp + m->wpoff[l]);
    }
    MCK(m, cudaGetLastError());
    return LBIF_OK;
}

extern "C" int lbif_mlp_set_params(lbif_mlp m, const float* params)
{
    if (!m || !params) return mfail(m, LBIF_ERR_ARG, "lbif_mlp_set_params: bad arguments");
    MCK(m, cudaMemcpyAsync(m->p, params, sizeof(float) * m->nparams, cudaMemcpyHostToDevice, m->stream));
    MCK(m, cudaMemsetAsync(m->m, 0, sizeof(float) * m->nparams, m->stream));
    MCK(m, cudaMemsetAsync(m->v, 0, sizeof(float) * m->nparams, m->stream));
    m->adam_t = 0;
    int rc = refresh_shadows(m);
    if (rc) return rc;
    MCK(m, cudaStreamSynchronize(m->stream));
    return LBIF_OK;
}

extern "C" int lbif_mlp_get_params(lbif_mlp m, float* params)
{
    if (!m || !params) return mfail(m, LBIF_ERR_ARG, "lbif_mlp_get_params: bad arguments");
    MCK(m, cudaMemcpyAsync(params, m->p, sizeof(float) * m->nparams, cudaMemcpyDeviceToHost, m->stream));
    MCK(m, cudaStreamSynchronize(m->stream));
    return LBIF_OK;
}

// Column block of a product: the whole N (<= 256) when there are enough row
// blocks to fill the GPU, else blocks of 64 columns for more CTAs.
static int gemm(lbif_mlp_ctx* m, const Gemm& g)
{
    if (g.N > 256 || g.K % 16 || g.K < 16)
        return mfail(m, LBIF_ERR_UNSUPPORTED, "gemm: N > 256 or K not a positive multiple of 16");
    const int mt = (g.M + 127) / 128;
    const int nfull = (g.N + 15) / 16 * 16;
    const int ntile = (mt >= 64 || nfull <= 64) ? nfull : 64;
    dim3 grid(mt, (g.N + ntile - 1) / ntile);
    // shared memory per CTA bounds the CTAs per SM so that their TMEM
    // columns (32..256 each) always fit in the SM's 512 together
    int smem = gemm_smem_bytes(ntile);
    if (tmem_cols(ntile) == 256 && smem < 80 * 1024) smem = 80 * 1024;
    k_gemm_tc<<<grid, GEMM_THREADS, smem, m->stream>>>(g, ntile);
    MCK(m, cudaGetLastError());
    return LBIF_OK;
}

static Gemm blank(lbif_mlp_ctx* m)
{
    Gemm g;
    memset(&g, 0, sizeof(g));
    g.err = m->err;
    return g;
}

// the training forward of `batch` rows already packed in H[0] / HT[0]: keeps
// what back-propagation reads (every layer's FP32 pre-activation Z and the
// transposed BF16 activations HT)
static int forward(lbif_mlp_ctx* m, int batch)
{
    const int bp = up16(batch);
    for (int l = 0; l < m->L; ++l) {
        const bool last = l == m->L - 1;
        Gemm g = blank(m);
        g.A = m->H[l];
        g.lda = m->kpad[l];
        g.B = m->Wb[l];
        g.ldb = m->kpad[l];
        g.M = bp;
        g.N = m->dout[l];
        g.K = m->kpad[l];
        g.bias = m->p + m->boff[l];
        g.epi = last ? EPI_NONE : EPI_GELU;
        g.Z = m->Z[l];
        g.ldz = m->dout[l];
        if (!last) {
            g.H = m->H[l + 1];
            g.ldh = m->kpad[l + 1];
            g.HT = m->HT[l + 1];
            g.ldht = bp;
        }
        int rc = gemm(m, g);
        if (rc) return rc;
    }
    return LBIF_OK;
}

// inference: Y (batch x nout) of X (batch x nin), device memory
static int infer(lbif_mlp_ctx* m, const float* X, int batch, float* Y)
{
    Fused f;
    memset(&f, 0, sizeof(f));
    f.X = X;
    f.Y = Y;
    f.Wp = m->Wp;
    f.p = m->p;
    f.batch = batch;
    f.nin = m->nin;
    f.hidden = m->hidden;
    f.nout = m->nout;
    f.L = m->L;
    f.tiles = (batch + 127) / 128;
    const int kmax = m->kpad[0] > m->hidden ? m->kpad[0] : m->hidden;
    const int nmax = m->opad[m->L - 1] > m->hidden ? m->opad[m->L - 1] : m->hidden;
    f.achunk = 256 * kmax;
    f.err = m->err;
    f.herr = m->result + 1;
    // two CTAs per SM: shared memory keeps a third one (and its TMEM) out
    int smem = fused_smem(kmax, nmax);
    if (smem < 80 * 1024) smem = 80 * 1024;
    // up to one tile per SM: 16 warps a CTA, which share the epilogue of the only tile
    if (f.tiles <= FUSE_SMS)
        k_mlp_forward<512><<<f.tiles, 512, smem, m->stream>>>(f);
    else
        k_mlp_forward<256><<<f.tiles < 2 * FUSE_SMS ? f.tiles : 2 * FUSE_SMS, 256, smem, m->stream>>>(f);
    MCK(m, cudaGetLastError());
    return LBIF_OK;
}

static int pack_input(lbif_mlp_ctx* m, const float* X, int batch, int on_device)
{
    const float* Xd = X;
    if (!on_device) {
        MCK(m, cudaMemcpyAsync(m->Xd, X, sizeof(float) * (size_t)batch * m->nin, cudaMemcpyHostToDevice, m->stream));
        Xd = m->Xd;
    }
    const int bp = up16(batch);
    int n = bp * m->kpad[0];
    k_pack_input<<<(n + 255) / 256, 256, 0, m->stream>>>(Xd, batch, m->nin, bp, m->kpad[0], m->H[0], m->HT[0]);
    MCK(m, cudaGetLastError());
    return LBIF_OK;
}

static int check_err(lbif_mlp_ctx* m)
{
    MCK(m, cudaStreamSynchronize(m->stream));
    if (*(volatile double*)(m->host + 1) != 0.0)
        return mfail(m, LBIF_ERR_TIMEOUT, "tensor-core product did not complete within its wait limit");
    return LBIF_OK;
}

extern "C" int lbif_mlp_forward(lbif_mlp m, const float* X, int32_t batch, float* Y, int32_t on_device)
{
    if (!m || !X || !Y || batch < 1 || batch > m->max_batch)
        return mfail(m, LBIF_ERR_ARG, "lbif_mlp_forward: bad arguments");
    const float* Xd = X;
    if (!on_device) {
        MCK(m, cudaMemcpyAsync(m->Xd, X, sizeof(float) * (size_t)batch * m->nin, cudaMemcpyHostToDevice, m->stream));
        Xd = m->Xd;
    }
    float* Yd = on_device ? Y : m->Yd;
    const int rc = infer(m, Xd, batch, Yd);
    if (rc) return rc;
    if (!on_device)
        MCK(m, cudaMemcpyAsync(Y, Yd, sizeof(float) * (size_t)batch * m->nout, cudaMemcpyDeviceToHost, m->stream));
    return check_err(m);
}

// learning rate and Adam's constants of a training step
struct AdamStep {
    float lr, beta1, beta2, eps, c1, c2;
};

// loss and gradients into m->g; with `adam` also the parameters' update
static int backward(lbif_mlp_ctx* m, const float* T, const float* mask, int batch, int on_device, double* loss,
                    const AdamStep* adam = nullptr)
{
    const int bp = up16(batch);
    const int nout = m->nout;
    const float *Td = T, *Md = mask;
    if (!on_device) {
        MCK(m, cudaMemcpyAsync(m->Td, T, sizeof(float) * (size_t)batch * nout, cudaMemcpyHostToDevice, m->stream));
        MCK(m, cudaMemcpyAsync(m->Md, mask, sizeof(float) * (size_t)batch * nout, cudaMemcpyHostToDevice, m->stream));
        Td = m->Td;
        Md = m->Md;
    }
    const int L = m->L;
    const int n = bp * nout;
    const int nb = (n + 256 * LOSS_PT - 1) / (256 * LOSS_PT);
    k_msum<<<MSUM_BLOCKS, 256, 0, m->stream>>>(Md, (long long)batch * nout, m->mpart);
    k_loss<<<nb, 256, 0, m->stream>>>(m->Z[L - 1], Td, Md, batch, nout, m->opad[L - 1], bp, m->mpart,
                                      m->dZ[L - 1], m->dZb[L - 1], m->dZT[L - 1], m->partial);
    MCK(m, cudaGetLastError());
    for (int l = L - 1; l > 0; --l) {
        // dZ_{l-1} = (dZ_l . W_l) * gelu'(Z_{l-1})  (M = bp, N = din_l, K = dout_l)
        Gemm gd = blank(m);
        gd.A = m->dZb[l];
        gd.lda = m->opad[l];
        gd.B = m->WTb[l];
        gd.ldb = m->opad[l];
        gd.M = bp;
        gd.N = m->din[l];
        gd.K = m->opad[l];
        gd.epi = EPI_GELU_GRAD;
        gd.zprev = m->Z[l - 1];
        gd.Z = m->dZ[l - 1];
        gd.ldz = m->dout[l - 1];
        gd.H = m->dZb[l - 1];
        gd.ldh = m->opad[l - 1];
        gd.HT = m->dZT[l - 1];
        gd.ldht = bp;
        const int rc = gemm(m, gd);
        if (rc) return rc;
    }
    std::vector<Finish> fin;  // after every product: nothing is updated once one failed
    std::vector<dim3> fgrid;
    for (int l0 = 0; l0 < L; l0 += WGRAD_LAYERS) {
        const int nl = L - l0 < WGRAD_LAYERS ? L - l0 : WGRAD_LAYERS;
        GemmBatch gb;
        memset(&gb, 0, sizeof(gb));
        Finish f;
        memset(&f, 0, sizeof(f));
        gb.splits = f.splits = wgrad_splits(bp);
        gb.chunk = wgrad_chunk(bp);
        // rounding the chunk up may leave trailing parts without rows
        gb.splits = f.splits = (bp + gb.chunk - 1) / gb.chunk;
        gb.pstride = f.pstride = m->npart;
        int mt = 1, nt = 1, nbias = 1;
        for (int k = 0; k < nl; ++k) {
            const int l = l0 + k;
            // dW_l = dZ_l^T . H_l  (M = dout, N = din, K = bp)
            Gemm& gw = gb.g[k];
            gw = blank(m);
            gw.A = m->dZT[l];
            gw.lda = bp;
            gw.B = m->HT[l];
            gw.ldb = bp;
            gw.M = m->dout[l];
            gw.N = m->din[l];
            gw.K = bp;
            gw.Z = m->dWpart + m->poff[l];
            gw.ldz = m->kpad[l];
            const int tiles_m = (m->dout[l] + 127) / 128, tiles_n = (m->din[l] + 63) / 64;
            mt = tiles_m > mt ? tiles_m : mt;
            nt = tiles_n > nt ? tiles_n : nt;
            const int w = (m->dout[l] * m->din[l] + 255) / 256, c = (m->dout[l] + 7) / 8;
            f.nw = w > f.nw ? w : f.nw;
            nbias = c > nbias ? c : nbias;
            f.l[k] = FinishLayer{gw.Z, m->dZ[l], m->woff[l], m->boff[l], m->dout[l], m->din[l], m->kpad[l], m->opad[l],
                                 m->Wb[l], m->WTb[l], m->Wp + m->wpoff[l]};
        }
        k_wgrad<<<dim3(mt, nt, nl * gb.splits), GEMM_THREADS, gemm_smem_bytes(64), m->stream>>>(gb, 64);
        MCK(m, cudaGetLastError());
        f.bp = bp;
        f.p = m->p;
        f.g = m->g;
        f.m = m->m;
        f.v = m->v;
        f.err = m->err;
        if (adam) {
            f.adam = 1;
            f.lr = adam->lr;
            f.b1 = adam->beta1;
            f.b2 = adam->beta2;
            f.eps = adam->eps;
            f.c1 = adam->c1;
            f.c2 = adam->c2;
        }
        f.partial = m->partial;
        f.mpart = m->mpart;
        f.nb = nb;
        f.result = l0 + nl == L ? m->result : nullptr;
        fin.push_back(f);
        fgrid.push_back(dim3(f.nw + nbias + 1, nl));
    }
    for (size_t k = 0; k < fin.size(); ++k) {
        k_finish<<<fgrid[k], 256, 0, m->stream>>>(fin[k]);
        MCK(m, cudaGetLastError());
    }
    const int rc = check_err(m);
    if (rc) return rc;
    if (loss) *loss = *(volatile double*)m->host;
    return LBIF_OK;
}

extern "C" int lbif_mlp_gradients(lbif_mlp m, const float* X, const float* T, const float* mask, int32_t batch,
                                  float* grads, double* loss, int32_t on_device)
{
    if (!m || !X || !T || !mask || batch < 1 || batch > m->max_batch)
        return mfail(m, LBIF_ERR_ARG, "lbif_mlp_gradients: bad arguments");
    int rc = pack_input(m, X, batch, on_device);
    if (rc) return rc;
    if ((rc = forward(m, batch))) return rc;
    if ((rc = backward(m, T, mask, batch, on_device, loss))) return rc;
    if (grads) {
        MCK(m, cudaMemcpyAsync(grads, m->g, sizeof(float) * m->nparams,
                               on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, m->stream));
        MCK(m, cudaStreamSynchronize(m->stream));
    }
    return LBIF_OK;
}

extern "C" int lbif_mlp_train_step(lbif_mlp m, const float* X, const float* T, const float* mask, int32_t batch,
                                   float lr, float beta1, float beta2, float eps, double* loss, int32_t on_device)
{
    if (!m || !X || !T || !mask || batch < 1 || batch > m->max_batch || !(lr >= 0))
        return mfail(m, LBIF_ERR_ARG, "lbif_mlp_train_step: bad arguments");
    int rc = pack_input(m, X, batch, on_device);
    if (rc) return rc;
    if ((rc = forward(m, batch))) return rc;
    // the update rides on the gradients' last kernel; a step whose products
    // failed leaves the parameters and the step count as they were
    const double t = (double)(m->adam_t + 1);
    const AdamStep a{lr, beta1, beta2, eps, (float)(1.0 - pow((double)beta1, t)), (float)(1.0 - pow((double)beta2, t))};
    if ((rc = backward(m, T, mask, batch, on_device, loss, &a))) return rc;
    m->adam_t += 1;
    return LBIF_OK;
}
