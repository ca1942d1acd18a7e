// Link-travel-time surrogate MLP on the 5th-generation tensor cores.
//
// Network: inputs (padded to 64) -> 256 -> 256 -> 256 -> 1, GELU after each
// hidden layer, BF16 weights and activations, FP32 accumulation, MSE loss,
// Adam.  Four kernels:
//   mlp_forward_fused  inference: all layers of a 128-row tile in one CTA
//   mlp_train_fused    training: forward and backward of a 128-row tile in a
//                      cluster of two CTAs (each half the columns of every layer)
//   mlp_wgrad          dW_l = dZ_l^T . H_{l-1}, split over the samples
//   mlp_update         split sums, gradients and the Adam step
// and a plain GEMM D = A . B^T (gemm_bf16_tn, the diagnostic entry).  All use
// TMA loads (128-byte swizzle) into mbarrier-guarded shared memory, one thread
// issuing tcgen05.mma into tensor memory and tcgen05.ld in the epilogues.
// Every wait on an mbarrier is bounded; on timeout the kernel records an
// error, stops issuing work and frees its tensor memory before returning.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <random>
#include <string>
#include <vector>

#include "../../include/lpsim_surrogate.h"
#include "ctx.h"

namespace {

int fail(int code, const std::string &m) { return lpsim_fail(code, m); }

#define CU(call)                                                                                            \
    do {                                                                                                    \
        cudaError_t e_ = (call);                                                                            \
        if (e_ != cudaSuccess) return fail(LPSIM_E_CUDA, std::string(#call ": ") + cudaGetErrorString(e_)); \
    } while (0)
#define TRY(x)                           \
    do {                                 \
        int rc_ = (x);                   \
        if (rc_ != LPSIM_OK) return rc_; \
    } while (0)

constexpr int kBM = 128;
constexpr int kBK = 64;  // one 128-byte swizzle atom of BF16
constexpr int kStages = 4;
constexpr uint32_t kSpinLimit = 1u << 26;

constexpr int kThreads = 256;  // eight warps: all take part in the epilogue

struct GemmArgs {
    int M, N, K;
    float *fout;  // M x N
    uint32_t *err;
};

// ----------------------------------------------------------- device helpers

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

// bounded wait for the phase with the given parity to complete; false on timeout
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity) {
    const uint32_t a = smem_u32(bar);
    for (uint32_t i = 0; i < kSpinLimit; i++) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, uint64_t *bar, int x, int y) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(
            smem_u32(dst)),
        "l"((uint64_t)map), "r"(smem_u32(bar)), "r"(x), "r"(y)
        : "memory");
}

// shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups
// 1024 bytes apart
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFF) >> 4);  // start address
    d |= (uint64_t)1 << 16;                   // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(1024 >> 4) << 32;         // stride byte offset
    d |= (uint64_t)1 << 46;                   // descriptor version
    d |= (uint64_t)2 << 61;                   // 128-byte swizzle
    return d;
}

// instruction descriptor: BF16 x BF16 -> F32, both K-major, M = 128, N = n
__host__ __device__ constexpr uint32_t umma_idesc(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kBM >> 4) << 24);
}

__device__ __forceinline__ void umma_f16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ void umma_commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}


// Writer of a staged 32 x 32 slice (row pitch 33 floats, so that a warp's
// accesses fall in 32 different banks): row r of the slice is output row
// rw0 + r, column j output column col0 + j; rows at or past M are skipped.
// Four columns per thread: a warp instruction writes 4 whole rows.
__device__ __forceinline__ void store_rows_f32(const float *stage, float *out, int N, int M, int rw0, int col0,
                                               int lane) {
#pragma unroll
    for (int it = 0; it < 8; it++) {
        const int r = it * 4 + (lane >> 3), q = (lane & 7) * 4;
        if (rw0 + r >= M) continue;
        const float *sp = stage + r * 33 + q;
        *reinterpret_cast<float4 *>(out + (size_t)(rw0 + r) * N + col0 + q) = make_float4(sp[0], sp[1], sp[2], sp[3]);
    }
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&p);
}

// Standard normal CDF for GELU(z) = z Phi(z), as a logistic of an odd
// polynomial: Phi(z) ~ 1 / (1 + 2^(z q(z^2))), q a quartic fitted toward the
// minimax of |z| |error| over [-14, 14] (fit_normal_cdf.py beside this file
// prints these coefficients and the errors): |z (Phi_a(z) - Phi(z))| < 3.1e-6
// and |Phi_a(z) - Phi(z)| < 6.8e-6 for every z, far below the BF16 rounding
// of the activations.  One hardware exp2, one hardware reciprocal and four
// multiply-adds; monotone in float32, 0 at -inf (2^s overflows to +inf and
// its reciprocal is 0) and 1 at +inf.
__device__ __forceinline__ float ex2_fast(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rcp_fast(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float norm_cdf(float z) {
    const float z2 = z * z;
    float q = __fmaf_rn(-3.231081337e-06f, z2, 8.827482816e-05f);
    q = __fmaf_rn(q, z2, 3.600096097e-04f);
    q = __fmaf_rn(q, z2, -1.052259058e-01f);
    q = __fmaf_rn(q, z2, -2.302046061e+00f);
    return rcp_fast(1.0f + ex2_fast(z * q));
}
// The same GELU for two activations at once on the paired FP32 instructions
// (add/mul/fma.rn.f32x2: one issue slot per pair, each lane rounded as the
// scalar instruction rounds it), so h0, h1 equal z * norm_cdf(z) bit for bit,
// z = acc + bias.
typedef unsigned long long f32x2_t;
__device__ __forceinline__ f32x2_t f2_pack(float lo, float hi) {
    f32x2_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void f2_unpack(f32x2_t v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f32x2_t f2_add(f32x2_t a, f32x2_t b) {
    f32x2_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2_t f2_mul(f32x2_t a, f32x2_t b) {
    f32x2_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2_t f2_fma(f32x2_t a, f32x2_t b, f32x2_t c) {
    f32x2_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ void gelu_pair(float acc0, float acc1, float b0, float b1, float &h0, float &h1) {
    const f32x2_t z = f2_add(f2_pack(acc0, acc1), f2_pack(b0, b1));
    const f32x2_t z2 = f2_mul(z, z);
    f32x2_t q = f2_fma(f2_pack(-3.231081337e-06f, -3.231081337e-06f), z2, f2_pack(8.827482816e-05f, 8.827482816e-05f));
    q = f2_fma(q, z2, f2_pack(3.600096097e-04f, 3.600096097e-04f));
    q = f2_fma(q, z2, f2_pack(-1.052259058e-01f, -1.052259058e-01f));
    q = f2_fma(q, z2, f2_pack(-2.302046061e+00f, -2.302046061e+00f));
    float s0, s1;
    f2_unpack(f2_mul(z, q), s0, s1);
    float d0, d1;
    f2_unpack(f2_add(f2_pack(1.0f, 1.0f), f2_pack(ex2_fast(s0), ex2_fast(s1))), d0, d1);
    f2_unpack(f2_mul(z, f2_pack(rcp_fast(d0), rcp_fast(d1))), h0, h1);
}

// standard normal density, phi(z) = 2^(-z^2 / (2 ln 2)) / sqrt(2 pi), for
// GELU'(z) = Phi(z) + z phi(z)
__device__ __forceinline__ float norm_pdf(float z) { return 0.3989422804f * ex2_fast(-0.7213475204f * (z * z)); }

// ------------------------------------------------------------- GEMM kernel
//
// D[M x N] = A[M x K] . B[N x K]^T, both operands K-major: one 128 x BN tile
// per CTA (BN = 256 or 64), K in 64-element slices through a ring of kStages.

template <int BN>
__global__ void __launch_bounds__(kThreads)
    gemm_bf16_tn(const __grid_constant__ CUtensorMap tA, const __grid_constant__ CUtensorMap tB, GemmArgs g) {
    constexpr uint32_t kABytes = kBM * kBK * 2;
    constexpr uint32_t kBBytes = BN * kBK * 2;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t *sA = smem;
    constexpr int ns = kStages;
    uint8_t *sB = smem + ns * kABytes;
    uint64_t *full = reinterpret_cast<uint64_t *>(sB + ns * kBBytes);
    uint64_t *empty = full + ns;
    uint64_t *done = empty + ns;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(done + 1);
    __shared__ int s_fail;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m0 = blockIdx.x * kBM, n0 = blockIdx.y * BN;
    const int nk = g.K / kBK;

    if (threadIdx.x == 0) {
        s_fail = 0;
        for (int s = 0; s < ns; s++) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(BN));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;

    if (warp == 0 && lane == 0) {
        // TMA producer
        for (int i = 0; i < nk; i++) {
            const int s = i % ns;
            if (i >= ns && !mbar_wait(&empty[s], ((i / ns) - 1) & 1)) {
                atomicOr(g.err, 1u);
                s_fail = 1;
                break;
            }
            if (s_fail) break;
            mbar_expect_tx(&full[s], kABytes + kBBytes);
            tma_load_2d(sA + s * kABytes, &tA, &full[s], i * kBK, m0);
            tma_load_2d(sB + s * kBBytes, &tB, &full[s], i * kBK, n0);
        }
    } else if (warp == 1 && lane == 0) {
        // MMA issuer
        const uint32_t idesc = umma_idesc(BN);
        for (int i = 0; i < nk; i++) {
            const int s = i % ns;
            if (!mbar_wait(&full[s], (i / ns) & 1)) {
                atomicOr(g.err, 2u);
                s_fail = 1;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t a0 = smem_u32(sA + s * kABytes), b0 = smem_u32(sB + s * kBBytes);
#pragma unroll
            for (int kk = 0; kk < kBK / 16; kk++)
                umma_f16(tmem, umma_desc(a0 + kk * 32), umma_desc(b0 + kk * 32), idesc, (i | kk) != 0);
            umma_commit(&empty[s]);
        }
        umma_commit(done);
    }
    __syncwarp();
    // Epilogue, all eight warps.  A warp may only read the tensor-memory
    // lanes of its quarter (warp % 4), i.e. accumulator rows
    // m0 + 32 (warp % 4) .. + 31, one row per thread; warps 0-3 take the
    // first half of the columns and warps 4-7 the second.  Every 32-column
    // slice is staged through shared memory (the operand ring is idle once
    // the last MMA has completed) so that the writes are whole rows.
    const bool ok = mbar_wait(done, 0);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (!ok) atomicOr(g.err, 4u);
    const int q = warp & 3, ch = warp >> 2;
    float *stage = reinterpret_cast<float *>(smem) + warp * (32 * 33);
    if (ok && !s_fail) {
#pragma unroll 1
        for (int cc = 0; cc < BN / 2; cc += 32) {
            const int c0 = ch * (BN / 2) + cc;
            uint32_t r[32];
            tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)c0, r);
#pragma unroll
            for (int j = 0; j < 32; j++) stage[lane * 33 + j] = __uint_as_float(r[j]);
            __syncwarp();
            store_rows_f32(stage, g.fout, g.N, g.M, m0 + q * 32, n0 + c0, lane);
            __syncwarp();
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(BN));
}


// ------------------------------------------------ fused inference forward
//
// All three hidden layers and the head of the inference forward in one
// persistent kernel.  Per 128-row tile two warps read the f32 inputs, round
// them and write the 128-byte-swizzled slice the first MMA reads (a packing
// pass before the kernel moved another 128 B per row out and back in); each
// layer's accumulator (128 x 256 f32) lives in tensor memory; the epilogue
// writes the layer's BF16 activations straight into shared memory in the
// 128-byte-swizzled K-major layout that the next layer's MMA reads, so the
// hidden activations never leave the SM and the forward moves only the
// inputs and the outputs (4 B per row) through HBM.  Weights stream from L2
// through a ring of 256 x 64 slices.  Roles: warp 0 lane 0 loads them, warp 1
// lane 0 issues the MMAs, warps 2-17 run the epilogues (four per tensor-memory
// lane quarter, each a quarter of the 256 columns), warps 18-19 the inputs.
//
// Two tiles are in flight per CTA, each with its own accumulator (the two
// fill the 512 tensor-memory columns) and its own activation buffer (the
// input slice lands in the buffer's first K slice): the jobs (tile, layer)
// run in the order A1 B1 A2 B2 A3 B3, then the next two tiles, so the MMAs of
// one tile's layer run while the epilogue warps work on the other tile's.

constexpr int kFwdEpiWarps = 16;
constexpr int kFwdInWarps = 2;
constexpr int kFwdThreads = (2 + kFwdEpiWarps + kFwdInWarps) * 32;
constexpr int kFwdBStages = 3;
constexpr uint32_t kSliceA = kBM * kBK * 2;  // one 64-wide K slice of a 128-row operand: 16 KB
constexpr uint32_t kSliceB = 256 * kBK * 2;  // one 64-wide K slice of a weight matrix: 32 KB
constexpr uint32_t kFwdBuf = 4 * kSliceA;    // a tile's activations (four K slices; the input in the first)
// two activation buffers, the weight ring, 14 mbarriers and the TMEM address
constexpr size_t kFwdSmem = 1024 + 2 * kFwdBuf + kFwdBStages * kSliceB + 128;
static_assert(kFwdSmem <= 232448, "fused forward exceeds the shared memory of a CTA");

struct FwdArgs {
    int n_tiles, n_rows, nf;
    const float *X;  // n_rows x nf
    int l1_k16;  // 16-wide K steps of layer 1 that hold real inputs (the rest of the 64 columns is zero padding)
    const float *b1, *b2, *b3, *w4, *b4;
    float *y;
    uint32_t *err;
};

__global__ void __launch_bounds__(kFwdThreads, 1)
    mlp_forward_fused(const __grid_constant__ CUtensorMap tW1, const __grid_constant__ CUtensorMap tW2,
                      const __grid_constant__ CUtensorMap tW3, FwdArgs g) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t *sA = smem;                  // two tiles' activation buffers (kFwdBuf each)
    uint8_t *sB = sA + 2 * kFwdBuf;      // weight-slice ring
    uint64_t *b_full = reinterpret_cast<uint64_t *>(sB + kFwdBStages * kSliceB);
    uint64_t *b_empty = b_full + kFwdBStages;
    uint64_t *x_full = b_empty + kFwdBStages;  // [2] input slice of the buffer's tile landed
    uint64_t *a_free = x_full + 2;             // [2] the buffer's last layer has read it (next input may land)
    uint64_t *acc_full = a_free + 2;           // [2] MMA -> epilogue: a layer's accumulator is complete
    uint64_t *ep_done = acc_full + 2;          // [2] epilogue -> MMA: accumulator drained (and activations written)
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(ep_done + 2);
    __shared__ volatile int s_fail;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // this CTA's tiles: blockIdx.x + j * gridDim.x, j < nt; tile j uses buffer j & 1
    const int nt = blockIdx.x < g.n_tiles ? (g.n_tiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    const int npairs = (nt + 1) / 2;
    if (threadIdx.x == 0) {
        s_fail = 0;
        for (int s = 0; s < kFwdBStages; s++) {
            mbar_init(&b_full[s], 1);
            mbar_init(&b_empty[s], 1);
        }
        for (int p = 0; p < 2; p++) {
            mbar_init(&x_full[p], kFwdInWarps);
            mbar_init(&a_free[p], 1);
            mbar_init(&acc_full[p], 1);
            mbar_init(&ep_done[p], kFwdEpiWarps);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            uint32_t bi = 0;
            for (int P = 0; P < npairs && !s_fail; P++) {
                for (int l = 0; l < 3 && !s_fail; l++) {
#pragma unroll
                    for (int p = 0; p < 2; p++) {
                        const int j = 2 * P + p;
                        if (j >= nt || s_fail) continue;
                        const CUtensorMap *tw = l == 0 ? &tW1 : l == 1 ? &tW2 : &tW3;
                        const int nks = l == 0 ? 1 : 4;
                        for (int ks = 0; ks < nks; ks++, bi++) {
                            const int s = bi % kFwdBStages;
                            if (bi >= kFwdBStages && !mbar_wait(&b_empty[s], ((bi / kFwdBStages) - 1) & 1)) {
                                atomicOr(g.err, 8u);
                                s_fail = 1;
                                break;
                            }
                            mbar_expect_tx(&b_full[s], kSliceB);
                            tma_load_2d(sB + s * kSliceB, tw, &b_full[s], ks * kBK, 0);
                        }
                    }
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t idesc = umma_idesc(256);
            uint32_t bi = 0;
            for (int P = 0; P < npairs && !s_fail; P++) {
                for (int l = 0; l < 3 && !s_fail; l++) {
#pragma unroll
                    for (int p = 0; p < 2; p++) {
                        const int j = 2 * P + p;
                        if (j >= nt || s_fail) continue;
                        // the accumulator is drained (and, past layer 1, this tile's activations written);
                        // layer 1 also waits for the input slice
                        const int n = 3 * P + l;  // the buffer's jobs before this one
                        if ((n > 0 && !mbar_wait(&ep_done[p], (n - 1) & 1)) ||
                            (l == 0 && !mbar_wait(&x_full[p], P & 1))) {
                            atomicOr(g.err, 16u);
                            s_fail = 1;
                            continue;
                        }
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        const uint32_t acc = tmem + (uint32_t)(p * 256);
                        const uint8_t *abuf = sA + p * kFwdBuf;
                        const int nks = l == 0 ? 1 : 4;
                        for (int ks = 0; ks < nks; ks++, bi++) {
                            const int s = bi % kFwdBStages;
                            if (!mbar_wait(&b_full[s], (bi / kFwdBStages) & 1)) {
                                atomicOr(g.err, 16u);
                                s_fail = 1;
                                break;
                            }
                            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                            const uint32_t a0 = smem_u32(abuf + ks * kSliceA);
                            const uint32_t b0 = smem_u32(sB + s * kSliceB);
                            // layer 1: only the K steps that hold real inputs (zero columns add nothing)
                            const int nkk = l == 0 ? g.l1_k16 : kBK / 16;
#pragma unroll
                            for (int kk = 0; kk < kBK / 16; kk++)
                                if (kk < nkk)
                                    umma_f16(acc, umma_desc(a0 + kk * 32), umma_desc(b0 + kk * 32), idesc,
                                             (ks | kk) != 0);
                            umma_commit(&b_empty[s]);
                        }
                        if (l == 2) umma_commit(&a_free[p]);
                        umma_commit(&acc_full[p]);
                    }
                }
            }
        }
    } else if (warp >= 2 + kFwdEpiWarps) {
        // inputs: two rows per thread, eight columns (one 16-byte chunk) at a time; the first 16 columns are on
        // their way while the buffer's previous tile finishes
        const int t0 = (int)threadIdx.x - (2 + kFwdEpiWarps) * 32;
        const int nch = 2 * g.l1_k16;
        for (int j = 0; j < nt; j++) {
            const int p = j & 1;
            const int r0 = ((int)blockIdx.x + j * (int)gridDim.x) * kBM;
            auto chunk = [&](int row, int ch) {
                const float *xp = g.X + (size_t)(r0 + row) * g.nf + ch * 8;
                float v[8];
#pragma unroll
                for (int i = 0; i < 8; i++) v[i] = r0 + row < g.n_rows && ch * 8 + i < g.nf ? xp[i] : 0.0f;
                return make_uint4(pack_bf16x2(v[0], v[1]), pack_bf16x2(v[2], v[3]), pack_bf16x2(v[4], v[5]),
                                  pack_bf16x2(v[6], v[7]));
            };
            uint8_t *xs = sA + p * kFwdBuf;
            auto put = [&](int row, int ch, uint4 v) {
                *reinterpret_cast<uint4 *>(xs + (row >> 3) * 1024 + (row & 7) * 128 + ((ch ^ (row & 7)) << 4)) = v;
            };
            uint4 first[2][2];
#pragma unroll
            for (int i = 0; i < 4; i++) first[i >> 1][i & 1] = chunk(t0 + 64 * (i >> 1), i & 1);
            // the buffer's previous tile has finished its last layer
            if (j >= 2 && !s_fail && !mbar_wait(&a_free[p], ((j >> 1) - 1) & 1)) {
                atomicOr(g.err, 8u);
                s_fail = 1;
            }
#pragma unroll
            for (int i = 0; i < 4; i++) put(t0 + 64 * (i >> 1), i & 1, first[i >> 1][i & 1]);
            for (int ch = 2; ch < nch; ch++) {
                put(t0, ch, chunk(t0, ch));
                put(t0 + 64, ch, chunk(t0 + 64, ch));
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&x_full[p]);
        }
    } else {
        // epilogue warps: rows q*32 + lane of the tile, columns [64 cq, 64 cq + 64)
        const int q = warp & 3, cq = (warp - 2) >> 2;
        const int row = q * 32 + lane;
        for (int P = 0; P < npairs; P++) {
            for (int l = 0; l < 3; l++) {
#pragma unroll
                for (int p = 0; p < 2; p++) {
                    const int j = 2 * P + p;
                    if (j >= nt) continue;
                    // the buffer's 3 P + l earlier jobs have completed the accumulator barrier's earlier phases
                    const bool ok = !s_fail && mbar_wait(&acc_full[p], (3 * P + l) & 1);
                    if (!ok) {
                        if (!s_fail) atomicOr(g.err, 32u);
                        s_fail = 1;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const float *bias = l == 0 ? g.b1 : l == 1 ? g.b2 : g.b3;
                    uint8_t *abuf = sA + p * kFwdBuf;
                    // the head's partial dot product over this warp's columns: even and odd
                    // columns in the two lanes of a paired accumulator
                    f32x2_t head2 = f2_pack(0.0f, 0.0f);
#pragma unroll 1
                    for (int c2 = 0; c2 < 2 && ok; c2++) {
                        const int c0 = cq * 64 + c2 * 32;
                        uint32_t r[32];
                        tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(p * 256 + c0), r);
                        uint32_t hp[16];
#pragma unroll
                        for (int q4 = 0; q4 < 8; q4++) {
                            const float4 b4v = reinterpret_cast<const float4 *>(bias + c0)[q4];
                            float4 w4v = make_float4(0.f, 0.f, 0.f, 0.f);
                            if (l == 2) w4v = reinterpret_cast<const float4 *>(g.w4 + c0)[q4];
                            const float bq[4] = {b4v.x, b4v.y, b4v.z, b4v.w};
                            const float wq[4] = {w4v.x, w4v.y, w4v.z, w4v.w};
                            float h[4];
                            gelu_pair(__uint_as_float(r[4 * q4]), __uint_as_float(r[4 * q4 + 1]), bq[0], bq[1], h[0],
                                      h[1]);
                            gelu_pair(__uint_as_float(r[4 * q4 + 2]), __uint_as_float(r[4 * q4 + 3]), bq[2], bq[3],
                                      h[2], h[3]);
                            // two activations per conversion, rounded to nearest as the training kernel does
                            const __nv_bfloat162 p0 = __floats2bfloat162_rn(h[0], h[1]);
                            const __nv_bfloat162 p1 = __floats2bfloat162_rn(h[2], h[3]);
                            if (l == 2) {
                                const float2 g0 = __bfloat1622float2(p0), g1 = __bfloat1622float2(p1);
                                head2 = f2_fma(f2_pack(g0.x, g0.y), f2_pack(wq[0], wq[1]), head2);
                                head2 = f2_fma(f2_pack(g1.x, g1.y), f2_pack(wq[2], wq[3]), head2);
                            }
                            hp[2 * q4] = *reinterpret_cast<const uint32_t *>(&p0);
                            hp[2 * q4 + 1] = *reinterpret_cast<const uint32_t *>(&p1);
                        }
                        if (l < 2) {
                            // next layer's A operand: K slice c0 / 64, 16-byte chunks (c0 % 64) / 8 .. + 3 of
                            // this row, at the 128-byte-swizzled positions (chunk ^ row % 8) TMA would have used
                            const int ch0 = (c0 & 63) >> 3;
                            uint8_t *rowp = abuf + (c0 >> 6) * kSliceA + (row >> 3) * 1024 + (row & 7) * 128;
#pragma unroll
                            for (int i = 0; i < 4; i++)
                                *reinterpret_cast<uint4 *>(rowp + (((ch0 + i) ^ (row & 7)) << 4)) =
                                    make_uint4(hp[4 * i], hp[4 * i + 1], hp[4 * i + 2], hp[4 * i + 3]);
                        }
                    }
                    // the activations written by the generic proxy are read by the tensor cores next
                    if (l < 2) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&ep_done[p]);
                    if (l == 2) {
                        // the head: the four column quarters of each row, added in order.  The partial
                        // sums sit in the buffer's last K slice: its last reader (this tile's layer-3
                        // MMA) is done, and the next writer is the epilogue of this buffer's next tile.
                        float *s_head = reinterpret_cast<float *>(abuf + 3 * kSliceA);
                        float he, ho;
                        f2_unpack(head2, he, ho);
                        s_head[cq * kBM + row] = he + ho;
                        asm volatile("bar.sync 1, %0;" ::"r"(kFwdEpiWarps * 32) : "memory");
                        if (cq == 0 && !s_fail && ((int)blockIdx.x + j * (int)gridDim.x) * kBM + row < g.n_rows)
                            g.y[((int)blockIdx.x + j * (int)gridDim.x) * kBM + row] =
                                (((s_head[row] + s_head[kBM + row]) + s_head[2 * kBM + row]) + s_head[3 * kBM + row]) +
                                *g.b4;
                        asm volatile("bar.sync 1, %0;" ::"r"(kFwdEpiWarps * 32) : "memory");
                    }
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

// ---------------------------------------------------------- small kernels

// GELU and its derivative as the epilogues compute them (diagnostics)
__global__ void gelu_eval(const float *z, uint64_t n, float *gelu, float *dgelu) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        const float cdf = norm_cdf(z[i]);
        gelu[i] = z[i] * cdf;
        dgelu[i] = cdf + z[i] * norm_pdf(z[i]);
    }
}

// bf16 copies of a weight matrix W (out x in, f32) and of its transpose
__global__ void weights_to_bf16(const float *W, int out, int in, __nv_bfloat16 *Wb, __nv_bfloat16 *WbT) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < out * in; i += gridDim.x * blockDim.x) {
        const int o = i / in, k = i % in;
        const __nv_bfloat16 b = __float2bfloat16_rn(W[i]);
        Wb[i] = b;
        if (WbT) WbT[(size_t)k * out + o] = b;
    }
}

// Shuffled passes over the training pool without storing a permutation: row
// p of pass q is perm_q(p), a bijection of [0, n) built from a four-round
// balanced Feistel network on [0, 4^h) (4^h >= n, round function SplitMix64
// of the seed, the pass and the round) with cycle walking back into [0, n)
// (Black and Rogaway, "Ciphers with arbitrary finite domains", 2002).  A
// walk longer than 4096 steps (probability below (3/4)^4096) sets an error
// bit instead of looping on.
__device__ __forceinline__ uint64_t mix64(uint64_t z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;  // SplitMix64 output function (Steele, Lea, Flood 2014)
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__device__ __forceinline__ uint64_t feistel(uint64_t x, uint32_t h, uint64_t key) {
    const uint64_t mask = (1ull << h) - 1ull;
    uint64_t L = x >> h, R = x & mask;
#pragma unroll
    for (uint32_t r = 0; r < 4; r++) {
        const uint64_t f = mix64(key ^ (0x9E3779B97F4A7C15ull * (r + 1)) ^ R) & mask;
        const uint64_t t = L ^ f;
        L = R;
        R = t;
    }
    return (L << h) | R;
}

// ------------------------------------------- fused training forward + backward
//
// The forward of a 128-row tile, its loss and the backward down to dZ1 in one
// cluster of two CTAs.  CTA r computes all 128 rows of columns
// [128 r, 128 r + 128) of every layer; each layer's input has to be whole, so
// a finished half goes to the partner's shared memory by bulk copy (32 KB per
// layer, in 4 KB pieces as the warps finish them) beside the CTA's own copy.
// A batch of 8192 rows is 64 tiles: one tile per CTA would leave 88 of the 152
// SMs idle while the others run a serial chain of five MMAs and five
// epilogues, so the chain itself is cut in two.
//
//   s = 0, 1   Z = A . W^T + b, H = GELU(Z)     MMA s -> T[s]
//   s = 2      the same, y = H . w4 + b4, dy, dZ3 = dy w4 GELU'(Z3)
//   s = 3, 4   dZ = (dZ_above . W) GELU'(Z)     MMA 3 -> T[3], MMA 4 -> T[2]
//
// T[0..3] are the four 128-column f32 accumulators that fill tensor memory:
// GELU'(Z1) and GELU'(Z2) replace Z1 and Z2 in place (f32, as computed) until
// the backward needs them, so only the BF16 operands of the weight gradients
// (X, H1, H2, dZ1..3, row-major) leave the chip, by TMA straight from the
// swizzled shared-memory tiles.  The column sums (bias gradients, dW4) are
// taken from those tiles while the next MMA runs and kept in registers
// over the CTA's tiles.  Training rows are drawn from the pool by the kernel
// itself (no gathered copy, no packing pass).
//
// Sums that decide a BF16 rounding keep one order whatever the tile's CTA: K
// ascending in every MMA, the head's 128 columns ascending per half, so dZ is the
// same wherever a row lands in a batch.
//
// Bound by latency: one tile's chain of five MMAs (0.55 us of tensor work
// each) and five epilogues.  (576 threads leave 96 registers each: 100 bytes
// are spilled, 128 reloaded, per thread.)  A training step of 8192 rows (this kernel, mlp_wgrad
// and mlp_update) takes 40.5 us, 155648 rows 440 us; with one GEMM launch per
// layer and gradient (transposed copies and f32 GELU' through memory, 47
// launches and memsets a step) it took 279 us and 908 us.
//
// The activation buffers alternate: X in 0, H1 in 1, H2 in 0, H3 in 1 (own
// half only), dZ3 in 0, dZ2 in 1, dZ1 in 0 (own half only).  A half may be
// written into the partner's buffer once the partner's MMA that last read
// that buffer is complete; the data received since then says so (its H1 follows
// its MMA 0, its head sum its MMA 2, and so on), except across tiles, where
// the partner reports the end of MMA 4 (peer_free).

constexpr int kTrEpiWarps = 16;
constexpr int kTrThreads = (2 + kTrEpiWarps) * 32;
constexpr int kTrBStages = 5;
constexpr uint32_t kTrSliceB = 128 * kBK * 2;  // one 64-wide K slice of half a weight matrix: 16 KB
constexpr size_t kTrSmem = 1024 + 2 * kFwdBuf + kTrBStages * kTrSliceB + 256;
constexpr int kSmall = 1026;  // per-cluster sums: db1, db2, db3, dW4 (256 each), squared errors, db4

struct TrainMaps {
    CUtensorMap w[5];   // operand B of MMA s: W1, W2, W3, W3^T, W2^T (boxes of 128 rows x 64)
    CUtensorMap x0;     // X (boxes of 128 x 64)
    CUtensorMap h[2];   // H1, H2 (boxes of 32 x 64)
    CUtensorMap dz[3];  // dZ1..3 (boxes of 32 x 64)
};

struct TrainArgs {
    int n_rows, n_tiles;  // rows of the batch; 128-row tiles that hold them (missing rows count as zero error)
    int nf, l1_k16;
    const float *X, *t;   // the batch, or the training pool
    uint64_t pool_n;      // 0: rows in order; else rows drawn from a pool of pool_n
    uint64_t seed, pos0;
    uint32_t h;
    const float *b1, *b2, *b3, *w4, *b4;
    float *small;         // clusters x kSmall
    uint32_t *err;
};

// bounded wait that also sees what the partner CTA wrote before completing the phase
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t *bar, uint32_t parity) {
    const uint32_t a = smem_u32(bar);
    for (uint32_t i = 0; i < kSpinLimit; i++) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
            " selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

__device__ __forceinline__ uint32_t mapa_u32(uint32_t saddr, uint32_t rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
    return r;
}

__device__ __forceinline__ void tma_store_2d(const CUtensorMap *map, const void *src, int x, int y) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"((uint64_t)map),
                 "r"(smem_u32(src)), "r"(x), "r"(y)
                 : "memory");
}

__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]),
        "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]),
        "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// GELU and GELU' of two activations on the paired FP32 instructions, each
// lane rounded as z * norm_cdf(z) and norm_cdf(z) + z * norm_pdf(z) round it
__device__ __forceinline__ void gelu_grad_pair(float acc0, float acc1, float b0, float b1, float &h0, float &h1,
                                               uint32_t &g0, uint32_t &g1) {
    const f32x2_t z = f2_add(f2_pack(acc0, acc1), f2_pack(b0, b1));
    const f32x2_t z2 = f2_mul(z, z);
    f32x2_t q = f2_fma(f2_pack(-3.231081337e-06f, -3.231081337e-06f), z2, f2_pack(8.827482816e-05f, 8.827482816e-05f));
    q = f2_fma(q, z2, f2_pack(3.600096097e-04f, 3.600096097e-04f));
    q = f2_fma(q, z2, f2_pack(-1.052259058e-01f, -1.052259058e-01f));
    q = f2_fma(q, z2, f2_pack(-2.302046061e+00f, -2.302046061e+00f));
    float s0, s1, d0, d1, p0, p1;
    f2_unpack(f2_mul(z, q), s0, s1);
    f2_unpack(f2_add(f2_pack(1.0f, 1.0f), f2_pack(ex2_fast(s0), ex2_fast(s1))), d0, d1);
    const float c0 = rcp_fast(d0), c1 = rcp_fast(d1);
    f2_unpack(f2_mul(z, f2_pack(c0, c1)), h0, h1);
    f2_unpack(f2_mul(f2_pack(-0.7213475204f, -0.7213475204f), z2), p0, p1);
    const f32x2_t pdf = f2_mul(f2_pack(0.3989422804f, 0.3989422804f), f2_pack(ex2_fast(p0), ex2_fast(p1)));
    float z0, z1, u0, u1;
    f2_unpack(z, z0, z1);
    f2_unpack(pdf, u0, u1);
    // scalar: a paired product and sum come out as one rounding
    g0 = __float_as_uint(__fadd_rn(c0, __fmul_rn(z0, u0)));
    g1 = __float_as_uint(__fadd_rn(c1, __fmul_rn(z1, u1)));
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kTrThreads, 1)
    mlp_train_fused(const __grid_constant__ TrainMaps mp, TrainArgs g) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t *sA = smem;              // two activation buffers (kFwdBuf each: four K slices of 128 rows)
    uint8_t *sB = sA + 2 * kFwdBuf;  // weight-slice ring
    uint64_t *b_full = reinterpret_cast<uint64_t *>(sB + kTrBStages * kTrSliceB);
    uint64_t *b_empty = b_full + kTrBStages;
    uint64_t *peer_full = b_empty + kTrBStages;  // [2] the partner's half of MMA s's input landed, s = 1, 3 / 2, 4
    uint64_t *acc_full = peer_full + 2;          // MMA -> epilogue
    uint64_t *ep_done = acc_full + 1;            // epilogue -> MMA: own half written, accumulator drained
    uint64_t *head_full = ep_done + 1;           // the partner's head sums landed
    uint64_t *peer_free = head_full + 1;         // the partner's MMA 4 of a tile is complete
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(peer_free + 1);
    __shared__ volatile int s_fail;
    __shared__ __align__(16) float s_par[4][128];  // b1, b2, b3, w4 of this CTA's columns
    __shared__ __align__(16) float s_hr[128];      // the partner's head sums
    __shared__ float s_sum[2][4];                  // squared errors and db4 of the four row quarters
    __shared__ float s_t[128], s_dy[128];
    __shared__ __align__(8) float s_col[8][128];   // column sums of the eight 16-row groups

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = blockIdx.x & 1u;  // clusters are pairs of neighbouring blocks
    const int cl = (int)(blockIdx.x >> 1), n_cl = (int)(gridDim.x >> 1);
    const int nt = cl < g.n_tiles ? (g.n_tiles - 1 - cl) / n_cl + 1 : 0;  // tiles cl + i n_cl
    if (threadIdx.x == 0) {
        s_fail = 0;
        for (int s = 0; s < kTrBStages; s++) {
            mbar_init(&b_full[s], 1);
            mbar_init(&b_empty[s], 1);
        }
        mbar_init(&peer_full[0], 1);
        mbar_init(&peer_full[1], 1);
        mbar_init(acc_full, 1);
        mbar_init(ep_done, kTrEpiWarps);
        mbar_init(head_full, 1);
        mbar_init(peer_free, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // the partner's barriers are initialised before anything is sent there
    asm volatile("barrier.cluster.arrive.release;\n barrier.cluster.wait.acquire;" ::: "memory");
    // the previous step's weights, and the buffers its weight gradients read
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    auto give_up = [&](uint32_t code) {
        atomicOr(g.err, code);
        s_fail = 1;
    };

    if (warp == 0) {
        if (lane == 0) {
            // weight slices in the order the MMAs take them
            uint32_t bi = 0;
            for (int ti = 0; ti < nt && !s_fail; ti++) {
                for (int s = 0; s < 5 && !s_fail; s++) {
                    const int nks = s == 0 ? 1 : 4;
                    for (int i = 0; i < nks && !s_fail; i++, bi++) {
                        const int st = bi % kTrBStages;
                        if (bi >= kTrBStages && !mbar_wait(&b_empty[st], ((bi / kTrBStages) - 1) & 1)) {
                            give_up(8u);
                            break;
                        }
                        mbar_expect_tx(&b_full[st], kTrSliceB);
                        tma_load_2d(sB + st * kTrSliceB, &mp.w[s], &b_full[st], i * kBK, 128 * (int)rank);
                    }
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t idesc = umma_idesc(128);
            uint32_t bi = 0;
            for (int ti = 0; ti < nt && !s_fail; ti++) {
                for (int s = 0; s < 5 && !s_fail; s++) {
                    if (!mbar_wait(ep_done, (5 * ti + s) & 1)) {
                        give_up(16u);
                        break;
                    }
                    // the half that comes from the partner: announced now, waited for before it is read
                    if (s > 0) mbar_expect_tx(&peer_full[(s - 1) & 1], 2 * kSliceA);
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint8_t *abuf = sA + ((s == 1 || s == 4) ? kFwdBuf : 0);
                    const uint32_t acc = tmem + (uint32_t)(s == 4 ? 2 : s) * 128u;
                    const int nks = s == 0 ? 1 : 4;
                    for (int i = 0; i < nks; i++, bi++) {
                        const int st = bi % kTrBStages;
                        // K slices 0, 1 come from CTA 0, slices 2, 3 from CTA 1
                        if ((s > 0 && i == 2 * (int)(rank ^ 1u) && !mbar_wait_cluster(&peer_full[(s - 1) & 1], (2 * ti + ((s - 1) >> 1)) & 1)) ||
                            !mbar_wait(&b_full[st], (bi / kTrBStages) & 1)) {
                            give_up(16u);
                            break;
                        }
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        const uint32_t a0 = smem_u32(abuf + i * kSliceA), b0 = smem_u32(sB + st * kTrSliceB);
                        const int nkk = s == 0 ? g.l1_k16 : kBK / 16;
#pragma unroll
                        for (int kk = 0; kk < kBK / 16; kk++)
                            if (kk < nkk)
                                umma_f16(acc, umma_desc(a0 + kk * 32), umma_desc(b0 + kk * 32), idesc, (i | kk) != 0);
                        umma_commit(&b_empty[st]);
                    }
                    umma_commit(acc_full);
                }
            }
        }
    } else {
        // epilogue: row q * 32 + lane of the tile, columns [32 cq, 32 cq + 32) of this CTA's half
        const int et = (int)threadIdx.x - 64;  // 0..511
        const int q = warp & 3, cq = (warp - 2) >> 2;
        const int row = q * 32 + lane;
        const uint32_t peer = rank ^ 1u;
        const uint32_t tlane = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(cq * 32);
        // the two warps of rows 32 q.. and K slice 2 rank + cq / 2 write one contiguous 4 KB piece;
        // lane 0 of the even one sends it on
        const int pair_bar = 2 + 2 * q + (cq >> 1);
        const bool sender = lane == 0 && (cq & 1) == 0;
        const uint32_t piece = (uint32_t)(2 * rank + (cq >> 1)) * kSliceA + (uint32_t)q * 4096u;
        const uint32_t rowoff = (uint32_t)(2 * rank + (cq >> 1)) * kSliceA + (uint32_t)(row >> 3) * 1024u +
                                (uint32_t)(row & 7) * 128u;
        const int ch0 = (cq & 1) * 4;
        auto put_row = [&](uint8_t *buf, const uint32_t(&hp)[16]) {
#pragma unroll
            for (int i = 0; i < 4; i++)
                *reinterpret_cast<uint4 *>(buf + rowoff + (((ch0 + i) ^ (row & 7)) << 4)) =
                    make_uint4(hp[4 * i], hp[4 * i + 1], hp[4 * i + 2], hp[4 * i + 3]);
        };
        auto wait_acc = [&](uint32_t n) {
            if (!s_fail && !mbar_wait(acc_full, n & 1)) give_up(32u);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        };
        // own half of buf written: to the MMA thread, to the partner (pf >= 0) and to global memory
        auto hand_over = [&](uint8_t *buf, int pf, const CUtensorMap *gm, int r0) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0 && pf >= 0) mbar_arrive(ep_done);
            asm volatile("bar.sync %0, 64;" ::"r"(pair_bar) : "memory");
            if (sender && !s_fail) {
                if (pf >= 0)
                    asm volatile(
                        "cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
                            "r"(mapa_u32(smem_u32(buf + piece), peer)),
                        "r"(smem_u32(buf + piece)), "r"(4096u), "r"(mapa_u32(smem_u32(&peer_full[pf]), peer))
                        : "memory");
                tma_store_2d(gm, buf + piece, (int)(2 * rank + (cq >> 1)) * kBK, r0 + q * 32);
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            }
        };
        // the TMA stores so far have read their tiles, for the pair of warps that writes there next
        auto tiles_read = [&]() {
            if (sender) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
            asm volatile("bar.sync %0, 64;" ::"r"(pair_bar) : "memory");
        };
        // sums over the tile's rows of this CTA's columns of buf, weighted by dy or not; thread et < 128 keeps column et
        auto column_sum = [&](const uint8_t *buf, bool weighted, float &sum) {
            asm volatile("bar.sync 1, %0;" ::"r"(kTrEpiWarps * 32) : "memory");
            const int cp = et & 63, rg = et >> 6;
            const uint8_t *base = buf + (size_t)(2 * rank + (cp >> 5)) * kSliceA + (cp & 3) * 4;
            const int chunk = (cp & 31) >> 2;
            float a0 = 0.0f, a1 = 0.0f;
#pragma unroll
            for (int i = 0; i < 16; i++) {
                const int r = rg * 16 + i;
                const uint32_t v = *reinterpret_cast<const uint32_t *>(base + (r >> 3) * 1024 + (r & 7) * 128 +
                                                                       ((chunk ^ (r & 7)) << 4));
                const float lo = __uint_as_float(v << 16), hi = __uint_as_float(v & 0xFFFF0000u);
                const float w = weighted ? s_dy[r] : 1.0f;
                a0 += weighted ? lo * w : lo;
                a1 += weighted ? hi * w : hi;
            }
            *reinterpret_cast<float2 *>(&s_col[rg][2 * cp]) = make_float2(a0, a1);
            asm volatile("bar.sync 1, %0;" ::"r"(kTrEpiWarps * 32) : "memory");
            if (et < 128) {
                float c = 0.0f;
#pragma unroll
                for (int i = 0; i < 8; i++) c += s_col[i][et];
                sum += c;
            }
        };
        const float scale = 2.0f / (float)g.n_rows;
        s_par[et >> 7][et & 127] = (et < 128 ? g.b1 : et < 256 ? g.b2 : et < 384 ? g.b3 : g.w4)[128 * rank + (et & 127)];
        const float b4 = *g.b4;
        float db1 = 0.0f, db2 = 0.0f, db3 = 0.0f, dw4 = 0.0f, sq = 0.0f, db4 = 0.0f;
        for (int ti = 0; ti < nt; ti++) {
            const int r0 = (cl + ti * n_cl) * 128;
            // the batch rows: four threads per row, 16 columns each
            tiles_read();
            asm volatile("bar.sync 1, %0;" ::"r"(kTrEpiWarps * 32) : "memory");
            {
                const int xr = et >> 2, sub = et & 3;
                const bool valid = r0 + xr < g.n_rows;
                uint64_t src = (uint64_t)(r0 + xr);
                if (g.pool_n && valid) {
                    const uint64_t pos = g.pos0 + src, pass = pos / g.pool_n;
                    const uint64_t key = mix64(g.seed ^ (pass * 0xD1B54A32D192ED03ull));
                    const uint64_t r_first = pos - pass * g.pool_n;
                    uint64_t r = r_first;
                    uint32_t walk = 0;
                    do {
                        r = feistel(r, g.h, key);
                    } while (r >= g.pool_n && ++walk < 4096u);
                    if (r >= g.pool_n) {
                        atomicOr(g.err, 64u);
                        r = r_first;
                    }
                    src = r;
                }
                const float *xp = g.X + src * (uint64_t)g.nf;
                float v[16];
#pragma unroll
                for (int i = 0; i < 16; i++) v[i] = valid && sub * 16 + i < g.nf ? xp[sub * 16 + i] : 0.0f;
                uint8_t *xrow = sA + (xr >> 3) * 1024 + (xr & 7) * 128;
#pragma unroll
                for (int i = 0; i < 2; i++)
                    *reinterpret_cast<uint4 *>(xrow + (((2 * sub + i) ^ (xr & 7)) << 4)) =
                        make_uint4(pack_bf16x2(v[8 * i], v[8 * i + 1]), pack_bf16x2(v[8 * i + 2], v[8 * i + 3]),
                                   pack_bf16x2(v[8 * i + 4], v[8 * i + 5]), pack_bf16x2(v[8 * i + 6], v[8 * i + 7]));
                if (sub == 0) s_t[xr] = valid ? g.t[src] : 0.0f;
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            asm volatile("bar.sync 1, %0;" ::"r"(kTrEpiWarps * 32) : "memory");
            if (lane == 0) mbar_arrive(ep_done);
            if (sender && q == 0 && cq == 0 && rank == 0 && !s_fail) {
                tma_store_2d(&mp.x0, sA, 0, r0);
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            }
            // layers 1 and 2
#pragma unroll 1
            for (int s = 0; s < 2; s++) {
                uint8_t *buf = sA + (s == 0 ? kFwdBuf : 0);
                tiles_read();
                wait_acc(5 * ti + s);
                // the partner's MMA 4 of the tile before: its buffer 1 may be written, and it has this CTA's dZ2
                if (s == 0 && ti > 0 && !s_fail && !mbar_wait_cluster(peer_free, (ti - 1) & 1)) give_up(32u);
                uint32_t r[32], hp[16];
                tmem_ld32(tlane + s * 128, r);
#pragma unroll
                for (int j = 0; j < 16; j++) {
                    const float2 b = *reinterpret_cast<const float2 *>(&s_par[s][cq * 32 + 2 * j]);
                    float h0, h1;
                    gelu_grad_pair(__uint_as_float(r[2 * j]), __uint_as_float(r[2 * j + 1]), b.x, b.y, h0, h1, r[2 * j],
                                   r[2 * j + 1]);
                    hp[j] = pack_bf16x2(h0, h1);
                }
                put_row(buf, hp);
                tmem_st32(tlane + s * 128, r);
                hand_over(buf, s, &mp.h[s], r0);
            }
            // layer 3, the head and dZ3
            tiles_read();
            wait_acc(5 * ti + 2);
            {
                uint32_t r[32], hp[16];
                tmem_ld32(tlane + 2 * 128, r);
#pragma unroll
                for (int j = 0; j < 16; j++) {
                    const float2 b = *reinterpret_cast<const float2 *>(&s_par[2][cq * 32 + 2 * j]);
                    float h0, h1;
                    gelu_grad_pair(__uint_as_float(r[2 * j]), __uint_as_float(r[2 * j + 1]), b.x, b.y, h0, h1, r[2 * j],
                                   r[2 * j + 1]);
                    hp[j] = pack_bf16x2(h0, h1);
                }
                put_row(sA + kFwdBuf, hp);
                if (et == 0) mbar_expect_tx(head_full, 512);
                asm volatile("bar.sync 1, %0;" ::"r"(kTrEpiWarps * 32) : "memory");
                if (cq == 0) {
                    // the head over this CTA's columns in ascending order, one thread per row
                    float own = 0.0f;
#pragma unroll 4
                    for (int c = 0; c < 16; c++) {
                        const uint4 hv = *reinterpret_cast<const uint4 *>(
                            sA + kFwdBuf + (size_t)(2 * rank + (c >> 3)) * kSliceA + (row >> 3) * 1024 +
                            (row & 7) * 128 + (((c & 7) ^ (row & 7)) << 4));
                        const float4 w0 = *reinterpret_cast<const float4 *>(&s_par[3][8 * c]);
                        const float4 w1 = *reinterpret_cast<const float4 *>(&s_par[3][8 * c + 4]);
                        own += __uint_as_float(hv.x << 16) * w0.x;
                        own += __uint_as_float(hv.x & 0xFFFF0000u) * w0.y;
                        own += __uint_as_float(hv.y << 16) * w0.z;
                        own += __uint_as_float(hv.y & 0xFFFF0000u) * w0.w;
                        own += __uint_as_float(hv.z << 16) * w1.x;
                        own += __uint_as_float(hv.z & 0xFFFF0000u) * w1.y;
                        own += __uint_as_float(hv.w << 16) * w1.z;
                        own += __uint_as_float(hv.w & 0xFFFF0000u) * w1.w;
                    }
                    if (!s_fail)
                        asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::
                                         "r"(mapa_u32(smem_u32(&s_hr[row]), peer)),
                                     "r"(__float_as_uint(own)), "r"(mapa_u32(smem_u32(head_full), peer))
                                     : "memory");
                    if (!s_fail && !mbar_wait_cluster(head_full, ti & 1)) give_up(32u);
                    const float e = r0 + row < g.n_rows ? (own + s_hr[row]) + b4 - s_t[row] : 0.0f;
                    s_dy[row] = scale * e;
                    sq += e * e;
                    db4 += scale * e;
                }
                asm volatile("bar.sync 1, %0;" ::"r"(kTrEpiWarps * 32) : "memory");
                const float dy = s_dy[row];
#pragma unroll
                for (int j = 0; j < 16; j++) {
                    const float2 w = *reinterpret_cast<const float2 *>(&s_par[3][cq * 32 + 2 * j]);
                    hp[j] = pack_bf16x2(dy * w.x * __uint_as_float(r[2 * j]), dy * w.y * __uint_as_float(r[2 * j + 1]));
                }
                put_row(sA, hp);
                hand_over(sA, 0, &mp.dz[2], r0);
            }
            column_sum(sA + kFwdBuf, true, dw4);
            column_sum(sA, false, db3);
            // dZ2 and dZ1
#pragma unroll 1
            for (int s = 3; s < 5; s++) {
                uint8_t *buf = sA + (s == 3 ? kFwdBuf : 0);
                tiles_read();
                wait_acc(5 * ti + s);
                if (s == 4 && et == 0 && !s_fail)
                    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(
                                     mapa_u32(smem_u32(peer_free), peer))
                                 : "memory");
                uint32_t r[32], gp[32], hp[16];
                tmem_ld32(tlane + (s == 3 ? 3 : 2) * 128, r);
                tmem_ld32(tlane + (s == 3 ? 1 : 0) * 128, gp);
#pragma unroll
                for (int j = 0; j < 16; j++)
                    hp[j] = pack_bf16x2(__uint_as_float(r[2 * j]) * __uint_as_float(gp[2 * j]),
                                        __uint_as_float(r[2 * j + 1]) * __uint_as_float(gp[2 * j + 1]));
                put_row(buf, hp);
                hand_over(buf, s == 3 ? 1 : -1, &mp.dz[s == 3 ? 1 : 0], r0);
                float db = 0.0f;
                column_sum(buf, false, db);
                if (s == 3) db2 += db;
                else db1 += db;
            }
        }
        // this cluster's sums
        float *sm = g.small + (size_t)cl * kSmall;
        if (et < 128) {
            const int c = 128 * (int)rank + et;
            sm[c] = db1;
            sm[256 + c] = db2;
            sm[512 + c] = db3;
            sm[768 + c] = dw4;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            sq += __shfl_xor_sync(0xFFFFFFFFu, sq, o);
            db4 += __shfl_xor_sync(0xFFFFFFFFu, db4, o);
        }
        asm volatile("bar.sync 1, %0;" ::"r"(kTrEpiWarps * 32) : "memory");
        if (cq == 0 && lane == 0) {
            s_sum[0][q] = sq;
            s_sum[1][q] = db4;
        }
        asm volatile("bar.sync 1, %0;" ::"r"(kTrEpiWarps * 32) : "memory");
        if (et == 0 && rank == 0) {
            sm[1024] = (s_sum[0][0] + s_sum[0][1]) + (s_sum[0][2] + s_sum[0][3]);
            sm[1025] = (s_sum[1][0] + s_sum[1][1]) + (s_sum[1][2] + s_sum[1][3]);
        }
        if (sender) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    // after a wait that gave up, copies may still be on their way: let them land before either CTA leaves
    if (s_fail)
        for (int i = 0; i < 1000; i++) __nanosleep(1000);
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
    asm volatile("barrier.cluster.arrive.release;\n barrier.cluster.wait.acquire;" ::: "memory");
}

// ------------------------------------------------------------ weight gradients
//
// dW_l = dZ_l^T . H_{l-1}, summed over the batch's rows.  Both operands are
// the row-major tiles the training kernel wrote, read as they are: a
// [64 rows][64 columns] box in the 128-byte swizzle is an MN-major operand
// whose K index is the row, so no transposed copies exist.  One CTA per
// 128 x 128 output tile (128 x 64 for layer 1: ten tiles in all) and split of
// the rows.  A split's even and odd 64-row slices go to an accumulator each,
// added at the end: half as many sums in the tensor core's own rounding (dW of
// 20,000 rows 1.5e-7 off the sums of 128-row blocks instead of 4.4e-7).  Partial
// sums go to global memory in the accumulator's own order (whole 512-byte lines
// per warp) and are added by mlp_update.

constexpr int kWgStages = 3;
constexpr uint32_t kWgBox = 64 * kBK * 2;  // 64 rows x 64 columns: 8 KB
constexpr size_t kWgSmem = 1024 + kWgStages * 4 * kWgBox + 128;
constexpr int kWgTiles = 10;                             // 4 of dW3, 4 of dW2, 2 of dW1
constexpr int kWgFloats = 8 * 128 * 128 + 2 * 128 * 64;  // partial sums of one split

struct WgradMaps {
    CUtensorMap dz[3], x0, h[2];  // boxes of 64 rows x 64 columns
};

// shared-memory matrix descriptor: MN-major, 128-byte swizzle; 64-element
// blocks of the MN index lbo bytes apart, 8-row groups of K 1024 bytes apart
__device__ __forceinline__ uint64_t umma_desc_mn(uint32_t saddr, uint32_t lbo) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
    d |= (uint64_t)(lbo >> 4) << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

__global__ void __launch_bounds__(kThreads, 2)
    mlp_wgrad(const __grid_constant__ WgradMaps mp, int kt_total, int kt_split, float *part, uint32_t *err) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + kWgStages * 4 * kWgBox);
    uint64_t *empty = full + kWgStages;
    uint64_t *done = empty + kWgStages;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(done + 1);
    __shared__ volatile int s_fail;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tile = blockIdx.x;
    const int layer = tile < 4 ? 2 : tile < 8 ? 1 : 0;
    const int mi = layer ? (tile >> 1) & 1 : tile - 8, ni = layer ? tile & 1 : 0;
    const int nb = layer ? 2 : 1;  // 64-column blocks of the B operand
    const int kt0 = blockIdx.y * kt_split, nk = min(kt_total, kt0 + kt_split) - kt0;
    if (threadIdx.x == 0) {
        s_fail = 0;
        for (int s = 0; s < kWgStages; s++) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(256));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const uint32_t tmem = *tmem_slot;

    if (warp == 0 && lane == 0) {
        const CUtensorMap *ta = &mp.dz[layer], *tb = layer == 2 ? &mp.h[1] : layer == 1 ? &mp.h[0] : &mp.x0;
        for (int i = 0; i < nk && !s_fail; i++) {
            const int s = i % kWgStages;
            if (i >= kWgStages && !mbar_wait(&empty[s], ((i / kWgStages) - 1) & 1)) {
                atomicOr(err, 1u);
                s_fail = 1;
                break;
            }
            uint8_t *st = smem + s * 4 * kWgBox;
            const int r = (kt0 + i) * 64;
            mbar_expect_tx(&full[s], (2 + nb) * kWgBox);
            tma_load_2d(st, ta, &full[s], mi * 128, r);
            tma_load_2d(st + kWgBox, ta, &full[s], mi * 128 + 64, r);
            tma_load_2d(st + 2 * kWgBox, tb, &full[s], ni * 128, r);
            if (nb == 2) tma_load_2d(st + 3 * kWgBox, tb, &full[s], ni * 128 + 64, r);
        }
    } else if (warp == 1 && lane == 0) {
        const uint32_t idesc = umma_idesc(nb * 64) | (1u << 15) | (1u << 16);  // A and B MN-major
        for (int i = 0; i < nk && !s_fail; i++) {
            const int s = i % kWgStages;
            if (!mbar_wait(&full[s], (i / kWgStages) & 1)) {
                atomicOr(err, 2u);
                s_fail = 1;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t a0 = smem_u32(smem + s * 4 * kWgBox), b0 = a0 + 2 * kWgBox;
#pragma unroll
            for (int kk = 0; kk < 4; kk++)  // 16 rows per instruction: two 8-row groups
                umma_f16(tmem + (uint32_t)(i & 1) * 128u, umma_desc_mn(a0 + kk * 2048, kWgBox),
                         umma_desc_mn(b0 + kk * 2048, kWgBox), idesc, i >= 2 || kk > 0);
            umma_commit(&empty[s]);
        }
        umma_commit(done);
    }
    __syncwarp();
    const bool ok = mbar_wait(done, 0);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (!ok) atomicOr(err, 4u);
    const int q = warp & 3, ch = warp >> 2;
    if (ok && !s_fail) {
        float4 *out = reinterpret_cast<float4 *>(part + (size_t)blockIdx.y * kWgFloats +
                                                 (layer ? tile * 16384 : 8 * 16384 + (tile - 8) * 8192));
#pragma unroll 1
        for (int c = 0; c < nb; c++) {
            const int cb = ch * nb + c;  // 32-column block
            uint32_t r[32];
            tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(cb * 32), r);
            if (nk > 1) {
                uint32_t r2[32];
                tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(128 + cb * 32), r2);
#pragma unroll
                for (int i = 0; i < 32; i++) r[i] = __float_as_uint(__uint_as_float(r[i]) + __uint_as_float(r2[i]));
            }
#pragma unroll
            for (int i = 0; i < 8; i++)
                out[((cb * 4 + q) * 8 + i) * 32 + lane] =
                    make_float4(__uint_as_float(r[4 * i]), __uint_as_float(r[4 * i + 1]), __uint_as_float(r[4 * i + 2]),
                                __uint_as_float(r[4 * i + 3]));
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256));
}

// ------------------------------------------------------------------- update
//
// The gradients as sums of the partial sums (in a fixed order: the splits of
// mlp_wgrad, the clusters of mlp_train_fused) and, with adam set, the Adam step
// (Kingma and Ba 2015, Algorithm 1) on the f32 master weights and the BF16
// copies of the new weights.  Parameters, moments and gradients are flat
// arrays in the order W1 b1 W2 b2 W3 b3 W4 b4.

__host__ __device__ constexpr int param_off(int t) {  // first element of tensor t (t = 8: their number)
    return (t > 0 ? 64 * 256 : 0) + (t > 1 ? 256 : 0) + (t > 2 ? 256 * 256 : 0) + (t > 3 ? 256 : 0) +
           (t > 4 ? 256 * 256 : 0) + (t > 5 ? 256 : 0) + (t > 6 ? 256 : 0) + (t > 7 ? 1 : 0);
}
constexpr int kUpdBlocks = kWgFloats / 4 / 256;  // four weights per thread
constexpr int kUpdSmallBlocks = (kSmall + 255) / 256;

struct UpdateArgs {
    const float *part, *small;
    int splits, clusters;
    float *G;       // nullable
    float *loss;    // sum of the squared errors (nullable)
    float *P, *Mo, *Ve;
    __nv_bfloat16 *Wb[3], *WbT[3];
    int adam;
    float lr, b1, b2, eps, c1, c2;
};

__device__ __forceinline__ float adam_one(const UpdateArgs &u, float gi, float &m, float &v, float p) {
    m = u.b1 * m + (1.0f - u.b1) * gi;
    v = u.b2 * v + (1.0f - u.b2) * gi * gi;
    return p - u.lr * (m / u.c1) / (sqrtf(v / u.c2) + u.eps);
}

__global__ void __launch_bounds__(256) mlp_update(UpdateArgs u) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (blockIdx.x < kUpdBlocks) {
        // four neighbouring weights of one row, in mlp_wgrad's order
        const int i4 = blockIdx.x * 256 + threadIdx.x;
        const int tile = i4 < 8 * 4096 ? i4 >> 12 : 8 + ((i4 - 8 * 4096) >> 11);
        const int layer = tile < 4 ? 2 : tile < 8 ? 1 : 0;
        const int mi = layer ? (tile >> 1) & 1 : tile - 8, ni = layer ? tile & 1 : 0;
        const int in_tile = layer ? i4 & 4095 : i4 & 2047;
        const int o = mi * 128 + ((in_tile >> 8) & 3) * 32 + (in_tile & 31);
        const int k = ni * 128 + (in_tile >> 10) * 32 + ((in_tile >> 5) & 7) * 4;
        const int n_in = layer ? 256 : 64;
        const int flat = param_off(2 * layer) + o * n_in + k;
        float4 gr = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        const float4 *pp = reinterpret_cast<const float4 *>(u.part) + i4;
#pragma unroll 8
        for (int s = 0; s < u.splits; s++) {
            const float4 a = pp[(size_t)s * (kWgFloats / 4)];
            gr.x += a.x;
            gr.y += a.y;
            gr.z += a.z;
            gr.w += a.w;
        }
        if (u.G) *reinterpret_cast<float4 *>(u.G + flat) = gr;
        if (u.adam) {
            float4 p = *reinterpret_cast<const float4 *>(u.P + flat);
            float4 m = *reinterpret_cast<const float4 *>(u.Mo + flat), v = *reinterpret_cast<const float4 *>(u.Ve + flat);
            p.x = adam_one(u, gr.x, m.x, v.x, p.x);
            p.y = adam_one(u, gr.y, m.y, v.y, p.y);
            p.z = adam_one(u, gr.z, m.z, v.z, p.z);
            p.w = adam_one(u, gr.w, m.w, v.w, p.w);
            *reinterpret_cast<float4 *>(u.P + flat) = p;
            *reinterpret_cast<float4 *>(u.Mo + flat) = m;
            *reinterpret_cast<float4 *>(u.Ve + flat) = v;
            const uint2 w = make_uint2(pack_bf16x2(p.x, p.y), pack_bf16x2(p.z, p.w));
            *reinterpret_cast<uint2 *>(u.Wb[layer] + o * n_in + k) = w;
            if (layer) {
                __nv_bfloat16 *wt = u.WbT[layer] + k * 256 + o;
                const float pv[4] = {p.x, p.y, p.z, p.w};
#pragma unroll
                for (int j = 0; j < 4; j++) wt[j * 256] = __float2bfloat16_rn(pv[j]);
            }
        }
        return;
    }
    const int i = (blockIdx.x - kUpdBlocks) * 256 + threadIdx.x;
    if (i >= kSmall) return;
    float gr = 0.0f;
#pragma unroll 8
    for (int c = 0; c < u.clusters; c++) gr += u.small[(size_t)c * kSmall + i];
    if (i == 1024) {
        if (u.loss) *u.loss = gr;
        return;
    }
    const int t = i == 1025 ? 7 : i >= 768 ? 6 : 2 * (i >> 8) + 1;
    const int flat = param_off(t) + (i == 1025 ? 0 : i & 255);
    if (u.G) u.G[flat] = gr;
    if (u.adam) {
        float m = u.Mo[flat], v = u.Ve[flat];
        u.P[flat] = adam_one(u, gr, m, v, u.P[flat]);
        u.Mo[flat] = m;
        u.Ve[flat] = v;
    }
}

// the Adam step with the gradients in u.G (the BF16 copies follow separately)
__global__ void adam_given(UpdateArgs u) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= param_off(8)) return;
    float m = u.Mo[i], v = u.Ve[i];
    u.P[i] = adam_one(u, u.G[i], m, v, u.P[i]);
    u.Mo[i] = m;
    u.Ve[i] = v;
}

// ------------------------------------------------------------- host side

PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;
std::once_flag g_encode_once;

int get_encode() {
    std::call_once(g_encode_once, [] {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    });
    if (!g_encode) return fail(LPSIM_E_CUDA, "cuTensorMapEncodeTiled is not available");
    return LPSIM_OK;
}

// K-major BF16 matrix [rows][cols] (cols contiguous) read in boxes of
// box_rows x 64 with 128-byte swizzle
int make_map(CUtensorMap *map, const void *ptr, uint64_t rows, uint64_t cols, uint32_t box_rows) {
    TRY(get_encode());
    if (cols % 64 != 0 || rows % box_rows != 0 || ((uintptr_t)ptr & 15) != 0)
        return fail(LPSIM_E_INVALID_ARG, "GEMM operand shape not a multiple of its tile");
    cuuint64_t dims[2] = {cols, rows};
    cuuint64_t strides[1] = {cols * 2};
    cuuint32_t box[2] = {64, box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(ptr), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(LPSIM_E_CUDA, "cuTensorMapEncodeTiled failed (" + std::to_string((int)r) + ")");
    return LPSIM_OK;
}

template <int BN>
int launch_gemm(const CUtensorMap &a, const CUtensorMap &b, const GemmArgs &g, cudaStream_t st) {
    const size_t smem = 1024 + kStages * (size_t)(kBM * kBK * 2 + BN * kBK * 2) + (2 * kStages + 1) * 8 + 16;
    CU(cudaFuncSetAttribute(gemm_bf16_tn<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    if (g.M % kBM != 0 || g.N % BN != 0) return fail(LPSIM_E_INVALID_ARG, "GEMM shape not a multiple of the tile");
    gemm_bf16_tn<BN><<<dim3(g.M / kBM, g.N / BN), kThreads, smem, st>>>(a, b, g);
    CU(cudaGetLastError());
    return LPSIM_OK;
}

// a launch that may start before the previous kernel of the stream has
// finished (the kernel waits for it itself, griddepcontrol)
template <class... P, class... A>
int launch_dependent(void (*kernel)(P...), dim3 grid, int block, size_t smem, cudaStream_t st, const A &...args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    CU(cudaLaunchKernelEx(&cfg, kernel, args...));
    return LPSIM_OK;
}

}  // namespace

// =================================================================== MLP

struct lpsim_mlp {
    int device = 0;
    int n_sm = 1;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    int nf = 9;       // real input features
    int B = 8192;     // rows per batch (multiple of 128)
    std::vector<void *> blocks;
    // parameters: f32 master, Adam moments, gradients; each one flat array in
    // the order W1 b1 W2 b2 W3 b3 W4 b4, P[i] the tensors of the first.  The
    // loss and the error word follow the gradients, so one copy brings all three
    float *Pf = nullptr, *Gf = nullptr, *Mf = nullptr, *Vf = nullptr, *P[8] = {};
    int sz[8] = {};
    // bf16 weights (W1..W3) and transposes (W2^T, W3^T)
    __nv_bfloat16 *Wb[3] = {}, *WbT[3] = {};
    // one batch: inputs as given, inputs and hidden activations in bf16, the
    // backward's dZ1..3
    float *Xf, *t, *y_block, *y;  // y follows an error word of its own, so one copy brings both
    __nv_bfloat16 *X0, *H[2], *dZ[3];
    float *small, *part;  // partial sums of mlp_train_fused (per cluster) and mlp_wgrad (per split)
    uint32_t *err;
    uint32_t failed = 0;  // error bits any call of this model has met
    CUtensorMap mW[3];
    TrainMaps tmaps;
    WgradMaps gmaps;
    std::vector<float> h_flat;  // gradients or parameters on their way to the caller's tensors
    int adam_t = 0;
    uint64_t launches = 0;
    // training pool: samples kept on the device (grown by doubling), and the
    // per-step batch losses of a training call
    float *pool_X = nullptr, *pool_t = nullptr;
    uint64_t pool_n = 0, pool_cap = 0;
    float *loss_hist = nullptr;
    uint32_t loss_cap = 0;
    // an inference call of more than a batch: outputs gathered on the device,
    // two pieces of inputs and the stream that copies them in
    float *y_all = nullptr;
    uint64_t y_all_cap = 0;
    float *in[2] = {};
    cudaStream_t in_stream = nullptr;
    cudaEvent_t in_here[2] = {}, in_used[2] = {};

    void *alloc(size_t bytes) {
        void *p = nullptr;
        if (cudaMalloc(&p, (bytes + 255) & ~size_t(255)) != cudaSuccess) return nullptr;
        blocks.push_back(p);
        return p;
    }
    ~lpsim_mlp() {
        if (stream) cudaStreamSynchronize(stream);
        for (void *b : blocks) cudaFree(b);
        cudaFree(pool_X);
        cudaFree(pool_t);
        cudaFree(loss_hist);
        cudaFree(y_all);
        if (in_stream) cudaStreamDestroy(in_stream);
        for (int b = 0; b < 2; b++) {
            cudaFree(in[b]);
            if (in_here[b]) cudaEventDestroy(in_here[b]);
            if (in_used[b]) cudaEventDestroy(in_used[b]);
        }
        if (own_stream) cudaStreamDestroy(stream);
    }
};

namespace {

const int kDims[5] = {64, 256, 256, 256, 1};

constexpr int kLossAt = (param_off(8) + 3) / 4 * 4, kErrAt = kLossAt + 1;  // in the gradients' flat array

int err_status(lpsim_mlp *m, uint32_t e) {
    e = m->failed |= e;
    if (e & 64u) return fail(LPSIM_E_TIMEOUT, "training-pool permutation walk exceeded its bound");
    if (e) return fail(LPSIM_E_TIMEOUT, "tensor-core GEMM wait gave up (code " + std::to_string(e) + ")");
    return LPSIM_OK;
}

int mlp_check_err(lpsim_mlp *m) {
    uint32_t e = 0;
    CU(cudaMemcpyAsync(&e, m->err, 4, cudaMemcpyDeviceToHost, m->stream));
    CU(cudaStreamSynchronize(m->stream));
    return err_status(m, e);
}

int refresh_weights(lpsim_mlp *m) {
    for (int l = 0; l < 3; l++) {
        weights_to_bf16<<<64, 256, 0, m->stream>>>(m->P[2 * l], kDims[l + 1], kDims[l], m->Wb[l], m->WbT[l]);
        m->launches++;
    }
    CU(cudaGetLastError());
    return LPSIM_OK;
}

// The next Adam step's constants: beta1 0.9, beta2 0.999, eps 1e-8 as FP32
// constants; the bias corrections 1 - beta^t are formed in double from those
// FP32 values and rounded once (in float arithmetic 1 - beta2^t loses most of
// its digits to cancellation).
void adam_constants(lpsim_mlp *m, float lr, UpdateArgs &u) {
    m->adam_t++;
    u.adam = 1;
    u.lr = lr;
    u.b1 = 0.9f;
    u.b2 = 0.999f;
    u.eps = 1e-8f;
    u.c1 = (float)(1.0 - std::pow((double)u.b1, (double)m->adam_t));
    u.c2 = (float)(1.0 - std::pow((double)u.b2, (double)m->adam_t));
}

// Splits of mlp_wgrad's rows (kt slices of 64): two CTAs per SM at most (ten
// tiles per split), and at least four slices each.  Measured, us per training
// step with caps of 15 / 30 splits: 8192 rows 41.6 / 40.5, 32768 rows 126 /
// 120, 155648 rows 455 / 440; with at least 2 / 4 / 16 slices: 1024 rows 34.9 /
// 36.4 / 39.6, 8192 rows 40.6 / 40.5 / 42.7.
int wgrad_splits(const lpsim_mlp *m, int kt) {
    return std::max(1, std::min(kt / 4, 2 * m->n_sm / kWgTiles));
}

// forward and backward of n rows (X, t: the batch in order, or drawn from a
// pool of pool_n rows from position pos0 of its shuffled passes on), leaving
// the partial sums for mlp_update
int train_core(lpsim_mlp *m, const float *X, const float *t, uint32_t n, uint64_t pool_n, uint32_t h, uint64_t seed,
               uint64_t pos0, UpdateArgs &u) {
    CU(cudaFuncSetAttribute(mlp_train_fused, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTrSmem));
    CU(cudaFuncSetAttribute(mlp_wgrad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWgSmem));
    TrainArgs g{};
    g.n_rows = (int)n;
    g.n_tiles = (int)((n + kBM - 1) / kBM);
    g.nf = m->nf;
    g.l1_k16 = (m->nf + 15) / 16;
    g.X = X;
    g.t = t;
    g.pool_n = pool_n;
    g.seed = seed;
    g.pos0 = pos0;
    g.h = h;
    g.b1 = m->P[1];
    g.b2 = m->P[3];
    g.b3 = m->P[5];
    g.w4 = m->P[6];
    g.b4 = m->P[7];
    g.small = m->small;
    g.err = m->err;
    u.clusters = std::min(g.n_tiles, m->n_sm / 2);
    TRY(launch_dependent(mlp_train_fused, dim3(2 * u.clusters), kTrThreads, kTrSmem, m->stream, m->tmaps, g));
    const int kt = 2 * g.n_tiles, want = wgrad_splits(m, kt), per = (kt + want - 1) / want;
    u.splits = (kt + per - 1) / per;
    TRY(launch_dependent(mlp_wgrad, dim3(kWgTiles, u.splits), kThreads, kWgSmem, m->stream, m->gmaps, kt, per, m->part,
                         m->err));
    m->launches += 2;
    u.part = m->part;
    u.small = m->small;
    u.P = m->Pf;
    u.Mo = m->Mf;
    u.Ve = m->Vf;
    for (int l = 0; l < 3; l++) {
        u.Wb[l] = m->Wb[l];
        u.WbT[l] = m->WbT[l];
    }
    return LPSIM_OK;
}

int train_update(lpsim_mlp *m, const UpdateArgs &u) {
    m->launches++;
    return launch_dependent(mlp_update, dim3(kUpdBlocks + kUpdSmallBlocks), 256, 0, m->stream, u);
}

// inference forward of n rows of m->nf inputs (device) into y
int forward_fused(lpsim_mlp *m, const float *X, uint64_t n, float *y, uint32_t *err) {
    CU(cudaFuncSetAttribute(mlp_forward_fused, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFwdSmem));
    FwdArgs g{};
    g.n_rows = (int)n;
    g.n_tiles = (int)((n + kBM - 1) / kBM);
    g.nf = m->nf;
    g.X = X;
    g.l1_k16 = (m->nf + 15) / 16;
    g.b1 = m->P[1];
    g.b2 = m->P[3];
    g.b3 = m->P[5];
    g.w4 = m->P[6];
    g.b4 = m->P[7];
    g.y = y;
    g.err = err;
    const int grid = std::min(g.n_tiles, m->n_sm);
    mlp_forward_fused<<<grid, kFwdThreads, kFwdSmem, m->stream>>>(m->mW[0], m->mW[1], m->mW[2], g);
    m->launches++;
    CU(cudaGetLastError());
    return LPSIM_OK;
}

// Inference calls of at most this many rows bring their outputs and the error
// word over in one copy, then copy the outputs on the host (a copy from the
// device costs some 8 us however small).
constexpr uint64_t kOneCopyRows = 16384;

// Rows per launch of a long inference call: four tiles per SM, whole waves, for
// which the kernel takes 35.5 us and the copy in 22 us.  (One launch per batch
// of 8192 rows kept 64 of the 152 SMs busy for 14.9 us each and the host with
// 735 calls: 2,000,003 rows 9.9 ms, now 1.08 ms, 0.92 ms of it the kernel.)
// Every tile's result is its own, so the split does not show in the outputs.
uint64_t forward_piece(const lpsim_mlp *m) { return 4ull * m->n_sm * kBM; }

// A long inference call: pieces of the rows, two on the device at once, so that
// one is copied in (on a stream of the model's own) while the other is computed.
// The copy stream is waited for before the caller's rows may go away.
int forward_pieces(lpsim_mlp *m, uint64_t n, const float *X, float *y) {
    const uint64_t piece = forward_piece(m);
    // the rows may be written by work on the caller's stream before this call (no one else has a
    // stream of the model's own)
    if (!m->own_stream) {
        CU(cudaEventRecord(m->in_used[0], m->stream));
        CU(cudaStreamWaitEvent(m->in_stream, m->in_used[0], 0));
    }
    for (uint64_t r0 = 0, i = 0; r0 < n; r0 += piece, i++) {
        const uint64_t nb = std::min(piece, n - r0);
        const int b = (int)(i & 1);
        if (i >= 2) CU(cudaStreamWaitEvent(m->in_stream, m->in_used[b], 0));
        CU(cudaMemcpyAsync(m->in[b], X + r0 * m->nf, nb * m->nf * 4, cudaMemcpyHostToDevice, m->in_stream));
        CU(cudaEventRecord(m->in_here[b], m->in_stream));
        CU(cudaStreamWaitEvent(m->stream, m->in_here[b], 0));
        TRY(forward_fused(m, m->in[b], nb, m->y_all + r0, m->err));
        CU(cudaEventRecord(m->in_used[b], m->stream));
    }
    CU(cudaMemcpyAsync(y, m->y_all, n * 4, cudaMemcpyDeviceToHost, m->stream));
    return LPSIM_OK;
}

// a flat parameter-shaped device array into the caller's tensors (each
// nullable): one copy, then host copies
int flat_to_tensors(lpsim_mlp *m, const float *flat, float *const *tensors) {
    m->h_flat.resize(std::max<size_t>(m->h_flat.size(), kErrAt + 1));
    CU(cudaMemcpyAsync(m->h_flat.data(), flat, (kErrAt + 1) * 4, cudaMemcpyDeviceToHost, m->stream));
    CU(cudaStreamSynchronize(m->stream));
    for (int i = 0; i < 8 && tensors; i++)
        if (tensors[i]) std::memcpy(tensors[i], m->h_flat.data() + param_off(i), (size_t)m->sz[i] * 4);
    return LPSIM_OK;
}

}  // namespace

extern "C" {

int lpsim_mlp_create(lpsim_mlp **out, uint32_t n_features, uint32_t batch, uint64_t seed, void *stream) {
    if (!out) return fail(LPSIM_E_INVALID_ARG, "out is NULL");
    *out = nullptr;
    if (n_features == 0 || n_features > 64) return fail(LPSIM_E_INVALID_ARG, "n_features must be 1..64");
    if (batch == 0 || batch % 128 != 0 || batch > (1u << 20))
        return fail(LPSIM_E_INVALID_ARG, "batch must be a positive multiple of 128 (at most 2^20)");
    auto *m = new (std::nothrow) lpsim_mlp();
    if (!m) return fail(LPSIM_E_OOM, "host allocation failed");
    auto bail = [&](int rc) {
        delete m;
        return rc;
    };
    cudaGetDevice(&m->device);
    cudaDeviceGetAttribute(&m->n_sm, cudaDevAttrMultiProcessorCount, m->device);
    m->stream = static_cast<cudaStream_t>(stream);
    if (!m->stream) {
        if (cudaStreamCreateWithFlags(&m->stream, cudaStreamNonBlocking) != cudaSuccess)
            return bail(fail(LPSIM_E_CUDA, "cannot create a stream"));
        m->own_stream = true;
    }
    m->nf = (int)n_features;
    m->B = (int)batch;
    const int B = m->B;
    for (int l = 0; l < 4; l++) {
        m->sz[2 * l] = kDims[l + 1] * kDims[l];
        m->sz[2 * l + 1] = kDims[l + 1];
    }
    const size_t flat = (size_t)(kErrAt + 1) * 4;
    m->Pf = (float *)m->alloc(flat);
    m->Gf = (float *)m->alloc(flat);
    m->Mf = (float *)m->alloc(flat);
    m->Vf = (float *)m->alloc(flat);
    const int max_kt = 2 * (B / kBM);
    m->small = (float *)m->alloc((size_t)std::max(1, std::min(B / kBM, m->n_sm / 2)) * kSmall * 4);
    m->part = (float *)m->alloc((size_t)wgrad_splits(m, max_kt) * kWgFloats * 4);
    if (!m->Pf || !m->Gf || !m->Mf || !m->Vf || !m->small || !m->part)
        return bail(fail(LPSIM_E_OOM, "device allocation failed"));
    for (int i = 0; i < 8; i++) m->P[i] = m->Pf + param_off(i);
    m->err = reinterpret_cast<uint32_t *>(m->Gf + kErrAt);
    for (int l = 0; l < 3; l++) {
        m->Wb[l] = (__nv_bfloat16 *)m->alloc(kDims[l + 1] * kDims[l] * 2);
        if (l > 0) m->WbT[l] = (__nv_bfloat16 *)m->alloc(kDims[l + 1] * kDims[l] * 2);
        if (l < 2) m->H[l] = (__nv_bfloat16 *)m->alloc((size_t)B * 256 * 2);
        m->dZ[l] = (__nv_bfloat16 *)m->alloc((size_t)B * 256 * 2);
        if (!m->Wb[l] || (l > 0 && !m->WbT[l]) || (l < 2 && !m->H[l]) || !m->dZ[l])
            return bail(fail(LPSIM_E_OOM, "device allocation failed"));
    }
    m->X0 = (__nv_bfloat16 *)m->alloc((size_t)B * 64 * 2);
    m->Xf = (float *)m->alloc((size_t)B * n_features * 4);
    m->y_block = (float *)m->alloc(((size_t)B + 4) * 4);
    m->y = m->y_block ? m->y_block + 4 : nullptr;
    m->t = (float *)m->alloc((size_t)B * 4);
    if (!m->X0 || !m->Xf || !m->y || !m->t) return bail(fail(LPSIM_E_OOM, "device allocation failed"));
    if (cudaMemsetAsync(m->err, 0, 4, m->stream) != cudaSuccess ||
        cudaMemsetAsync(m->y_block, 0, 16, m->stream) != cudaSuccess) return bail(fail(LPSIM_E_CUDA, "memset"));
    // tensor maps of every operand
    int rc;
    TrainMaps &tm = m->tmaps;
    WgradMaps &gm = m->gmaps;
    const __nv_bfloat16 *wsrc[5] = {m->Wb[0], m->Wb[1], m->Wb[2], m->WbT[2], m->WbT[1]};
    if ((rc = make_map(&tm.x0, m->X0, B, 64, kBM)) || (rc = make_map(&gm.x0, m->X0, B, 64, 64))) return bail(rc);
    for (int s = 0; s < 5; s++)
        if ((rc = make_map(&tm.w[s], wsrc[s], 256, s == 0 ? 64 : 256, 128))) return bail(rc);
    for (int l = 0; l < 3; l++) {
        if ((rc = make_map(&m->mW[l], m->Wb[l], 256, kDims[l], 256)) ||
            (rc = make_map(&tm.dz[l], m->dZ[l], B, 256, 32)) || (rc = make_map(&gm.dz[l], m->dZ[l], B, 256, 64)))
            return bail(rc);
        if (l < 2 && ((rc = make_map(&tm.h[l], m->H[l], B, 256, 32)) || (rc = make_map(&gm.h[l], m->H[l], B, 256, 64))))
            return bail(rc);
    }
    // He initialisation (host, seeded), then upload
    std::mt19937_64 gen(seed);
    std::normal_distribution<double> nd(0.0, 1.0);
    for (int l = 0; l < 4; l++) {
        const int fan_in = l == 0 ? (int)n_features : kDims[l];
        std::vector<float> w(m->sz[2 * l]), b(m->sz[2 * l + 1], 0.0f);
        for (int o = 0; o < kDims[l + 1]; o++)
            for (int k = 0; k < kDims[l]; k++)
                w[(size_t)o * kDims[l] + k] =
                    (l == 0 && k >= (int)n_features) ? 0.0f : (float)(nd(gen) * std::sqrt(2.0 / fan_in));
        if (cudaMemcpy(m->P[2 * l], w.data(), w.size() * 4, cudaMemcpyHostToDevice) != cudaSuccess ||
            cudaMemcpy(m->P[2 * l + 1], b.data(), b.size() * 4, cudaMemcpyHostToDevice) != cudaSuccess)
            return bail(fail(LPSIM_E_CUDA, "parameter upload failed"));
    }
    cudaMemsetAsync(m->Mf, 0, flat, m->stream);
    cudaMemsetAsync(m->Vf, 0, flat, m->stream);
    if ((rc = refresh_weights(m))) return bail(rc);
    if (cudaStreamSynchronize(m->stream) != cudaSuccess) return bail(fail(LPSIM_E_CUDA, "init failed"));
    *out = m;
    return LPSIM_OK;
}

int lpsim_mlp_set_params(lpsim_mlp *m, const float *const *tensors) {
    if (!m || !tensors) return fail(LPSIM_E_INVALID_ARG, "NULL argument");
    for (int i = 0; i < 8; i++) {
        if (!tensors[i]) return fail(LPSIM_E_INVALID_ARG, "parameter tensor is NULL");
        CU(cudaMemcpyAsync(m->P[i], tensors[i], m->sz[i] * 4, cudaMemcpyHostToDevice, m->stream));
    }
    CU(cudaMemsetAsync(m->Mf, 0, param_off(8) * 4, m->stream));
    CU(cudaMemsetAsync(m->Vf, 0, param_off(8) * 4, m->stream));
    m->adam_t = 0;
    TRY(refresh_weights(m));
    CU(cudaStreamSynchronize(m->stream));
    return LPSIM_OK;
}

int lpsim_mlp_get_params(lpsim_mlp *m, float *const *tensors) {
    if (!m || !tensors) return fail(LPSIM_E_INVALID_ARG, "NULL argument");
    return flat_to_tensors(m, m->Pf, tensors);
}

int lpsim_mlp_forward(lpsim_mlp *m, uint64_t n, const float *X, float *y) {
    if (!m || !X || !y) return fail(LPSIM_E_INVALID_ARG, "NULL argument");
    if (n <= (uint64_t)m->B) {
        if (n == 0) return mlp_check_err(m);
        CU(cudaMemcpyAsync(m->Xf, X, n * m->nf * 4, cudaMemcpyHostToDevice, m->stream));
        if (n <= kOneCopyRows) {
            m->h_flat.resize(std::max<size_t>(m->h_flat.size(), n + 4));
            TRY(forward_fused(m, m->Xf, n, m->y, reinterpret_cast<uint32_t *>(m->y_block)));
            CU(cudaMemcpyAsync(m->h_flat.data(), m->y_block, (n + 4) * 4, cudaMemcpyDeviceToHost, m->stream));
            CU(cudaStreamSynchronize(m->stream));
            uint32_t e;
            std::memcpy(&e, m->h_flat.data(), 4);
            TRY(err_status(m, e));
            std::memcpy(y, m->h_flat.data() + 4, n * 4);
            return LPSIM_OK;
        }
        TRY(forward_fused(m, m->Xf, n, m->y, m->err));
        CU(cudaMemcpyAsync(y, m->y, n * 4, cudaMemcpyDeviceToHost, m->stream));
        return mlp_check_err(m);
    }
    if (n > m->y_all_cap) {
        CU(cudaStreamSynchronize(m->stream));
        cudaFree(m->y_all);
        m->y_all = nullptr;
        m->y_all_cap = 0;
        if (cudaMalloc(&m->y_all, n * 4) != cudaSuccess) {
            m->y_all = nullptr;
            return fail(LPSIM_E_OOM, "device allocation of the outputs failed");
        }
        m->y_all_cap = n;
    }
    if (!m->in_stream) {
        const size_t bytes = forward_piece(m) * m->nf * 4;
        for (int b = 0; b < 2; b++) {
            if (!m->in[b] && cudaMalloc(&m->in[b], bytes) != cudaSuccess) {
                m->in[b] = nullptr;
                return fail(LPSIM_E_OOM, "device allocation of the input pieces failed");
            }
            if (!m->in_here[b]) CU(cudaEventCreateWithFlags(&m->in_here[b], cudaEventDisableTiming));
            if (!m->in_used[b]) CU(cudaEventCreateWithFlags(&m->in_used[b], cudaEventDisableTiming));
        }
        CU(cudaStreamCreateWithFlags(&m->in_stream, cudaStreamNonBlocking));
    }
    const int rc = forward_pieces(m, n, X, y);
    const cudaError_t e = cudaStreamSynchronize(m->in_stream);
    const int rc2 = mlp_check_err(m);
    if (rc) return rc;
    if (e != cudaSuccess) return fail(LPSIM_E_CUDA, std::string("input copies: ") + cudaGetErrorString(e));
    return rc2;
}

int lpsim_mlp_grad(lpsim_mlp *m, uint64_t n, const float *X, const float *t, float *loss, float *const *grads) {
    if (!m || !X || !t) return fail(LPSIM_E_INVALID_ARG, "NULL argument");
    if (n == 0 || n > (uint64_t)m->B) return fail(LPSIM_E_INVALID_ARG, "n must be 1..batch");
    CU(cudaMemcpyAsync(m->Xf, X, n * m->nf * 4, cudaMemcpyHostToDevice, m->stream));
    CU(cudaMemcpyAsync(m->t, t, n * 4, cudaMemcpyHostToDevice, m->stream));
    UpdateArgs u{};
    TRY(train_core(m, m->Xf, m->t, (uint32_t)n, 0, 0, 0, 0, u));
    u.G = m->Gf;
    u.loss = m->Gf + kLossAt;
    TRY(train_update(m, u));
    TRY(flat_to_tensors(m, m->Gf, grads));
    uint32_t e;
    std::memcpy(&e, &m->h_flat[kErrAt], 4);
    TRY(err_status(m, e));
    if (loss) *loss = m->h_flat[kLossAt] / (float)n;
    return LPSIM_OK;
}

int lpsim_mlp_pool_clear(lpsim_mlp *m) {
    if (!m) return fail(LPSIM_E_INVALID_ARG, "NULL argument");
    m->pool_n = 0;
    return LPSIM_OK;
}

uint64_t lpsim_mlp_pool_size(const lpsim_mlp *m) { return m ? m->pool_n : 0; }

int lpsim_mlp_pool_add(lpsim_mlp *m, uint64_t n, const float *X, const float *t) {
    if (!m || (n && (!X || !t))) return fail(LPSIM_E_INVALID_ARG, "NULL argument");
    if (n == 0) return LPSIM_OK;
    const uint64_t need = m->pool_n + n;
    if (need >= (1ull << 40)) return fail(LPSIM_E_INVALID_ARG, "training pool too large");
    if (need > m->pool_cap) {
        // grow by doubling; the rows so far move to the new buffers
        const uint64_t cap = std::max<uint64_t>(need, std::max<uint64_t>(2 * m->pool_cap, 1u << 16));
        float *nx = nullptr, *nt = nullptr;
        if (cudaMalloc(&nx, cap * m->nf * 4) != cudaSuccess || cudaMalloc(&nt, cap * 4) != cudaSuccess) {
            cudaFree(nx);
            return fail(LPSIM_E_OOM, "device allocation of the training pool failed");
        }
        if (m->pool_n) {
            CU(cudaMemcpyAsync(nx, m->pool_X, m->pool_n * m->nf * 4, cudaMemcpyDeviceToDevice, m->stream));
            CU(cudaMemcpyAsync(nt, m->pool_t, m->pool_n * 4, cudaMemcpyDeviceToDevice, m->stream));
        }
        CU(cudaStreamSynchronize(m->stream));
        cudaFree(m->pool_X);
        cudaFree(m->pool_t);
        m->pool_X = nx;
        m->pool_t = nt;
        m->pool_cap = cap;
    }
    CU(cudaMemcpyAsync(m->pool_X + m->pool_n * m->nf, X, n * m->nf * 4, cudaMemcpyHostToDevice, m->stream));
    CU(cudaMemcpyAsync(m->pool_t + m->pool_n, t, n * 4, cudaMemcpyHostToDevice, m->stream));
    CU(cudaStreamSynchronize(m->stream));
    m->pool_n = need;
    return LPSIM_OK;
}

int lpsim_mlp_train_pool(lpsim_mlp *m, uint32_t steps, float lr, uint64_t shuffle_seed, float *losses) {
    if (!m) return fail(LPSIM_E_INVALID_ARG, "NULL argument");
    const uint64_t n = m->pool_n;
    if (n == 0) return fail(LPSIM_E_INVALID_ARG, "no samples in the training pool");
    if (steps > m->loss_cap) {
        cudaFree(m->loss_hist);
        m->loss_hist = nullptr;
        m->loss_cap = 0;
        if (cudaMalloc(&m->loss_hist, (size_t)steps * 4) != cudaSuccess)
            return fail(LPSIM_E_OOM, "device allocation of the loss record failed");
        m->loss_cap = steps;
    }
    uint32_t h = 1;
    while ((1ull << (2 * h)) < n) h++;
    const uint32_t nb = (uint32_t)std::min<uint64_t>(m->B, n);
    cudaStream_t st = m->stream;
    for (uint32_t s = 0; s < steps; s++) {
        // the next minibatch of the shuffled passes, drawn by the training kernel
        UpdateArgs u{};
        TRY(train_core(m, m->pool_X, m->pool_t, nb, n, h, shuffle_seed, (uint64_t)s * nb, u));
        adam_constants(m, lr, u);
        u.loss = m->loss_hist + s;
        TRY(train_update(m, u));
    }
    CU(cudaGetLastError());
    if (losses && steps) {
        CU(cudaMemcpyAsync(losses, m->loss_hist, (size_t)steps * 4, cudaMemcpyDeviceToHost, st));
        CU(cudaStreamSynchronize(st));
        for (uint32_t s = 0; s < steps; s++) losses[s] /= (float)nb;
    }
    CU(cudaStreamSynchronize(st));
    return mlp_check_err(m);
}

int lpsim_mlp_train(lpsim_mlp *m, uint64_t n, const float *X, const float *t, uint32_t steps, float lr,
                    uint64_t shuffle_seed, float *losses) {
    if (!m || !X || !t) return fail(LPSIM_E_INVALID_ARG, "NULL argument");
    if (n == 0) return fail(LPSIM_E_INVALID_ARG, "no samples");
    TRY(lpsim_mlp_pool_clear(m));
    TRY(lpsim_mlp_pool_add(m, n, X, t));
    return lpsim_mlp_train_pool(m, steps, lr, shuffle_seed, losses);
}

int lpsim_mlp_apply_grads(lpsim_mlp *m, const float *const *grads, float lr) {
    if (!m || !grads) return fail(LPSIM_E_INVALID_ARG, "NULL argument");
    if (!(lr >= 0.0f) || !std::isfinite(lr)) return fail(LPSIM_E_INVALID_ARG, "lr must be finite and >= 0");
    for (int i = 0; i < 8; i++)
        if (!grads[i]) return fail(LPSIM_E_INVALID_ARG, "gradient tensor is NULL");
    CU(cudaStreamSynchronize(m->stream));
    for (int i = 0; i < 8; i++)
        CU(cudaMemcpyAsync(m->Gf + param_off(i), grads[i], m->sz[i] * 4, cudaMemcpyHostToDevice, m->stream));
    UpdateArgs u{};
    u.G = m->Gf;
    u.P = m->Pf;
    u.Mo = m->Mf;
    u.Ve = m->Vf;
    adam_constants(m, lr, u);
    adam_given<<<(param_off(8) + 255) / 256, 256, 0, m->stream>>>(u);
    m->launches++;
    CU(cudaGetLastError());
    TRY(refresh_weights(m));
    CU(cudaStreamSynchronize(m->stream));
    return LPSIM_OK;
}

int lpsim_mlp_gemm_test(uint32_t M, uint32_t N, uint32_t K, const uint16_t *A, const uint16_t *B, float *D) {
    if (!A || !B || !D) return fail(LPSIM_E_INVALID_ARG, "NULL argument");
    if (M == 0 || M % 128 || (N != 64 && N % 256) || K == 0 || K % 64)
        return fail(LPSIM_E_INVALID_ARG, "M % 128, K % 64 must be 0 and N 64 or a multiple of 256");
    void *dA = nullptr, *dB = nullptr, *dD = nullptr, *dE = nullptr;
    int rc = LPSIM_OK;
    cudaStream_t st = nullptr;
    if (cudaMalloc(&dA, (size_t)M * K * 2) || cudaMalloc(&dB, (size_t)N * K * 2) || cudaMalloc(&dD, (size_t)M * N * 4) ||
        cudaMalloc(&dE, 16))
        rc = fail(LPSIM_E_OOM, "device allocation failed");
    CUtensorMap ma, mb;
    if (!rc) {
        cudaMemcpy(dA, A, (size_t)M * K * 2, cudaMemcpyHostToDevice);
        cudaMemcpy(dB, B, (size_t)N * K * 2, cudaMemcpyHostToDevice);
        cudaMemset(dD, 0, (size_t)M * N * 4);
        cudaMemset(dE, 0, 16);
        rc = make_map(&ma, dA, M, K, kBM);
        if (!rc) rc = make_map(&mb, dB, N, K, N == 64 ? 64 : 256);
    }
    if (!rc) {
        GemmArgs g{};
        g.M = (int)M;
        g.N = (int)N;
        g.K = (int)K;
        g.fout = (float *)dD;
        g.err = (uint32_t *)dE;
        rc = N == 64 ? launch_gemm<64>(ma, mb, g, st) : launch_gemm<256>(ma, mb, g, st);
    }
    if (!rc) {
        uint32_t e = 0;
        if (cudaDeviceSynchronize() != cudaSuccess) rc = fail(LPSIM_E_CUDA, cudaGetErrorString(cudaGetLastError()));
        else {
            cudaMemcpy(&e, dE, 4, cudaMemcpyDeviceToHost);
            cudaMemcpy(D, dD, (size_t)M * N * 4, cudaMemcpyDeviceToHost);
            if (e) rc = fail(LPSIM_E_TIMEOUT, "GEMM wait gave up (code " + std::to_string(e) + ")");
        }
    }
    cudaFree(dA);
    cudaFree(dB);
    cudaFree(dD);
    cudaFree(dE);
    return rc;
}

int lpsim_mlp_time(lpsim_mlp *m, uint32_t iters, double *fwd_ms, double *train_ms) {
    if (!m || iters == 0) return fail(LPSIM_E_INVALID_ARG, "bad argument");
    cudaEvent_t e0, e1;
    CU(cudaEventCreate(&e0));
    CU(cudaEventCreate(&e1));
    // whatever the batch buffers hold is a valid input; warm up once
    TRY(forward_fused(m, m->Xf, (uint64_t)m->B, m->y, m->err));
    CU(cudaEventRecord(e0, m->stream));
    for (uint32_t i = 0; i < iters; i++) TRY(forward_fused(m, m->Xf, (uint64_t)m->B, m->y, m->err));
    CU(cudaEventRecord(e1, m->stream));
    CU(cudaEventSynchronize(e1));
    float ms = 0.0f;
    CU(cudaEventElapsedTime(&ms, e0, e1));
    if (fwd_ms) *fwd_ms = ms / iters;
    if (train_ms) {
        CU(cudaEventRecord(e0, m->stream));
        for (uint32_t i = 0; i < iters; i++) {
            UpdateArgs u{};
            TRY(train_core(m, m->Xf, m->t, (uint32_t)m->B, 0, 0, 0, 0, u));
            u.G = m->Gf;
            u.loss = m->Gf + kLossAt;
            TRY(train_update(m, u));
        }
        CU(cudaEventRecord(e1, m->stream));
        CU(cudaEventSynchronize(e1));
        CU(cudaEventElapsedTime(&ms, e0, e1));
        *train_ms = ms / iters;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return mlp_check_err(m);
}

int lpsim_mlp_gelu_eval(uint64_t n, const float *z, float *gelu, float *dgelu) {
    if (!z || !gelu || !dgelu) return fail(LPSIM_E_INVALID_ARG, "NULL argument");
    if (n == 0) return LPSIM_OK;
    float *dz = nullptr;
    CU(cudaMalloc(&dz, n * 12));
    cudaError_t e = cudaMemcpy(dz, z, n * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        gelu_eval<<<(unsigned)std::min<uint64_t>((n + 255) / 256, 4096), 256>>>(dz, n, dz + n, dz + 2 * n);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(gelu, dz + n, n * 4, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(dgelu, dz + 2 * n, n * 4, cudaMemcpyDeviceToHost);
    cudaFree(dz);
    if (e != cudaSuccess) return fail(LPSIM_E_CUDA, std::string("gelu_eval: ") + cudaGetErrorString(e));
    return LPSIM_OK;
}

void lpsim_mlp_destroy(lpsim_mlp *m) { delete m; }

}  // extern "C"
