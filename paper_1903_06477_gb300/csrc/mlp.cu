// mlp.cu -- the learned warm start: a 3-layer MLP trained and evaluated
// entirely by the kernels in this file (see include/superscs_mlp.h).
//
// Every product is C = A B^T in BF16 with FP32 accumulation, on one of two
// kernels: gemm_tc (default), tcgen05.mma fed by TMA with the accumulators in
// tensor memory, whose operands may be stored K-contiguous or row-contiguous
// (the backward pass reads the activations and weights as they are), or
// gemm_nt, the warp-level MMA (m16n8k16) on 128x128x32 tiles staged by
// cp.async, which takes K-contiguous operands only (the backward pass then
// works on transposed copies made by a tiled transpose kernel).
#include <cuda.h>  // CUtensorMap and its enums (types only: the encoder is reached through the runtime)
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <atomic>
#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cstdint>
#include <mutex>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "../../include/superscs.h"
#include "../../include/superscs_mlp.h"

namespace sscs {
void record_error(const char* msg);
}

namespace {

typedef __nv_bfloat16 bf16;

constexpr int BM = 128, BN = 128, BK = 32, NTH = 256, SROW = BK + 8;  // 80-byte smem rows: ldmatrix conflict-free

struct Epi {
    const float* bias;  // per column, or null
    const bf16* mask;   // relu' mask (value > 0 keeps), row-major with ldm, or null
    int ldm;
    int relu;
    float* C32;         // FP32 output or null
    int ldc;
    bf16* C16;          // BF16 output or null
    int ldc16;
    float* Y;           // gemm_tc: second FP32 output, (value) * std + mean per column (row stride ldc), or null
    const float* ystd;
    const float* ymean;
};

__device__ __forceinline__ unsigned sa(const void* p) { return static_cast<unsigned>(__cvta_generic_to_shared(p)); }

// 16-byte async copy with zero fill of the bytes past src_bytes
__device__ __forceinline__ void cp16(void* dst, const void* src, int src_bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sa(dst)), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_wait1() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }
__device__ __forceinline__ void cp_wait0() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

__device__ __forceinline__ void ldsm_x4(unsigned& r0, unsigned& r1, unsigned& r2, unsigned& r3, const void* p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(sa(p)));
}

__device__ __forceinline__ void mma_bf16(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// C[M x N] = A[M x K] * B[N x K]^T.  lda, ldb multiples of 8, A and B 16-byte
// aligned; tails in M, N and K are zero-filled on load and masked on store.
__global__ void __launch_bounds__(NTH) gemm_nt(int M, int N, int K, const bf16* __restrict__ A, int lda,
                                               const bf16* __restrict__ Bm, int ldb, Epi e)
{
    __shared__ __align__(16) bf16 As[2][BM][SROW];
    __shared__ __align__(16) bf16 Bs[2][BN][SROW];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wm = warp >> 2, wn = warp & 3;  // 2 x 4 warps, 64 x 32 each
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    float acc[4][4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.f;

    auto load = [&](int st, int k0) {
        for (int c = tid; c < BM * (BK / 8); c += NTH) {
            const int r = c >> 2, kc = (c & 3) * 8;
            const int gk = k0 + kc;
            int gm = m0 + r;
            int bytes = (gm < M && gk < K) ? min(16, (K - gk) * 2) : 0;
            const bf16* src = bytes ? A + (size_t)gm * lda + gk : A;
            cp16(&As[st][r][kc], src, bytes);
            const int gn = n0 + r;
            bytes = (gn < N && gk < K) ? min(16, (K - gk) * 2) : 0;
            src = bytes ? Bm + (size_t)gn * ldb + gk : Bm;
            cp16(&Bs[st][r][kc], src, bytes);
        }
    };

    const int KT = (K + BK - 1) / BK;
    load(0, 0);
    cp_commit();
    for (int kt = 0; kt < KT; ++kt) {
        const int st = kt & 1;
        if (kt + 1 < KT) {
            load(st ^ 1, (kt + 1) * BK);
            cp_commit();
            cp_wait1();
        } else {
            cp_wait0();
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BK; kk += 16) {
            unsigned af[4][4];
#pragma unroll
            for (int mi = 0; mi < 4; ++mi) {
                const int row = wm * 64 + mi * 16 + (lane & 15);
                const int col = kk + (lane >> 4) * 8;
                ldsm_x4(af[mi][0], af[mi][1], af[mi][2], af[mi][3], &As[st][row][col]);
            }
            unsigned bfr[4][2];
#pragma unroll
            for (int nj = 0; nj < 4; nj += 2) {
                const int row = wn * 32 + nj * 8 + (lane & 7) + (lane >> 4) * 8;
                const int col = kk + ((lane >> 3) & 1) * 8;
                ldsm_x4(bfr[nj][0], bfr[nj][1], bfr[nj + 1][0], bfr[nj + 1][1], &Bs[st][row][col]);
            }
#pragma unroll
            for (int mi = 0; mi < 4; ++mi)
#pragma unroll
                for (int ni = 0; ni < 4; ++ni) mma_bf16(acc[mi][ni], af[mi], bfr[ni][0], bfr[ni][1]);
        }
        __syncthreads();
    }
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int mi = 0; mi < 4; ++mi)
#pragma unroll
        for (int ni = 0; ni < 4; ++ni)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int m = m0 + wm * 64 + mi * 16 + g + h * 8;
                if (m >= M) continue;
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int n = n0 + wn * 32 + ni * 8 + 2 * t + q;
                    if (n >= N) continue;
                    float v = acc[mi][ni][h * 2 + q];
                    if (e.bias) v += e.bias[n];
                    if (e.mask && !((float)e.mask[(size_t)m * e.ldm + n] > 0.f)) v = 0.f;
                    if (e.relu) v = fmaxf(v, 0.f);
                    if (e.C32) e.C32[(size_t)m * e.ldc + n] = v;
                    if (e.C16) e.C16[(size_t)m * e.ldc16 + n] = __float2bfloat16(v);
                }
            }
}

// ---------------------------------------------------------------------------
// The same product C = A B^T on the fifth-generation tensor cores.
//
// Operands arrive by TMA from 2D tensor maps with the 128-byte swizzle, zeros
// past M, N and K, so the kernel needs no tail logic.  An operand stored with
// K contiguous is copied in boxes of 64 K by its tile's rows; one stored with
// its rows contiguous (AMN, BMN) in boxes of 64 rows by 64 K, and the MMA is
// told that it is row-major ("MN-major").  A CTA computes an (MT * 128) x bn
// tile.  A ring of stages (one K block of 64 of both operands each) is filled
// by one producer lane (warp 0) and drained by one MMA lane (warp 1), which
// issues the 128 x bn x 16 tcgen05.mma of a stage from shared-memory
// descriptors and commits them to the stage's "empty" barrier, which frees it
// for the producer.  After the last stage a commit to the "done" barrier hands
// the accumulators in tensor memory to the eight epilogue warps (2..9), two a
// lane quarter (warp % 4): each reads 32 columns at a time with tcgen05.ld,
// turns the 32 x 32 values through shared memory (the idle ring) and then works
// on rows, four columns a lane: bias, ReLU mask, ReLU, FP32 / BF16 /
// denormalised output, in 16-byte stores.
//
// K is cut into `splits` ranges whose FP32 partial sums are added in order (a
// fixed order, so results do not depend on the tile shape).  Up to spc of them
// run in one CTA, one after the other, each with accumulators of its own in
// tensor memory; with more (grid z > 1) every range goes to a workspace that a
// second kernel adds up before the same epilogue.  tc_plan chooses.  Every wait
// is bounded; on expiry *err is set (1; 2 if copies or MMAs in flight did not
// drain either) and the tile is not written.
//
// Batch 256, network 2000-1024-1024-22004, against 128 x 128 tiles one CTA an
// SM with scalar epilogue stores and K-contiguous copies: see tc_plan.
// ---------------------------------------------------------------------------
constexpr int TC_BK = 64, TC_NTH = 320, TC_MAX_STAGES = 8;
constexpr int TC_BOX = 128 * TC_BK * 2;                    // bytes of 128 rows of one K block (16 KB)
constexpr int TC_CHUNK = 64 * TC_BK * 2;                   // bytes of one 64 x 64 box (8 KB)
constexpr int TC_STG = 36;                                 // row stride (floats) of an epilogue warp's 32 x 32 values
constexpr int TC_SMEM_MAX = 220 * 1024;                    // dynamic shared memory a CTA may take
constexpr unsigned long long TC_WAIT_NS = 2000000000ull;
// kind::f16 instruction descriptor: D FP32 (bits 4-5 = 1), A and B BF16
// (bits 7-9 = 1, 10-12 = 1), bits 15 / 16: A / B row-major, N >> 3 in bits
// 17-22, M >> 4 in bits 24-28
constexpr unsigned TC_IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(128 >> 4) << 24);

struct TcPlan {
    int mt;       // 128-row sub-tiles of a CTA (1 or 2)
    int bn;       // columns of a CTA's tile (a multiple of 32, at most 256)
    int stages;   // ring depth
    int per;      // K blocks of one range
    int splits;   // ranges
    int spc;      // ranges of one CTA (grid z = ceil(splits / spc))
    int cols;     // tensor memory columns (a power of two)
};

__device__ __forceinline__ unsigned long long tc_now()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ bool tc_try_wait(unsigned bar, unsigned parity)
{
    unsigned ok;
    asm volatile(
        "{\n .reg .pred P;\n mbarrier.try_wait.parity.shared::cta.b64 P, [%1], %2;\n selp.b32 %0, 1, 0, P;\n}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ bool tc_wait(unsigned bar, unsigned parity)
{
    if (tc_try_wait(bar, parity)) return true;
    const unsigned long long t0 = tc_now();
    while (!tc_try_wait(bar, parity))
        if (tc_now() - t0 > TC_WAIT_NS) return false;
    return true;
}
// Shared-memory matrix descriptor with the 128-byte swizzle: start >> 4 (bits
// 0-13), leading offset >> 4 (bits 16-29), stride offset >> 4 (bits 32-45),
// descriptor version 1 (bits 46-47), swizzle mode 2 = 128 bytes (bits 61-63).
// K-contiguous: the stride is the 1024 bytes between groups of 8 rows (no
// leading offset in a swizzled layout).  Row-contiguous: the stride is the 1024
// bytes between groups of 8 K, the leading offset that between 64-row boxes.
__device__ __forceinline__ unsigned long long tc_desc(unsigned addr, unsigned leading)
{
    return (unsigned long long)((addr >> 4) & 0x3FFFu) | ((unsigned long long)((leading >> 4) & 0x3FFFu) << 16) |
           ((unsigned long long)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
__device__ __forceinline__ void tc_mma(unsigned tmem, unsigned long long ad, unsigned long long bd, unsigned idesc,
                                       unsigned acc)
{
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem),
        "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
        : "memory");
}
__device__ __forceinline__ void tc_tma_2d(unsigned dst, const CUtensorMap* map, int x, int y, unsigned bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            dst),
        "l"(map), "r"(x), "r"(y), "r"(bar)
        : "memory");
}

// one output element through the epilogue
__device__ __forceinline__ void epi_store(const Epi& e, int m, int n, float x)
{
    if (e.bias) x += e.bias[n];
    if (e.mask && !((float)e.mask[(size_t)m * e.ldm + n] > 0.f)) x = 0.f;
    if (e.relu) x = fmaxf(x, 0.f);
    if (e.C32) e.C32[(size_t)m * e.ldc + n] = x;
    if (e.C16) e.C16[(size_t)m * e.ldc16 + n] = __float2bfloat16(x);
    if (e.Y) e.Y[(size_t)m * e.ldc + n] = x * e.ystd[n] + e.ymean[n];
}

// What an epilogue does with a value, fixed at compile time: with the fields of Epi tested for every
// four elements (a constant load, a compare and a branch each) a 32 x 32 chunk took 2400 cycles.
enum EpiKind {
    EK_WS,       // partial sum of one range to the workspace
    EK_C32,      // FP32
    EK_BIAS32,   // + bias, FP32
    EK_BIAS32Y,  // the same, and value * std + mean
    EK_RELU16,   // + bias, ReLU, BF16
    EK_MASK      // ReLU mask, FP32 and BF16
};
static int epi_kind(const Epi& e)
{
    if (e.mask) return EK_MASK;
    if (e.relu) return EK_RELU16;
    if (e.Y) return EK_BIAS32Y;
    return e.bias ? EK_BIAS32 : EK_C32;
}

// four elements of one row, columns n..n+3; bias, sd, mu: the columns' values
template <int KIND>
__device__ __forceinline__ void epi_store4(const Epi& e, size_t m, int n, float4 x, float4 b, float4 sd, float4 mu)
{
    if constexpr (KIND == EK_BIAS32 || KIND == EK_BIAS32Y || KIND == EK_RELU16)
        x = make_float4(x.x + b.x, x.y + b.y, x.z + b.z, x.w + b.w);
    if constexpr (KIND == EK_MASK) {
        const uint2 k = *reinterpret_cast<const uint2*>(e.mask + m * e.ldm + n);
        const __nv_bfloat162 k0 = *reinterpret_cast<const __nv_bfloat162*>(&k.x), k1 = *reinterpret_cast<const __nv_bfloat162*>(&k.y);
        if (!(__low2float(k0) > 0.f)) x.x = 0.f;
        if (!(__high2float(k0) > 0.f)) x.y = 0.f;
        if (!(__low2float(k1) > 0.f)) x.z = 0.f;
        if (!(__high2float(k1) > 0.f)) x.w = 0.f;
    }
    if constexpr (KIND == EK_RELU16) x = make_float4(fmaxf(x.x, 0.f), fmaxf(x.y, 0.f), fmaxf(x.z, 0.f), fmaxf(x.w, 0.f));
    if constexpr (KIND != EK_RELU16) *reinterpret_cast<float4*>(e.C32 + m * e.ldc + n) = x;
    if constexpr (KIND == EK_RELU16 || KIND == EK_MASK) {
        const __nv_bfloat162 a = __floats2bfloat162_rn(x.x, x.y), c = __floats2bfloat162_rn(x.z, x.w);
        uint2 v;
        v.x = *reinterpret_cast<const unsigned*>(&a);
        v.y = *reinterpret_cast<const unsigned*>(&c);
        *reinterpret_cast<uint2*>(e.C16 + m * e.ldc16 + n) = v;
    }
    if constexpr (KIND == EK_BIAS32Y)
        *reinterpret_cast<float4*>(e.Y + m * e.ldc + n) =
            make_float4(x.x * sd.x + mu.x, x.y * sd.y + mu.y, x.z * sd.z + mu.z, x.w * sd.w + mu.w);
}
template <int KIND>
__device__ __forceinline__ void epi_columns(const Epi& e, int n, float4& b, float4& sd, float4& mu)
{
    b = sd = mu = make_float4(0.f, 0.f, 0.f, 0.f);
    if constexpr (KIND == EK_BIAS32 || KIND == EK_BIAS32Y || KIND == EK_RELU16) b = *reinterpret_cast<const float4*>(e.bias + n);
    if constexpr (KIND == EK_BIAS32Y) {
        sd = *reinterpret_cast<const float4*>(e.ystd + n);
        mu = *reinterpret_cast<const float4*>(e.ymean + n);
    }
}
// whether rows of the outputs may be stored four elements at a time
__host__ __device__ inline bool epi_vec(const Epi& e)
{
    auto al = [](const void* p, int bytes) { return p == nullptr || (reinterpret_cast<uintptr_t>(p) & (bytes - 1)) == 0; };
    return al(e.bias, 16) && al(e.C32, 16) && al(e.Y, 16) && al(e.ystd, 16) && al(e.ymean, 16) && al(e.mask, 8) &&
           al(e.C16, 8) && (!(e.C32 || e.Y) || e.ldc % 4 == 0) && (!e.mask || e.ldm % 4 == 0) &&
           (!e.C16 || e.ldc16 % 4 == 0);
}

// The kernels of a step are queued with programmatic stream serialization (launch_next): one may be
// launched while its predecessor drains, and waits here, before its first access to global memory, until
// that has completed and its writes are visible.  Only then does it let its own successor start, so what
// is two kernels back is complete as well.  A step is a row of short kernels (six for the forward pass)
// and each boundary costs its launch and ramp otherwise (2000 x 1024 x 1024 x 22004, batch 256: forward 53
// -> 41.6 us, training step 343 -> 324 us).
__device__ __forceinline__ void after_predecessor()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <int MT, bool AMN, bool BMN, int KIND>
__global__ void __launch_bounds__(TC_NTH) gemm_tc(const __grid_constant__ CUtensorMap ta,
                                                   const __grid_constant__ CUtensorMap tb, int M, int N, int K, TcPlan p,
                                                   const __grid_constant__ Epi e, int vec, float* ws, int* err)
{
    extern __shared__ unsigned char tc_dyn[];
    __shared__ __align__(8) unsigned long long bar_full[TC_MAX_STAGES], bar_empty[TC_MAX_STAGES], bar_done;
    __shared__ unsigned tmem_slot;
    __shared__ int fail_s, issued_s;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int m0 = blockIdx.y * (128 * MT), n0 = blockIdx.x * p.bn;
    const int KB = (K + TC_BK - 1) / TC_BK;
    const int s0 = blockIdx.z * p.spc, s1 = min(p.splits, s0 + p.spc);  // this CTA's ranges
    const int kb0 = s0 * p.per, nk = min(KB, s1 * p.per) - kb0;
    // the ring starts at the first 1024-byte boundary (the swizzle pattern follows address bits)
    const unsigned ring = (sa(tc_dyn) + 1023u) & ~1023u;
    const int bchunks = (p.bn + 63) / 64;
    const unsigned b_bytes = BMN ? (unsigned)bchunks * TC_CHUNK : (unsigned)p.bn * TC_BK * 2;
    const unsigned stage_bytes = MT * TC_BOX + b_bytes;
    auto full = [&](int s) { return sa(&bar_full[s]); };
    auto empty = [&](int s) { return sa(&bar_empty[s]); };
    if (tid == 0) {
        for (int s = 0; s < p.stages; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(full(s)) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(empty(s)) : "memory");
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sa(&bar_done)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fail_s = 0;
        issued_s = nk;
    }
    if (warp == 0 && lane == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(&ta) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tb) : "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sa(&tmem_slot)),
                     "r"(p.cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const unsigned tmem = tmem_slot;
    after_predecessor();
    if (warp == 0 && lane == 0) {
        // producer: one stage = K block kb0 + i of both operands
        unsigned a_s = ring, fb = full(0), eb = empty(0);
        int kx = kb0 * TC_BK;  // innermost coordinates: multiples of 32 elements, 64 bytes
        for (int i = 0, s = 0, round = 0; i < nk; ++i, kx += TC_BK) {
            if (round > 0 && !tc_wait(eb, (unsigned)(round - 1) & 1u)) {
                issued_s = i;
                atomicExch(&fail_s, 1);
                break;
            }
            const unsigned b_s = a_s + MT * TC_BOX;
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb), "r"(stage_bytes) : "memory");
            if constexpr (AMN) {
#pragma unroll
                for (int c = 0; c < 2 * MT; ++c) tc_tma_2d(a_s + c * TC_CHUNK, &ta, m0 + 64 * c, kx, fb);
            } else {
                tc_tma_2d(a_s, &ta, kx, m0, fb);  // MT * 128 rows
            }
            if constexpr (BMN) {
                for (int c = 0; c < bchunks; ++c) tc_tma_2d(b_s + c * TC_CHUNK, &tb, n0 + 64 * c, kx, fb);
            } else {
                tc_tma_2d(b_s, &tb, kx, n0, fb);
            }
            a_s += stage_bytes;
            fb += 8;
            eb += 8;
            if (++s == p.stages) {
                s = 0;
                ++round;
                a_s = ring;
                fb = full(0);
                eb = empty(0);
            }
        }
    } else if (warp == 1 && lane == 0) {
        // MMA lane; descriptors differ from stage to stage and K step to K step in their low word only
        const unsigned idesc = TC_IDESC | (AMN ? 1u << 15 : 0u) | (BMN ? 1u << 16 : 0u) | ((unsigned)(p.bn >> 3) << 17);
        constexpr unsigned a_step = (AMN ? 2048u : 32u) >> 4, b_step = (BMN ? 2048u : 32u) >> 4;  // 16 K further
        const unsigned long long a0 = tc_desc(ring, AMN ? TC_CHUNK : 16u), b0 = tc_desc(ring + MT * TC_BOX, BMN ? TC_CHUNK : 16u);
        unsigned off = 0, fb = full(0), eb = empty(0), d = tmem;
        for (int i = 0, s = 0, round = 0, in = 0; i < nk; ++i) {
            if (!tc_wait(fb, (unsigned)round & 1u)) {
                atomicExch(&fail_s, 1);
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
            for (int t = 0; t < MT; ++t)
#pragma unroll
                for (int j = 0; j < TC_BK / 16; ++j)
                    tc_mma(d + (unsigned)(t * p.bn), a0 + (off + (unsigned)(t * (TC_BOX >> 4)) + j * a_step),
                           b0 + (off + j * b_step), idesc, (in | j) != 0);
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(eb) : "memory");
            if (++in == p.per) {  // the next range
                in = 0;
                d += (unsigned)(MT * p.bn);
            }
            off += stage_bytes >> 4;
            fb += 8;
            eb += 8;
            if (++s == p.stages) {
                s = 0;
                ++round;
                off = 0;
                fb = full(0);
                eb = empty(0);
            }
        }
        // completion of the last commit implies completion of every earlier MMA
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                         sa(&bar_done))
                     : "memory");
    } else if (warp >= 2) {
        // epilogue: wait for the accumulators, then lane quarter warp % 4 = rows 32 (warp % 4) + lane of each sub-tile
        // the tcgen05.ld below is warp-collective: decide once per warp
        const bool ok = __all_sync(0xffffffffu, tc_wait(sa(&bar_done), 0u));
        if (!ok && lane == 0) atomicExch(&fail_s, 1);
        const int failed = __shfl_sync(0xffffffffu, *(volatile int*)&fail_s, 0);
        if (ok && !failed) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int q = warp & 3, half = (warp - 2) >> 2;  // two warps a quarter, every other chunk of columns
            float* stg = reinterpret_cast<float*>(tc_dyn + (ring - sa(tc_dyn))) + (size_t)(warp - 2) * 32 * TC_STG;
            const int nacc = s1 - s0;
            const int col = 4 * (lane & 7), row = lane >> 3;
#pragma unroll 1
            for (int t = 0; t < MT; ++t) {
                const int mr0 = m0 + 128 * t + 32 * q;
                if (mr0 >= M) break;
#pragma unroll 1
                for (int c0 = 32 * half; c0 < p.bn && n0 + c0 < N; c0 += 64)
#pragma unroll 1
                    for (int z0 = 0; z0 < (KIND == EK_WS ? nacc : 1); ++z0) {
                        float x[32];
#pragma unroll 1
                        for (int z = z0; z < (KIND == EK_WS ? z0 + 1 : nacc); ++z) {
                            unsigned v[32];
                            asm volatile(
                                "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
                                "%11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, "
                                "%28, %29, %30, %31}, [%32];"
                                : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
                                  "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]),
                                  "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]),
                                  "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
                                  "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]),
                                  "=r"(v[31])
                                : "r"(tmem + ((unsigned)(q * 32) << 16) + (unsigned)((z * MT + t) * p.bn + c0)));
                            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                            if (z == z0) {
#pragma unroll
                                for (int i = 0; i < 32; ++i) x[i] = __uint_as_float(v[i]);
                            } else {
#pragma unroll
                                for (int i = 0; i < 32; ++i) x[i] += __uint_as_float(v[i]);
                            }
                        }
                        // lane = row here; stored as rows, then read back 4 columns a lane, 8 lanes a row
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            *reinterpret_cast<float4*>(stg + lane * TC_STG + 4 * i) =
                                make_float4(x[4 * i], x[4 * i + 1], x[4 * i + 2], x[4 * i + 3]);
                        __syncwarp();
                        float4 f[8];
#pragma unroll
                        for (int it = 0; it < 8; ++it)
                            f[it] = *reinterpret_cast<const float4*>(stg + (it * 4 + row) * TC_STG + col);
                        const int n = n0 + c0 + col, m = mr0 + row;
                        if constexpr (KIND == EK_WS) {
                            float* w = ws + ((size_t)(s0 + z0) * M + m) * N + n;
                            if ((N & 3) == 0) {
                                if (n < N)
#pragma unroll
                                    for (int it = 0; it < 8; ++it)
                                        if (m + 4 * it < M) *reinterpret_cast<float4*>(w + (size_t)(4 * it) * N) = f[it];
                            } else {
#pragma unroll 1
                                for (int it = 0; it < 8; ++it)
                                    for (int j = 0; j < 4; ++j)
                                        if (m + 4 * it < M && n + j < N)
                                            w[(size_t)(4 * it) * N + j] = stg[(it * 4 + row) * TC_STG + col + j];
                            }
                        } else if (vec && n + 3 < N) {
                            float4 b, sd, mu;
                            epi_columns<KIND>(e, n, b, sd, mu);
#pragma unroll
                            for (int it = 0; it < 8; ++it)
                                if (m + 4 * it < M) epi_store4<KIND>(e, (size_t)(m + 4 * it), n, f[it], b, sd, mu);
                        } else if (n < N) {
#pragma unroll 1
                            for (int it = 0; it < 8; ++it)
#pragma unroll 1
                                for (int j = 0; j < 4; ++j)
                                    if (m + 4 * it < M && n + j < N)
                                        epi_store(e, m + 4 * it, n + j, stg[(it * 4 + row) * TC_STG + col + j]);
                        }
                        __syncwarp();
                    }
            }
        }
    }
    __syncwarp();
    __syncthreads();
    if (*(volatile int*)&fail_s && tid == 0) {
        // before the stages and the tensor memory are released, copies still in flight and
        // MMAs still in flight must finish: the producer reuses a stage only after its MMAs
        // consumed it, so only the last `stages` issued copies can be pending (each completes
        // the phase (i / stages) of its stage's "full" barrier), and the "done" commit,
        // made after the MMA lane's last issue, completes once every MMA has
        bool drained = true;
        const int issued = issued_s;
        for (int i = max(0, issued - p.stages); i < issued; ++i)
            if (!tc_wait(full(i % p.stages), (unsigned)(i / p.stages) & 1u)) drained = false;
        if (!tc_wait(sa(&bar_done), 0u)) drained = false;
        atomicMax(err, drained ? 1 : 2);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(p.cols) : "memory");
}

// split-K: C = epilogue(sum over z of ws[z]) in a fixed order; vec: four columns a thread (N a multiple of 4)
template <int KIND>
__global__ void __launch_bounds__(256) splitk_epilogue(const float* ws, int splits, int M, int N,
                                                       const __grid_constant__ Epi e, int vec)
{
    const long long total = (long long)M * N;
    after_predecessor();
    if (vec) {
        for (long long i = 4 * (blockIdx.x * (long long)blockDim.x + threadIdx.x); i < total;
             i += 4ll * gridDim.x * blockDim.x) {
            float4 acc = *reinterpret_cast<const float4*>(ws + i);
#pragma unroll 4
            for (int z = 1; z < splits; ++z) {
                const float4 v = *reinterpret_cast<const float4*>(ws + (size_t)z * total + i);
                acc.x += v.x;
                acc.y += v.y;
                acc.z += v.z;
                acc.w += v.w;
            }
            const int n = (int)(i % N);
            float4 b, sd, mu;
            epi_columns<KIND>(e, n, b, sd, mu);
            epi_store4<KIND>(e, (size_t)(i / N), n, acc, b, sd, mu);
        }
        return;
    }
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        float acc = 0.f;
        for (int z = 0; z < splits; ++z) acc += ws[(size_t)z * total + i];
        epi_store(e, (int)(i / N), (int)(i % N), acc);
    }
}

// out (C x R, ld_out) = in (R x C, ld_in)^T, BF16, 32 x 32 tiles
__global__ void transpose_bf16(const bf16* in, int R, int C, int ld_in, bf16* out, int ld_out)
{
    __shared__ bf16 tile[32][33];
    const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
    for (int i = threadIdx.y; i < 32; i += blockDim.y) {
        const int r = r0 + i, c = c0 + threadIdx.x;
        if (r < R && c < C) tile[i][threadIdx.x] = in[(size_t)r * ld_in + c];
    }
    __syncthreads();
    for (int i = threadIdx.y; i < 32; i += blockDim.y) {
        const int c = c0 + i, r = r0 + threadIdx.x;
        if (r < R && c < C) out[(size_t)c * ld_out + r] = tile[threadIdx.x][i];
    }
}

constexpr int MAX_GRID_Y = 32768;  // rows of blocks in the elementwise kernels, which loop beyond

// Xn (bf16, ld) = (X - mean) / std, X row-major B x d; a row of blocks a row
__global__ void normalize_to_bf16(const float* X, int B, int d, const float* mean, const float* istd, bf16* out, int ld)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    after_predecessor();
    if (c >= d) return;
    for (int r = blockIdx.y; r < B; r += gridDim.y)
        out[(size_t)r * ld + c] = __float2bfloat16((X[(size_t)r * d + c] - mean[c]) * istd[c]);
}

// loss partials and dy = (y - (t - mean)/std) / (B d): dy32 (B x d), dy16 (ld16).
// A thread has four columns (vec: 16-byte accesses) of LG_ROWS rows.  The
// squares are summed as exact FP32 products in a two-word (hi, lo) sum, about
// 48 bits, and in FP64 from there on: adding each square in FP64 took 18 us of
// the FP64 pipe for 256 x 22004 values, the memory traffic 12 us.  A thread
// whose sum leaves FP32's range (errors above 1.8e19, infinities, NaN) adds its
// squares again in FP64.  (Squares below that range, whose low words are lost,
// are below the FP32 loss's last digit.)
constexpr int LG_ROWS = 8;
__global__ void loss_grad(const float* y, const float* tgt, int B, int d, const float* mean, const float* istd,
                          float* dy32, bf16* dy16, int ld16, double* part, int vec)
{
    after_predecessor();
    const float scale = 1.0f / (float)((long long)B * d);
    const int c = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
    float hi = 0.f, lo = 0.f;
    auto add = [&](float diff) {  // (hi, lo) += diff^2
        const float p = diff * diff, pe = fmaf(diff, diff, -p);
        const float t = hi + p, z = t - hi;
        lo += ((hi - (t - z)) + (p - z)) + pe;
        hi = t;
    };
    if (c < d) {
        const int nc = min(4, d - c);
        float mu[4], is[4];
        for (int j = 0; j < 4; ++j) {
            mu[j] = j < nc ? mean[c + j] : 0.f;
            is[j] = j < nc ? istd[c + j] : 0.f;
        }
        for (int r0 = blockIdx.y * LG_ROWS; r0 < B; r0 += (int)gridDim.y * LG_ROWS)
        for (int r = r0; r < min(B, r0 + LG_ROWS); ++r) {
            const size_t i = (size_t)r * d + c;
            float g[4];
            if (vec && nc == 4) {
                const float4 a = *reinterpret_cast<const float4*>(y + i), t = *reinterpret_cast<const float4*>(tgt + i);
                g[0] = a.x - (t.x - mu[0]) * is[0];
                g[1] = a.y - (t.y - mu[1]) * is[1];
                g[2] = a.z - (t.z - mu[2]) * is[2];
                g[3] = a.w - (t.w - mu[3]) * is[3];
                for (int j = 0; j < 4; ++j) {
                    add(g[j]);
                    g[j] *= scale;
                }
                *reinterpret_cast<float4*>(dy32 + i) = make_float4(g[0], g[1], g[2], g[3]);
                const __nv_bfloat162 b0 = __floats2bfloat162_rn(g[0], g[1]), b1 = __floats2bfloat162_rn(g[2], g[3]);
                uint2 w;
                w.x = *reinterpret_cast<const unsigned*>(&b0);
                w.y = *reinterpret_cast<const unsigned*>(&b1);
                *reinterpret_cast<uint2*>(dy16 + (size_t)r * ld16 + c) = w;
            } else {
                for (int j = 0; j < nc; ++j) {
                    const float diff = y[i + j] - (tgt[i + j] - mu[j]) * is[j];
                    add(diff);
                    dy32[i + j] = diff * scale;
                    dy16[(size_t)r * ld16 + c + j] = __float2bfloat16(diff * scale);
                }
            }
        }
    }
    double acc = (double)hi + (double)lo;
    if (!(hi <= FLT_MAX)) {
        acc = 0.0;
        for (int r0 = blockIdx.y * LG_ROWS; r0 < B; r0 += (int)gridDim.y * LG_ROWS)
            for (int r = r0; r < min(B, r0 + LG_ROWS); ++r)
                for (int k = c; k < min(d, c + 4); ++k) {
                    const size_t i = (size_t)r * d + k;
                    const double diff = y[i] - (tgt[i] - mean[k]) * istd[k];
                    acc += diff * diff;
                }
    }
    __shared__ double red[32];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
        part[blockIdx.y * gridDim.x + blockIdx.x] = s;
    }
}

// The bias gradients and the loss, one launch: blocks [first[k], first[k+1]) sum BS_COLS columns
// each of D[k] (B x d[k]) into out[k], row after row with 16 rows' loads in flight; the last block adds
// the nb loss partials.
constexpr int BS_COLS = 64;
struct Sums {
    const float* D[3];
    float* out[3];
    int d[3], first[4];
    const double* part;
    int nb;
    double scale;
    double* loss;
};
__global__ void __launch_bounds__(BS_COLS) bias_sums(const __grid_constant__ Sums a, int B)
{
    after_predecessor();
    if ((int)blockIdx.x == a.first[3]) {
        double s = 0.0;
        for (int i = threadIdx.x; i < a.nb; i += BS_COLS) s += a.part[i];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        __shared__ double red[BS_COLS / 32];
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0;
            for (int w = 0; w < BS_COLS / 32; ++w) t += red[w];
            *a.loss = t * a.scale;
        }
        return;
    }
    const int k = (int)blockIdx.x >= a.first[2] ? 2 : ((int)blockIdx.x >= a.first[1] ? 1 : 0);
    const int d = a.d[k], c = BS_COLS * ((int)blockIdx.x - a.first[k]) + threadIdx.x;
    if (c >= d) return;
    const float* D = a.D[k] + c;
    float s = 0.f;
    int r = 0;
    for (; r + 16 <= B; r += 16) {
        float v[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = D[(size_t)(r + i) * d];
#pragma unroll
        for (int i = 0; i < 16; ++i) s += v[i];
    }
    for (; r < B; ++r) s += D[(size_t)r * d];
    a.out[k][c] = s;
}

// Adam on all parameters, four at a time (segments start at multiples of 4); refreshes the BF16
// copies of the weight matrices.  Does nothing once a GEMM of this step or an earlier one reported an
// error, and then says so in *skipped (host memory); else counts the step in *applied.
// Bound by memory: 7 words and a BF16 copy a parameter, 0.77 GB for 25.6 M of them, 115 us at the
// copy rate; one element a thread with a search of its segment took 199 us.
struct Seg {
    long long off, len;
    bf16* w16;  // BF16 copy or null for biases
    int cols;   // row length of the matrix
    int ld16;   // leading dimension of the BF16 copy
};
struct Segs {
    Seg s[6];
};
__global__ void __launch_bounds__(256) adam(float* p, const float* g, float* m, float* v, long long n, float lr, float b1c,
                                            float b2c, Segs segs, const int* err, int* applied, int* skipped)
{
    after_predecessor();
    const bool first = blockIdx.x == 0 && threadIdx.x == 0;
    if (*err) {
        if (first) *(volatile int*)skipped = 1;
        return;
    }
    if (first) ++*applied;
    auto step = [&](float pi, float gi, float& mi, float& vi) {
        mi = 0.9f * mi + 0.1f * gi;
        vi = 0.999f * vi + 0.001f * gi * gi;
        return pi - lr * (mi / b1c) / (sqrtf(vi / b2c) + 1e-8f);
    };
    for (long long i = 4 * (blockIdx.x * (long long)blockDim.x + threadIdx.x); i < n; i += 4ll * gridDim.x * blockDim.x) {
        const int cnt = (int)min(4ll, n - i);
        float w[4];
        if (cnt == 4) {
            const float4 p4 = *reinterpret_cast<const float4*>(p + i), g4 = *reinterpret_cast<const float4*>(g + i);
            float4 m4 = *reinterpret_cast<const float4*>(m + i), v4 = *reinterpret_cast<const float4*>(v + i);
            w[0] = step(p4.x, g4.x, m4.x, v4.x);
            w[1] = step(p4.y, g4.y, m4.y, v4.y);
            w[2] = step(p4.z, g4.z, m4.z, v4.z);
            w[3] = step(p4.w, g4.w, m4.w, v4.w);
            *reinterpret_cast<float4*>(m + i) = m4;
            *reinterpret_cast<float4*>(v + i) = v4;
            *reinterpret_cast<float4*>(p + i) = make_float4(w[0], w[1], w[2], w[3]);
        } else {
            for (int j = 0; j < cnt; ++j) {
                w[j] = step(p[i + j], g[i + j], m[i + j], v[i + j]);
                p[i + j] = w[j];
            }
        }
        int k = 0;
        while (k < 5 && i >= segs.s[k + 1].off) ++k;
        const Seg& sg = segs.s[k];
        if (!sg.w16) continue;
        const long long j0 = i - sg.off;
        if (sg.cols == sg.ld16) {
            const __nv_bfloat162 b0 = __floats2bfloat162_rn(w[0], w[1]), b1 = __floats2bfloat162_rn(w[2], w[3]);
            uint2 o;
            o.x = *reinterpret_cast<const unsigned*>(&b0);
            o.y = *reinterpret_cast<const unsigned*>(&b1);
            *reinterpret_cast<uint2*>(sg.w16 + j0) = o;
        } else {
            for (int j = 0; j < cnt; ++j)
                sg.w16[((j0 + j) / sg.cols) * sg.ld16 + (j0 + j) % sg.cols] = __float2bfloat16(w[j]);
        }
    }
}

__device__ __forceinline__ unsigned long long mix64(unsigned long long z)
{
    z += 0x9e3779b97f4a7c15ull;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}
// uniform(-a, a) from a counter-based hash of (seed, index); zero outside [off, off+len) of weights
__global__ void init_uniform(float* p, long long off, long long len, float a, unsigned long long seed)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < len; i += (long long)gridDim.x * blockDim.x) {
        const unsigned long long h = mix64(seed ^ mix64((unsigned long long)(off + i)));
        const double u = (double)(h >> 11) * (1.0 / 9007199254740992.0);
        p[off + i] = (float)((2.0 * u - 1.0) * a);
    }
}

// out (rows x cols, ld) = in (rows x cols, packed)
__global__ void f32_to_bf16_2d(const float* in, long long rows, int cols, bf16* out, int ld)
{
    const long long n = rows * cols;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        out[(i / cols) * ld + i % cols] = __float2bfloat16(in[i]);
}

// Y = y * std + mean (output units)
__global__ void denormalize(const float* y, int B, int d, const float* mean, const float* stdv, float* Y)
{
    const long long total = (long long)B * d;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(i % d);
        Y[i] = y[i] * stdv[c] + mean[c];
    }
}

// per-column mean and inverse std (two passes in FP64), std < 1e-6 -> 1
__global__ void col_stats(const float* X, long long rows, int d, float* mean, float* stdv, float* istd)
{
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < d; c += gridDim.x * blockDim.x) {
        double s = 0.0;
        for (long long r = 0; r < rows; ++r) s += X[(size_t)r * d + c];
        const double mu = s / (double)rows;
        double q = 0.0;
        for (long long r = 0; r < rows; ++r) {
            const double e = X[(size_t)r * d + c] - mu;
            q += e * e;
        }
        double sd = sqrt(q / (double)rows);
        if (!(sd >= 1e-6)) sd = 1.0;
        mean[c] = (float)mu;
        stdv[c] = (float)sd;
        istd[c] = (float)(1.0 / sd);
    }
}

__global__ void fill_f32(float* p, long long n, float v)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) p[i] = v;
}

int pad8(int x) { return (x + 7) & ~7; }
int grid1d(long long n, int th = 256) { return (int)std::max<long long>(1, std::min<long long>((n + th - 1) / th, 8192)); }

}  // namespace

struct scs_mlp {
    int din, dh, dout, maxB;
    int ldin, ldout;  // padded leading dimensions (multiples of 8)
    cudaStream_t st;
    long long np;
    long long oW1, ob1, oW2, ob2, oW3, ob3;
    float *p, *g, *m, *v;                // parameters, gradients, Adam moments
    bf16 *W1, *W2, *W3, *W2t, *W3t;      // BF16 copies (W2t: h x h, W3t: h x ldout)
    float *in_mean, *in_std, *in_istd, *out_mean, *out_std, *out_istd;
    bf16 *Xn, *Xnt, *h1, *h1t, *h2, *h2t, *dy16, *dyt, *dh2_16, *dh2t, *dh1_16, *dh1t;
    float *y, *dy32, *dh2_32, *dh1_32;
    double *part, *loss;
    int* err;  // set by a tensor-core GEMM whose bounded wait expired; beside *loss, so one copy reads all three
    int* applied;           // Adam steps made
    struct Report {
        double loss;
        int err, applied;
    }* report;              // pinned host copy of (*loss, *err, *applied)
    cudaEvent_t reported;   // that copy has arrived
    int* skipped;           // pinned, beside it: set by an Adam step that found *err set and did nothing
    int step;               // Adam steps queued; those made, after an error
    int gemm_impl;  // SCS_MLP_GEMM_MMA or SCS_MLP_GEMM_TCGEN05
    int lastB;      // rows of the last batch that went through forward()
    float* ws;      // split-K partial tiles of the tensor-core GEMMs
    size_t ws_floats;
    char* arena;
};

static int mlp_err(const char* what, cudaError_t e)
{
    char buf[256];
    snprintf(buf, sizeof buf, "%s: %s", what, cudaGetErrorString(e));
    sscs::record_error(buf);
    return SCS_ECUDA;
}
#define MCU(x)                                          \
    do {                                                \
        cudaError_t e_ = (x);                           \
        if (e_ != cudaSuccess) return mlp_err(#x, e_); \
    } while (0)

// Set once a tensor-core GEMM reported that its MMAs did not drain before the
// tensor memory was released: that memory may since have been written behind
// another CTA's back, so no later GEMM of this process is trusted.
static std::atomic<bool> g_tc_fatal{false};
static const char* const TC_FATAL_MSG =
    "mlp: a tensor-core GEMM released tensor memory while its MMAs may still have been running; "
    "results of this CUDA context can no longer be trusted, every later GEMM call fails";

// cuTensorMapEncodeTiled, looked up once through the runtime (no link against the driver library)
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static EncodeTiledFn tensor_map_encoder()
{
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)p;
    });
    return fn;
}

// tensor map of a BF16 matrix of `outer` rows of `inner` contiguous elements (row stride ld):
// boxes of box_outer rows x 64 elements, 128-byte swizzle, zero fill past the extents
static int operand_map(CUtensorMap* map, const bf16* base, int inner, int outer, int ld, int box_outer)
{
    EncodeTiledFn enc = tensor_map_encoder();
    if (!enc) {
        sscs::record_error("mlp: cuTensorMapEncodeTiled is unavailable");
        return SCS_ECUDA;
    }
    const cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)outer};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * sizeof(bf16)};
    const cuuint32_t box[2] = {64, (cuuint32_t)box_outer};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void*)base, dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        char buf[128];
        snprintf(buf, sizeof buf, "mlp: cuTensorMapEncodeTiled failed (%d)", (int)r);
        sscs::record_error(buf);
        return SCS_ECUDA;
    }
    return SCS_OK;
}

static int device_sms()
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 1;
    return sms > 0 ? sms : 1;
}

// The tile and the K ranges of a tcgen05 product.
//  - K ranges: where the product's 128 x 128 tiles would leave half the SMs idle and K is deep, as
//    many as fill the SMs with such tiles, of at least 4 K blocks; else one.  They fix the order of
//    the sums, so results do not depend on the rest of the plan.
//  - At most 4 ranges of a shallow K (64 blocks), or no room for their sums: all in one CTA,
//    accumulators side by side in tensor memory -- no workspace, no second kernel -- and 128 x 32
//    tiles, which are many (256 x 1024 x 1024: 10.2 us, against 6.2 + 3.5 us with the second kernel;
//    256 x 1024 x 2000, 8 ranges: 14.4 against 6.2 + 3.5 us).
//  - Else the tile (1 or 2 sub-tiles of 128 rows, a width in steps of 32) that makes waves x bytes
//    of a K block least, each range on CTAs of its own; products of many tiles and few K blocks in
//    two CTAs an SM, so that one's epilogue runs under the other's copies.
static TcPlan tc_plan(int M, int N, int K, bool bmn, int sms, size_t ws_floats)
{
    TcPlan p{};
    const int KB = (K + TC_BK - 1) / TC_BK;
    auto up = [](int a, int b) { return (a + b - 1) / b; };
    auto b_bytes = [&](int bn) { return bmn ? up(bn, 64) * TC_CHUNK : bn * TC_BK * 2; };
    const int tiles = up(M, 128) * up(N, 128);
    p.mt = 1;
    p.splits = 1;
    p.per = KB;
    if (2 * tiles <= sms && KB >= 8) {
        int sp = std::min(up(sms, tiles), KB / 4);
        if (KB > 64)
            while (sp > 1 && (size_t)sp * M * N > ws_floats) --sp;
        p.per = up(KB, sp);
        p.splits = up(KB, p.per);
    }
    p.spc = 1;
    if (p.splits > 1 && KB <= 64 && (p.splits <= 4 || (size_t)p.splits * M * N > ws_floats)) {
        p.bn = 32;
        p.spc = p.splits;  // at most 16: 512 columns
    } else {
        long long best = -1;
        for (int mt = M > 128 ? 2 : 1; mt >= 1; --mt)
            for (int bn = 256; bn >= 32; bn -= 32) {
                const int ctas = up(M, 128 * mt) * up(N, bn) * p.splits;
                if (mt == 2 && ctas > sms) continue;
                const long long cost = (long long)up(ctas, sms) * (mt * TC_BOX + b_bytes(bn));
                if (best < 0 || cost < best) {
                    best = cost;
                    p.mt = mt;
                    p.bn = bn;
                }
            }
        if (tiles > 2 * sms && KB <= 8) {
            p.mt = 1;
            p.bn = 128;
        }
    }
    const int stage = p.mt * TC_BOX + b_bytes(p.bn);
    const bool two = up(M, 128 * p.mt) * up(N, p.bn) * p.splits / p.spc > sms && p.mt * p.bn * p.spc <= 256;
    p.stages = std::max(2, std::min({TC_MAX_STAGES, (two ? TC_SMEM_MAX / 2 - 2048 : TC_SMEM_MAX) / stage, std::max(2, KB)}));
    p.cols = 32;
    while (p.cols < p.mt * p.bn * p.spc) p.cols *= 2;
    return p;
}
// dynamic shared memory: the ring, aligned to 1024 bytes; at least the epilogue's staging
static size_t tc_smem(const TcPlan& p, bool bmn)
{
    const size_t stage = (size_t)p.mt * TC_BOX + (bmn ? (size_t)(p.bn + 63) / 64 * TC_CHUNK : (size_t)p.bn * TC_BK * 2);
    return std::max(p.stages * stage, (size_t)(TC_NTH / 32 - 2) * 32 * TC_STG * sizeof(float)) + 1024;
}

// A kernel that begins with after_predecessor(), queued so that it may start while its predecessor drains.
template <class... P, class... A>
static cudaError_t launch_next(void (*fn)(P...), dim3 grid, int block, size_t smem, cudaStream_t st, A... a)
{
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fn, static_cast<P>(a)...);
}

typedef void (*GemmTc)(const CUtensorMap, const CUtensorMap, int, int, int, TcPlan, const Epi, int, float*, int*);
typedef void (*SplitkEpi)(const float*, int, int, int, const Epi, int);
template <int KIND>
static GemmTc gemm_tc_of(int mt, bool amn, bool bmn)
{
    if (mt == 2) return amn ? (bmn ? gemm_tc<2, true, true, KIND> : gemm_tc<2, true, false, KIND>)
                            : (bmn ? gemm_tc<2, false, true, KIND> : gemm_tc<2, false, false, KIND>);
    return amn ? (bmn ? gemm_tc<1, true, true, KIND> : gemm_tc<1, true, false, KIND>)
               : (bmn ? gemm_tc<1, false, true, KIND> : gemm_tc<1, false, false, KIND>);
}
static GemmTc gemm_tc_kernel(int kind, int mt, bool amn, bool bmn)
{
    switch (kind) {
        case EK_WS: return gemm_tc_of<EK_WS>(mt, amn, bmn);
        case EK_BIAS32: return gemm_tc_of<EK_BIAS32>(mt, amn, bmn);
        case EK_BIAS32Y: return gemm_tc_of<EK_BIAS32Y>(mt, amn, bmn);
        case EK_RELU16: return gemm_tc_of<EK_RELU16>(mt, amn, bmn);
        case EK_MASK: return gemm_tc_of<EK_MASK>(mt, amn, bmn);
        default: return gemm_tc_of<EK_C32>(mt, amn, bmn);
    }
}
static SplitkEpi splitk_kernel(int kind)
{
    switch (kind) {
        case EK_BIAS32: return splitk_epilogue<EK_BIAS32>;
        case EK_BIAS32Y: return splitk_epilogue<EK_BIAS32Y>;
        case EK_RELU16: return splitk_epilogue<EK_RELU16>;
        case EK_MASK: return splitk_epilogue<EK_MASK>;
        default: return splitk_epilogue<EK_C32>;
    }
}

// C = A B^T.  amn (bmn): A (B) is stored K x M (K x N) with lda (ldb) the stride of a K row, else
// M x K (N x K); the legacy kernel takes the latter only.
static int launch_gemm(int impl, cudaStream_t st, int* err, int M, int N, int K, const bf16* A, int lda, bool amn,
                       const bf16* B, int ldb, bool bmn, const Epi& e, float* ws = nullptr, size_t ws_floats = 0)
{
    if (g_tc_fatal) {
        sscs::record_error(TC_FATAL_MSG);
        return SCS_ECUDA;
    }
    if (impl == SCS_MLP_GEMM_TCGEN05) {
        const TcPlan p = tc_plan(M, N, K, bmn, device_sms(), ws_floats);
        CUtensorMap ta, tb;
        int rc;
        if ((rc = amn ? operand_map(&ta, A, M, K, lda, 64) : operand_map(&ta, A, K, M, lda, 128 * p.mt)) ||
            (rc = bmn ? operand_map(&tb, B, N, K, ldb, 64) : operand_map(&tb, B, K, N, ldb, p.bn)))
            return rc;
        const int z = (p.splits + p.spc - 1) / p.spc;
        const GemmTc fn = gemm_tc_kernel(z > 1 ? (int)EK_WS : epi_kind(e), p.mt, amn, bmn);
        const size_t smem = tc_smem(p, bmn);
        const int vec = epi_vec(e) ? 1 : 0;
        // a per-device attribute: set before every launch (a host call of about a microsecond)
        MCU(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM_MAX + 1024));
        dim3 grid((N + p.bn - 1) / p.bn, (M + 128 * p.mt - 1) / (128 * p.mt), z);
        cudaError_t ce = launch_next(fn, grid, TC_NTH, smem, st, ta, tb, M, N, K, p, e, vec, ws, err);
        if (ce != cudaSuccess) return mlp_err("gemm_tc launch", ce);
        if (z > 1) {
            const long long total = (long long)M * N;
            const int v4 = vec && N % 4 == 0;
            ce = launch_next(splitk_kernel(epi_kind(e)),
                             (int)std::min<long long>(8192, (total / (v4 ? 4 : 1) + 255) / 256), 256, 0, st, ws, p.splits,
                             M, N, e, v4);
            if (ce != cudaSuccess) return mlp_err("splitk_epilogue launch", ce);
        }
        return SCS_OK;
    }
    dim3 grid((N + BN - 1) / BN, (M + BM - 1) / BM);
    gemm_nt<<<grid, NTH, 0, st>>>(M, N, K, A, lda, B, ldb, e);
    const cudaError_t ce = cudaGetLastError();
    return ce == cudaSuccess ? SCS_OK : mlp_err("gemm_nt launch", ce);
}
static int gemm(scs_mlp* n, int M, int N, int K, const bf16* A, int lda, bool amn, const bf16* B, int ldb, bool bmn,
                const Epi& e)
{
    return launch_gemm(n->gemm_impl, n->st, n->err, M, N, K, A, lda, amn, B, ldb, bmn, e, n->ws, n->ws_floats);
}
// Waits for the stream and reads (and clears) the tensor-core GEMMs' timeout flag.  After an error the
// steps that Adam skipped no longer count.
static int check_err_flag(scs_mlp* n)
{
    scs_mlp::Report r{};
    MCU(cudaMemcpyAsync(&r, n->loss, sizeof r, cudaMemcpyDeviceToHost, n->st));
    MCU(cudaStreamSynchronize(n->st));
    if (r.err) {
        MCU(cudaMemsetAsync(n->err, 0, sizeof(int), n->st));
        n->step = r.applied;
        *(volatile int*)n->skipped = 0;
        if (r.err >= 2) g_tc_fatal = true;
        sscs::record_error(r.err >= 2 ? TC_FATAL_MSG : "mlp: a tensor-core GEMM wait timed out; its output tile was not written");
        return SCS_ECUDA;
    }
    return SCS_OK;
}
// An error of an earlier call that did not wait for its own (a step without a loss), once an Adam step has
// been skipped for it: the host sees it without waiting.
static int earlier_error(scs_mlp* n) { return *(volatile int*)n->skipped ? check_err_flag(n) : SCS_OK; }
static void transpose(scs_mlp* n, const bf16* in, int R, int C, int ld_in, bf16* out, int ld_out)
{
    dim3 grid((C + 31) / 32, (R + 31) / 32), block(32, 8);
    transpose_bf16<<<grid, block, 0, n->st>>>(in, R, C, ld_in, out, ld_out);
}
static Epi epi(const float* bias, const bf16* mask, int ldm, int relu, float* C32, int ldc, bf16* C16, int ldc16)
{
    Epi e;
    e.bias = bias;
    e.mask = mask;
    e.ldm = ldm;
    e.relu = relu;
    e.C32 = C32;
    e.ldc = ldc;
    e.C16 = C16;
    e.ldc16 = ldc16;
    e.Y = nullptr;
    e.ystd = e.ymean = nullptr;
    return e;
}

// blocks of loss_grad, each with one loss partial
static dim3 loss_grid(int dout, int B) { return dim3((dout + 1023) / 1024, std::min((B + LG_ROWS - 1) / LG_ROWS, MAX_GRID_Y)); }

extern "C" int scs_mlp_create(int32_t din, int32_t dh, int32_t dout, int32_t maxB, uint64_t seed, void* stream,
                              scs_mlp** out)
{
    if (!out || din <= 0 || dh <= 0 || dout <= 0 || maxB <= 0 || dh % 8 != 0) {
        sscs::record_error("scs_mlp_create: bad sizes (all positive, d_hidden a multiple of 8)");
        return SCS_EINVAL;
    }
    *out = nullptr;
    scs_mlp* n = new (std::nothrow) scs_mlp();
    if (!n) return SCS_ENOMEM;
    memset(n, 0, sizeof(*n));
    n->din = din;
    n->dh = dh;
    n->dout = dout;
    n->maxB = maxB;
    n->ldin = pad8(din);
    n->ldout = pad8(dout);
    n->gemm_impl = SCS_MLP_GEMM_TCGEN05;
    n->st = (cudaStream_t)stream;
    const int Bp = pad8(maxB);
    n->oW1 = 0;
    n->ob1 = n->oW1 + (long long)dh * din;
    n->oW2 = n->ob1 + dh;
    n->ob2 = n->oW2 + (long long)dh * dh;
    n->oW3 = n->ob2 + dh;
    n->ob3 = n->oW3 + (long long)dout * dh;
    n->np = n->ob3 + dout;
    // one arena
    size_t off = 0;
    std::vector<std::pair<void**, size_t>> plan;
    auto take = [&](void** ptr, size_t bytes) { plan.push_back({ptr, bytes}); };
    take((void**)&n->p, sizeof(float) * n->np);
    take((void**)&n->g, sizeof(float) * n->np);
    take((void**)&n->m, sizeof(float) * n->np);
    take((void**)&n->v, sizeof(float) * n->np);
    take((void**)&n->W1, sizeof(bf16) * (size_t)dh * n->ldin);
    take((void**)&n->W2, sizeof(bf16) * (size_t)dh * dh);
    take((void**)&n->W3, sizeof(bf16) * (size_t)dout * dh);
    take((void**)&n->W2t, sizeof(bf16) * (size_t)dh * dh);
    take((void**)&n->W3t, sizeof(bf16) * (size_t)dh * n->ldout);
    take((void**)&n->in_mean, sizeof(float) * din);
    take((void**)&n->in_std, sizeof(float) * din);
    take((void**)&n->in_istd, sizeof(float) * din);
    take((void**)&n->out_mean, sizeof(float) * dout);
    take((void**)&n->out_std, sizeof(float) * dout);
    take((void**)&n->out_istd, sizeof(float) * dout);
    take((void**)&n->Xn, sizeof(bf16) * (size_t)maxB * n->ldin);
    take((void**)&n->Xnt, sizeof(bf16) * (size_t)din * Bp);
    take((void**)&n->h1, sizeof(bf16) * (size_t)maxB * dh);
    take((void**)&n->h1t, sizeof(bf16) * (size_t)dh * Bp);
    take((void**)&n->h2, sizeof(bf16) * (size_t)maxB * dh);
    take((void**)&n->h2t, sizeof(bf16) * (size_t)dh * Bp);
    take((void**)&n->dy16, sizeof(bf16) * (size_t)maxB * n->ldout);
    take((void**)&n->dyt, sizeof(bf16) * (size_t)dout * Bp);
    take((void**)&n->dh2_16, sizeof(bf16) * (size_t)maxB * dh);
    take((void**)&n->dh2t, sizeof(bf16) * (size_t)dh * Bp);
    take((void**)&n->dh1_16, sizeof(bf16) * (size_t)maxB * dh);
    take((void**)&n->dh1t, sizeof(bf16) * (size_t)dh * Bp);
    take((void**)&n->y, sizeof(float) * (size_t)maxB * dout);
    take((void**)&n->dy32, sizeof(float) * (size_t)maxB * dout);
    take((void**)&n->dh2_32, sizeof(float) * (size_t)maxB * dh);
    take((void**)&n->dh1_32, sizeof(float) * (size_t)maxB * dh);
    take((void**)&n->part, sizeof(double) * (size_t)loss_grid(dout, maxB).x * loss_grid(dout, maxB).y);
    take((void**)&n->loss, sizeof(scs_mlp::Report));
    // split-K workspace: 20 partial sums of a max_batch-row product, room for the 19 ranges that fill 152 SMs
    // with the 8 tiles of up to 128 rows by 1024 columns (256 rows take 10); thinner products get fewer ranges
    // than would fill the SMs
    n->ws_floats = (size_t)20 * maxB * (size_t)std::max(std::max(dh, din), 128);
    take((void**)&n->ws, sizeof(float) * n->ws_floats);
    for (auto& pl : plan) off += (pl.second + 255) & ~size_t(255);
    cudaError_t e = cudaMalloc((void**)&n->arena, off);
    if (e != cudaSuccess) {
        delete n;
        return mlp_err("cudaMalloc", e);
    }
    size_t o = 0;
    for (auto& pl : plan) {
        *pl.first = n->arena + o;
        o += (pl.second + 255) & ~size_t(255);
    }
    n->err = reinterpret_cast<int*>(n->loss + 1);
    n->applied = n->err + 1;
    auto fail = [&](int rc) { scs_mlp_destroy(n); return rc; };
    if (cudaMallocHost((void**)&n->report, sizeof(scs_mlp::Report) + sizeof(int)) != cudaSuccess ||
        cudaEventCreateWithFlags(&n->reported, cudaEventDisableTiming) != cudaSuccess)
        return fail(mlp_err("cudaMallocHost", cudaGetLastError()));
    n->skipped = reinterpret_cast<int*>(n->report + 1);
    *n->skipped = 0;
    if (cudaMemsetAsync(n->arena, 0, off, n->st) != cudaSuccess) return fail(mlp_err("memset", cudaGetLastError()));
    init_uniform<<<grid1d((long long)dh * din), 256, 0, n->st>>>(n->p, n->oW1, (long long)dh * din, 1.f / sqrtf((float)din), seed);
    init_uniform<<<grid1d((long long)dh * dh), 256, 0, n->st>>>(n->p, n->oW2, (long long)dh * dh, 1.f / sqrtf((float)dh), seed);
    init_uniform<<<grid1d((long long)dout * dh), 256, 0, n->st>>>(n->p, n->oW3, (long long)dout * dh, 1.f / sqrtf((float)dh), seed);
    fill_f32<<<grid1d(din), 256, 0, n->st>>>(n->in_std, din, 1.f);
    fill_f32<<<grid1d(din), 256, 0, n->st>>>(n->in_istd, din, 1.f);
    fill_f32<<<grid1d(dout), 256, 0, n->st>>>(n->out_std, dout, 1.f);
    fill_f32<<<grid1d(dout), 256, 0, n->st>>>(n->out_istd, dout, 1.f);
    int rc = scs_mlp_set_params(n, nullptr);
    if (rc) return fail(rc);
    *out = n;
    return SCS_OK;
}

// refresh the BF16 copies from the FP32 parameters
static int refresh_bf16(scs_mlp* n)
{
    f32_to_bf16_2d<<<grid1d((long long)n->dh * n->din), 256, 0, n->st>>>(n->p + n->oW1, n->dh, n->din, n->W1, n->ldin);
    f32_to_bf16_2d<<<grid1d((long long)n->dh * n->dh), 256, 0, n->st>>>(n->p + n->oW2, n->dh, n->dh, n->W2, n->dh);
    f32_to_bf16_2d<<<grid1d((long long)n->dout * n->dh), 256, 0, n->st>>>(n->p + n->oW3, n->dout, n->dh, n->W3, n->dh);
    MCU(cudaGetLastError());
    return SCS_OK;
}

// the transposed copies of W2 and W3, made each time they are read, by the legacy GEMM kernel's backward
// pass or by scs_mlp_read: the host cannot know that they are current, since a captured step updates W2
// and W3 at every replay
static void refresh_transposed(scs_mlp* n)
{
    transpose(n, n->W2, n->dh, n->dh, n->dh, n->W2t, n->dh);
    transpose(n, n->W3, n->dout, n->dh, n->dh, n->W3t, n->ldout);
}

extern "C" int64_t scs_mlp_num_params(const scs_mlp* n) { return n ? n->np : 0; }

extern "C" int scs_mlp_get_params(scs_mlp* n, float* params)
{
    if (!n || !params) return SCS_EINVAL;
    MCU(cudaMemcpyAsync(params, n->p, sizeof(float) * n->np, cudaMemcpyDefault, n->st));
    MCU(cudaStreamSynchronize(n->st));
    return SCS_OK;
}

extern "C" int scs_mlp_set_params(scs_mlp* n, const float* params)
{
    if (!n) return SCS_EINVAL;
    if (params) MCU(cudaMemcpyAsync(n->p, params, sizeof(float) * n->np, cudaMemcpyDefault, n->st));
    int rc = refresh_bf16(n);
    if (rc) return rc;
    MCU(cudaStreamSynchronize(n->st));
    return SCS_OK;
}

extern "C" int scs_mlp_fit_normalization(scs_mlp* n, const float* X, const float* Y, int64_t rows)
{
    if (!n || !X || !Y || rows <= 0) return SCS_EINVAL;
    col_stats<<<grid1d(n->din, 128), 128, 0, n->st>>>(X, rows, n->din, n->in_mean, n->in_std, n->in_istd);
    col_stats<<<grid1d(n->dout, 128), 128, 0, n->st>>>(Y, rows, n->dout, n->out_mean, n->out_std, n->out_istd);
    MCU(cudaGetLastError());
    MCU(cudaStreamSynchronize(n->st));
    return SCS_OK;
}

// Y: also the output in its own units, or null
static int forward(scs_mlp* n, const float* X, int B, float* Y = nullptr)
{
    int rc;
    n->lastB = B;
    MCU(launch_next(normalize_to_bf16, dim3((n->din + 255) / 256, std::min(B, MAX_GRID_Y)), 256, 0, n->st, X, B, n->din,
                    n->in_mean, n->in_istd, n->Xn, n->ldin));
    if ((rc = gemm(n, B, n->dh, n->din, n->Xn, n->ldin, false, n->W1, n->ldin, false,
                   epi(n->p + n->ob1, nullptr, 0, 1, nullptr, 0, n->h1, n->dh))))
        return rc;
    if ((rc = gemm(n, B, n->dh, n->dh, n->h1, n->dh, false, n->W2, n->dh, false,
                   epi(n->p + n->ob2, nullptr, 0, 1, nullptr, 0, n->h2, n->dh))))
        return rc;
    Epi e3 = epi(n->p + n->ob3, nullptr, 0, 0, n->y, n->dout, nullptr, 0);
    const bool fused = n->gemm_impl == SCS_MLP_GEMM_TCGEN05;
    if (Y && fused) {
        e3.Y = Y;
        e3.ystd = n->out_std;
        e3.ymean = n->out_mean;
    }
    if ((rc = gemm(n, B, n->dout, n->dh, n->h2, n->dh, false, n->W3, n->dh, false, e3))) return rc;
    if (Y && !fused) {
        denormalize<<<grid1d((long long)B * n->dout), 256, 0, n->st>>>(n->y, B, n->dout, n->out_mean, n->out_std, Y);
        MCU(cudaGetLastError());
    }
    return SCS_OK;
}

// loss (*n->loss) and gradients (n->g) of the last forward batch, queued
static int backward(scs_mlp* n, const float* Y, int B)
{
    const int Bp = pad8(B);
    const dim3 lg = loss_grid(n->dout, B);
    const bool tc = n->gemm_impl == SCS_MLP_GEMM_TCGEN05;
    const int vec = n->dout % 4 == 0 && (reinterpret_cast<uintptr_t>(Y) & 15) == 0 ? 1 : 0;
    int rc;
    MCU(launch_next(loss_grad, lg, 256, 0, n->st, n->y, Y, B, n->dout, n->out_mean, n->out_istd, n->dy32, n->dy16, n->ldout,
                    n->part, vec));
    if (!tc) {
        refresh_transposed(n);
        transpose(n, n->dy16, B, n->dout, n->ldout, n->dyt, Bp);
        transpose(n, n->h2, B, n->dh, n->dh, n->h2t, Bp);
        transpose(n, n->h1, B, n->dh, n->dh, n->h1t, Bp);
        transpose(n, n->Xn, B, n->din, n->ldin, n->Xnt, Bp);
    }
    // layer 3: gW3 = dy^T h2, dh2 = (dy W3) * [h2 > 0]
    const Epi g3 = epi(nullptr, nullptr, 0, 0, n->g + n->oW3, n->dh, nullptr, 0);
    const Epi e2 = epi(nullptr, n->h2, n->dh, 0, n->dh2_32, n->dh, n->dh2_16, n->dh);
    if ((rc = tc ? gemm(n, n->dout, n->dh, B, n->dy16, n->ldout, true, n->h2, n->dh, true, g3)
                 : gemm(n, n->dout, n->dh, B, n->dyt, Bp, false, n->h2t, Bp, false, g3)) ||
        (rc = tc ? gemm(n, B, n->dh, n->dout, n->dy16, n->ldout, false, n->W3, n->dh, true, e2)
                 : gemm(n, B, n->dh, n->dout, n->dy16, n->ldout, false, n->W3t, n->ldout, false, e2)))
        return rc;
    // layer 2
    const Epi g2 = epi(nullptr, nullptr, 0, 0, n->g + n->oW2, n->dh, nullptr, 0);
    const Epi e1 = epi(nullptr, n->h1, n->dh, 0, n->dh1_32, n->dh, n->dh1_16, n->dh);
    if (!tc) transpose(n, n->dh2_16, B, n->dh, n->dh, n->dh2t, Bp);
    if ((rc = tc ? gemm(n, n->dh, n->dh, B, n->dh2_16, n->dh, true, n->h1, n->dh, true, g2)
                 : gemm(n, n->dh, n->dh, B, n->dh2t, Bp, false, n->h1t, Bp, false, g2)) ||
        (rc = tc ? gemm(n, B, n->dh, n->dh, n->dh2_16, n->dh, false, n->W2, n->dh, true, e1)
                 : gemm(n, B, n->dh, n->dh, n->dh2_16, n->dh, false, n->W2t, n->dh, false, e1)))
        return rc;
    // layer 1
    const Epi g1 = epi(nullptr, nullptr, 0, 0, n->g + n->oW1, n->din, nullptr, 0);
    if (!tc) transpose(n, n->dh1_16, B, n->dh, n->dh, n->dh1t, Bp);
    if ((rc = tc ? gemm(n, n->dh, n->din, B, n->dh1_16, n->dh, true, n->Xn, n->ldin, true, g1)
                 : gemm(n, n->dh, n->din, B, n->dh1t, Bp, false, n->Xnt, Bp, false, g1)))
        return rc;
    Sums sm;
    const float* Ds[3] = {n->dy32, n->dh2_32, n->dh1_32};
    float* outs[3] = {n->g + n->ob3, n->g + n->ob2, n->g + n->ob1};
    const int ds[3] = {n->dout, n->dh, n->dh};
    sm.first[0] = 0;
    for (int k = 0; k < 3; ++k) {
        sm.D[k] = Ds[k];
        sm.out[k] = outs[k];
        sm.d[k] = ds[k];
        sm.first[k + 1] = sm.first[k] + (ds[k] + BS_COLS - 1) / BS_COLS;
    }
    sm.part = n->part;
    sm.nb = (int)(lg.x * lg.y);
    sm.scale = 0.5 / ((double)B * n->dout);
    sm.loss = n->loss;
    MCU(launch_next(bias_sums, sm.first[3] + 1, BS_COLS, 0, n->st, sm, B));
    return SCS_OK;
}

// queues the copy of (*loss, *err, *applied) to the host; report_wait reads it once it has arrived
static int report_queue(scs_mlp* n)
{
    MCU(cudaMemcpyAsync(n->report, n->loss, sizeof(scs_mlp::Report), cudaMemcpyDeviceToHost, n->st));
    MCU(cudaEventRecord(n->reported, n->st));
    return SCS_OK;
}
static int report_wait(scs_mlp* n, float* loss)
{
    MCU(cudaEventSynchronize(n->reported));
    if (n->report->err) return check_err_flag(n);
    if (loss) *loss = (float)n->report->loss;
    return SCS_OK;
}

extern "C" int scs_mlp_forward(scs_mlp* n, const float* X, int32_t B, float* Y)
{
    if (!n || !X || !Y || B <= 0 || B > n->maxB) {
        sscs::record_error("scs_mlp_forward: bad arguments");
        return SCS_EINVAL;
    }
    const int rc = earlier_error(n);
    return rc ? rc : forward(n, X, B, Y);
}

extern "C" int scs_mlp_gradients(scs_mlp* n, const float* X, const float* Y, int32_t B, float* grad, float* loss)
{
    if (!n || !X || !Y || B <= 0 || B > n->maxB) {
        sscs::record_error("scs_mlp_gradients: bad arguments");
        return SCS_EINVAL;
    }
    int rc = earlier_error(n);
    if (!rc) rc = forward(n, X, B);
    if (!rc) rc = backward(n, Y, B);
    if (rc) return rc;
    if (grad) MCU(cudaMemcpyAsync(grad, n->g, sizeof(float) * n->np, cudaMemcpyDefault, n->st));
    if ((rc = report_queue(n))) return rc;
    return report_wait(n, loss);
}

extern "C" int scs_mlp_train_step(scs_mlp* n, const float* X, const float* Y, int32_t B, float lr, float* loss)
{
    if (!n || !X || !Y || B <= 0 || B > n->maxB) {
        sscs::record_error("scs_mlp_train_step: bad arguments");
        return SCS_EINVAL;
    }
    int rc = earlier_error(n);
    if (!rc) rc = forward(n, X, B);
    if (!rc) rc = backward(n, Y, B);
    // the loss is on its way before Adam runs, so that the next step can be queued under it
    if (!rc && loss) rc = report_queue(n);
    if (rc) return rc;
    n->step++;
    // bias corrections 1 - beta^t in FP64: in FP32, 1 - 0.999f^t loses five digits to cancellation
    const float b1c = (float)(1.0 - pow(0.9, (double)n->step)), b2c = (float)(1.0 - pow(0.999, (double)n->step));
    Segs segs;
    segs.s[0] = {n->oW1, (long long)n->dh * n->din, n->W1, n->din, n->ldin};
    segs.s[1] = {n->ob1, n->dh, nullptr, 1, 1};
    segs.s[2] = {n->oW2, (long long)n->dh * n->dh, n->W2, n->dh, n->dh};
    segs.s[3] = {n->ob2, n->dh, nullptr, 1, 1};
    segs.s[4] = {n->oW3, (long long)n->dout * n->dh, n->W3, n->dh, n->dh};
    segs.s[5] = {n->ob3, n->dout, nullptr, 1, 1};
    MCU(launch_next(adam, grid1d((n->np + 3) / 4), 256, 0, n->st, n->p, n->g, n->m, n->v, n->np, lr, b1c, b2c, segs, n->err,
                    n->applied, n->skipped));
    return loss ? report_wait(n, loss) : SCS_OK;
}

extern "C" int scs_mlp_set_gemm(scs_mlp* n, int32_t impl)
{
    if (!n || (impl != SCS_MLP_GEMM_MMA && impl != SCS_MLP_GEMM_TCGEN05)) {
        sscs::record_error("scs_mlp_set_gemm: bad arguments");
        return SCS_EINVAL;
    }
    n->gemm_impl = impl;
    return SCS_OK;
}

extern "C" int scs_mlp_gemm_nt(int32_t impl, int32_t M, int32_t N, int32_t K, const void* A, int32_t lda,
                               const void* B, int32_t ldb, float* C, int32_t ldc, void* stream)
{
    // with K = 0 the operands are never read (C = 0) and may be null
    const bool aligned = ((reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B)) & 15) == 0;
    const bool operands_ok = K == 0 || (A && B && aligned);
    if ((impl != SCS_MLP_GEMM_MMA && impl != SCS_MLP_GEMM_TCGEN05) || M < 0 || N < 0 || K < 0 || !operands_ok ||
        !C || lda < K || ldb < K || lda % 8 || ldb % 8 || ldc < N) {
        sscs::record_error("scs_mlp_gemm_nt: bad arguments");
        return SCS_EINVAL;
    }
    if (M == 0 || N == 0) return SCS_OK;
    cudaStream_t st = (cudaStream_t)stream;
    if (K == 0) {  // empty sum: no kernel reads the (possibly null) operands
        MCU(cudaMemset2DAsync(C, sizeof(float) * (size_t)ldc, 0, sizeof(float) * (size_t)N, (size_t)M, st));
        MCU(cudaStreamSynchronize(st));
        return SCS_OK;
    }
    int* err = nullptr;
    MCU(cudaMalloc((void**)&err, sizeof(int)));
    // the split-K workspace this product would use (tensor-core kernel only)
    float* ws = nullptr;
    size_t ws_floats = 0;
    if (impl == SCS_MLP_GEMM_TCGEN05) {
        const TcPlan p = tc_plan(M, N, K, false, device_sms(), (size_t)1 << 40);
        if (p.spc < p.splits) {
            ws_floats = (size_t)p.splits * M * N;
            if (cudaMalloc((void**)&ws, sizeof(float) * ws_floats) != cudaSuccess) {
                cudaFree(err);
                return mlp_err("cudaMalloc", cudaGetLastError());
            }
        }
    }
    int rc = SCS_OK;
    if (cudaMemsetAsync(err, 0, sizeof(int), st) != cudaSuccess) rc = mlp_err("memset", cudaGetLastError());
    if (!rc)
        rc = launch_gemm(impl, st, err, M, N, K, static_cast<const bf16*>(A), lda, false, static_cast<const bf16*>(B), ldb,
                         false,                         epi(nullptr, nullptr, 0, 0, C, ldc, nullptr, 0), ws, ws_floats);
    int h = 0;
    if (!rc && cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess)
        rc = mlp_err("copy", cudaGetLastError());
    if (!rc && cudaStreamSynchronize(st) != cudaSuccess) rc = mlp_err("gemm", cudaGetLastError());
    cudaFree(err);
    if (ws) cudaFree(ws);
    if (!rc && h) {
        if (h >= 2) g_tc_fatal = true;
        sscs::record_error(h >= 2 ? TC_FATAL_MSG : "scs_mlp_gemm_nt: a tensor-core wait timed out");
        rc = SCS_ECUDA;
    }
    return rc;
}

extern "C" int scs_mlp_read(scs_mlp* n, int32_t what, void* out, int64_t* rows, int64_t* cols, int32_t* elem_bytes)
{
    if (!n) {
        sscs::record_error("scs_mlp_read: NULL network");
        return SCS_EINVAL;
    }
    const void* src = nullptr;
    long long r = 1, c = 0, ld = 0;
    int eb = 4;
    const long long B = n->lastB;
    switch (what) {
        case SCS_MLP_READ_PARAMS: src = n->p; c = n->np; break;
        case SCS_MLP_READ_GRAD: src = n->g; c = n->np; break;
        case SCS_MLP_READ_ADAM_M: src = n->m; c = n->np; break;
        case SCS_MLP_READ_ADAM_V: src = n->v; c = n->np; break;
        case SCS_MLP_READ_IN_MEAN: src = n->in_mean; c = n->din; break;
        case SCS_MLP_READ_IN_STD: src = n->in_std; c = n->din; break;
        case SCS_MLP_READ_OUT_MEAN: src = n->out_mean; c = n->dout; break;
        case SCS_MLP_READ_OUT_STD: src = n->out_std; c = n->dout; break;
        case SCS_MLP_READ_XN: src = n->Xn; r = B; c = n->din; ld = n->ldin; eb = 2; break;
        case SCS_MLP_READ_H1: src = n->h1; r = B; c = n->dh; eb = 2; break;
        case SCS_MLP_READ_H2: src = n->h2; r = B; c = n->dh; eb = 2; break;
        case SCS_MLP_READ_Y: src = n->y; r = B; c = n->dout; break;
        case SCS_MLP_READ_DY: src = n->dy32; r = B; c = n->dout; break;
        case SCS_MLP_READ_DY16: src = n->dy16; r = B; c = n->dout; ld = n->ldout; eb = 2; break;
        case SCS_MLP_READ_DH2: src = n->dh2_32; r = B; c = n->dh; break;
        case SCS_MLP_READ_DH2_16: src = n->dh2_16; r = B; c = n->dh; eb = 2; break;
        case SCS_MLP_READ_DH1: src = n->dh1_32; r = B; c = n->dh; break;
        case SCS_MLP_READ_DH1_16: src = n->dh1_16; r = B; c = n->dh; eb = 2; break;
        case SCS_MLP_READ_W1: src = n->W1; r = n->dh; c = n->din; ld = n->ldin; eb = 2; break;
        case SCS_MLP_READ_W2: src = n->W2; r = n->dh; c = n->dh; eb = 2; break;
        case SCS_MLP_READ_W3: src = n->W3; r = n->dout; c = n->dh; eb = 2; break;
        case SCS_MLP_READ_W2T: refresh_transposed(n); src = n->W2t; r = n->dh; c = n->dh; eb = 2; break;
        case SCS_MLP_READ_W3T: refresh_transposed(n); src = n->W3t; r = n->dh; c = n->dout; ld = n->ldout; eb = 2; break;
        default:
            sscs::record_error("scs_mlp_read: unknown buffer");
            return SCS_EINVAL;
    }
    if (ld == 0) ld = c;
    if (rows) *rows = r;
    if (cols) *cols = c;
    if (elem_bytes) *elem_bytes = eb;
    if (!out || r == 0 || c == 0) return SCS_OK;
    MCU(cudaMemcpy2DAsync(out, (size_t)c * eb, src, (size_t)ld * eb, (size_t)c * eb, (size_t)r, cudaMemcpyDefault,
                          n->st));
    MCU(cudaStreamSynchronize(n->st));
    return SCS_OK;
}

extern "C" void scs_mlp_destroy(scs_mlp* n)
{
    if (!n) return;
    if (n->arena) cudaFree(n->arena);  // waits for the device: a queued step may still write the pinned report
    if (n->reported) cudaEventDestroy(n->reported);
    if (n->report) cudaFreeHost(n->report);
    delete n;
}
