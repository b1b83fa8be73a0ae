// solver.cuh -- device-resident SuperSCS (Sopasakis, Menounou, Patrinos,
// arXiv 1903.06477), generic over the bulk precision T (double or float)
// and over the execution team (one CTA, or every CTA of a cooperative grid).
//
// Structure of one outer iteration (Algorithm 1):
//   termination test (Sec. 4.3)       2 SpMVs + 1 reduction
//   direction d (Sec. 4.4, AA or RB)   passes over the N x mem buffers
//   d~ = (I+Q)^{-1} d                  CG on I + A^T A (Sec. 4.1)
//   K0 | line search with K1/K2        fused projection + residual passes
// HSDE vectors keep their tau entry in FP64 whatever T is.
#pragma once

#include <vector>

#include "common.cuh"
#include "team.cuh"

namespace sscs {

constexpr int MAXMEM = 64;   // direction memory cap (RB)
constexpr int AAMAX = 32;    // Anderson memory cap (Gram matrix kept in shared memory)
constexpr int PSD_MAX = 64;  // largest PSD order decomposed in shared memory
constexpr int PSD_BIG_MAX = 1024;    // largest PSD order (orders above PSD_MAX use a global-memory workspace)

enum Mode { MODE_SETUP = 0, MODE_SOLVE = 1, MODE_LINSYS = 2, MODE_PROJECT = 3, MODE_APPLY_T = 4, MODE_PROFILE = 5,
            MODE_RESID = 6, MODE_SPMV = 7, MODE_FACTOR = 8 };
enum { ST_SOLVED = 1, ST_INFEASIBLE = -1, ST_UNBOUNDED = -2, ST_MAX_ITERS = -3, ST_TIME_LIMIT = -4,
       ST_NUMERICAL = -5, ST_STALLED = -6 };

template <typename T>
struct HV {  // HSDE vector: (chi, psi) bulk of n+m entries in T, tau in FP64
    T* v;
    double* t;
};

struct DevSettings {
    int direction, mem;
    double eps, c0, c1, q, sigma, lambda, thetabar;
    int max_iters, ls_max, cg_max, check_every;
    double cg_rtol, aa_reg;
    double time_limit_ns;  // <= 0: none
    int stall_iters;       // > 0: stop when ||Ru|| has not dropped 10% below its best for this many iterations
    int use_warm;
    double switch_kkt;     // > 0: stop (hand over) once max(pr,dr,gap) <= switch_kkt
    double cg_adapt;       // > 0: CG inside the loop also stops at ||res|| <= cg_adapt ||Ru||
    int keep_ws;           // 1: keep the CG warm starts found in ws (handed over by the FP32 phase)
    int warm_fallback;     // > 0 with a warm start: restart cold if ||Ru|| is not below the cold
                           // start's ||Ru0|| after this many iterations
    int save_state;        // 1: write the loop state to W.res when the solve ends (FP32 phase of SCS_MIXED)
    int resume;            // 1: continue from the loop state in W.res instead of starting Algorithm 1 afresh
    int stall_after_tau;   // 1: the stall count starts only once tau_ > 0 (FP32 phase of SCS_MIXED)
    int refine;            // 1 (FP64 data only): linear systems by iterative refinement, FP64 residuals
                           // and FP32 CG corrections on the FP32 copy of A (W.ir)
    double psd_tol;        // FP32 eigensolves: a PSD block whose FP64-evaluated relative eigen-residual
                           // exceeds this is decomposed again in FP64
};

// State of Algorithm 1 at the end of the FP32 phase of SCS_MIXED, so that the
// FP64 phase continues the same iteration (direction memory, the K0/K1
// references eta, eta0, r_safe and the outer index nu) instead of restarting.
struct Resume {
    int valid, count, have_pair, nu;
    long long inserted;
    double eta, eta0, r_safe, nz2;
    double G[AAMAX * AAMAX];  // AA Gram matrix of the stored pairs
};

struct DevState {
    int status, iters, k0, k1, k2, backtracks;
    long long cg_iters;
    double pr, dr, gap, ic, uc, pobj, dobj, nRu, hg;
    int setup_cg, pad;
    long long mat_passes;  // SpMV passes over A or A^T
    double psd_resid;      // largest ||X V - V L||_F / ||X||_F of the FP32 eigensolves, in FP64
    int fallback;          // 1 if the warm start was abandoned for the cold start
    int pad2;
    long long mat_passes_ir;  // FP32 passes of the refinement corrections (FP64 phase)
    long long cg_iters_ir;    // FP32 CG iterations of the refinement corrections (FP64 phase)
    long long ir_sweeps;      // refinement sweeps (FP32 correction solves)
    // device time (globaltimer, read by the leader thread between team barriers) of the parts of
    // Algorithm 1: [0] termination tests, [1] directions, [2] linear solves (all of minv / its
    // refinement variant), [3] the CG loops inside them, [4] everything else (K0 steps, line
    // searches, projections, updates)
    double part_ns[5];
    long long psd_redo;    // PSD blocks of the FP32 phase decomposed again in FP64 (eigen-residual above psd_tol)
};

// Column-blocked sliced ELL, the grid team's layout for large matrices.  CTA b
// owns the contiguous rows [rbnd[b], rbnd[b+1]); the columns are cut into ncb
// blocks of cw.  A "segment" is one (CTA, column block) pair: the CTA's rows
// that have entries in the block, sorted by their count there (descending),
// packed as slices of H = 32 / V rows (V chosen for each segment) with element j of slice row r at
// step (slice start + j / V), lane (j % V) * H + r, 32 entries per step, and
// its column stored as a 16-bit offset inside the block (padding: value 0,
// offset 0).  The slices of a segment are dealt to the CTA's warps (largest
// first to the least-loaded warp) and stored warp by warp.  The entries of
// segment g = b * ncb + k are contiguous, [E0, E1) of col / val.
//
// Each segment has ms 32-bit words of metadata at meta + g * ms:
//   [0] E0   [1] E1   [2], [3] E0, E1 of the CTA's segment (k + S) mod ncb
//   [4] ns slices + (H << 16)   [5 .. 5+nw] first slice of each warp (nw+1 values)
//   [6+nw .. 6+nw+ns] slice start steps from E0 (ns+1 values)
//   then ns * H 16-bit row indices inside the CTA's range (0xFFFF: none),
//   two per word, low half first.
//
// The product streams segments through a ring of S shared-memory stages,
// warp-specialised: the CTA's last warp is the producer, which copies a
// segment's metadata, its slice of the multiplied vector and its entries with
// bulk (TMA) copies completing on the stage's "full" mbarrier as soon as the
// stage's "empty" mbarrier says every compute warp is done with it; the
// other nw warps compute, so the random reads of the vector and the matrix
// stream are all shared-memory reads.  The rows of one segment are distinct,
// and the partial sums are double-buffered by segment parity: a compute warp
// starts segment j once segment j-2 is finished by every warp (its "empty"
// barrier), so warps may run one segment apart without two of them ever
// updating the same sum, and each sum is accumulated in a fixed order
// (deterministic).  CTA b visits the column blocks in the order b, b+1, ...
// (mod ncb), so at any moment the CTAs read different slices of the vector.
// The CTA adds its two partial-sum buffers after the last block.
template <typename T>
struct Cblk {
    int ncb;          // column blocks (0: layout absent)
    int cw;           // columns per block (multiple of 4)
    int cols;         // columns of the matrix
    int nw;           // compute warps per CTA (the CTA has nw + 1 warps)
    int V;            // lanes per row (tiles; the segments name their own)
    int acc_rows;     // partial-sum entries per buffer (largest row range); 2 buffers per vector
    int ms;           // metadata words per segment (multiple of 4)
    int S;            // stages in the copy ring (2..CB_MAX_STAGES)
    int stage_off;    // byte offset of stage 0 in dynamic shared memory
    int stage_bytes;  // bytes per stage (multiple of 16)
    int off_x, off_col, off_val;  // byte offsets inside a stage (tiles: off_x = the vector slice's offset
                                  // in dynamic shared memory, after the tile's row sums)
    const int* rbnd;
    const int* meta;
    const unsigned short* col;
    const T* val;
    // two-dimensional tiles (tile = 1; layout in cb_layout.h): R row blocks of
    // rbnd, ncb column blocks, tile g = r * ncb + k on CTA g with chunks
    // [cbeg[g], cbeg[g+1]) of meta; part holds two buffers of nv x ncb x rows
    // partial sums
    int tile, R, rows, nv;
    const int* cbeg;
    T* part;
};

// Sliced ELL with row sorting (SELL-H-sigma) and V lanes per row, H = 32 / V
// rows per slice: element j of the slice's row r sits at ptr[s] + j*H + r,
// so lane q*H + r of a warp reads element t*V + q of row r at
// ptr[s] + 32 t + lane -- every load of a warp is one coalesced 32-element
// segment, and each lane streams its own run of independent loads.
template <typename T>
struct Sell {
    int rows, V, nslices;
    const int* ptr;    // nslices + 1 offsets (multiples of 32)
    const int* col;    // padded column indices
    const T* val;      // padded values (0 in padding)
    const int* perm;   // sorted position -> original row (nslices * H entries, -1 past the end)
    const int* wbnd;   // grid team only: warp w owns slices [wbnd[w], wbnd[w+1]) (nnz-balanced), else null
    Cblk<T> cb;        // grid team only: column-blocked copy (cb.ncb > 0), used instead of the above
    int l1;            // block team: the padded matrix is small enough (48 KB) to keep in L1 across products
};

constexpr int TMA_CH = 8;  // t-steps (of 32 elements) per staged chunk
template <typename T>
__host__ __device__ constexpr int tma_stage_bytes()
{
    return TMA_CH * 32 * (4 + (int)sizeof(T));
}

template <typename T>
struct DevProb {
    int n, m;
    Sell<T> A;   // A   (m rows)
    Sell<T> AT;  // A^T (n rows)
    const T *b, *c;
    double nb, nc;
    int f, l, nq, ns;
    const int* q_off;  // nq+1 row offsets of the SOCs inside s
    const int* s_dim;  // ns PSD orders
    const int* s_off;  // ns row offsets of the PSD blocks inside s
    int ep, ed;        // primal / dual exponential cones (3 rows each)
    int e_off;         // row offset of the first exponential cone inside s
    // PSD blocks above PSD_MAX: the Jacobi workspace of block k starts at psd_big + big_off[k]
    // bytes (laid out by psd_layout below; big_off[k] < 0 for blocks decomposed in shared memory)
    unsigned char* psd_big;
    const long long* big_off;
    const long long* v_off;  // byte offset of each PSD block's warm-start eigenvectors in DevWork::psd_v
    int psd_order;           // the largest PSD order
    int psd_small;           // the largest one up to PSD_MAX (0: none)
};

// Iterative refinement of the FP64 linear solves (SCS_MIXED, FP64 phase): the
// FP32 copies of A and A^T and FP32 vectors for the correction solves.
struct IrBufs {
    Sell<float> A, AT;
    float *r, *p, *q, *x;  // n
    float* tm;             // m
};

template <typename T>
struct DevWork {
    IrBufs ir;
    Resume* res;  // loop state handed from the FP32 to the FP64 phase (SCS_MIXED)
    T* dinv;      // direct solves: L^{-1} and its transpose, I + A^T A = L L^T, n x n (else null)
    int* dinv_fail;  // set by MODE_FACTOR if a pivot was not positive (the factor is then not used)
    HV<T> u, ut, ub, Ru, d, dt, wb, Rw, zp, xip, zt;
    T* g;       // n+m: g = M^{-1}(c, b)
    T* ws[2];   // CG warm starts (n) for the u~ and d~ systems
    T *cr, *cp, *cq, *tn;  // n
    T *tm, *py;            // m
    T* Zv;
    double* Zt;  // mem columns (AA: z^i; RB: z^i)
    T* Xv;
    double* Xt;  // mem columns (AA: xi^i; RB: z~^i)
    T* Qv;
    double* Qt;  // AA with QR: mem orthonormal columns, Xi (oldest first) = Q R
    double *io_in, *io_out, *io_out2;      // N-vectors of the single-operator entries
    double* warm;                          // N: warm start (FP64)
    double *x_out, *y_out, *s_out, *u_out; // results (FP64)
    unsigned char* psd_v;  // PSD blocks: eigenvectors of the last converged decomposition (warm starts)
    int* psd_vok;          // per PSD block: 0 if psd_v holds nothing, else warm-start generations
    double* partials;      // [2][KMAX][blocks] block partials
    unsigned* bar;
    int* abort_flag;
    DevState* st;
};

template <typename T>
struct Args {
    DevProb<T> P;
    DevWork<T> W;
    DevSettings S;
    int mode;
    int slot;
};

__device__ __forceinline__ float fmaT(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fmaT(double a, double b, double c) { return fma(a, b, c); }

// ---------------------------------------------------------------------------
// sparse products on the sliced-ELL layout: warps of the team take slices in
// turn; xf(c) supplies the gathered vector entry, epi(row, sum) consumes the
// row result (only lanes q = 0 call it)
// ---------------------------------------------------------------------------
// Matrix entries of the sliced-ELL products: streamed past L1 (evict-first in
// L2), except for a block-team instance small enough to stay in L1 across the
// products of its solve (Sell::l1), whose entries are cached there.
template <typename V>
__device__ __forceinline__ V ldm(const V* p, unsigned long long pol, bool l1)
{
    return l1 ? ro(p) : ld_stream(p, pol);
}

template <typename T, class Team, class XF, class Epi>
__device__ __forceinline__ void sell_v(const Team& tm, const Sell<T>& S, XF& xf, Epi& epi)
{
    const int H = 32 / S.V;
    const int lane = threadIdx.x & 31;
    const int nw = tm.size() >> 5;
    const unsigned long long pol = evict_first_policy();
    const bool l1 = !Team::kGrid && S.l1;
    for (int s = tm.rank() >> 5; s < S.nslices; s += nw) {
        const int p0 = ro(S.ptr + s);
        const int tc = (ro(S.ptr + s + 1) - p0) >> 5;
        const int* cp = S.col + p0 + lane;
        const T* vp = S.val + p0 + lane;
        T a0 = 0, a1 = 0;
        int t = 0;
        for (; t + 4 <= tc; t += 4) {
            const int c0 = ldm(cp + 32 * t, pol, l1), c1 = ldm(cp + 32 * (t + 1), pol, l1),
                      c2 = ldm(cp + 32 * (t + 2), pol, l1), c3 = ldm(cp + 32 * (t + 3), pol, l1);
            const T v0 = ldm(vp + 32 * t, pol, l1), v1 = ldm(vp + 32 * (t + 1), pol, l1),
                    v2 = ldm(vp + 32 * (t + 2), pol, l1), v3 = ldm(vp + 32 * (t + 3), pol, l1);
            const T x0 = xf(c0), x1 = xf(c1), x2 = xf(c2), x3 = xf(c3);
            a0 = fmaT(v0, x0, a0);
            a1 = fmaT(v1, x1, a1);
            a0 = fmaT(v2, x2, a0);
            a1 = fmaT(v3, x3, a1);
        }
        for (; t < tc; ++t) a0 += ldm(vp + 32 * t, pol, l1) * xf(ldm(cp + 32 * t, pol, l1));
        T acc = a0 + a1;
        for (int o = H; o < 32; o <<= 1) acc += __shfl_xor_sync(FULL_MASK, acc, o);
        const int pos = s * H + lane;
        if (lane < H && pos < S.rows) epi(ro(S.perm + pos), acc);
    }
}

template <typename T, class Team, class XF1, class XF2, class Epi>
__device__ __forceinline__ void sell2_v(const Team& tm, const Sell<T>& S, XF1& xf1, XF2& xf2, Epi& epi)
{
    const int H = 32 / S.V;
    const int lane = threadIdx.x & 31;
    const int nw = tm.size() >> 5;
    const unsigned long long pol = evict_first_policy();
    const bool l1 = !Team::kGrid && S.l1;
    for (int s = tm.rank() >> 5; s < S.nslices; s += nw) {
        const int p0 = ro(S.ptr + s);
        const int tc = (ro(S.ptr + s + 1) - p0) >> 5;
        const int* cp = S.col + p0 + lane;
        const T* vp = S.val + p0 + lane;
        T a1 = 0, a2 = 0, b1 = 0, b2 = 0;
        int t = 0;
        for (; t + 2 <= tc; t += 2) {
            const int c0 = ldm(cp + 32 * t, pol, l1), c1 = ldm(cp + 32 * (t + 1), pol, l1);
            const T v0 = ldm(vp + 32 * t, pol, l1), v1 = ldm(vp + 32 * (t + 1), pol, l1);
            a1 += v0 * xf1(c0);
            a2 += v0 * xf2(c0);
            b1 += v1 * xf1(c1);
            b2 += v1 * xf2(c1);
        }
        if (t < tc) {
            const int c0 = ldm(cp + 32 * t, pol, l1);
            const T v0 = ldm(vp + 32 * t, pol, l1);
            a1 += v0 * xf1(c0);
            a2 += v0 * xf2(c0);
        }
        a1 += b1;
        a2 += b2;
        for (int o = H; o < 32; o <<= 1) {
            a1 += __shfl_xor_sync(FULL_MASK, a1, o);
            a2 += __shfl_xor_sync(FULL_MASK, a2, o);
        }
        const int pos = s * H + lane;
        if (lane < H && pos < S.rows) epi(ro(S.perm + pos), a1, a2);
    }
}

// Sparse product with the matrix stream staged through shared memory by TMA
// bulk copies: each warp owns a contiguous, nnz-balanced run of slices,
// copies it in chunks of TMA_CH t-steps into a two-stage buffer (one
// mbarrier per stage) and computes chunk k while chunk k+1 is in flight, so
// the HBM stream never waits on the gathers.  Waits are bounded: on timeout
// the abort flag is set, the warp waits (bounded) for its other copy and
// leaves the product unfinished.
template <typename T, class Team, class XF, class Epi>
__device__ __forceinline__ void sell_tma(const Team& tm, const Sell<T>& S, XF& xf, Epi& epi)
{
    const int H = 32 / S.V;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int gw = tm.rank() >> 5;
    const int s0 = ro(S.wbnd + gw), s1 = ro(S.wbnd + gw + 1);
    if (s0 >= s1) return;
    const int e0 = ro(S.ptr + s0);
    const int total_t = (ro(S.ptr + s1) - e0) >> 5;
    constexpr int SB = tma_stage_bytes<T>();
    unsigned char* wbuf = tm.stage + (size_t)wib * 2 * SB;
    const unsigned bar0 = smem_addr(&tm.mbar[2 * wib]), bar1 = smem_addr(&tm.mbar[2 * wib + 1]);
    unsigned ph = tm.ph[wib];
    const unsigned long long pol = evict_first_policy();
    const int nch = (total_t + TMA_CH - 1) / TMA_CH;
    auto issue = [&](int k) {
        const int t_lo = k * TMA_CH;
        const int nt = min(TMA_CH, total_t - t_lo);
        unsigned char* dst = wbuf + (k & 1) * SB;
        const unsigned bar = (k & 1) ? bar1 : bar0;
        const unsigned bc = (unsigned)nt * 32u * 4u, bv = (unsigned)nt * 32u * (unsigned)sizeof(T);
        fence_proxy_async();
        mbar_expect_tx(bar, bc + bv);
        tma_load_1d(smem_addr(dst), S.col + e0 + 32 * t_lo, bc, bar, pol);
        tma_load_1d(smem_addr(dst + TMA_CH * 32 * 4), S.val + e0 + 32 * t_lo, bv, bar, pol);
    };
    auto finalize = [&](int sl, T a) {
        for (int o = H; o < 32; o <<= 1) a += __shfl_xor_sync(FULL_MASK, a, o);
        const int pos = sl * H + lane;
        if (lane < H && pos < S.rows) epi(ro(S.perm + pos), a);
    };
    if (nch > 0 && lane == 0) issue(0);
    int cur = s0;
    int bound = (ro(S.ptr + cur + 1) - e0) >> 5;
    T acc = 0;
    for (int k = 0; k < nch; ++k) {
        const bool more = k + 1 < nch;
        if (more) {
            __syncwarp();
            if (lane == 0) issue(k + 1);
        }
        const unsigned bar = (k & 1) ? bar1 : bar0;
        bool ok = mbar_wait(bar, (ph >> (k & 1)) & 1u, tm.abort_flag);
        ok = __all_sync(FULL_MASK, ok);
        ph ^= 1u << (k & 1);
        if (!ok) {
            if (more) {
                const unsigned obar = (k & 1) ? bar0 : bar1;
                mbar_wait(obar, (ph >> ((k + 1) & 1)) & 1u, nullptr);
                ph ^= 1u << ((k + 1) & 1);
            }
            if (lane == 0) tm.ph[wib] = ph;
            __syncwarp();
            return;
        }
        const int t_lo = k * TMA_CH;
        const int nt = min(TMA_CH, total_t - t_lo);
        const int* sc = (const int*)(wbuf + (k & 1) * SB);
        const T* sv = (const T*)(wbuf + (k & 1) * SB + TMA_CH * 32 * 4);
        int cs[TMA_CH];
        T vs[TMA_CH], xs[TMA_CH];
#pragma unroll
        for (int t = 0; t < TMA_CH; ++t) {
            cs[t] = t < nt ? sc[t * 32 + lane] : 0;
            vs[t] = t < nt ? sv[t * 32 + lane] : T(0);
        }
#pragma unroll
        for (int t = 0; t < TMA_CH; ++t) xs[t] = xf(cs[t]);
#pragma unroll
        for (int t = 0; t < TMA_CH; ++t) {
            if (t < nt) {
                const int tg = t_lo + t;
                while (tg == bound) {
                    finalize(cur, acc);
                    acc = 0;
                    ++cur;
                    bound = (ro(S.ptr + cur + 1) - e0) >> 5;
                }
                acc = fmaT(vs[t], xs[t], acc);
            }
        }
    }
    while (cur < s1) {
        finalize(cur, acc);
        acc = 0;
        ++cur;
    }
    if (lane == 0) tm.ph[wib] = ph;
    __syncwarp();
}

// ---------------------------------------------------------------------------
// column-blocked product (grid team): y = M x (NV = 1) or M x1, M x2 (NV = 2)
// ---------------------------------------------------------------------------

// One segment from its stage: compute warp w runs its slices (matrix
// entries, the vector slice and the metadata all in shared memory); row sums
// are reduced over the V = 32 / H lanes of a row and added to acc (rows of a
// segment are distinct, so plain read-modify-writes do not race).  Operands
// are byte offsets into the dynamic shared memory, indexed through the
// shared array itself so the loads are 32-bit-addressed shared loads and the
// hot loop touches no local memory.
template <typename T>
__device__ __forceinline__ void cb_segment(int nw, unsigned mt_off, unsigned xs_off, unsigned col_off,
                                           unsigned val_off, unsigned acc_off)
{
    extern __shared__ __align__(128) unsigned char cb_sm[];
    const int* mt = (const int*)(cb_sm + mt_off);
    const T* xs = (const T*)(cb_sm + xs_off);
    const unsigned short* scol = (const unsigned short*)(cb_sm + col_off);
    const T* sval = (const T*)(cb_sm + val_off);
    T* acc = (T*)(cb_sm + acc_off);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int ns = mt[4] & 0xFFFF, H = mt[4] >> 16;
    const int* wl = mt + 5;
    const int* st = wl + nw + 1;
    const unsigned short* sr = (const unsigned short*)(st + ns + 1);
    const int s_hi = wl[w + 1];
    int s0 = wl[w];
    if constexpr (sizeof(T) == 4) {
        // FP32, two slices at a time: their steps interleave four by four, so a warp keeps
        // eight independent offset -> gather -> FMA chains in flight instead of four (the
        // slices are short: about six steps at the benchmark's row lengths)
        for (; s0 + 1 < s_hi; s0 += 2) {
            int ta = st[s0];
            const int ta1 = st[s0 + 1];
            int tb = ta1;
            const int tb1 = st[s0 + 2];
            T a0 = 0, a1 = 0, a2 = 0, a3 = 0, b0 = 0, b1 = 0, b2 = 0, b3 = 0;
            for (; ta < ta1 || tb < tb1; ta += 4, tb += 4) {
                const bool p0 = ta < ta1, p1 = ta + 1 < ta1, p2 = ta + 2 < ta1, p3 = ta + 3 < ta1;
                const bool q0 = tb < tb1, q1 = tb + 1 < tb1, q2 = tb + 2 < tb1, q3 = tb + 3 < tb1;
                const int c0 = p0 ? (int)scol[ta * 32 + lane] : 0;
                const int c1 = p1 ? (int)scol[ta * 32 + 32 + lane] : 0;
                const int c2 = p2 ? (int)scol[ta * 32 + 64 + lane] : 0;
                const int c3 = p3 ? (int)scol[ta * 32 + 96 + lane] : 0;
                const int d0 = q0 ? (int)scol[tb * 32 + lane] : 0;
                const int d1 = q1 ? (int)scol[tb * 32 + 32 + lane] : 0;
                const int d2 = q2 ? (int)scol[tb * 32 + 64 + lane] : 0;
                const int d3 = q3 ? (int)scol[tb * 32 + 96 + lane] : 0;
                const T v0 = p0 ? sval[ta * 32 + lane] : T(0);
                const T v1 = p1 ? sval[ta * 32 + 32 + lane] : T(0);
                const T v2 = p2 ? sval[ta * 32 + 64 + lane] : T(0);
                const T v3 = p3 ? sval[ta * 32 + 96 + lane] : T(0);
                const T u0 = q0 ? sval[tb * 32 + lane] : T(0);
                const T u1 = q1 ? sval[tb * 32 + 32 + lane] : T(0);
                const T u2 = q2 ? sval[tb * 32 + 64 + lane] : T(0);
                const T u3 = q3 ? sval[tb * 32 + 96 + lane] : T(0);
                a0 = fmaT(v0, xs[c0], a0);
                a1 = fmaT(v1, xs[c1], a1);
                a2 = fmaT(v2, xs[c2], a2);
                a3 = fmaT(v3, xs[c3], a3);
                b0 = fmaT(u0, xs[d0], b0);
                b1 = fmaT(u1, xs[d1], b1);
                b2 = fmaT(u2, xs[d2], b2);
                b3 = fmaT(u3, xs[d3], b3);
            }
            T a = (a0 + a2) + (a1 + a3), b = (b0 + b2) + (b1 + b3);
            for (int o = H; o < 32; o <<= 1) {
                a += __shfl_xor_sync(FULL_MASK, a, o);
                b += __shfl_xor_sync(FULL_MASK, b, o);
            }
            if (lane < H) {
                const int ra = sr[s0 * H + lane], rb = sr[(s0 + 1) * H + lane];
                if (ra != 0xFFFF) acc[ra] += a;
                if (rb != 0xFFFF) acc[rb] += b;
            }
        }
    }
    for (int s = s0; s < s_hi; ++s) {
        const int t1 = st[s + 1];
        int t = st[s];
        if constexpr (sizeof(T) == 4) {
            // FP32: four steps per trip, the tail predicated (offset 0, value 0)
            T a0 = 0, a1 = 0, a2 = 0, a3 = 0;
            for (; t < t1; t += 4) {
                const bool o1 = t + 1 < t1, o2 = t + 2 < t1, o3 = t + 3 < t1;
                const int c0 = scol[t * 32 + lane];
                const int c1 = o1 ? (int)scol[t * 32 + 32 + lane] : 0;
                const int c2 = o2 ? (int)scol[t * 32 + 64 + lane] : 0;
                const int c3 = o3 ? (int)scol[t * 32 + 96 + lane] : 0;
                const T v0 = sval[t * 32 + lane];
                const T v1 = o1 ? sval[t * 32 + 32 + lane] : T(0);
                const T v2 = o2 ? sval[t * 32 + 64 + lane] : T(0);
                const T v3 = o3 ? sval[t * 32 + 96 + lane] : T(0);
                a0 = fmaT(v0, xs[c0], a0);
                a1 = fmaT(v1, xs[c1], a1);
                a2 = fmaT(v2, xs[c2], a2);
                a3 = fmaT(v3, xs[c3], a3);
            }
            T a = (a0 + a2) + (a1 + a3);
            for (int o = H; o < 32; o <<= 1) a += __shfl_xor_sync(FULL_MASK, a, o);
            if (lane < H) {
                const int r = sr[s * H + lane];
                if (r != 0xFFFF) acc[r] += a;
            }
        } else {
            // FP64: two chains.  The row index is read ahead of them: after the sum, with H (lanes per row) in a
            // register only since the segments choose it, it cost the product 1 us (1e7 nonzeros, A, A^T and a CG
            // iteration: 41.1, 44.0 and 93.6 us with one H for the matrix, 43.3, 45.0 and 95.4 with H by segment,
            // 42.5, 44.5 and 94.0 so)
            const int r = lane < H ? sr[s * H + lane] : 0xFFFF;
            T a0 = 0, a1 = 0;
            for (; t + 2 <= t1; t += 2) {
                const int c0 = scol[t * 32 + lane], c1 = scol[t * 32 + 32 + lane];
                const T v0 = sval[t * 32 + lane], v1 = sval[t * 32 + 32 + lane];
                a0 = fmaT(v0, xs[c0], a0);
                a1 = fmaT(v1, xs[c1], a1);
            }
            if (t < t1) a0 = fmaT(sval[t * 32 + lane], xs[scol[t * 32 + lane]], a0);
            T a = a0 + a1;
            for (int o = H; o < 32; o <<= 1) a += __shfl_xor_sync(FULL_MASK, a, o);
            if (r != 0xFFFF) acc[r] += a;
        }
    }
}

// acc[0, R) + acc[acc_rows, acc_rows + R) = (rows of this CTA's range) . x
// over all column blocks (even segments into the first buffer, odd into the
// second), through the ring of S stages: full barriers tm.mbar[0..S-1], empty
// barriers tm.mbar[CB_MAX_STAGES + s]; tm.ph[s] counts the stage's past uses,
// so use u of this pass waits on parity (ph[s] + u) & 1.  Every field the
// loops need is read once into registers (the structs live in local memory,
// which misses the small L1 left beside the stages).  Returns false if a wait
// ran out of time (the abort flag is then set and the copies still in
// flight are waited for, bounded, before returning).
template <typename T>
__device__ bool cb_pass(const GridTeam& tm, const Cblk<T>& C, const T* x, T* acc, unsigned long long pol)
{
    constexpr int E = 16 / (int)sizeof(T);
    const int S = C.S, ncb = C.ncb, nw = C.nw, ms = C.ms, cw = C.cw, cols = C.cols;
    const int off_x = C.off_x, off_col = C.off_col, off_val = C.off_val, ar = C.acc_rows;
    const int* meta = C.meta;
    const unsigned short* gcol = C.col;
    const T* gval = C.val;
    unsigned char* const tm_dsm = tm.dsm;
    unsigned char* st0 = tm_dsm + C.stage_off;
    const unsigned acc_off = (unsigned)((unsigned char*)acc - tm_dsm);
    const int stage_bytes = C.stage_bytes;
    unsigned long long* mbar = tm.mbar;
    unsigned* ph = tm.ph;
    int* abort_flag = tm.abort_flag;
    const int g0 = blockIdx.x * ncb;
    const int k0 = blockIdx.x % ncb;  // first column block of this CTA
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int mis = (int)(((uintptr_t)x & 15) / sizeof(T));
    auto stage = [=](int s) { return st0 + (size_t)s * stage_bytes; };
    auto full = [=](int s) { return smem_addr(&mbar[s]); };
    auto empty = [=](int s) { return smem_addr(&mbar[CB_MAX_STAGES + s]); };
    auto blk = [=](int j) { return (k0 + j) % ncb; };  // column block of the j-th segment visited
    __syncthreads();  // stages free, acc zeroed, ph current
    bool ok = true;
    int issued = 0;
    if (w == nw) {
        // producer warp: lane 0 issues every copy
        if (lane == 0) {
            auto issue = [=](int j, int e0, int e1) {
                const int s = j % S, k = blk(j);
                unsigned char* d = stage(s);
                const int len = min(cw, cols - k * cw);
                const unsigned xb = (unsigned)((mis + len + E - 1) / E) * 16u;
                const unsigned ne = (unsigned)(e1 - e0);
                const unsigned mb = (unsigned)ms * 4u;
                mbar_expect_tx(full(s), mb + xb + ne * (2u + (unsigned)sizeof(T)));
                tma_load_1d_plain(smem_addr(d), meta + (size_t)(g0 + k) * ms, mb, full(s));
                tma_load_1d_plain(smem_addr(d + off_x), x + (size_t)k * cw - mis, xb, full(s));
                if (ne) {
                    tma_load_1d(smem_addr(d + off_col), gcol + e0, ne * 2u, full(s), pol);
                    tma_load_1d(smem_addr(d + off_val), gval + e0, ne * (unsigned)sizeof(T), full(s), pol);
                }
            };
            // x was written by generic stores (other CTAs, before the last
            // grid barrier) and is read here by the async proxy
            fence_proxy_async_all();
            const int npro = min(S, ncb);
            int e0a = 0, e1a = 0, e0b = 0, e1b = 0, e0c = 0, e1c = 0, e0d = 0, e1d = 0;
            e0a = ro(meta + (size_t)(g0 + blk(0)) * ms);
            e1a = ro(meta + (size_t)(g0 + blk(0)) * ms + 1);
            if (npro > 1) {
                e0b = ro(meta + (size_t)(g0 + blk(1)) * ms);
                e1b = ro(meta + (size_t)(g0 + blk(1)) * ms + 1);
            }
            if (npro > 2) {
                e0c = ro(meta + (size_t)(g0 + blk(2)) * ms);
                e1c = ro(meta + (size_t)(g0 + blk(2)) * ms + 1);
            }
            if (npro > 3) {
                e0d = ro(meta + (size_t)(g0 + blk(3)) * ms);
                e1d = ro(meta + (size_t)(g0 + blk(3)) * ms + 1);
            }
            issue(0, e0a, e1a);
            if (npro > 1) issue(1, e0b, e1b);
            if (npro > 2) issue(2, e0c, e1c);
            if (npro > 3) issue(3, e0d, e1d);
            issued = npro;
            for (int j = S; j < ncb; ++j) {
                const int s = j % S;
                if (!mbar_wait(empty(s), (ph[s] + j / S - 1) & 1u, abort_flag)) {
                    ok = false;
                    break;
                }
                // the stage's header names the segment visited S after its own
                const int* h = (const int*)stage(s);
                const int ne0 = h[2], ne1 = h[3];
                fence_proxy_async();  // the stage was read through the generic proxy
                issue(j, ne0, ne1);
                issued = j + 1;
            }
        }
    } else {
        for (int j = 0; j < ncb; ++j) {
            const int s = j % S;
            if (!mbar_wait(full(s), (ph[s] + j / S) & 1u, abort_flag)) {
                ok = false;
                break;
            }
            if (j >= 2) {  // every warp is done with segment j-2 (same partial-sum buffer)
                const int s2 = (j - 2) % S;
                if (!mbar_wait(empty(s2), (ph[s2] + (j - 2) / S) & 1u, abort_flag)) {
                    ok = false;
                    break;
                }
            }
            const unsigned so = (unsigned)(stage(s) - tm_dsm);
            cb_segment<T>(nw, so, so + off_x + mis * (unsigned)sizeof(T), so + off_col, so + off_val,
                          acc_off + (unsigned)((j & 1) * ar * (int)sizeof(T)));
            __syncwarp();
            if (lane == 0) mbar_arrive(empty(s));
        }
    }
    const bool all_ok = __syncthreads_and(ok);
    if (!all_ok && w == nw && lane == 0) {
        // copies of the last S issued segments may still be in flight
        for (int j = max(0, issued - S); j < issued; ++j) mbar_wait(full(j % S), (ph[j % S] + j / S) & 1u, nullptr);
    }
    __syncthreads();  // everyone has read ph for this pass
    if (threadIdx.x == 0 && all_ok)
        for (int s = 0; s < S; ++s) ph[s] += (unsigned)((ncb - s + S - 1) / S);
    return all_ok;
}

// The product: one pass per multiplied vector (NV = 2: x1 into acc1, then x2
// into acc2), then epi(row, sum) (or epi(row, sum1, sum2)) for every row of
// the CTA's range.
template <typename T, int NV, class Epi>
__device__ void cb_spmv(const GridTeam& tm, const Cblk<T>& C, const T* x1, const T* x2, Epi& epi)
{
    const int b = blockIdx.x;
    const int r0 = ro(C.rbnd + b), R = ro(C.rbnd + b + 1) - r0;
    const int ar = C.acc_rows;
    T* acc1 = (T*)tm.dsm;      // two buffers of ar
    T* acc2 = acc1 + 2 * ar;   // two more for the second vector
    const unsigned long long pol = evict_first_policy();
    __syncthreads();  // shared memory is free (earlier users done)
    for (int r = threadIdx.x; r < R; r += blockDim.x) {
        acc1[r] = 0;
        acc1[ar + r] = 0;
        if constexpr (NV == 2) {
            acc2[r] = 0;
            acc2[ar + r] = 0;
        }
    }
    if (!cb_pass<T>(tm, C, x1, acc1, pol)) return;
    if constexpr (NV == 2) {
        if (!cb_pass<T>(tm, C, x2, acc2, pol)) return;
    }
    for (int r = threadIdx.x; r < R; r += blockDim.x) {
        if constexpr (NV == 1)
            epi(r0 + r, acc1[r] + acc1[ar + r]);
        else
            epi(r0 + r, acc1[r] + acc1[ar + r], acc2[r] + acc2[ar + r]);
    }
}

// ---------------------------------------------------------------------------
// two-dimensional tiled product (grid team): y = M x (NV = 1) or M x1, M x2
// ---------------------------------------------------------------------------

// One chunk from its stage: compute warp w runs its slices against the
// resident vector slice xs; each row's sum (reduced over its V lanes) is
// final and is stored to the tile's row array at the start of dynamic shared
// memory (every row of a tile lies in exactly one slice, so the stores never
// meet).
template <typename T>
__device__ __forceinline__ void tile_chunk(int nw, int H, unsigned mt_off, unsigned xs_off, unsigned col_off,
                                           unsigned val_off)
{
    extern __shared__ __align__(128) unsigned char cb_sm[];
    const int* mt = (const int*)(cb_sm + mt_off);
    const T* xs = (const T*)(cb_sm + xs_off);
    const unsigned short* scol = (const unsigned short*)(cb_sm + col_off);
    const T* sval = (const T*)(cb_sm + val_off);
    T* acc = (T*)cb_sm;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int ns = mt[4];
    const int* wl = mt + 5;
    const int* st = wl + nw + 1;
    const unsigned short* sr = (const unsigned short*)(st + ns + 1);
    const int s_hi = wl[w + 1];
    for (int s = wl[w]; s < s_hi; ++s) {
        const int t1 = st[s + 1];
        int t = st[s];
        T a0 = 0, a1 = 0;
        if constexpr (sizeof(T) == 4) {
            // four steps per trip, the tail predicated (offset 0, value 0)
            T a2 = 0, a3 = 0;
            for (; t < t1; t += 4) {
                const bool o1 = t + 1 < t1, o2 = t + 2 < t1, o3 = t + 3 < t1;
                const int c0 = scol[t * 32 + lane];
                const int c1 = o1 ? (int)scol[t * 32 + 32 + lane] : 0;
                const int c2 = o2 ? (int)scol[t * 32 + 64 + lane] : 0;
                const int c3 = o3 ? (int)scol[t * 32 + 96 + lane] : 0;
                const T v0 = sval[t * 32 + lane];
                const T v1 = o1 ? sval[t * 32 + 32 + lane] : T(0);
                const T v2 = o2 ? sval[t * 32 + 64 + lane] : T(0);
                const T v3 = o3 ? sval[t * 32 + 96 + lane] : T(0);
                a0 = fmaT(v0, xs[c0], a0);
                a1 = fmaT(v1, xs[c1], a1);
                a2 = fmaT(v2, xs[c2], a2);
                a3 = fmaT(v3, xs[c3], a3);
            }
            a0 += a2;
            a1 += a3;
        } else {
            for (; t + 2 <= t1; t += 2) {
                const int c0 = scol[t * 32 + lane], c1 = scol[t * 32 + 32 + lane];
                const T v0 = sval[t * 32 + lane], v1 = sval[t * 32 + 32 + lane];
                a0 = fmaT(v0, xs[c0], a0);
                a1 = fmaT(v1, xs[c1], a1);
            }
            if (t < t1) a0 = fmaT(sval[t * 32 + lane], xs[scol[t * 32 + lane]], a0);
        }
        T a = a0 + a1;
        for (int o = H; o < 32; o <<= 1) a += __shfl_xor_sync(FULL_MASK, a, o);
        if (lane < H) {
            const int r = sr[s * H + lane];
            if (r != 0xFFFF) acc[r] = a;
        }
    }
}

// This CTA's tile of M x: the vector slice is copied once (completing on
// mbarrier 2 CB_MAX_STAGES, its uses counted in ph[CB_MAX_STAGES]), the
// chunks stream through the ring of S stages as the column-blocked segments
// do (full barriers tm.mbar[0..S-1], empty barriers tm.mbar[CB_MAX_STAGES +
// s]), the row sums collect in shared memory and go to part[k][rows of the
// block] at the end.  Returns false if a wait ran out of time (the abort
// flag is then set and the copies still in flight are waited for, bounded,
// before returning).
template <typename T>
__device__ bool tile_pass(const GridTeam& tm, const Cblk<T>& C, const T* x, T* part, unsigned long long pol)
{
    constexpr int E = 16 / (int)sizeof(T);
    const int S = C.S, ncb = C.ncb, nw = C.nw, H = 32 / C.V, ms = C.ms, cw = C.cw, cols = C.cols, rows = C.rows;
    const int off_col = C.off_col, off_val = C.off_val, stage_bytes = C.stage_bytes, off_x = C.off_x;
    const int* meta = C.meta;
    const unsigned short* gcol = C.col;
    const T* gval = C.val;
    unsigned char* const dsm = tm.dsm;
    unsigned char* st0 = dsm + C.stage_off;
    unsigned long long* mbar = tm.mbar;
    unsigned* ph = tm.ph;
    int* abort_flag = tm.abort_flag;
    const int g = blockIdx.x;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (g >= C.R * ncb) return true;  // no tile on this CTA (uniform in the CTA)
    const int r = g / ncb, k = g % ncb;
    const int r0 = ro(C.rbnd + r), Rr = ro(C.rbnd + r + 1) - r0;
    const int c0 = ro(C.cbeg + g), nch = ro(C.cbeg + g + 1) - c0;
    const int mis = (int)(((uintptr_t)x & 15) / sizeof(T));
    T* acc = (T*)dsm;
    auto stage = [=](int s) { return st0 + (size_t)s * stage_bytes; };
    auto full = [=](int s) { return smem_addr(&mbar[s]); };
    auto empty = [=](int s) { return smem_addr(&mbar[CB_MAX_STAGES + s]); };
    const unsigned xbar = smem_addr(&mbar[2 * CB_MAX_STAGES]);
    __syncthreads();  // shared memory free (earlier users done), ph current
    for (int i = threadIdx.x; i < Rr; i += blockDim.x) acc[i] = 0;
    __syncthreads();  // the row sums are zero before any warp stores one
    bool ok = true;
    int issued = 0;
    if (nch > 0) {
        if (w == nw) {
            // producer warp: lane 0 issues every copy
            if (lane == 0) {
                auto issue = [=](int j, int e0, int e1) {
                    const int s = j % S;
                    unsigned char* d = stage(s);
                    const unsigned ne = (unsigned)(e1 - e0);
                    const unsigned mb = (unsigned)ms * 4u;
                    mbar_expect_tx(full(s), mb + ne * (2u + (unsigned)sizeof(T)));
                    tma_load_1d_plain(smem_addr(d), meta + (size_t)(c0 + j) * ms, mb, full(s));
                    if (ne) {
                        tma_load_1d(smem_addr(d + off_col), gcol + e0, ne * 2u, full(s), pol);
                        tma_load_1d(smem_addr(d + off_val), gval + e0, ne * (unsigned)sizeof(T), full(s), pol);
                    }
                };
                // x was written by generic stores (other CTAs, before the last
                // grid barrier) and is read here by the async proxy
                fence_proxy_async_all();
                const int len = min(cw, cols - k * cw);
                const unsigned xb = (unsigned)((mis + len + E - 1) / E) * 16u;
                mbar_expect_tx(xbar, xb);
                tma_load_1d_plain(smem_addr(dsm + off_x), x + (size_t)k * cw - mis, xb, xbar);
                const int npro = min(S, nch);
                for (int j = 0; j < npro; ++j)
                    issue(j, ro(meta + (size_t)(c0 + j) * ms), ro(meta + (size_t)(c0 + j) * ms + 1));
                issued = npro;
                for (int j = S; j < nch; ++j) {
                    const int s = j % S;
                    if (!mbar_wait(empty(s), (ph[s] + j / S - 1) & 1u, abort_flag)) {
                        ok = false;
                        break;
                    }
                    // the stage's header names the chunk S after its own
                    const int* h = (const int*)stage(s);
                    const int ne0 = h[2], ne1 = h[3];
                    fence_proxy_async();  // the stage was read through the generic proxy
                    issue(j, ne0, ne1);
                    issued = j + 1;
                }
            }
        } else {
            if (!mbar_wait(xbar, ph[CB_MAX_STAGES] & 1u, abort_flag)) ok = false;
            for (int j = 0; ok && j < nch; ++j) {
                const int s = j % S;
                if (!mbar_wait(full(s), (ph[s] + j / S) & 1u, abort_flag)) {
                    ok = false;
                    break;
                }
                const unsigned so = (unsigned)(stage(s) - dsm);
                tile_chunk<T>(nw, H, so, (unsigned)off_x + mis * (unsigned)sizeof(T), so + off_col, so + off_val);
                __syncwarp();
                if (lane == 0) mbar_arrive(empty(s));
            }
        }
    }
    const bool all_ok = __syncthreads_and(ok);
    if (!all_ok && w == nw && lane == 0 && nch > 0) {
        // the slice copy and the copies of the last S issued chunks may still be in flight
        mbar_wait(xbar, ph[CB_MAX_STAGES] & 1u, nullptr);
        for (int j = max(0, issued - S); j < issued; ++j) mbar_wait(full(j % S), (ph[j % S] + j / S) & 1u, nullptr);
    }
    __syncthreads();  // everyone has read ph for this pass
    if (threadIdx.x == 0 && nch > 0) {
        for (int s = 0; s < S; ++s) ph[s] += (unsigned)((nch - s + S - 1) / S);
        ph[CB_MAX_STAGES] += 1u;
    }
    if (!all_ok) return false;
    T* out = part + (size_t)k * rows + r0;
    for (int i = threadIdx.x; i < Rr; i += blockDim.x) out[i] = acc[i];
    return true;
}

// The tiled product: one tile pass per vector into its partial sums, a grid
// barrier, then epi(row, sum) (or epi(row, sum1, sum2)) for every row, the
// sum over the column blocks taken in block order (deterministic), rows dealt
// like the team's vector loops.  The partial sums alternate between two
// buffers by the parity of the barrier count at entry: the next product of
// this matrix either starts one barrier later (the other buffer) or after a
// barrier that every CTA reaches only once it has read this one.
template <typename T, int NV, class Epi>
__device__ void tile_spmv(GridTeam& tm, const Cblk<T>& C, const T* x1, const T* x2, Epi& epi)
{
    const unsigned long long pol = evict_first_policy();
    const int rows = C.rows, ncb = C.ncb;
    T* part = C.part + (size_t)(tm.epoch & 1ull) * C.nv * ncb * rows;
    if (!tile_pass<T>(tm, C, x1, part, pol)) return;
    if constexpr (NV == 2) {
        if (!tile_pass<T>(tm, C, x2, part + (size_t)ncb * rows, pol)) return;
    }
    tm.sync();
    for (int i = tm.rank(); i < rows; i += tm.size()) {
        T s1 = 0;
        for (int k = 0; k < ncb; ++k) s1 += part[(size_t)k * rows + i];
        if constexpr (NV == 1) {
            epi(i, s1);
        } else {
            T s2 = 0;
            for (int k = 0; k < ncb; ++k) s2 += part[(size_t)(ncb + k) * rows + i];
            epi(i, s1, s2);
        }
    }
}

template <typename T, class Team, class XF, class Epi>
__device__ __forceinline__ void spmv_f(const Team& tm, const Sell<T>& S, XF xf, Epi epi)
{
    if (S.wbnd != nullptr && tm.stage != nullptr)
        sell_tma(tm, S, xf, epi);
    else
        sell_v(tm, S, xf, epi);
}

template <typename T, class Team, class Epi>
__device__ __forceinline__ void spmv(Team& tm, const Sell<T>& S, const T* x, Epi epi)
{
    if constexpr (Team::kGrid) {
        if (S.cb.ncb > 0) {
            if (S.cb.tile)
                tile_spmv<T, 1>(tm, S.cb, x, x, epi);
            else
                cb_spmv<T, 1>(tm, S.cb, x, x, epi);
            return;
        }
    }
    auto f = [x](int c) { return x[c]; };
    spmv_f(tm, S, f, epi);
}

template <typename T, class Team, class Epi>
__device__ __forceinline__ void spmv2(Team& tm, const Sell<T>& S, const T* x1, const T* x2, Epi epi)
{
    if constexpr (Team::kGrid) {
        if (S.cb.ncb > 0) {
            if (S.cb.tile)
                tile_spmv<T, 2>(tm, S.cb, x1, x2, epi);
            else
                cb_spmv<T, 2>(tm, S.cb, x1, x2, epi);
            return;
        }
    }
    auto f1 = [x1](int c) { return x1[c]; };
    auto f2 = [x2](int c) { return x2[c]; };
    sell2_v(tm, S, f1, f2, epi);
}

// ---------------------------------------------------------------------------
// CG on (I + A^T A) x = rhs from the residual r = rhs - (I + A^T A) x of the
// start x, rr = ||r||^2 (already reduced), stopping at ||r|| <= tol or after
// cg_max iterations.  One reduction per iteration: <p,q>, <r,q>, <q,q> are
// reduced together, ||r - alpha q||^2 = rr - 2 alpha <r,q> + alpha^2 <q,q>
// gives beta, and x, r, p are updated in one pass; the exact ||r||^2 of the
// updated r rides along with the next reduction and replaces the recurrence
// value before it is used for alpha.  Returns the iterations.
// ---------------------------------------------------------------------------
template <typename T>
struct CgBufs {
    T *r, *p, *q;  // n
    T* tm;         // m
};

template <typename T, class Team>
__device__ int cg_loop(Team& tm, const Sell<T>& A, const Sell<T>& AT, int n, CgBufs<T> b, T* x, double rr,
                       double tol, int cg_max)
{
    T* p = b.p;
    T* q = b.q;
    T* r = b.r;
    T* tmv = b.tm;
    for (int j = tm.rank(); j < n; j += tm.size()) p[j] = r[j];
    tm.sync();
    int it = 0;
    T rr_part = 0;
    bool have_part = false;
    while (it < cg_max) {
        if (tm.aborted()) break;
        spmv(tm, A, p, [&](int i, T s) { tmv[i] = s; });
        tm.sync();
        T pq = 0, rq = 0, qq = 0;
        spmv(tm, AT, tmv, [&](int j, T s) {
            const T qj = p[j] + s;
            q[j] = qj;
            pq += p[j] * qj;
            rq += r[j] * qj;
            qq += qj * qj;
        });
        double red[4] = {(double)pq, (double)rq, (double)qq, (double)rr_part};
        tm.reduce(red);
        ++it;
        // The scalar step (two FP64 divisions, a square root) is evaluated by
        // one thread per CTA and handed to the others through shared memory:
        // the FP64 pipe is a small fraction of the FP32 one, and every thread
        // of every warp evaluating it costs more than the extra CTA barrier.
        // The values are the same bits either way (rr lives in thread 0).
        double* bc = tm.bcast();
        if (threadIdx.x == 0) {
            if (have_part) rr = red[3];
            const double alpha = rr / red[0];
            double rr_new = rr - 2.0 * alpha * red[1] + alpha * alpha * red[2];
            if (rr_new < 0.0) rr_new = 0.0;
            reinterpret_cast<T*>(bc)[0] = (T)alpha;
            reinterpret_cast<T*>(bc)[1] = (T)(rr_new / rr);
            reinterpret_cast<int*>(bc + 2)[0] = (!(sqrt(rr_new) > tol) || it >= cg_max) ? 1 : 0;
            rr = rr_new;
        }
        __syncthreads();
        const T ta = reinterpret_cast<const T*>(bc)[0];
        const T tb = reinterpret_cast<const T*>(bc)[1];
        const bool done = reinterpret_cast<const int*>(bc + 2)[0] != 0;
        rr_part = 0;
        if (done) {
            for (int j = tm.rank(); j < n; j += tm.size()) x[j] += ta * p[j];
        } else {
            for (int j = tm.rank(); j < n; j += tm.size()) {
                const T pj = p[j];
                x[j] += ta * pj;
                const T rj = r[j] - ta * q[j];
                r[j] = rj;
                p[j] = rj + tb * pj;
                rr_part += rj * rj;
            }
        }
        have_part = true;
        tm.sync();
        if (done) break;
    }
    return it;
}

// ---------------------------------------------------------------------------
// Direct solves of (I + A^T A) x = b (the "direct" alternative Sec. 4.1 names
// beside CG), for one CTA per instance: the matrix is formed column by column
// as e_j + A^T (A e_j) with the solver's own sparse products, factored L L^T,
// and the factor inverted in place, once, at setup; a solve is then
// x = L^{-T} (L^{-1} b), two triangular products.
//
// Why L^{-1} and not L: both take n^2 multiply-adds and n^2 words a solve, but
// triangular solves are a chain of n divisions and 4 n / 32 CTA barriers, and
// on this GPU an FP64 instruction occupies the SM's FP64 pipe for 16 cycles
// whether one lane needs it or all 32 do.  Why not the inverse of the whole
// matrix (one product): its residual grows with cond(I + A^T A), by orders of
// magnitude where b lies in the range of A^T, as the solver's right-hand sides
// do; with L^{-1} it grows with cond(L), the square root (300 columns, FP64,
// residual over |b| at cond 5e3: triangular solves 9e-15, L^{-1} 1.7e-14, full
// inverse 1.3e-13; at 5e5: 8e-14, 1.6e-13, 8.5e-12), and the error of x and of
// A x is that of the triangular solves.
// ---------------------------------------------------------------------------
constexpr int DIR_B = 32;  // tile of the factorisation: DIR_B^2 values fit each of the two shared arrays

// The lower triangle of the n x n row-major matrix L, positive definite, is
// replaced by the inverse of its Cholesky factor, n^3 / 3 multiply-adds in
// 32 x 32 tiles: right-looking factorisation whose diagonal blocks are inverted
// at once (W_kk; panels are A_ik W_kk^T), then the inverse by block rows,
// W_ij = -W_ii sum_k L_ik W_kj.  S1 and S2 are DIR_B^2 values of shared memory
// each.  Returns (in warp 0) false if a pivot was not positive.
template <typename T, class Team>
__device__ bool direct_factor(Team& tm, T* L, int n, T* S1, T* S2)
{
    const int tid = tm.rank(), nt = tm.size(), lane = threadIdx.x & 31;
    const int nb = (n + DIR_B - 1) / DIR_B;
    bool good = true;
    // tiles in shared memory hold element (r, c) at r DIR_B + (c xor r): rows and columns hit distinct banks
    auto sw = [](int r, int c) { return r * DIR_B + (c ^ r); };
    auto at = [&](int gi, int gj) -> T { return gi < n && gj <= gi ? L[(size_t)gi * n + gj] : T(0); };
    auto stage = [&](T* S, int i, int k, bool transposed) {  // tile (i, k) of the lower triangle, zeros elsewhere
        for (int e = tid; e < DIR_B * DIR_B; e += nt) {
            const int r = e / DIR_B, c = e % DIR_B;
            S[transposed ? sw(c, r) : sw(r, c)] = at(i * DIR_B + r, k * DIR_B + c);
        }
    };
    // tile (i, j) <- keep * tile (i, j) + sign * S1 S2, four rows r, r + 8, ... of one column a thread
    auto product = [&](int i, int j, bool keep, T sign) {
        for (int e = tid; e < DIR_B * DIR_B / 4; e += nt) {
            const int r = e / DIR_B, c = e % DIR_B;
            T acc[4] = {0, 0, 0, 0};
            for (int q = 0; q < DIR_B; ++q) {
                const T v = S2[sw(q, c)];
#pragma unroll
                for (int h = 0; h < 4; ++h) acc[h] = fmaT(S1[sw(r + 8 * h, q)], v, acc[h]);
            }
            const int gj = j * DIR_B + c;
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const int gi = i * DIR_B + r + 8 * h;
                if (gi < n && gj <= gi) {
                    T& x = L[(size_t)gi * n + gj];
                    x = fmaT(sign, acc[h], keep ? x : T(0));
                }
            }
        }
    };
    for (int k = 0; k < nb; ++k) {
        const int w = min(DIR_B, n - k * DIR_B);
        stage(S1, k, k, false);
        tm.sync();
        if (tid < 32) {
            // the diagonal block's factor, a row a lane, in S1 ...
            for (int p = 0; p < w; ++p) {
                const T d = S1[sw(p, p)];
                if (!(d > T(0))) good = false;
                const T rs = d > T(0) ? sqrt(d) : T(1);
                __syncwarp();
                T l = 0;
                if (lane >= p && lane < w) S1[sw(lane, p)] = l = lane == p ? rs : S1[sw(lane, p)] / rs;
                __syncwarp();
                for (int c = p + 1; c < w; ++c) {
                    const T lc = S1[sw(c, p)];
                    if (lane >= c && lane < w) S1[sw(lane, c)] -= l * lc;
                }
                __syncwarp();
            }
            // ... and its inverse, a column a lane, transposed in S2 (zero outside w x w)
            for (int r = 0; r < DIR_B; ++r) {
                T a0 = r == lane && r < w ? T(1) : T(0), a1 = 0;
                if (r < w) {
                    for (int q = 0; q + 1 < r; q += 2) {
                        a0 -= S1[sw(r, q)] * S2[sw(lane, q)];
                        a1 -= S1[sw(r, q + 1)] * S2[sw(lane, q + 1)];
                    }
                    if (r & 1) a0 -= S1[sw(r, r - 1)] * S2[sw(lane, r - 1)];
                    a0 = (a0 + a1) / S1[sw(r, r)];
                }
                S2[sw(lane, r)] = a0;
            }
        }
        tm.sync();
        for (int e = tid; e < DIR_B * DIR_B; e += nt) {  // W_kk in place of A_kk
            const int r = e / DIR_B, c = e % DIR_B;
            if (r < w && c <= r) L[(size_t)(k * DIR_B + r) * n + k * DIR_B + c] = S2[sw(c, r)];
        }
        for (int i = k + 1; i < nb; ++i) {  // L_ik = A_ik W_kk^T
            tm.sync();
            stage(S1, i, k, false);
            tm.sync();
            product(i, k, false, T(1));
        }
        for (int i = k + 1; i < nb; ++i)  // A_ij -= L_ik L_jk^T
            for (int j = k + 1; j <= i; ++j) {
                tm.sync();
                if (j == k + 1) stage(S1, i, k, false);
                stage(S2, j, k, true);
                tm.sync();
                product(i, j, true, T(-1));
            }
        tm.sync();
    }
    for (int i = 1; i < nb; ++i) {
        // tile (i, j) <- sum over k = j .. i - 1 of L_ik W_kj: once L_ik is in S1 its tile starts as the first term
        for (int k = 0; k < i; ++k)
            for (int j = k; j >= 0; --j) {
                tm.sync();
                if (j == k) stage(S1, i, k, false);
                stage(S2, k, j, false);
                tm.sync();
                product(i, j, j < k, T(1));
            }
        for (int j = 0; j < i; ++j) {  // W_ij = -W_ii times it
            tm.sync();
            if (j == 0) stage(S1, i, i, false);
            stage(S2, i, j, false);
            tm.sync();
            product(i, j, false, T(-1));
        }
        tm.sync();
    }
    return good;
}

template <typename T, class Team>
__device__ void direct_setup(Team& tm, const DevProb<T>& P, const DevWork<T>& W, double* s1, double* s2)
{
    const int n = P.n;
    T* L = W.dinv;
    T* ej = W.cp;
    T* y = W.tm;
    for (int j = 0; j < n; ++j) {
        for (int i = tm.rank(); i < n; i += tm.size()) ej[i] = i == j ? T(1) : T(0);
        tm.sync();
        spmv(tm, P.A, ej, [&](int i, T v) { y[i] = v; });
        tm.sync();
        spmv(tm, P.AT, y, [&](int i, T v) {
            if (i >= j) L[(size_t)i * n + j] = v + (i == j ? T(1) : T(0));
        });
        tm.sync();
    }
    const bool good = direct_factor<T>(tm, L, n, reinterpret_cast<T*>(s1), reinterpret_cast<T*>(s2));
    // L^{-1} in the lower triangle, its transpose in the upper one: both products of a solve read rows
    for (int i = tm.rank() >> 5; i < n; i += tm.size() >> 5)
        for (int j = threadIdx.x & 31; j < i; j += 32) L[(size_t)j * n + i] = L[(size_t)i * n + j];
    if (threadIdx.x == 0 && !good) atomicExch(W.dinv_fail, 1);
    tm.sync();
}

// out = (or +=) the product of L^{-1} (lower: column j of the upper triangle
// down to row j) or of its transpose (column j of the lower triangle from row
// j on) with v.  A column belongs to a lane: a warp reads 32 consecutive words
// of each row.  Group q of 32 columns (counted from the short end) has 4 (q + 1)
// units of 8 rows; all units, group after group, are dealt to the warps in
// equal runs, and the sums of a group's runs are added through shared memory
// (part, DIR_PART values: run w of group q at slot w + q).  Where the slots do
// not suffice, warps take whole groups, longest first and to and fro.
constexpr int DIR_PART = 1024;

template <typename T, class Team>
__device__ __forceinline__ void direct_product(Team& tm, const T* D, int n, const T* v, bool lower, T* out, bool add, T* part)
{
    const int lane = threadIdx.x & 31, warp = tm.rank() >> 5, nw = tm.size() >> 5, ng = (n + 31) >> 5;
    // the sum of column 32 c + lane over units [u0, u1) of its group q
    auto column = [&](int q, int u0, int u1) -> T {
        const int c = lower ? q : ng - 1 - q, j = 32 * c + lane;
        if (j >= n) return T(0);
        int i = lower ? 8 * u0 : 32 * ng - 8 * u1;
        const int e = min(n, lower ? 8 * u1 : 32 * ng - 8 * u0);
        const T* d = D + j;
        T a[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        auto across = [&](int hi) {  // rows of the diagonal block
            for (; i < hi; i += 4)
#pragma unroll
                for (int h = 0; h < 4; ++h)
                    if (i + h < hi && (lower ? i + h <= j : i + h >= j)) a[h] = fmaT(d[(size_t)(i + h) * n], v[i + h], a[h]);
        };
        auto whole = [&](int hi) {
            for (; i + 8 <= hi; i += 8)
#pragma unroll
                for (int h = 0; h < 8; ++h) a[h] = fmaT(d[(size_t)(i + h) * n], v[i + h], a[h]);
            for (; i < hi; ++i) a[0] = fmaT(d[(size_t)i * n], v[i], a[0]);
        };
        if (lower) {
            whole(min(e, 32 * c));
            across(e);
        } else {
            across(min(e, 32 * c + 32));
            whole(e);
        }
        return ((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7]));
    };
    const int room = DIR_PART / 32 + 1 - ng;  // warps whose slots fit
    if (room >= min(nw, 8)) {
        const int units = 2 * ng * (ng + 1), nwe = min(nw, room), per = (units + nwe - 1) / nwe;
        if (warp < nwe) {
            int u = warp * per, q = 0;
            const int u1 = min(units, u + per);
            while (2 * (q + 1) * (q + 2) <= u) ++q;
            for (; u < u1; ++q) {
                const int g0 = 2 * q * (q + 1), e = min(u1, g0 + 4 * (q + 1));
                part[(warp + q) * 32 + lane] = column(q, u - g0, e - g0);
                u = e;
            }
        }
        tm.sync();
        for (int k = tm.rank(); k < n; k += tm.size()) {
            const int q = lower ? k >> 5 : ng - 1 - (k >> 5);
            const int w1 = (2 * (q + 1) * (q + 2) - 1) / per;
            T s = 0;
            for (int w = 2 * q * (q + 1) / per; w <= w1; ++w) s += part[(w + q) * 32 + (k & 31)];
            out[k] = add ? out[k] + s : s;
        }
    } else {
        for (int t = 0; t * nw < ng; ++t) {
            const int q = ng - 1 - (t * nw + (t & 1 ? nw - 1 - warp : warp));
            if (q < 0) continue;
            const int j = 32 * (lower ? q : ng - 1 - q) + lane;
            const T s = column(q, 0, 4 * (q + 1));
            if (j < n) out[j] = add ? out[j] + s : s;
        }
    }
    tm.sync();
}

// x += (I + A^T A)^{-1} r; y: n words.  Bound by the FP64 pipe (n^2 / 2 cycles an SM, and 16 n for the diagonal
// blocks, of which each product uses half) or by reading the matrix from L2.  1024 portfolio instances of 20 to 400
// columns, 20 iterations in FP64: 24.3 ms with triangular solves, 17.4 ms with the whole inverse, 17.8 ms so (19.5 with
// whole columns to a warp); one instance of 560 columns, 16 iterations: 23.9, 14.2 and 14.5 ms (15.3).  Setup of that
// instance 81, 43 and 33 ms.
template <typename T, class Team>
__device__ void direct_solve(Team& tm, const T* D, int n, const T* r, T* x, T* y, T* part)
{
    direct_product<T>(tm, D, n, r, true, y, false, part);
    direct_product<T>(tm, D, n, y, false, x, true, part);
}

// ---------------------------------------------------------------------------
// M^{-1}(a, e) for M = [I A^T; -A I]: x = (I + A^T A)^{-1}(a - A^T e) by CG
// warm-started from x (in place), y = e + A x written to W.py.  Returns the CG
// iterations; htp = <c, x> + <b, y>.  CG stops when ||res|| <= rtol ||rhs||.
// (Block elimination of the linear-system step of Eq. drs; Sec. 4.1 names CG.)
// ---------------------------------------------------------------------------
template <typename T, class Team>
__device__ __forceinline__ bool direct_available(const Team&, const DevWork<T>& W)
{
    if constexpr (Team::kGrid) return false;
    else return W.dinv != nullptr;
}

template <typename T, class Team>
__device__ int minv(Team& tm, const DevProb<T>& P, const DevWork<T>& W, const T* a, const T* e, T* x, double rtol,
                    int cg_max, double& htp, double atol = 0.0)
{
    const int n = P.n;
    T* tmv = W.tm;
    T* r = W.cr;
    spmv(tm, P.A, x, [&](int i, T s) { tmv[i] = s; });
    tm.sync();
    T acc_b = 0, acc_r = 0;
    spmv2(tm, P.AT, e, tmv, [&](int j, T s1, T s2) {
        const T rhs = a[j] - s1;
        const T res = rhs - x[j] - s2;
        r[j] = res;
        acc_b += rhs * rhs;
        acc_r += res * res;
    });
    double red2[2] = {(double)acc_b, (double)acc_r};
    tm.reduce(red2);
    const double rhs2 = red2[0];
    const double rr = red2[1];
    const double tol = fmax(rtol * sqrt(rhs2), atol);
    int it = 0;
    if (rhs2 == 0.0) {
        for (int j = tm.rank(); j < n; j += tm.size()) x[j] = 0;
        tm.sync();
    } else if (direct_available(tm, W)) {
        // direct: the residual of the warm start solved exactly; the shared scratch is the AA
        // direction's Cholesky array, idle during a linear solve
        if constexpr (!Team::kGrid) direct_solve<T>(tm, W.dinv, n, r, x, W.cp, reinterpret_cast<T*>(tm.scratch));
    } else if (sqrt(rr) > tol) {
        const unsigned long long tc0 = tm.leader() ? gtimer() : 0ull;
        it = cg_loop<T>(tm, P.A, P.AT, n, CgBufs<T>{r, W.cp, W.cq, tmv}, x, rr, tol, cg_max);
        if (tm.leader()) W.st->part_ns[3] += (double)(gtimer() - tc0);
    }
    T hb = 0, hc = 0;
    T* py = W.py;
    spmv(tm, P.A, x, [&](int i, T s) {
        const T yi = e[i] + s;
        py[i] = yi;
        hb += ro(P.b + i) * yi;
    });
    for (int j = tm.rank(); j < n; j += tm.size()) hc += ro(P.c + j) * x[j];
    double red4[2] = {(double)hb, (double)hc};
    tm.reduce(red4);
    htp = red4[0] + red4[1];
    if (tm.leader()) W.st->mat_passes += 3 + 2 * it;
    return it;
}

// The same M^{-1}(a, e) in FP64 by iterative refinement (SCS_MIXED, FP64
// phase): the residual r = rhs - (I + A^T A) x is formed in FP64 with the FP64
// matrix, the correction solves (I + A^T A) dx = r / ||r|| in FP32 with the
// FP32 copy of A by the same CG from dx = 0, and x += ||r|| dx in FP64; then
// the FP64 residual is formed again, until ||r|| <= tol.  Where the requested
// accuracy relative to ||r|| is looser than IR_VERIFY (the solves inside the
// loop under cg_adapt) one correction is taken without the checking residual:
// its FP32 rounding (about 1e-7 of ||r|| times the growth of the products) is
// far below what was asked.  Each correction is asked for at most IR_FLOOR
// relative accuracy, about what FP32 CG reaches reliably.  Returns the FP32
// CG iterations.
constexpr double IR_VERIFY = 1e-3;
constexpr double IR_FLOOR = 1e-5;
constexpr int IR_MAX_SWEEPS = 6;

template <class Team>
__device__ int minv_ir(Team& tm, const DevProb<double>& P, const DevWork<double>& W, const double* a,
                       const double* e, double* x, double rtol, int cg_max, double& htp, double atol)
{
    const int n = P.n;
    double* tmv = W.tm;
    double* r = W.cr;
    double* rhs = W.tn;
    const IrBufs& ir = W.ir;
    spmv(tm, P.A, x, [&](int i, double s) { tmv[i] = s; });
    tm.sync();
    double acc_b = 0, acc_r = 0;
    spmv2(tm, P.AT, e, tmv, [&](int j, double s1, double s2) {
        const double rh = a[j] - s1;
        const double res = rh - x[j] - s2;
        rhs[j] = rh;
        r[j] = res;
        acc_b += rh * rh;
        acc_r += res * res;
    });
    double red2[2] = {acc_b, acc_r};
    tm.reduce(red2);
    const double rhs2 = red2[0];
    double rr = red2[1];
    const double tol = fmax(rtol * sqrt(rhs2), atol);
    long long passes64 = 3, passes32 = 0, sweeps = 0;
    int it = 0;
    if (rhs2 == 0.0) {
        for (int j = tm.rank(); j < n; j += tm.size()) x[j] = 0;
        tm.sync();
    } else {
        for (int sw = 0; sw < IR_MAX_SWEEPS && sqrt(rr) > tol && it < cg_max && !tm.aborted(); ++sw) {
            const double nr = sqrt(rr);
            const double want = tol / nr;  // relative accuracy asked of this correction
            // the scaled residual in FP32, the correction from zero
            float acc32 = 0.f;
            const double inv = 1.0 / nr;
            for (int j = tm.rank(); j < n; j += tm.size()) {
                const float rj = (float)(r[j] * inv);
                ir.r[j] = rj;
                ir.x[j] = 0.f;
                acc32 += rj * rj;
            }
            double red3[1] = {(double)acc32};
            tm.reduce(red3);
            const unsigned long long tc0 = tm.leader() ? gtimer() : 0ull;
            const int k = cg_loop<float>(tm, ir.A, ir.AT, n, CgBufs<float>{ir.r, ir.p, ir.q, ir.tm}, ir.x, red3[0],
                                         fmax(want, IR_FLOOR) * sqrt(red3[0]), cg_max - it);
            if (tm.leader()) W.st->part_ns[3] += (double)(gtimer() - tc0);
            it += k;
            passes32 += 2 * k;
            ++sweeps;
            if (want >= IR_VERIFY) {
                for (int j = tm.rank(); j < n; j += tm.size()) x[j] += nr * (double)ir.x[j];
                tm.sync();
                break;
            }
            for (int j = tm.rank(); j < n; j += tm.size()) x[j] += nr * (double)ir.x[j];
            tm.sync();
            // FP64 residual of the corrected x
            spmv(tm, P.A, x, [&](int i, double s) { tmv[i] = s; });
            tm.sync();
            double acc = 0;
            spmv(tm, P.AT, tmv, [&](int j, double s) {
                const double res = rhs[j] - x[j] - s;
                r[j] = res;
                acc += res * res;
            });
            double red4[1] = {acc};
            tm.reduce(red4);
            rr = red4[0];
            passes64 += 2;
        }
    }
    double hb = 0, hc = 0;
    double* py = W.py;
    spmv(tm, P.A, x, [&](int i, double s) {
        const double yi = e[i] + s;
        py[i] = yi;
        hb += ro(P.b + i) * yi;
    });
    for (int j = tm.rank(); j < n; j += tm.size()) hc += ro(P.c + j) * x[j];
    double red5[2] = {hb, hc};
    tm.reduce(red5);
    htp = red5[0] + red5[1];
    if (tm.leader()) {
        W.st->mat_passes += passes64 + 1;
        W.st->mat_passes_ir += passes32;
        W.st->cg_iters_ir += it;
        W.st->ir_sweeps += sweeps;
    }
    return it;
}

// out = (I+Q)^{-1} r via tau = (r_tau + h^T M^{-1} r) / (1 + h^T g), (x,y) = M^{-1} r - tau g.
// r and out must not share storage of the bulk part.
template <typename T, class Team>
__device__ int linsys(Team& tm, const DevProb<T>& P, const DevWork<T>& W, HV<T> r, HV<T> out, int slot,
                      double rtol, int cg_max, double hg, double atol = 0.0, bool refine = false)
{
    const int n = P.n, m = P.m;
    const double rtau = *r.t;
    T* x = W.ws[slot];
    double htp;
    int it;
    const unsigned long long tl0 = tm.leader() ? gtimer() : 0ull;
    if constexpr (sizeof(T) == sizeof(double)) {
        it = refine ? minv_ir(tm, P, W, r.v, r.v + n, x, rtol, cg_max, htp, atol)
                    : minv(tm, P, W, r.v, r.v + n, x, rtol, cg_max, htp, atol);
    } else {
        it = minv(tm, P, W, r.v, r.v + n, x, rtol, cg_max, htp, atol);
    }
    const double tau = (rtau + htp) / (1.0 + hg);
    const T tt = (T)tau;
    for (int i = tm.rank(); i < n; i += tm.size()) out.v[i] = x[i] - tt * W.g[i];
    for (int i = tm.rank(); i < m; i += tm.size()) out.v[n + i] = W.py[i] - tt * W.g[n + i];
    if (tm.leader()) *out.t = tau;
    tm.sync();
    if (tm.leader()) W.st->part_ns[2] += (double)(gtimer() - tl0);
    return it;
}

// ---------------------------------------------------------------------------
// Projection on C = R^n x K* x R_+ fused with the DRS residual (Eq. drs):
// for each element the op supplies (w, w~), the pass forms v = 2 w~ - w,
// projects it (identity on chi and zero-cone rows, max(0,.) on the orthant,
// closed form per SOC with one warp per cone, eigen-decomposition per PSD
// block with one CTA per block) and hands (w, w~, w_) back to the op.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int svec_index(int d, int i, int j)  // i >= j
{
    return j * d - j * (j - 1) / 2 + (i - j);
}

// The warps of a CTA that share one PSD block: consecutive threads with a named barrier of their own.
struct PsdTeam {
    int tid, nt, bar;
    __device__ __forceinline__ void sync() const { asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(nt) : "memory"); }
};

// the sum of x over the team, in every thread; red: 33 doubles of shared memory.  The warps' sums are
// added by one warp: every thread adding them itself kept the FP64 pipe busy for 4000 cycles.
__device__ __forceinline__ double block_sum(double x, double* red, const PsdTeam& g)
{
    const int lane = g.tid & 31, wid = g.tid >> 5, nw = g.nt >> 5;
    x = warp_sum(x);
    g.sync();
    if (lane == 0) red[wid] = x;
    g.sync();
    if (wid == 0) {
        const double s = warp_sum(lane < nw ? red[lane] : 0.0);
        if (lane == 0) red[32] = s;
    }
    g.sync();
    return red[32];
}

// Parallel two-sided Jacobi (round-robin pairing, dp/2 disjoint rotations per
// round) on a symmetric dp x dp matrix.
//
// Round r pairs index r + k with r - k (mod dp - 1; pair 0: r with dp - 1).
// The matrix is stored by pairs, not by indices: "slot" 2k / 2k+1 is the first
// / second member of pair k, and a "cell" (k, l), k > l, holds the four values
// of pair k's rows and pair l's columns, updated from both sides by one thread.
// The pairs of round r+1 are those of round r with every member moved one slot
// on (next_slot), the same move in every round, so a thread reads its cell
// from one buffer and writes the four values to their places of the next round
// in the other, at addresses that never change; consecutive threads touch
// consecutive words.  The cells (k+1, k-1) hold the next round's pair k: their
// threads also compute its rotation, straight from the register.  So a round
// takes one CTA barrier and no index arithmetic.  (Three passes over an indexed
// matrix with a barrier each: 4400 cycles a round for order 64 in FP32, 12000 in
// FP64; one pass over the indexed lower triangle: 2400 and 10800; the cells: 1160
// and 6540.  512 blocks of order 64 in FP32, one projection: 10.0, 6.5 and 4.6 ms;
// one block of order 120 in FP64, four iterations: 129, 76 and 42 ms, 45 with the
// sweeps out of line.)
//
// FP64: the FP64 pipe (2 multiply-adds a cycle and SM) is the bound, so the
// rotations are applied in scaled form (fast Givens): X = D X^ D and V = V^ D
// with D diagonal, x^_p -= al x^_q, x^_q += be x^_p -- one multiply-add per
// element instead of a product and a multiply-add -- and D is multiplied in
// after each sweep (its entries shrink by at most sqrt(2) a round).  The angle
// is found in FP32 -- any t with c = 1/sqrt(1 + t^2), s = t c is a rotation,
// and c, the scales and the diagonal are FP64 for the t that was taken; an
// angle 1e-7 off leaves 1e-7 of the element for the next sweep.  Once the
// off-diagonal part is below 3e-6 of the whole, a Newton step in FP64 makes
// the angle exact to 1e-14: what the last sweep leaves is the projection's
// error, and with FP32 angles it stopped just under the test (mean error over
// |X| of random blocks, by a simulation on the CPU, FP64 angles / FP32 angles /
// so: order 2 1.1e-16, 2.7e-15, 1.5e-16; order 5 2.8e-15, 5.5e-15, 1.1e-15;
// order 17 4.2e-15, 5.2e-15, 3.2e-15; order 32 6.6e-15, 3.8e-15, 3.6e-15),
// often after one sweep more.  The line lies where a sweep's quadratic remainder
// begins to fall below 1e-7 of what it started from; at 1e-4 two sweeps of a warm
// start took the step instead of one (a tenth of a rotation's chain each).
//
// V (columns contiguous, stride ldv) receives the eigenvectors; its update is
// left to the warps that compute no rotations, a round's longest chain.
template <typename T>
struct Jacobi {
    T* cell[2];   // two buffers of 4 x ncell values: component c of cell i at c * ncell + i
    T* V;
    T* rot;       // [2][dp/2][2]: rotations of a round, (c, s), or (al, be) in FP64
    T* dg;        // [2][dp]: the diagonal by slots
    T *sc, *isc;  // FP64: [2][dp], the scales D and 1 / D by slots
    T *e, *def;   // dp/2 each: the pairs' own off-diagonal values at a sweep's start; after their rotation
    int dp, half, ncell, ldv;
    static constexpr int scratch_words(int dp) { return 9 * dp; }
    __host__ __device__ static constexpr int cells(int dp) { return (dp / 2) * (dp / 2 - 1) / 2; }
    __device__ Jacobi(T* c0, T* c1, T* v, T* scratch, int dp_, int ldv_)
        : V(v), rot(scratch), dg(scratch + 2 * dp_), sc(scratch + 4 * dp_), isc(scratch + 6 * dp_), e(scratch + 8 * dp_),
          def(e + dp_ / 2), dp(dp_), half(dp_ / 2), ncell(cells(dp_)), ldv(ldv_)
    {
        cell[0] = c0;
        cell[1] = c1;
    }
    __device__ __forceinline__ int slot_of(int i) const  // of index i at a sweep's start
    {
        return i == dp - 1 ? 1 : (i < half ? 2 * i : 2 * (dp - 1 - i) + 1);
    }
    // offset of the value at slots (a, b) of two different pairs
    __device__ __forceinline__ int at(int a, int b) const
    {
        const int k = a >> 1, l = b >> 1;
        return k > l ? ((a & 1) * 2 + (b & 1)) * ncell + k * (k - 1) / 2 + l
                     : ((b & 1) * 2 + (a & 1)) * ncell + l * (l - 1) / 2 + k;
    }
    // the slot of the next round
    __device__ __forceinline__ int next_slot(int a) const
    {
        const int k = a >> 1;
        if (a & 1) return k == 0 ? 1 : (k == half - 1 ? a - 1 : a + 2);
        return k == 0 ? 3 : a - 2;
    }
    // entry (i, j) of the matrix at the start (any i, j of the lower triangle, once each)
    __device__ __forceinline__ void put(int i, int j, T x) const
    {
        const int a = slot_of(i), b = slot_of(j);
        if (i == j)
            dg[a] = x;
        else if ((a >> 1) == (b >> 1))
            e[a >> 1] = x;
        else
            cell[0][at(a, b)] = x;
    }
};

// tan of the rotation that annihilates apq, the smaller root of t^2 + 2 th t - 1
// = 0 with th = diff / (2 apq), by the hardware's approximate reciprocal and
// square root: it is on the round's critical path, and any t is a rotation.
__device__ __forceinline__ float jacobi_tan(float diff, float apq)
{
    if (apq == 0.f) return 0.f;
    const float th = __fdividef(0.5f * diff, apq), at = fabsf(th);
    if (!(at < 1e18f)) return at < 1e38f ? __fdividef(0.5f, th) : 0.f;
    float root;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(root) : "f"(fmaf(th, th, 1.f)));
    return copysignf(__fdividef(1.f, at + root), th);
}

// Sweeps until the off-diagonal mass is below tol2 times the total, at most
// max_sweeps (FP32: V is updated only, so it must hold the start basis; the
// matrix has been put).  Returns whether it is (the same value in every
// thread); dg[slot_of(i)] of buffer `cur` then is eigenvalue i.
//
// A function of its own: inlined at its five places it made the solver's kernels so large that their
// other loops ran slower (sparse program of 1e7 nonzeros in FP64, ten iterations: 28.3 ms, 27.4 ms so; 27.1 since
// a slice's row index is read ahead).
template <typename T>
__device__ __noinline__ bool jacobi_sweeps(const Jacobi<T> J, double* red, double tol2, int max_sweeps, int& cur,
                                           const PsdTeam g)
{
    constexpr bool kFast = sizeof(T) == 8;
    constexpr int VW = 16 / (int)sizeof(T);  // rows of V a thread moves at a time
    constexpr int NC = 3;                    // cells of a thread, besides the owned one, whose addresses are kept
    const int tid = g.tid, nt = g.nt, nw = nt >> 5;
    const int dp = J.dp, half = J.half, ncell = J.ncell;
    struct Cell {
        int k, l, src, dst[4];
    };
    auto make_cell = [&](int idx) {
        Cell c;
        if (idx < half) {  // the cells that hold next round's pairs
            c.k = min(idx + 1, half - 1);
            c.l = idx == half - 1 ? half - 2 : max(idx - 1, 0);
        } else if (idx < 2 * half - 3) {  // neighbours (k - l = 1) but the first and the last
            c.k = idx - half + 2;
            c.l = c.k - 1;
        } else {  // k - l >= 3: a triangle
            const int i = idx - (2 * half - 3);
            int r = (int)((sqrtf(8.0f * (float)i + 1.0f) - 1.0f) * 0.5f);
            while ((r + 1) * (r + 2) / 2 <= i) ++r;
            while (r * (r + 1) / 2 > i) --r;
            c.k = r + 3;
            c.l = i - r * (r + 1) / 2;
        }
        c.src = c.k * (c.k - 1) / 2 + c.l;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int a = J.next_slot(2 * c.k + (q >> 1)), b = J.next_slot(2 * c.l + (q & 1));
            c.dst[q] = (a >> 1) == (b >> 1) ? -1 : J.at(a, b);
        }
        return c;
    };
    // Roles: the first `own` warps have the cells that hold the next round's pairs and their rotations,
    // a round's longest chain; the other cells and V go to the other warps, where there are any.
    const int own = (half + 31) >> 5;
    const bool split = nw > own;
    const int ostep = split ? 32 * own : nt, vt0 = split ? 32 * own : 0, vn = nt - vt0, vtid = tid - vt0;
    const bool owner = tid < ostep && half >= 3;
    Cell mine{}, kept[NC];
    if (owner && tid < half) mine = make_cell(tid);
#pragma unroll
    for (int n = 0; n < NC; ++n)
        if (vtid >= 0 && half + vtid + n * vn < ncell) kept[n] = make_cell(half + vtid + n * vn);
    T* const buf0 = J.cell[0];  // (an indexed J.cell would live in local memory)
    T* const buf1 = J.cell[1];
    // a pair's members' slots in the round before, and where its own value goes in the next
    auto from_a = [&](int k) { return k < half - 1 ? 2 * k + 2 : 2 * half - 1; };
    auto from_b = [&](int k) { return k == 0 ? 1 : (k == 1 ? 0 : 2 * k - 1); };
    auto def_to = [&](int k) { return J.at(J.next_slot(2 * k), J.next_slot(2 * k + 1)); };
    const int my_a = from_a(tid), my_b = from_b(tid), my_def = owner && tid < half ? def_to(tid) : 0;
    // what a rotation needs of the round before: loaded ahead of the cell that holds its value
    struct Own {
        T app, aqq, sp, sq, ep, eq;
    };
    auto ahead = [&](int fr, int a, int b) {
        Own o;
        o.app = J.dg[fr * dp + a];
        o.aqq = J.dg[fr * dp + b];
        if constexpr (kFast) {
            o.sp = J.sc[fr * dp + a];
            o.sq = J.sc[fr * dp + b];
            o.ep = J.isc[fr * dp + a];
            o.eq = J.isc[fr * dp + b];
        }
        return o;
    };
    bool fine = false;  // FP64: the angles of this sweep in FP64
    // rotation of pair k, whose off-diagonal value is x, into buffer `to`
    auto rotate = [&](int k, T x, const Own& o, int to) {
        T *dgt = J.dg + to * dp + 2 * k, *sct = J.sc + to * dp + 2 * k, *ist = J.isc + to * dp + 2 * k;
        T* rt = J.rot + (to * half + k) * 2;
        const T app = o.app, aqq = o.aqq, diff = aqq - app;
        if constexpr (kFast) {
            const T sp = o.sp, sq = o.sq, ep = o.ep, eq = o.eq;
            const T apq = x * (sp * sq);
            const float tf = jacobi_tan((float)diff, (float)apq);
            T t = (T)tf;
            if (fine) {  // one Newton step on apq t^2 + diff t - apq, its slope in FP32
                const float slope = fmaf(2.f * (float)apq, tf, (float)diff);
                if (fabsf(slope) > 1e-30f) t = fma(-fma(t, fma(apq, t, diff), -apq), (T)__fdividef(1.f, slope), t);
            }
            const T al = t * (sq * ep), be = t * (sp * eq);
            rt[0] = al;
            rt[1] = be;
            // the factors c^2 of the rotation and 1 / c^2 of the scales cancel
            J.def[k] = fma(fma(-t, t, T(1)), apq, -t * diff) * (ep * eq);
            // c = 1 / sqrt(1 + t^2) from its FP32 value: (1 + d)^-1/2 to second order in d = 1e-7
            const T a2 = fma(t, t, T(1)), c0 = (T)rsqrtf(fmaf(tf, tf, 1.f)), d = fma(a2 * c0, c0, T(-1));
            const T c = c0 * fma(d, fma(d, T(0.375), T(-0.5)), T(1)), ic = a2 * c;
            const T del = (c * c) * (t * fma(t, diff, T(-2) * apq));
            dgt[0] = app + del;
            dgt[1] = aqq - del;
            sct[0] = c * sp;
            sct[1] = c * sq;
            ist[0] = ic * ep;
            ist[1] = ic * eq;
        } else {
            // c as the quotient of two correctly rounded operations, each by one Newton step from the
            // hardware's approximation (Markstein, 1990; a in [1, 2]): V's slow loss of
            // orthogonality depends on how c is rounded, and stays what it was
            const T t = jacobi_tan(diff, x), a2 = t * t + T(1);
            const T y = rsqrtf(a2), g0 = a2 * y, g = fmaf(fmaf(-g0, g0, a2), T(0.5) * y, g0);
            const T c0 = __fdividef(1.f, g), c = fmaf(fmaf(-g, c0, 1.f), c0, c0), s = t * c;
            rt[0] = c;
            rt[1] = s;
            const T xpp = c * app - s * x, xpq = s * app + c * x;  // columns, then rows
            const T xqp = c * x - s * aqq, xqq = s * x + c * aqq;
            dgt[0] = c * xpp - s * xqp;
            J.def[k] = c * xpq - s * xqq;
            dgt[1] = s * xpq + c * xqq;
        }
    };
    auto turn = [](T& xp, T& xq, T r0, T r1) {  // (x_p, x_q) through one rotation
        const T a = xp, b = xq;
        if constexpr (kFast) {
            xp = fma(-r0, b, a);
            xq = fma(r1, a, b);
        } else {
            xp = r0 * a - r1 * b;
            xq = r1 * a + r0 * b;
        }
    };
    // the whole matrix is put; its total, and in FP64 a power of four that scales it to about 1 for
    // the FP32 angles (through the first D)
    auto square_sum = [&](int buf) {
        double s = 0.0;
        const T* c = buf ? buf1 : buf0;
        for (int i = tid; i < 4 * ncell; i += nt) s += (double)c[i] * (double)c[i];
        for (int i = tid; i < half; i += nt) s += (double)J.e[i] * (double)J.e[i];
        return 2.0 * s;
    };
    g.sync();
    double total = square_sum(0);
    for (int i = tid; i < dp; i += nt) total += (double)J.dg[i] * (double)J.dg[i];
    total = block_sum(total, red, g);
    const int quad = kFast && total > 0.0 && isfinite(total) ? ilogb(total) / 4 : 0;
    if constexpr (kFast) {
        for (int i = tid; i < dp; i += nt) {
            J.dg[i] = scalbn(J.dg[i], -2 * quad);
            J.sc[i] = scalbn(1.0, -quad);
        }
        total = scalbn(total, -4 * quad);
        g.sync();
    }
    // V: a thread has VW rows and every ng-th pair, or all pairs of several row groups
    const int groups = J.ldv / VW;
    const bool wide = vn >= groups;
    const int vi0 = vtid < 0 ? groups : (wide ? vtid % groups : vtid), vstep = wide ? groups : vn;
    const int ng = wide ? vn / groups : 1, vg = wide ? vtid / groups : 0;
    bool conv = false;
    cur = 0;
    for (int sweep = 0; sweep <= max_sweeps; ++sweep) {
        if constexpr (kFast) {
            T* c = cur ? buf1 : buf0;
            const T* sc = J.sc + cur * dp;
            for (int i = tid; i < ncell; i += nt) {
                int k = (int)((sqrtf(8.0f * (float)i + 1.0f) + 1.0f) * 0.5f);
                while (k * (k + 1) / 2 <= i) ++k;
                while (k * (k - 1) / 2 > i) --k;
                const int l = i - k * (k - 1) / 2;
#pragma unroll
                for (int q = 0; q < 4; ++q) c[q * ncell + i] *= sc[2 * k + (q >> 1)] * sc[2 * l + (q & 1)];
            }
            for (int i = tid; i < half; i += nt) J.e[i] *= sc[2 * i] * sc[2 * i + 1];
            if (sweep > 0)
                for (int j = tid >> 5; j < dp; j += nw) {
                    const T f = sc[J.slot_of(j)];
                    for (int i = tid & 31; i < dp; i += 32) J.V[j * J.ldv + i] *= f;
                }
            g.sync();
        }
        const double off = block_sum(square_sum(cur), red, g);
        conv = off <= tol2 * total || off == 0.0;
        if (conv || sweep == max_sweeps) break;
        if constexpr (kFast) fine = off <= 1e-11 * total;
        for (int k = tid; k < half; k += nt) {
            if constexpr (kFast) {
                J.sc[cur * dp + 2 * k] = J.sc[cur * dp + 2 * k + 1] = T(1);
                J.isc[cur * dp + 2 * k] = J.isc[cur * dp + 2 * k + 1] = T(1);
            }
            rotate(k, J.e[k], ahead(cur, 2 * k, 2 * k + 1), cur);
        }
        g.sync();
        for (int rnd = 0; rnd < dp - 1; ++rnd) {
            const T* rot = J.rot + cur * dp;
            const T* src = cur ? buf1 : buf0;
            T* dst = cur ? buf0 : buf1;
            const bool last = rnd == dp - 2;
            // a cell's four values through its two rotations
            auto load_turn = [&](const Cell& c, T(&x)[4]) {
                const T ck = rot[2 * c.k], sk = rot[2 * c.k + 1], cl = rot[2 * c.l], sl = rot[2 * c.l + 1];
#pragma unroll
                for (int q = 0; q < 4; ++q) x[q] = src[q * ncell + c.src];
                turn(x[0], x[1], cl, sl);
                turn(x[2], x[3], cl, sl);
                turn(x[0], x[2], ck, sk);
                turn(x[1], x[3], ck, sk);
            };
            auto run_cell = [&](const Cell& c) {
                T x[4];
                load_turn(c, x);
#pragma unroll
                for (int q = 0; q < 4; ++q) dst[c.dst[q]] = x[q];
            };
            auto run_owned = [&](const Cell& c, int k, int a, int b, int to_def) {
                dst[to_def] = J.def[k];  // the pair's own value, rotated before this round
                const Own o = ahead(cur, a, b);
                T x[4], v = 0;
                load_turn(c, x);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    v = c.dst[q] < 0 ? x[q] : v;
                    if (c.dst[q] >= 0) dst[c.dst[q]] = x[q];
                }
                if (last)
                    J.e[k] = v;
                else
                    rotate(k, v, o, cur ^ 1);
            };
            if (owner) {
                if (tid < half) run_owned(mine, tid, my_a, my_b, my_def);
                for (int k = tid + ostep; k < half; k += ostep)
                    run_owned(make_cell(k), k, from_a(k), from_b(k), def_to(k));
            } else if (half < 3 && tid == 0) {
                if (half == 1) {
                    J.e[0] = J.def[0];
                } else {  // one cell, which holds both of the next pairs: (a1, b0) and (b1, a0)
                    Cell c;
                    c.k = 1;
                    c.l = c.src = 0;
                    T x[4];
                    load_turn(c, x);
                    dst[J.at(3, 1)] = J.def[0];
                    dst[J.at(0, 2)] = J.def[1];
                    dst[J.at(0, 3)] = x[0];
                    dst[J.at(2, 1)] = x[3];
                    if (last) {
                        J.e[0] = x[1];
                        J.e[1] = x[2];
                    } else {
                        rotate(0, x[1], ahead(cur, from_a(0), from_b(0)), cur ^ 1);
                        rotate(1, x[2], ahead(cur, from_a(1), from_b(1)), cur ^ 1);
                    }
                }
            }
            if (vtid >= 0 && half >= 3) {
#pragma unroll
                for (int n = 0; n < NC; ++n)
                    if (half + vtid + n * vn < ncell) run_cell(kept[n]);
                for (int idx = half + vtid + NC * vn; idx < ncell; idx += vn) run_cell(make_cell(idx));
            }
            if (vg < ng)
                for (int i = vi0; i < groups; i += vstep) {
                    struct alignas(16) Vec {
                        T x[VW];
                    };
                    T* Vi = J.V + i * VW;
                    for (int k = vg; k < half; k += ng) {
                        const T c = rot[2 * k], sn = rot[2 * k + 1];
                        int a = rnd, b = dp - 1;
                        if (k > 0) {
                            a = rnd + k;
                            if (a >= dp - 1) a -= dp - 1;
                            b = rnd - k;
                            if (b < 0) b += dp - 1;
                        }
                        Vec va = *reinterpret_cast<const Vec*>(Vi + a * J.ldv), vb = *reinterpret_cast<const Vec*>(Vi + b * J.ldv);
#pragma unroll
                        for (int h = 0; h < VW; ++h) turn(va.x[h], vb.x[h], c, sn);
                        *reinterpret_cast<Vec*>(Vi + a * J.ldv) = va;
                        *reinterpret_cast<Vec*>(Vi + b * J.ldv) = vb;
                    }
                }
            cur ^= 1;
            if (last)  // the diagonal (and the scales) of round dp - 2, by the slots of the next sweep
                for (int a = tid; a < dp; a += nt) {
                    const int b = half == 1 ? a : J.next_slot(a);
                    J.dg[cur * dp + b] = J.dg[(cur ^ 1) * dp + a];
                    if constexpr (kFast) {
                        J.sc[cur * dp + b] = J.sc[(cur ^ 1) * dp + a];
                        J.isc[cur * dp + b] = J.isc[(cur ^ 1) * dp + a];
                    }
                }
            g.sync();
        }
    }
    if constexpr (kFast) {
        for (int i = tid; i < dp; i += nt) J.dg[cur * dp + i] = scalbn(J.dg[cur * dp + i], 2 * quad);
        g.sync();
    }
    return conv;
}

// ---------------------------------------------------------------------------
// Exponential cone K = cl{(x1, x2, x3) : x1 >= x2 exp(x3 / x2), x2 > 0}
// (Sec. 2, cone (v)), one cone per thread, in FP64 whatever T is.  With
// (r, s, t) = (x3, x2, x1): a point inside K is kept, a point of the polar
// cone -K* goes to 0, a point with r <= 0 and s <= 0 goes to the face
// (r, 0, max(t, 0)).  Any other point projects on the boundary: either on the
// face {s = 0, r <= 0, t >= 0}, whose nearest point is (min(r,0), 0,
// max(t,0)), or on a ray c (rho, 1, e^rho), c > 0, where the distance is
// stationary in rho, i.e. where
//   F(rho) = r (1 + (1-rho) e^{2rho}) - s (rho + e^{2rho}) + t e^rho (rho^2 - rho + 1)
// vanishes.  The sign changes of F (evaluated as F e^{-2rho} for rho > 0)
// are found on a grid of step 1/4 over [-60, 60] (its roots lie at least
// about 3 apart) and by doubling brackets outside it, each root is bisected
// to full precision, and the nearest of the candidates (origin, face point,
// ray points) is returned.  On the 240 cones of an l1-logistic problem (one
// CTA) a projection took 5.3 ms with every evaluation in FP64 and the sides
// doubled up to overflow (about 3000 FP64 evaluations a cone), 0.45 ms now.  The
// dual cone K* = cl{y3 < 0, -y3 exp(y2/y3) <= e y1}
// is projected through Moreau's decomposition, Pi_{K*}(v) = v + Pi_K(-v).
// ---------------------------------------------------------------------------
// F for rho <= 0 given e = e^rho, and for rho > 0 given em = e^-rho (scaled by e^-2rho)
static __device__ __forceinline__ double expc_Fn(double rho, double e, double r, double s, double t)
{
    const double e2 = e * e;
    return r * (1.0 + (1.0 - rho) * e2) - s * (rho + e2) + t * e * (rho * rho - rho + 1.0);
}
static __device__ __forceinline__ double expc_Fp(double rho, double em, double r, double s, double t)
{
    const double em2 = em * em;
    return r * ((1.0 - rho) + em2) - s * (rho * em2 + 1.0) + t * em * (rho * rho - rho + 1.0);
}
static __device__ __forceinline__ double expc_F(double rho, double r, double s, double t)
{
    return rho <= 0.0 ? expc_Fn(rho, exp(rho), r, s, t) : expc_Fp(rho, exp(-rho), r, s, t);
}

// Root of F in [lo, hi] (a sign change) to adjacent doubles: regula falsi with the
// Illinois modification (the retained end's value is halved when the same end is
// kept twice), a bisection step every fourth iteration so the bracket at least halves
// that often.  Converges in a dozen evaluations where bisection needs about sixty.
static __device__ double expc_root(double lo, double hi, double flo, double r, double s, double t)
{
    // both ends exactly (the grid's values carry the incremental exponentials' roundings)
    flo = expc_F(lo, r, s, t);
    if (flo == 0.0) return lo;
    double fhi = expc_F(hi, r, s, t);
    if (fhi == 0.0) return hi;
    int kept = 0;  // -1: lo kept last time, +1: hi kept last time
    for (int it = 0; it < 400; ++it) {
        const double mid = 0.5 * (lo + hi);
        if (!(mid > lo && mid < hi)) break;
        double x = mid;
        if ((it & 3) != 3) {
            const double sec = (lo * fhi - hi * flo) / (fhi - flo);
            if (sec > lo && sec < hi) x = sec;
        }
        const double fx = expc_F(x, r, s, t);
        if (fx == 0.0) return x;
        if ((fx > 0.0) == (flo > 0.0)) {
            lo = x;
            flo = fx;
            if (kept == 1) fhi *= 0.5;
            kept = 1;
        } else {
            hi = x;
            fhi = fx;
            if (kept == -1) flo *= 0.5;
            kept = -1;
        }
    }
    return 0.5 * (lo + hi);
}

// candidate on the ray of slope rho: the ray's nearest point to (r, s, t) if it lies on the open ray
static __device__ void expc_try_ray(double rho, double r, double s, double t, double& br, double& bs, double& bt, double& bd)
{
    double a0, a1, a2;  // the ray direction scaled by 1 / max(1, e^rho)
    if (rho <= 0.0) {
        a0 = rho;
        a1 = 1.0;
        a2 = exp(rho);
    } else {
        const double em = exp(-rho);
        a0 = rho * em;
        a1 = em;
        a2 = 1.0;
    }
    const double c = (r * a0 + s * a1 + t * a2) / (a0 * a0 + a1 * a1 + a2 * a2);
    if (!(c > 0.0)) return;
    const double pr = c * a0, ps = c * a1, pt = c * a2;
    const double d = (r - pr) * (r - pr) + (s - ps) * (s - ps) + (t - pt) * (t - pt);
    if (d < bd) {
        bd = d;
        br = pr;
        bs = ps;
        bt = pt;
    }
}

// x = (x1, x2, x3) <- Pi_K(x)
static __device__ void expc_project(double& x1, double& x2, double& x3)
{
    const double r = x3, s = x2, t = x1;
    if (s > 0.0 ? s * exp(r / s) <= t : (s == 0.0 && r <= 0.0 && t >= 0.0)) return;  // in K
    if (r > 0.0 ? r * exp(s / r) <= -2.718281828459045 * t : (r == 0.0 && s <= 0.0 && t <= 0.0)) {
        x1 = x2 = x3 = 0.0;  // in the polar cone
        return;
    }
    if (r <= 0.0 && s <= 0.0) {
        x1 = t > 0.0 ? t : 0.0;
        x2 = 0.0;
        return;
    }
    double br = 0.0, bs = 0.0, bt = 0.0, bd = r * r + s * s + t * t;  // the origin
    {
        const double fr = fmin(r, 0.0), ft = fmax(t, 0.0);
        const double d = (r - fr) * (r - fr) + s * s + (t - ft) * (t - ft);
        if (d < bd) {
            bd = d;
            br = fr;
            bs = 0.0;
            bt = ft;
        }
    }
    // Outside the grid F is dominated by its linear part: at most one sign change on each side.
    // Past |rho| = 800 the exponential is exactly 0 and F is r - s rho (left), r (1 - rho) - s
    // (right), monotone in rho also as rounded: once its sign is that of its limit, no later
    // doubling changes it.
    for (int side = 0; side < 2; ++side) {
        double a = side == 0 ? -60.0 : 60.0;
        double fa = expc_F(a, r, s, t);
        const double slope = side == 0 ? s : -r, rest = side == 0 ? r : -s;  // the limit's sign, or F itself
        for (int k = 0; k < 1100; ++k) {
            const double b = 2.0 * a;
            if (!isfinite(b)) break;
            const double fb = expc_F(b, r, s, t);
            if (fb != 0.0 && (fb > 0.0) != (fa > 0.0)) {
                const double rho = side == 0 ? expc_root(b, a, fb, r, s, t) : expc_root(a, b, fa, r, s, t);
                expc_try_ray(rho, r, s, t, br, bs, bt, bd);
                break;
            }
            if (fabs(b) > 800.0 && isfinite(fb) && (slope == 0.0 ? rest != 0.0 : (fb != 0.0 && (fb > 0.0) == (slope > 0.0))))
                break;
            a = b;
            fa = fb;
        }
    }
    // The grid.  Only the signs of F matter, and they are found in FP32 (the FP64 pipe runs at
    // 1/64 of the FP32 rate): with (r, s, t) scaled to a largest entry of 1, the FP32 value of F
    // is off by less than 8e-6 of the sum of its terms' magnitudes, so where it is larger its
    // sign is F's; nearer a root F is evaluated in FP64.  (A term is an input rounded to FP32, a
    // polynomial in rho that is exact, since rho is a multiple of 1/4 up to 60, and e or e^2, e
    // within 2 ulp: at most 8 roundings a term and 4 in the sums, 7e-7 of the magnitudes.  Where
    // e^2 or an input underflows, its term is below 1e-38 beside one of 3e-23 at least.)  The sign
    // changes are noted first and refined afterwards, so that the lanes of a warp (one cone each)
    // refine theirs together.
    const double big = fmax(fabs(r), fmax(fabs(s), fabs(t)));
    const bool scan32 = isfinite(big) && big > 1e-290;
    const double sc = scan32 ? 1.0 / big : 0.0;
    const float rf = (float)(r * sc), sf = (float)(s * sc), tf = (float)(t * sc);
    auto sign_at = [&](int k) {  // -1 (also NaN), 0 or 1
        const float x = -60.0f + 0.25f * (float)k;
        const float e = expf(k <= 240 ? x : -x), e2 = e * e, q = e * (x * x - x + 1.0f);
        const float u = k <= 240 ? 1.0f : e2, v = k <= 240 ? e2 : 1.0f;  // F's e^0 and e^2 weights
        // r (1 + (1 - x) e2) - s (x + e2) + t q, or for x > 0 the same times e^-2x
        const float ra = k <= 240 ? (1.0f - x) * e2 : 1.0f - x;
        const float f = rf * (u + ra) - sf * (x * u + v) + tf * q;
        const float mag = fabsf(rf) * (u + fabsf(ra)) + fabsf(sf) * (fabsf(x) * u + v) + fabsf(tf) * q;
        if (scan32 && fabsf(f) > 8e-6f * mag) return f > 0.0f ? 1 : -1;
        const double F = expc_F(-60.0 + 0.25 * k, r, s, t);
        return F == 0.0 ? 0 : (F > 0.0 ? 1 : -1);
    };
    constexpr int PEND = 6;
    unsigned long long pend = 0;  // 10 bits a noted point: its k, and bit 9 if F is 0 there
    int np = 0;
    auto refine = [&]() {
        for (int i = 0; i < np; ++i, pend >>= 10) {
            const int k = (int)(pend & 511u);
            const double xb = -60.0 + 0.25 * k;
            expc_try_ray((pend & 512u) ? xb : expc_root(xb - 0.25, xb, 0.0, r, s, t), r, s, t, br, bs, bt, bd);
        }
        pend = 0;
        np = 0;
    };
    int ga = sign_at(0);
    for (int k = 1; k <= 480; ++k) {
        const int gb = sign_at(k);
        if (gb == 0 || (ga != 0 && gb != ga)) {
            if (np == PEND) refine();
            pend |= (unsigned long long)(k | (gb == 0 ? 512 : 0)) << (10 * np);
            ++np;
        }
        ga = gb;
    }
    refine();
    x1 = bt;
    x2 = bs;
    x3 = br;
}

// Shared memory of a CTA's PSD projections, and where a block's matrices are:
// all in shared memory up to order PSD_MAX; larger orders in the block's global
// workspace, with the Jacobi scratch in shared memory.
template <typename T>
struct PsdSmem {
    T* X0;        // the input matrix, full, row stride dp + 1; FP64: later the second cell buffer
    T* V;         // X Vp while a warm start is formed (row stride dp + 1), then the eigenvectors (columns, stride ldv)
    T* cell[2];
    double* V64;  // FP32 eigensolves only: the eigenvectors in FP64 (row stride dp + 1), for the recheck
    T* scratch;   // Jacobi's scratch, 8 bytes a word in either precision
    T* lam;
    double* red;
};

// stride of V's columns: whole 16-byte vectors
template <typename T>
__host__ __device__ constexpr int psd_ldv(int dp)
{
    return sizeof(T) == 4 ? (dp + 3) & ~3 : dp;
}
__host__ __device__ constexpr size_t psd_round(size_t bytes) { return (bytes + 15) & ~size_t(15); }
template <typename T>
__host__ __device__ constexpr size_t psd_matrix_bytes(int dp)  // matrices of one block of (even) order dp
{
    return 2 * psd_round(sizeof(T) * (size_t)dp * (dp + 2)) + (sizeof(T) == 4 ? 2 : 1) * psd_round(sizeof(T) * 4 * (size_t)Jacobi<T>::cells(dp)) +
           (sizeof(T) == 4 ? psd_round(sizeof(double) * (size_t)dp * (dp + 1)) : 0);
}
__host__ __device__ constexpr size_t psd_scratch_bytes(int dp) { return sizeof(double) * (64 + 10 * (size_t)dp); }
// dynamic shared memory of a CTA that projects a block of order d; not monotone: largest at PSD_MAX
template <typename T>
__host__ __device__ constexpr size_t psd_smem_bytes(int d)
{
    return psd_scratch_bytes(d + (d & 1)) + (d <= PSD_MAX ? psd_matrix_bytes<T>(d + (d & 1)) : 0);
}
// workspace of one PSD block of order d > PSD_MAX in global memory
template <typename T>
__host__ __device__ constexpr size_t psd_big_bytes(int d)
{
    return psd_matrix_bytes<T>(d + (d & 1));
}
// warm-start eigenvectors of one PSD block: dp columns
template <typename T>
__host__ __device__ constexpr size_t psd_v_bytes(int d)
{
    const int dp = d + (d & 1);
    return psd_round(sizeof(T) * (size_t)dp * psd_ldv<T>(dp));
}

// How a CTA of `threads` threads shares out its PSD blocks, ns of at most order d over `ctas` CTAs, in at
// most `limit` bytes of shared memory: several blocks at a time, each by a group of its threads, where a
// CTA has several.  `small` is the largest order up to PSD_MAX (0: none): beside larger orders, whose
// matrices are elsewhere, it is what sizes a group's memory.  A round of the Jacobi sweeps is a chain of latencies and a block's matrix is small, so
// a group of 256 threads is hardly slower than 512 (order 64 in FP32, 512 blocks, one group a CTA: 4.0
// and 3.65 ms; in FP64, where more warps only crowd the pipe, 13.7 and 17.3 ms) and 128 do for small
// orders (20: 1.01 and 1.10 ms).  A CTA with one block gives it 256 threads, FP32 above order 48 all.
struct PsdPlan {
    int threads, groups;
    unsigned bytes;  // of one group
};
template <typename T>
__host__ __device__ inline PsdPlan psd_plan(int d, int small, int ns, int ctas, int threads, unsigned limit)
{
    const size_t top = psd_smem_bytes<T>(d), mid = psd_smem_bytes<T>(small);
    PsdPlan p{threads, 1, (unsigned)(top > mid ? top : mid)};
    if (d > PSD_MAX || ns == 0) return p;
    const int per = (ns + ctas - 1) / ctas;
    int t = d <= 24 ? 128 : 256;
    if (per == 1 && (d <= 24 || sizeof(T) == 4)) t = sizeof(T) == 4 && d > 48 ? threads : 256;
    if (t >= threads || threads % t) return p;
    p.threads = t;
    const int room = (int)(limit / p.bytes), most = threads / t < per ? threads / t : per;
    p.groups = room < most ? (room > 1 ? room : 1) : most;
    return p;
}
// the orders that size it: the largest, and the largest up to PSD_MAX (0: none)
inline void psd_orders(const std::vector<int>& orders, int& order, int& small)
{
    order = small = 0;
    for (int d : orders) {
        order = d > order ? d : order;
        small = d <= PSD_MAX && d > small ? d : small;
    }
}
__device__ __forceinline__ unsigned dyn_smem_size()
{
    unsigned n;
    asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(n));
    return n;
}

// smem: the CTA's shared region; big: the block's global workspace, or null
template <typename T>
__host__ __device__ PsdSmem<T> psd_layout(unsigned char* smem, unsigned char* big, int dp)
{
    PsdSmem<T> s;
    s.red = (double*)smem;
    s.scratch = (T*)(s.red + 64);
    s.lam = (T*)(s.red + 64 + 9 * dp);
    unsigned char* m = big ? big : smem + psd_scratch_bytes(dp);
    s.V64 = (double*)m;
    if (sizeof(T) == 4) m += psd_round(sizeof(double) * (size_t)dp * (dp + 1));
    s.X0 = (T*)m;
    m += psd_round(sizeof(T) * (size_t)dp * (dp + 2));
    s.V = (T*)m;
    m += psd_round(sizeof(T) * (size_t)dp * (dp + 2));
    s.cell[0] = (T*)m;
    s.cell[1] = sizeof(T) == 4 ? (T*)(m + psd_round(sizeof(T) * 4 * (size_t)Jacobi<T>::cells(dp))) : s.X0;
    return s;
}

// Where the FP32 eigensolves report to: the largest relative eigen-residual
// (FP64-evaluated), the count of blocks decomposed again in FP64, and the
// bound above which that happens.
struct PsdCheck {
    double* resid;
    long long* redo;
    double tol;
    // warm starts: block k's eigenvectors of its last converged decomposition are kept at
    // vbase + voff[k] bytes (dp columns of psd_ldv elements of the bulk type); vok[k] = 0: none, else the
    // number of decompositions since the last cold one
    unsigned char* vbase;
    const long long* voff;
    int* vok;
};

// FP64 Jacobi of the input block X0 (FP32 eigensolves only): the cells in the
// place of the FP32 V and cells, which are dead, the eigenvectors in V64
// (columns, stride dp), the positive parts of the eigenvalues in lam64.
static __device__ __noinline__ void psd_redo_fp64(PsdSmem<float>& sm, int dp, double* lam64, const PsdTeam& g)
{
    double* c0 = reinterpret_cast<double*>(sm.V);
    const Jacobi<double> J(c0, c0 + 4 * Jacobi<double>::cells(dp), sm.V64, reinterpret_cast<double*>(sm.scratch), dp, dp);
    const int lane = g.tid & 31, warp = g.tid >> 5, nw = g.nt >> 5;
    g.sync();
    for (int j = warp; j < dp; j += nw)
        for (int i = lane; i < dp; i += 32) {
            if (i >= j) J.put(i, j, (double)sm.X0[i * (dp + 1) + j]);
            J.V[j * dp + i] = i == j ? 1.0 : 0.0;
        }
    int cur;
    jacobi_sweeps<double>(J, sm.red, 1e-26, 20, cur, g);
    for (int i = g.tid; i < dp; i += g.nt) lam64[i] = fmax(J.dg[cur * dp + J.slot_of(i)], 0.0);
    g.sync();
}

// V diag(l) V^T, the entries (i, j), i >= j, of its leading d x d part, from V's columns (stride
// ldv): four rows of one column a thread; eigenvectors with l = 0 are skipped.
template <typename T, class Emit>
__device__ __forceinline__ void psd_rebuild(const T* V, const T* l, int d, int dp, int ldv, const PsdTeam& g, Emit emit)
{
    const int lane = g.tid & 31, warp = g.tid >> 5, nw = g.nt >> 5;
    for (int i0 = 4 * warp; i0 < d; i0 += 4 * nw)
        for (int j = lane; j < min(i0 + 4, d); j += 32) {
            T a[4] = {0, 0, 0, 0};
            for (int k = 0; k < dp; ++k) {
                if (l[k] == T(0)) continue;
                const T* c = V + k * ldv;
                const T v = l[k] * c[j];
#pragma unroll
                for (int h = 0; h < 4; ++h) a[h] = fmaT(c[min(i0 + h, d - 1)], v, a[h]);
            }
#pragma unroll
            for (int h = 0; h < 4; ++h)
                if (i0 + h < d && j <= i0 + h) emit(i0 + h, j, a[h]);
        }
}

template <typename T, class Team, class Op>
__device__ void project_pass(Team& tm, const DevProb<T>& P, Op& op, unsigned char* psd_base,
                             PsdCheck ck = PsdCheck{nullptr, nullptr, 0.0})
{
    const int n = P.n;
    const int lin = n + P.f + P.l;
    const int fz = n + P.f;
    for (int i = tm.rank(); i < lin; i += tm.size()) {
        T w, wt;
        op.load(i, w, wt);
        const T v = T(2) * wt - w;
        const T wb = (i >= fz) ? (v > T(0) ? v : T(0)) : v;
        op.store(i, w, wt, wb);
    }
    // second-order cones, t last: one warp per cone
    const int lane = threadIdx.x & 31;
    const int nw = tm.size() >> 5;
    for (int k = tm.rank() >> 5; k < P.nq; k += nw) {
        const int o = n + ro(P.q_off + k);
        const int dim = ro(P.q_off + k + 1) - ro(P.q_off + k);
        T ss = 0;
        for (int j = lane; j < dim - 1; j += 32) {
            T w, wt;
            op.load(o + j, w, wt);
            const T v = T(2) * wt - w;
            ss += v * v;
        }
        T wT, wtT;
        op.load(o + dim - 1, wT, wtT);
        const T tv = T(2) * wtT - wT;
        const double nx = sqrt((double)warp_sum(ss));
        const double t = (double)tv;
        int mode;
        double a = 0.0, tb = 0.0;
        if (nx <= t) mode = 0;
        else if (nx <= -t) mode = 1;
        else {
            mode = 2;
            a = (nx + t) / (2.0 * nx);
            tb = a * nx;
        }
        for (int j = lane; j < dim - 1; j += 32) {
            T w, wt;
            op.load(o + j, w, wt);
            const T v = T(2) * wt - w;
            const T wb = mode == 0 ? v : (mode == 1 ? T(0) : (T)(a * (double)v));
            op.store(o + j, w, wt, wb);
        }
        if (lane == 0) op.store(o + dim - 1, wT, wtT, mode == 0 ? tv : (mode == 1 ? T(0) : (T)tb));
        __syncwarp();
    }
    // PSD blocks: one group of a CTA's threads per block (psd_plan), Jacobi
    // eigen-decomposition in shared memory (orders above PSD_MAX: in the block's
    // workspace in global memory)
    if (P.ns > 0) {
        __syncthreads();  // shared memory is free (earlier users done)
        const PsdPlan plan = psd_plan<T>(P.psd_order, P.psd_small, P.ns, tm.nblocks(), blockDim.x, dyn_smem_size());
        const int gid = threadIdx.x / plan.threads;
        const PsdTeam g{(int)threadIdx.x - gid * plan.threads, plan.threads, 1 + gid};
        const int lane = g.tid & 31, warp = g.tid >> 5, nwb = g.nt >> 5;
        const int k0 = gid < plan.groups ? tm.block() + gid * tm.nblocks() : P.ns;
        for (int k = k0; k < P.ns; k += plan.groups * tm.nblocks()) {
            const int d = ro(P.s_dim + k);
            const int o = n + ro(P.s_off + k);
            const int dp = d + (d & 1);
            const int ld = dp + 1;  // odd row stride: column walks are free of bank conflicts
            const int ldv = psd_ldv<T>(dp);
            PsdSmem<T> sm = psd_layout<T>(psd_base + gid * plan.bytes, d > PSD_MAX ? P.psd_big + ro(P.big_off + k) : nullptr, dp);
            const Jacobi<T> J(sm.cell[0], sm.cell[1], sm.V, sm.scratch, dp, ldv);
            const double isq2 = 0.70710678118654752440;
            // Warm start: successive projections of a block see nearby matrices, so the
            // eigenvectors Vp of the last converged decomposition nearly diagonalise this one.
            // The sweeps run on Vp^T X Vp and accumulate onto V = Vp: the same eigenpairs, found in
            // a few sweeps instead of a dozen.  vok[k] counts the generations since the last cold
            // start; V loses orthogonality by a few roundings per generation, so every
            // PSD_WARM_GEN-th decomposition starts cold again.
            constexpr int PSD_WARM_GEN = sizeof(T) == 4 ? 16 : 64;
            T* Vp = ck.vbase ? reinterpret_cast<T*>(ck.vbase + ro(ck.voff + k)) : nullptr;
            const int gen = Vp ? *(volatile const int*)(ck.vok + k) : 0;
            const bool warm = gen > 0 && gen < PSD_WARM_GEN;
            g.sync();
            for (int j = warp; j < dp; j += nwb)  // column j of the lower triangle: consecutive in svec
                for (int i = j + lane; i < dp; i += 32) {
                    T val = 0;
                    if (i < d) {
                        T w, wt;
                        op.load(o + svec_index(d, i, j), w, wt);
                        const T v = T(2) * wt - w;
                        val = i == j ? v : (T)((double)v * isq2);
                    }
                    if (warm || sizeof(T) == 4) {
                        sm.X0[i * ld + j] = val;
                        sm.X0[j * ld + i] = val;
                    }
                    if (!warm) J.put(i, j, val);
                }
            if (warm) {
                constexpr int VW = 16 / (int)sizeof(T);
                struct alignas(16) Vec {
                    T x[VW];
                };
                g.sync();
                for (int j0 = 4 * warp; j0 < dp; j0 += 4 * nwb)  // T <- X Vp, four columns a thread
                    for (int i = lane; i < dp; i += 32) {
                        T a[4] = {0, 0, 0, 0};
                        for (int l = 0; l < dp; l += VW) {
                            Vec v[4];
#pragma unroll
                            for (int h = 0; h < 4; ++h)
                                v[h] = *reinterpret_cast<const Vec*>(Vp + min(j0 + h, dp - 1) * ldv + l);
#pragma unroll
                            for (int u = 0; u < VW; ++u) {
                                const T x = l + u < dp ? sm.X0[(l + u) * ld + i] : T(0);
#pragma unroll
                                for (int h = 0; h < 4; ++h) a[h] = l + u < dp ? fmaT(x, v[h].x[u], a[h]) : a[h];
                            }
                        }
#pragma unroll
                        for (int h = 0; h < 4; ++h)
                            if (j0 + h < dp) sm.V[i * ld + j0 + h] = a[h];
                    }
                g.sync();
                for (int i0 = 4 * warp; i0 < dp; i0 += 4 * nwb)  // Vp^T T, lower triangle
                    for (int j = lane; j < min(i0 + 4, dp); j += 32) {
                        T a[4] = {0, 0, 0, 0};
                        for (int l = 0; l < dp; l += VW) {
                            Vec v[4];
#pragma unroll
                            for (int h = 0; h < 4; ++h)
                                v[h] = *reinterpret_cast<const Vec*>(Vp + min(i0 + h, dp - 1) * ldv + l);
#pragma unroll
                            for (int u = 0; u < VW; ++u) {
                                const T x = l + u < dp ? sm.V[(l + u) * ld + j] : T(0);
#pragma unroll
                                for (int h = 0; h < 4; ++h) a[h] = l + u < dp ? fmaT(v[h].x[u], x, a[h]) : a[h];
                            }
                        }
#pragma unroll
                        for (int h = 0; h < 4; ++h)
                            if (i0 + h < dp && j <= i0 + h) J.put(i0 + h, j, a[h]);
                    }
                g.sync();
                for (int i = g.tid; i < dp * ldv; i += g.nt) sm.V[i] = Vp[i];
            } else {
                for (int j = warp; j < dp; j += nwb)
                    for (int i = lane; i < ldv; i += 32) sm.V[j * ldv + i] = i == j ? T(1) : T(0);
            }
            int cur;
            const bool conv = jacobi_sweeps<T>(J, sm.red, sizeof(T) == 8 ? 1e-26 : 1e-11,
                                               d > PSD_MAX ? 30 : (sizeof(T) == 8 ? 20 : 15), cur, g);
            if (Vp) {
                if (conv)
                    for (int i = g.tid; i < dp * ldv; i += g.nt) Vp[i] = sm.V[i];
                if (g.tid == 0) ck.vok[k] = conv ? (warm ? gen + 1 : 1) : 0;
            }
            for (int i = g.tid; i < dp; i += g.nt) {
                const T l = J.dg[cur * dp + J.slot_of(i)];
                sm.lam[i] = l > T(0) ? l : T(0);
            }
            if constexpr (sizeof(T) == 4) {
                // Recheck of the FP32 eigenpairs: ||X V - V diag(l)||_F / ||X||_F.  X, V and l are FP32,
                // so a product is two FP32 words exactly, and the sums are kept in three words by
                // error-free additions (Knuth's two-sum), more than FP64's bits; FP64 from there on.
                // The d^3 multiply-adds in FP64 took as long as the sweeps did (FP64 pipe: 131k cycles
                // of the SM for order 64; 512 such blocks, one projection: 4.6 ms, 3.8 ms
                // so).  X is scaled by a power of two so that no word overflows or loses bits to underflow.
                float* VR = reinterpret_cast<float*>(sm.V64);  // V by rows (stride ld)
                for (int j = warp; j < dp; j += nwb)
                    for (int i = lane; i < dp; i += 32) VR[i * ld + j] = sm.V[j * ldv + i];
                double x2 = 0.0, r2 = 0.0;
                for (int i = warp; i < dp; i += nwb)
                    for (int j = lane; j < dp; j += 32) x2 += (double)sm.X0[i * ld + j] * (double)sm.X0[i * ld + j];
                x2 = block_sum(x2, sm.red, g);
                const int e2 = x2 > 0.0 && isfinite(x2) ? ilogb(x2) / 2 : 0;
                const float sc1 = scalbnf(1.0f, -(e2 / 2)), sc2 = scalbnf(1.0f, -(e2 - e2 / 2));  // (each in range)
                const int nk = (dp + 31) >> 5;
                for (int it = warp; it < nk * ((dp + 3) >> 2); it += nwb) {
                    // 4 rows by 32 columns a warp, a column a lane
                    const int i0 = 4 * (it / nk), k = 32 * (it % nk) + lane, kk = min(k, dp - 1);
                    const float lk = J.dg[cur * dp + J.slot_of(kk)] * sc1 * sc2;
                    float hi[4] = {0.f, 0.f, 0.f, 0.f}, lo[4] = {0.f, 0.f, 0.f, 0.f}, lo2[4] = {0.f, 0.f, 0.f, 0.f};
                    auto two_sum = [](float& a, float b) {  // a + b = (a, returned error)
                        const float t = a + b, z = t - a, e = (a - (t - z)) + (b - z);
                        a = t;
                        return e;
                    };
                    auto add = [&](int h, float x, float v) {  // (hi, lo, lo2) += x v
                        const float p = x * v, pe = fmaf(x, v, -p);
                        const float e = two_sum(hi[h], p);
                        lo2[h] += two_sum(lo[h], e) + two_sum(lo[h], pe);
                    };
#pragma unroll
                    for (int h = 0; h < 4; ++h) add(h, -lk, VR[min(i0 + h, dp - 1) * ld + kk]);
                    for (int j = 0; j < dp; ++j) {
                        const float v = VR[j * ld + kk];
#pragma unroll
                        for (int h = 0; h < 4; ++h) add(h, sm.X0[j * ld + min(i0 + h, dp - 1)] * sc1 * sc2, v);
                    }
#pragma unroll
                    for (int h = 0; h < 4; ++h)
                        if (k < dp && i0 + h < dp) {
                            const double a = (double)hi[h] + ((double)lo[h] + (double)lo2[h]);
                            r2 += a * a;
                        }
                }
                r2 = scalbn(block_sum(r2, sm.red, g), 2 * e2);
                // block_sum hands every thread the same sums, so the decision
                // to decompose the block again in FP64 is uniform in the group
                const double rel = x2 > 0.0 ? sqrt(r2 / x2) : 0.0;
                if (g.tid == 0 && ck.resid)
                    atomicMax((unsigned long long*)ck.resid, (unsigned long long)__double_as_longlong(rel));
                if (rel > ck.tol && ck.redo) {
                    double* lam64 = reinterpret_cast<double*>(sm.lam);
                    psd_redo_fp64(sm, dp, lam64, g);
                    if (g.tid == 0) {
                        atomicAdd((unsigned long long*)ck.redo, 1ull);
                        if (Vp) ck.vok[k] = 0;  // the FP32 eigenvectors were not good enough to start from
                    }
                    psd_rebuild<double>(sm.V64, lam64, d, dp, dp, g, [&](int i, int j, double x) {
                        const int e = o + svec_index(d, i, j);
                        T w, wt;
                        op.load(e, w, wt);
                        op.store(e, w, wt, (T)(i == j ? x : x * 1.41421356237309504880));
                    });
                    g.sync();
                    continue;
                }
            }
            g.sync();
            psd_rebuild<T>(sm.V, sm.lam, d, dp, ldv, g, [&](int i, int j, T x) {
                const int e = o + svec_index(d, i, j);
                T w, wt;
                op.load(e, w, wt);
                op.store(e, w, wt, i == j ? x : (T)((double)x * 1.41421356237309504880));
            });
            g.sync();
        }
    }
    // exponential cones, one per thread: the psi part lies in K*, so a primal
    // block projects on the dual cone (Moreau: v + Pi_K(-v)) and a dual block on K
    for (int k = tm.rank(); k < P.ep + P.ed; k += tm.size()) {
        const int o = n + P.e_off + 3 * k;
        T w[3], wt[3];
        double v[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            op.load(o + j, w[j], wt[j]);
            v[j] = 2.0 * (double)wt[j] - (double)w[j];
        }
        if (k < P.ep) {
            double m1 = -v[0], m2 = -v[1], m3 = -v[2];
            expc_project(m1, m2, m3);
            v[0] += m1;
            v[1] += m2;
            v[2] += m3;
        } else {
            expc_project(v[0], v[1], v[2]);
        }
#pragma unroll
        for (int j = 0; j < 3; ++j) op.store(o + j, w[j], wt[j], (T)v[j]);
    }
    if (tm.leader()) {
        double w, wt;
        op.load_tau(w, wt);
        const double v = 2.0 * wt - w;
        op.store_tau(w, wt, v > 0.0 ? v : 0.0);
    }
}

// ---- ops of the projection pass ----
// residual at (u, u~): u_ = Pi(2u~ - u), R = u~ - u_;  acc0 = ||R||^2
template <typename T>
struct OpResidual {
    HV<T> u, ut, ub, R;
    T acc0;
    __device__ void load(int i, T& w, T& wt) const { w = u.v[i]; wt = ut.v[i]; }
    __device__ void store(int i, T, T wt, T wb)
    {
        ub.v[i] = wb;
        const T r = wt - wb;
        R.v[i] = r;
        acc0 += r * r;
    }
    __device__ void load_tau(double& w, double& wt) const { w = *u.t; wt = *ut.t; }
    __device__ void store_tau(double, double wt, double wb)
    {
        *ub.t = wb;
        const double r = wt - wb;
        *R.t = r;
        acc0 += (T)(r * r);
    }
};

// K0 (blind step): u <- u + d, u~ <- u~ + d~, then the residual of the new
// point; secant pair z = d, xi = R_new - R_old; acc0 = ||R_new||^2, acc1 = ||d||^2
template <typename T>
struct OpK0 {
    HV<T> u, ut, ub, Ru, d, dt, zp, xip;
    T acc0, acc1;
    __device__ void load(int i, T& w, T& wt) const { w = u.v[i] + d.v[i]; wt = ut.v[i] + dt.v[i]; }
    __device__ void store(int i, T w, T wt, T wb)
    {
        const T di = d.v[i];
        u.v[i] = w;
        ut.v[i] = wt;
        ub.v[i] = wb;
        const T r = wt - wb;
        xip.v[i] = r - Ru.v[i];
        zp.v[i] = di;
        Ru.v[i] = r;
        acc0 += r * r;
        acc1 += di * di;
    }
    __device__ void load_tau(double& w, double& wt) const { w = *u.t + *d.t; wt = *ut.t + *dt.t; }
    __device__ void store_tau(double w, double wt, double wb)
    {
        const double di = *d.t;
        *u.t = w;
        *ut.t = wt;
        *ub.t = wb;
        const double r = wt - wb;
        *xip.t = r - *Ru.t;
        *zp.t = di;
        *Ru.t = r;
        acc0 += (T)(r * r);
        acc1 += (T)(di * di);
    }
};

// line-search trial at w = u + alpha d, w~ = u~ + alpha d~ (linearity trick,
// Sec. 4.2): stores w_ and Rw; acc0 = ||Rw||^2, acc1 = <Rw, Rw - alpha d>
template <typename T>
struct OpTrial {
    HV<T> u, ut, d, dt, wb, Rw;
    double alpha;
    T acc0, acc1;
    __device__ void load(int i, T& w, T& wt) const
    {
        const T a = (T)alpha;
        w = u.v[i] + a * d.v[i];
        wt = ut.v[i] + a * dt.v[i];
    }
    __device__ void store(int i, T, T wt, T wbv)
    {
        wb.v[i] = wbv;
        const T r = wt - wbv;
        Rw.v[i] = r;
        acc0 += r * r;
        acc1 += r * (r - (T)alpha * d.v[i]);
    }
    __device__ void load_tau(double& w, double& wt) const
    {
        w = *u.t + alpha * *d.t;
        wt = *ut.t + alpha * *dt.t;
    }
    __device__ void store_tau(double, double wt, double wbv)
    {
        *wb.t = wbv;
        const double r = wt - wbv;
        *Rw.t = r;
        acc0 += (T)(r * r);
        acc1 += (T)(r * (r - alpha * *d.t));
    }
};

// plain projection: v -> Pi_C(v) (as w = -v, w~ = 0)
template <typename T>
struct OpProject {
    const T* vin;
    const double* tin;
    T* out;
    double* tout;
    __device__ void load(int i, T& w, T& wt) const { w = -vin[i]; wt = 0; }
    __device__ void store(int i, T, T, T wb) { out[i] = wb; }
    __device__ void load_tau(double& w, double& wt) const { w = -*tin; wt = 0.0; }
    __device__ void store_tau(double, double, double wb) { *tout = wb; }
};

// ---------------------------------------------------------------------------
// elementwise helpers on HSDE vectors
// ---------------------------------------------------------------------------

// ---------------------------------------------------------------------------
// Termination (Sec. 4.3) on (u, u~, u_).  Returns a status (0 = continue).
// Certificates use the reading ic = ||b|| ||A^T psi_|| / (-<b, psi_>) and
// uc = ||c|| ||A chi_ + sigma_|| / (-<c, chi_>) on unscaled vectors.
// ---------------------------------------------------------------------------
struct TermOut {
    double pr, dr, gap, ic, uc, pobj, dobj, bpsi, cchi;
    bool time_up;
};

template <typename T, class Team>
__device__ int termination(Team& tm, const DevProb<T>& P, const DevWork<T>& W, double eps, double deadline_ns,
                           TermOut& o)
{
    const int n = P.n, m = P.m;
    const T* chib = W.ub.v;
    const T* psib = W.ub.v + n;
    const T* psit = W.ut.v + n;
    const T* psi = W.u.v + n;
    const double taub = *W.ub.t;
    T* tmv = W.tm;
    T* tnv = W.tn;
    spmv(tm, P.A, chib, [&](int i, T s) { tmv[i] = s; });
    spmv(tm, P.AT, psib, [&](int j, T s) { tnv[j] = s; });
    tm.sync();
    if (tm.leader()) W.st->mat_passes += 2;
    const bool pos = taub > 0.0;
    const T inv = pos ? (T)(1.0 / taub) : T(0);
    T a0 = 0, a1 = 0, a2 = 0, a3 = 0, a4 = 0, a5 = 0;
    for (int i = tm.rank(); i < m; i += tm.size()) {
        const T sig = psib[i] - T(2) * psit[i] + psi[i];
        const T bi = ro(P.b + i);
        if (pos) {
            const T e = tmv[i] * inv + sig * inv - bi;
            a0 += e * e;
        }
        const T f = tmv[i] + sig;
        a4 += f * f;
        a3 += bi * psib[i];
    }
    for (int j = tm.rank(); j < n; j += tm.size()) {
        const T cj = ro(P.c + j);
        if (pos) {
            const T gq = tnv[j] * inv + cj;
            a1 += gq * gq;
        }
        a2 += cj * chib[j];
        a5 += tnv[j] * tnv[j];
    }
    double tflag = 0.0;
    if (tm.leader() && deadline_ns > 0.0 && (double)gtimer() > deadline_ns) tflag = 1.0;
    double red[7] = {(double)a0, (double)a1, (double)a2, (double)a3, (double)a4, (double)a5, tflag};
    tm.reduce(red);
    o.time_up = red[6] > 0.0;
    o.cchi = red[2];
    o.bpsi = red[3];
    o.pr = o.dr = o.gap = INFINITY;
    o.pobj = o.dobj = NAN;
    int status = 0;
    if (pos) {
        o.pr = sqrt(red[0]) / (1.0 + P.nb);
        o.dr = sqrt(red[1]) / (1.0 + P.nc);
        const double cx = red[2] / taub, by = red[3] / taub;
        o.gap = fabs(cx + by) / (1.0 + fabs(cx) + fabs(by));
        o.pobj = cx;
        o.dobj = -by;
        if (o.pr <= eps && o.dr <= eps && o.gap <= eps) status = ST_SOLVED;
    }
    o.ic = red[3] < 0.0 ? P.nb * sqrt(red[5]) / (-red[3]) : INFINITY;
    o.uc = red[2] < 0.0 ? P.nc * sqrt(red[4]) / (-red[2]) : INFINITY;
    if (!status) {
        if (o.ic < eps) status = ST_INFEASIBLE;
        else if (o.uc < eps) status = ST_UNBOUNDED;
    }
    return status;
}

// ---------------------------------------------------------------------------
// directions (Sec. 4.4)
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ HV<T> col(T* base, double* tb, int k, int nm)
{
    return HV<T>{base + (size_t)k * nm, tb + k};
}

// small dense Cholesky solve by warp 0 of every block (k <= 32):
// (G + reg I) t = rhs with reg raised tenfold up to 8 times; false on failure
static __device__ bool small_chol(const double* G, const double* rhs, double* L, double* t, int k, double reg0)
{
    __shared__ int ok_s;
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        bool ok = false;
        double reg = reg0;
        for (int attempt = 0; attempt < 8 && !ok; ++attempt, reg *= 10.0) {
            ok = true;
            for (int j = 0; j < k; ++j) {
                double s = (lane < j) ? L[j * AAMAX + lane] * L[j * AAMAX + lane] : 0.0;
                s = warp_sum(s);
                const double dj = G[j * AAMAX + j] + reg - s;
                if (!(dj > 0.0)) {
                    ok = false;
                    break;
                }
                const double ljj = sqrt(dj);
                if (lane > j && lane < k) {
                    double e = G[lane * AAMAX + j];
                    for (int p = 0; p < j; ++p) e -= L[lane * AAMAX + p] * L[j * AAMAX + p];
                    L[lane * AAMAX + j] = e / ljj;
                }
                if (lane == 0) L[j * AAMAX + j] = ljj;
                __syncwarp();
            }
            __syncwarp();
        }
        if (lane == 0) {
            if (ok) {
                for (int i = 0; i < k; ++i) {
                    double e = rhs[i];
                    for (int p = 0; p < i; ++p) e -= L[i * AAMAX + p] * t[p];
                    t[i] = e / L[i * AAMAX + i];
                }
                for (int i = k - 1; i >= 0; --i) {
                    double e = t[i];
                    for (int p = i + 1; p < k; ++p) e -= L[p * AAMAX + i] * t[p];
                    t[i] = e / L[i * AAMAX + i];
                }
            }
            ok_s = ok ? 1 : 0;
        }
    }
    __syncthreads();
    return ok_s != 0;
}

struct DirState {
    int count;     // stored pairs
    long long inserted;
};

// Anderson's acceleration: d = -Ru - (Z - Xi) t, t = argmin ||Xi t - Ru|| by
// regularised normal equations; ring buffer of the last mem pairs.
template <typename T, class Team>
__device__ void aa_direction(Team& tm, const DevProb<T>& P, const DevWork<T>& W, const DevSettings& S,
                             bool have_pair, double nz2, DirState& ds, double* G, double* sm_rhs, double* sm_L,
                             double* sm_t)
{
    const int nm = P.n + P.m;
    const int mem = S.mem;
    if (have_pair && mem > 0 && nz2 > 0.0) {
        const int slot = (int)(ds.inserted % mem);
        HV<T> Zs = col(W.Zv, W.Zt, slot, nm), Xs = col(W.Xv, W.Xt, slot, nm);
        for (int i = tm.rank(); i < nm; i += tm.size()) {
            Zs.v[i] = W.zp.v[i];
            Xs.v[i] = W.xip.v[i];
        }
        if (tm.leader()) {
            *Zs.t = *W.zp.t;
            *Xs.t = *W.xip.t;
        }
        ds.inserted++;
        if (ds.count < mem) ds.count++;
        tm.sync();
        // new Gram row: <xi_slot, xi_j> for all stored j, in chunks of 8
        for (int j0 = 0; j0 < ds.count; j0 += 8) {
            T a[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) a[q] = 0;
            for (int i = tm.rank(); i < nm; i += tm.size()) {
                const T xs = Xs.v[i];
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    if (j0 + q < ds.count) a[q] += xs * W.Xv[(size_t)(j0 + q) * nm + i];
            }
            double red[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) red[q] = (double)a[q];
            if (tm.leader()) {
                const double xt = *Xs.t;
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    if (j0 + q < ds.count) red[q] += xt * W.Xt[j0 + q];
            }
            tm.reduce(red);
            if (threadIdx.x == 0) {
                for (int q = 0; q < 8 && j0 + q < ds.count; ++q) {
                    G[slot * AAMAX + j0 + q] = red[q];
                    G[(j0 + q) * AAMAX + slot] = red[q];
                }
            }
        }
    }
    const int k = ds.count;
    if (k == 0) {
        for (int i = tm.rank(); i < nm; i += tm.size()) W.d.v[i] = -W.Ru.v[i];
        if (tm.leader()) *W.d.t = -*W.Ru.t;
        tm.sync();
        return;
    }
    // rhs_j = <xi_j, Ru>
    for (int j0 = 0; j0 < k; j0 += 8) {
        T a[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) a[q] = 0;
        for (int i = tm.rank(); i < nm; i += tm.size()) {
            const T r = W.Ru.v[i];
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (j0 + q < k) a[q] += r * W.Xv[(size_t)(j0 + q) * nm + i];
        }
        double red[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) red[q] = (double)a[q];
        if (tm.leader()) {
            const double rt = *W.Ru.t;
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (j0 + q < k) red[q] += rt * W.Xt[j0 + q];
        }
        tm.reduce(red);
        if (threadIdx.x == 0)
            for (int q = 0; q < 8 && j0 + q < k; ++q) sm_rhs[j0 + q] = red[q];
    }
    __syncthreads();
    double tr = 0.0;
    for (int j = 0; j < k; ++j) tr += G[j * AAMAX + j];
    bool ok = false;
    if (tr > 0.0) ok = small_chol(G, sm_rhs, sm_L, sm_t, k, S.aa_reg * tr / k);
    // d = -Ru - sum_j t_j (Z_j - Xi_j)
    for (int i = tm.rank(); i < nm; i += tm.size()) {
        T di = -W.Ru.v[i];
        if (ok)
            for (int j = 0; j < k; ++j) di -= (T)sm_t[j] * (W.Zv[(size_t)j * nm + i] - W.Xv[(size_t)j * nm + i]);
        W.d.v[i] = di;
    }
    if (tm.leader()) {
        double di = -*W.Ru.t;
        if (ok)
            for (int j = 0; j < k; ++j) di -= sm_t[j] * (W.Zt[j] - W.Xt[j]);
        *W.d.t = di;
    }
    tm.sync();
}

// Anderson's acceleration with the least squares min ||Xi t - Ru|| solved
// through Xi = Q R (Sec. 4.4: an updated QR factorisation in place of the
// normal equations).  Q's columns are kept oldest first in W.Qv/W.Qt, R
// (upper triangular, row stride AAMAX) in the CTA's shared array G; Z and Xi
// stay in their ring slots (the oldest pair at (inserted - count) mod mem).
//  - a full window drops its oldest pair: R without its first column is upper
//    Hessenberg; Givens rotations (j, j+1), j = 0..k-2, restore the triangle
//    (computed by thread 0 of every CTA from identical data) and one pass
//    applies them to Q's columns, carrying column j+1 in a register;
//  - a new pair enters by two rounds of classical Gram-Schmidt (dots in
//    chunks of 8 per reduction); a remainder below 1e-14 ||xi|| is rank
//    deficient and the pair is not stored;
//  - t solves R t = Q^T Ru, d = -Ru - sum_j t_j (Z_j - Xi_j).
template <typename T, class Team>
__device__ void aa_qr_direction(Team& tm, const DevProb<T>& P, const DevWork<T>& W, const DevSettings& S,
                                bool have_pair, double nz2, DirState& ds, double* R, double* sm_h, double* sm_cs,
                                double* sm_t)
{
    const int nm = P.n + P.m;
    const int mem = S.mem;
    auto qcol = [&](int j) { return W.Qv + (size_t)j * nm; };
    auto slot_of = [&](int j) { return (int)((ds.inserted - ds.count + j) % mem); };  // ring slot of pair j
    if (have_pair && mem > 0 && nz2 > 0.0) {
        if (ds.count == mem) {
            const int k = ds.count;
            if (threadIdx.x == 0) {
                for (int j = 0; j + 1 < k; ++j) {
                    const double a = R[j * AAMAX + j + 1], b = R[(j + 1) * AAMAX + j + 1];
                    const double h = hypot(a, b);
                    const double c = h > 0.0 ? a / h : 1.0, sn = h > 0.0 ? b / h : 0.0;
                    for (int col = j + 1; col < k; ++col) {
                        const double x = R[j * AAMAX + col], y = R[(j + 1) * AAMAX + col];
                        R[j * AAMAX + col] = c * x + sn * y;
                        R[(j + 1) * AAMAX + col] = -sn * x + c * y;
                    }
                    sm_cs[2 * j] = c;
                    sm_cs[2 * j + 1] = sn;
                }
                for (int r = 0; r + 1 < k; ++r)
                    for (int col = 0; col + 1 < k; ++col) R[r * AAMAX + col] = col >= r ? R[r * AAMAX + col + 1] : 0.0;
                for (int col = 0; col < k; ++col) R[(k - 1) * AAMAX + col] = 0.0;
            }
            __syncthreads();
            for (int i = tm.rank(); i < nm; i += tm.size()) {
                T x = qcol(0)[i];
                for (int j = 0; j + 1 < k; ++j) {
                    const T y = qcol(j + 1)[i];
                    const T c = (T)sm_cs[2 * j], sn = (T)sm_cs[2 * j + 1];
                    qcol(j)[i] = c * x + sn * y;
                    x = -sn * x + c * y;
                }
            }
            if (tm.leader()) {
                double x = W.Qt[0];
                for (int j = 0; j + 1 < k; ++j) {
                    const double y = W.Qt[j + 1];
                    W.Qt[j] = sm_cs[2 * j] * x + sm_cs[2 * j + 1] * y;
                    x = -sm_cs[2 * j + 1] * x + sm_cs[2 * j] * y;
                }
            }
            ds.count = k - 1;
            tm.sync();
        }
        // append xi: the new column k of Q is built in place
        const int k = ds.count;
        const T* xi = W.xip.v;
        const double xit = *W.xip.t;
        T* w = qcol(k);
        double nxi2 = 0.0;
        for (int round = 0; round < 2; ++round) {
            const T* src = round == 0 ? xi : w;
            const double srct = round == 0 ? xit : W.Qt[k];
            // h_j = <q_j, src>, chunks of 8 (the first chunk of round 0 also reduces ||xi||^2)
            for (int j0 = 0; j0 < (k > 0 ? k : 1); j0 += 8) {
                T a[8];
                T x2 = 0;
#pragma unroll
                for (int q = 0; q < 8; ++q) a[q] = 0;
                for (int i = tm.rank(); i < nm; i += tm.size()) {
                    const T v = src[i];
                    if (round == 0 && j0 == 0) x2 += v * v;
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        if (j0 + q < k) a[q] += qcol(j0 + q)[i] * v;
                }
                double red[9];
#pragma unroll
                for (int q = 0; q < 8; ++q) red[q] = (double)a[q];
                red[8] = (double)x2;
                if (tm.leader()) {
                    if (round == 0 && j0 == 0) red[8] += srct * srct;
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        if (j0 + q < k) red[q] += W.Qt[j0 + q] * srct;
                }
                tm.reduce(red);
                if (round == 0 && j0 == 0) nxi2 = red[8];
                if (threadIdx.x == 0)
                    for (int q = 0; q < 8 && j0 + q < k; ++q) sm_h[j0 + q] = red[q];
            }
            __syncthreads();
            // w = src - Q h (and ||w||^2 after the second round); R's new column accumulates h
            T ww = 0;
            for (int i = tm.rank(); i < nm; i += tm.size()) {
                T v = src[i];
                for (int j = 0; j < k; ++j) v -= (T)sm_h[j] * qcol(j)[i];
                w[i] = v;
                ww += v * v;
            }
            double red2[1] = {(double)ww};
            if (tm.leader()) {
                double v = srct;
                for (int j = 0; j < k; ++j) v -= sm_h[j] * W.Qt[j];
                W.Qt[k] = v;
                red2[0] += v * v;
            }
            tm.reduce(red2);
            if (threadIdx.x == 0)
                for (int j = 0; j < k; ++j) R[j * AAMAX + k] = (round == 0 ? 0.0 : R[j * AAMAX + k]) + sm_h[j];
            if (round == 1 && threadIdx.x == 0) sm_t[0] = red2[0];  // ||w||^2 after the second round
            __syncthreads();
        }
        const double rkk = sqrt(sm_t[0]);
        if (rkk > 1e-14 * sqrt(nxi2)) {
            const T inv = (T)(1.0 / rkk);
            const int slot = (int)(ds.inserted % mem);
            HV<T> Zs = col(W.Zv, W.Zt, slot, nm), Xs = col(W.Xv, W.Xt, slot, nm);
            for (int i = tm.rank(); i < nm; i += tm.size()) {
                w[i] *= inv;
                Zs.v[i] = W.zp.v[i];
                Xs.v[i] = xi[i];
            }
            if (tm.leader()) {
                W.Qt[k] /= rkk;
                *Zs.t = *W.zp.t;
                *Xs.t = xit;
            }
            if (threadIdx.x == 0) R[k * AAMAX + k] = rkk;
            ds.inserted++;
            ds.count++;
        }
        tm.sync();
    }
    const int k = ds.count;
    if (k == 0) {
        for (int i = tm.rank(); i < nm; i += tm.size()) W.d.v[i] = -W.Ru.v[i];
        if (tm.leader()) *W.d.t = -*W.Ru.t;
        tm.sync();
        return;
    }
    // Q^T Ru, then R t = Q^T Ru by back substitution (thread 0 of every CTA)
    for (int j0 = 0; j0 < k; j0 += 8) {
        T a[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) a[q] = 0;
        for (int i = tm.rank(); i < nm; i += tm.size()) {
            const T r = W.Ru.v[i];
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (j0 + q < k) a[q] += qcol(j0 + q)[i] * r;
        }
        double red[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) red[q] = (double)a[q];
        if (tm.leader()) {
            const double rt = *W.Ru.t;
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (j0 + q < k) red[q] += W.Qt[j0 + q] * rt;
        }
        tm.reduce(red);
        if (threadIdx.x == 0)
            for (int q = 0; q < 8 && j0 + q < k; ++q) sm_t[j0 + q] = red[q];
    }
    if (threadIdx.x == 0)
        for (int j = k - 1; j >= 0; --j) {
            double e = sm_t[j];
            for (int p = j + 1; p < k; ++p) e -= R[j * AAMAX + p] * sm_t[p];
            sm_t[j] = e / R[j * AAMAX + j];
        }
    __syncthreads();
    for (int i = tm.rank(); i < nm; i += tm.size()) {
        T di = -W.Ru.v[i];
        for (int j = 0; j < k; ++j) {
            const size_t o = (size_t)slot_of(j) * nm + i;
            di -= (T)sm_t[j] * (W.Zv[o] - W.Xv[o]);
        }
        W.d.v[i] = di;
    }
    if (tm.leader()) {
        double di = -*W.Ru.t;
        for (int j = 0; j < k; ++j) di -= sm_t[j] * (W.Zt[slot_of(j)] - W.Xt[slot_of(j)]);
        *W.d.t = di;
    }
    tm.sync();
}

// Restarted Broyden, Algorithm 2 (readings: m' = stored pairs; restart when
// m' = mem empties the buffers without storing the current pair; the
// denominator of z~ is <z, H xi~>; sgn(0) = 1).
template <typename T, class Team>
__device__ void rb_direction(Team& tm, const DevProb<T>& P, const DevWork<T>& W, const DevSettings& S,
                             bool have_pair, double nz2, DirState& ds)
{
    const int nm = P.n + P.m;
    HV<T> d = W.d, zt = W.zt, Ru = W.Ru, z = W.zp, xi = W.xip;
    if (!have_pair || !(nz2 > 0.0)) {
        for (int i = tm.rank(); i < nm; i += tm.size()) d.v[i] = -Ru.v[i];
        if (tm.leader()) *d.t = -*Ru.t;
        tm.sync();
        return;
    }
    const int cnt = ds.count;
    // pass 0: d = -Ru, zt = xi; dots with the first stored z (or with z when none)
    {
        const T* z0 = cnt > 0 ? W.Zv : z.v;
        const double z0t = cnt > 0 ? W.Zt[0] : *z.t;
        T a = 0, b = 0;
        for (int i = tm.rank(); i < nm; i += tm.size()) {
            const T di = -Ru.v[i], zi = xi.v[i];
            d.v[i] = di;
            zt.v[i] = zi;
            a += z0[i] * zi;
            b += z0[i] * di;
        }
        double red[2] = {(double)a, (double)b};
        if (tm.leader()) {
            *d.t = -*Ru.t;
            *zt.t = *xi.t;
            red[0] += z0t * *xi.t;
            red[1] += z0t * (-*Ru.t);
        }
        tm.reduce(red);
        double ca = red[0], cb = red[1];
        // stored pairs: zt += <z^k, zt> z~^k ; d += <z^k, d> z~^k, dots for the next pair fused
        for (int k = 0; k < cnt; ++k) {
            const T* zk1 = (k + 1 < cnt) ? W.Zv + (size_t)(k + 1) * nm : z.v;
            const double zk1t = (k + 1 < cnt) ? W.Zt[k + 1] : *z.t;
            const T* ztk = W.Xv + (size_t)k * nm;
            const T ta = (T)ca, tb = (T)cb;
            T a2 = 0, b2 = 0;
            for (int i = tm.rank(); i < nm; i += tm.size()) {
                const T zti = zt.v[i] + ta * ztk[i];
                const T di = d.v[i] + tb * ztk[i];
                zt.v[i] = zti;
                d.v[i] = di;
                a2 += zk1[i] * zti;
                b2 += zk1[i] * di;
            }
            double red2[2] = {(double)a2, (double)b2};
            if (tm.leader()) {
                const double zti = *zt.t + ca * W.Xt[k];
                const double di = *d.t + cb * W.Xt[k];
                *zt.t = zti;
                *d.t = di;
                red2[0] += zk1t * zti;
                red2[1] += zk1t * di;
            }
            tm.reduce(red2);
            ca = red2[0];
            cb = red2[1];
        }
        // now ca = <z, H xi>, cb = <z, H(-r)>
        const double gamma = ca / nz2;
        const double sg = gamma >= 0.0 ? 1.0 : -1.0;
        const double theta = fabs(gamma) >= S.thetabar ? 1.0 : (1.0 - sg * S.thetabar) / (1.0 - gamma);
        // z~ = (z - ((1-theta) z + theta H xi)) / <z, (1-theta) z + theta H xi>
        const double den = (1.0 - theta) * nz2 + theta * ca;
        const bool store = cnt < S.mem;
        T* ztn = W.Xv + (size_t)cnt * nm;  // used only when storing
        T* zsn = W.Zv + (size_t)cnt * nm;
        const T f1 = (T)(theta / den);
        const T tcb = (T)cb;
        for (int i = tm.rank(); i < nm; i += tm.size()) {
            const T zi = z.v[i];
            const T zn = f1 * (zi - zt.v[i]);
            d.v[i] += tcb * zn;
            if (store) {
                ztn[i] = zn;
                zsn[i] = zi;
            }
        }
        if (tm.leader()) {
            const double zi = *z.t;
            const double zn = (theta / den) * (zi - *zt.t);
            *d.t += cb * zn;
            if (store) {
                W.Xt[cnt] = zn;
                W.Zt[cnt] = zi;
            }
        }
        tm.sync();
        ds.count = store ? cnt + 1 : 0;
    }
}

// ---------------------------------------------------------------------------
// outputs (Sec. 3.1 recovery rules)
// ---------------------------------------------------------------------------
template <typename T, class Team>
__device__ void write_outputs(Team& tm, const DevProb<T>& P, const DevWork<T>& W, int status, const TermOut& o)
{
    const int n = P.n, m = P.m;
    const double taub = *W.ub.t;
    const T* chib = W.ub.v;
    const T* psib = W.ub.v + n;
    for (int i = tm.rank(); i < m; i += tm.size()) {
        const double sig = (double)psib[i] - 2.0 * (double)W.ut.v[n + i] + (double)W.u.v[n + i];
        double yv, sv;
        if (status == ST_INFEASIBLE) {
            yv = (double)psib[i] / (-o.bpsi);
            sv = NAN;
        } else if (status == ST_UNBOUNDED) {
            yv = NAN;
            sv = sig / (-o.cchi);
        } else if (taub > 0.0) {
            yv = (double)psib[i] / taub;
            sv = sig / taub;
        } else {
            yv = NAN;
            sv = NAN;
        }
        W.y_out[i] = yv;
        W.s_out[i] = sv;
    }
    for (int j = tm.rank(); j < n; j += tm.size()) {
        double xv;
        if (status == ST_INFEASIBLE) xv = NAN;
        else if (status == ST_UNBOUNDED) xv = (double)chib[j] / (-o.cchi);
        else if (taub > 0.0) xv = (double)chib[j] / taub;
        else xv = NAN;
        W.x_out[j] = xv;
    }
    for (int i = tm.rank(); i < n + m; i += tm.size()) W.u_out[i] = (double)W.u.v[i];
    if (tm.leader()) W.u_out[n + m] = *W.u.t;
}

// ---------------------------------------------------------------------------
// Algorithm 1 with the linearity trick (Sec. 4.2).  Readings where the paper
// is silent: u0 = (0,0,1) unless warm; q^nu with nu the outer index; at most
// ls_max halvings, then alpha = 0 (the KM step); ||Rw|| = 0 is accepted as
// K1; secant pair z = w - u, xi = Rw - Ru of the last evaluated w; after K2
// the new u~ is solved from the new u; termination before the direction.
// ---------------------------------------------------------------------------
// Returns 1 (and writes no result) when a warm start is abandoned for the
// cold start; the caller then runs it again cold with the counts carried over.
template <typename T, class Team>
__device__ int superscs(Team& tm, const DevProb<T>& P, const DevWork<T>& W, const DevSettings& S, double* G,
                        double* sm_rhs, double* sm_L, double* sm_t, unsigned char* psd, bool use_warm,
                        int iter_base, long long cg_base, int& iters_out, long long& cg_out)
{
    const int n = P.n, m = P.m, nm = n + m;
    const double hg = W.st->hg;
    long long cg_total = cg_base;
    int k0 = 0, k1 = 0, k2 = 0, bt = 0;
    const double deadline = S.time_limit_ns > 0.0 ? (double)gtimer() + S.time_limit_ns : 0.0;
    // CG warm starts from zero unless the previous phase handed them over
    if (!S.keep_ws)
        for (int i = tm.rank(); i < n; i += tm.size()) {
            W.ws[0][i] = T(0);
            W.ws[1][i] = T(0);
        }
    // the PSD eigensolves' warm starts live within one solve: a solve neither depends on nor
    // profits from an earlier one (the flags are read after the next team barrier)
    if (W.psd_vok)
        for (int k = tm.rank(); k < P.ns; k += tm.size()) W.psd_vok[k] = 0;
    if (tm.leader() && iter_base == 0) {
        W.st->mat_passes = 0;
        W.st->mat_passes_ir = 0;
        W.st->cg_iters_ir = 0;
        W.st->ir_sweeps = 0;
        for (int k = 0; k < 5; ++k) W.st->part_ns[k] = 0.0;
        W.st->psd_resid = 0.0;
        W.st->psd_redo = 0;
        W.st->fallback = 0;
    }
    // residual of the cold start, the yardstick of the warm-start fallback
    double nRu_cold = INFINITY;
    const bool watch = use_warm && S.warm_fallback > 0;
    if (watch) {
        for (int i = tm.rank(); i < nm; i += tm.size()) W.u.v[i] = T(0);
        if (tm.leader()) *W.u.t = 1.0;
        tm.sync();
        cg_total += linsys(tm, P, W, W.u, W.ut, 0, S.cg_rtol, S.cg_max, hg, 0.0, S.refine != 0);
        OpResidual<T> op{W.u, W.ut, W.ub, W.Ru, T(0)};
        project_pass(tm, P, op, psd, PsdCheck{&W.st->psd_resid, &W.st->psd_redo, S.psd_tol, W.psd_v, P.v_off, W.psd_vok});
        double red[1] = {(double)op.acc0};
        tm.reduce(red);
        nRu_cold = sqrt(red[0]);
    }
    // u0
    for (int i = tm.rank(); i < nm; i += tm.size()) W.u.v[i] = use_warm ? (T)W.warm[i] : T(0);
    if (tm.leader()) *W.u.t = use_warm ? W.warm[nm] : 1.0;
    tm.sync();
    cg_total += linsys(tm, P, W, W.u, W.ut, 0, S.cg_rtol, S.cg_max, hg, 0.0, S.refine != 0);
    double nRu;
    {
        OpResidual<T> op{W.u, W.ut, W.ub, W.Ru, T(0)};
        project_pass(tm, P, op, psd, PsdCheck{&W.st->psd_resid, &W.st->psd_redo, S.psd_tol, W.psd_v, P.v_off, W.psd_vok});
        double red[1] = {(double)op.acc0};
        tm.reduce(red);
        nRu = sqrt(red[0]);
    }
    double eta0 = nRu, r_safe = nRu, eta = nRu, nz2 = 0.0;
    bool have_pair = false;
    DirState ds{0, 0};
    int nu_q = 0;  // outer iterations before this launch (the exponent of q^nu continues)
    if (S.resume && W.res->valid) {
        // continue the FP32 phase's iteration: its direction memory (Z, Xi and
        // the pending secant pair were widened by the hand-over), the Gram
        // matrix, and the K0/K1 references; u~, u_ and Ru were just evaluated
        // in this precision at the handed-over u
        const Resume* R = W.res;
        eta0 = R->eta0;
        eta = R->eta;
        r_safe = R->r_safe;
        nz2 = R->nz2;
        have_pair = R->have_pair != 0;
        ds.count = R->count;
        ds.inserted = R->inserted;
        nu_q = R->nu;
        if (S.direction == 0 || S.direction == 3)  // the Gram matrix, or R of the QR variant
            for (int i = threadIdx.x; i < AAMAX * AAMAX; i += blockDim.x) G[i] = R->G[i];
        __syncthreads();
    }
    int status = ST_MAX_ITERS;
    TermOut to;
    to.pr = to.dr = to.gap = to.ic = to.uc = INFINITY;
    to.pobj = to.dobj = NAN;
    to.bpsi = to.cchi = 0.0;
    double best_kkt = INFINITY;
    int best_it = 0;
    const int check_every = S.check_every > 0 ? S.check_every : 1;
    bool need_final_check = true;
    int nu;
    for (nu = 0; nu < S.max_iters - iter_base; ++nu) {
        if (tm.aborted()) break;
        if (watch && nu == S.warm_fallback && !(nRu < nRu_cold)) {
            iters_out = iter_base + nu;
            cg_out = cg_total;
            return 1;
        }
        if (!isfinite(nRu)) {
            if (watch) {
                iters_out = iter_base + nu;
                cg_out = cg_total;
                return 1;
            }
            status = ST_NUMERICAL;
            break;
        }
        unsigned long long tp = tm.leader() ? gtimer() : 0ull;  // start of this part
        auto part_end = [&](int k) {
            if (tm.leader()) {
                const unsigned long long t = gtimer();
                W.st->part_ns[k] += (double)(t - tp);
                tp = t;
            }
        };
        if (nu % check_every == 0) {
            const int st = termination(tm, P, W, S.eps, deadline, to);
            part_end(0);
            if (st != 0) {
                status = st;
                need_final_check = false;
                break;
            }
            if (to.time_up) {
                status = ST_TIME_LIMIT;
                need_final_check = false;
                break;
            }
            if (S.switch_kkt > 0.0 && fmax(to.pr, fmax(to.dr, to.gap)) <= S.switch_kkt) {
                status = ST_STALLED;  // hand over to the FP64 phase
                need_final_check = false;
                break;
            }
            if (S.stall_iters > 0) {
                // FP32 phase of SCS_MIXED: stop once ||Ru|| has not dropped 10% below
                // its best value for stall_iters iterations (the FP32 floor).  While
                // tau_ = 0 the residuals of Sec. 4.3 are undefined and the iterate is
                // still turning away from the tau axis, where ||Ru|| can plateau
                // without any floor being reached; a plateau with max(pr, dr, gap) still
                // above 100 times the hand-over level is not the FP32 floor either (the
                // FP32 phases measured here level off within a few times of it).  In
                // both cases the window is five times longer.
                const double kkt = fmax(to.pr, fmax(to.dr, to.gap));
                const bool far = !isfinite(to.pr) || (S.switch_kkt > 0.0 && kkt > 100.0 * S.switch_kkt);
                const int window = (S.stall_after_tau && far) ? 5 * S.stall_iters : S.stall_iters;
                if (nRu < 0.9 * best_kkt) {
                    best_kkt = nRu;
                    best_it = nu;
                } else if (nu - best_it >= window) {
                    status = ST_STALLED;
                    need_final_check = false;
                    break;
                }
            }
        }
        // direction d (Sec. 4.4)
        part_end(4);
        if (S.direction == 0)
            aa_direction(tm, P, W, S, have_pair, nz2, ds, G, sm_rhs, sm_L, sm_t);
        else if (S.direction == 3)
            aa_qr_direction(tm, P, W, S, have_pair, nz2, ds, G, sm_rhs, sm_L, sm_t);
        else if (S.direction == 1)
            rb_direction(tm, P, W, S, have_pair, nz2, ds);
        else {
            for (int i = tm.rank(); i < nm; i += tm.size()) W.d.v[i] = T(0);
            if (tm.leader()) *W.d.t = 0.0;
            tm.sync();
        }
        part_end(1);
        const double atol = S.cg_adapt > 0.0 ? S.cg_adapt * nRu : 0.0;
        cg_total += linsys(tm, P, W, W.d, W.dt, 1, S.cg_rtol, S.cg_max, hg, atol, S.refine != 0);
        double lin0 = 0.0;  // linear-solve time so far (a K2 step adds its own below)
        if (tm.leader()) {
            tp = gtimer();  // the linear solve timed itself
            lin0 = W.st->part_ns[2];
        }
        if (nRu <= S.c0 * eta) {
            // K0
            eta = nRu;
            OpK0<T> op{W.u, W.ut, W.ub, W.Ru, W.d, W.dt, W.zp, W.xip, T(0), T(0)};
            project_pass(tm, P, op, psd, PsdCheck{&W.st->psd_resid, &W.st->psd_redo, S.psd_tol, W.psd_v, P.v_off, W.psd_vok});
            double red[2] = {(double)op.acc0, (double)op.acc1};
            tm.reduce(red);
            nRu = sqrt(red[0]);
            nz2 = red[1];
            ++k0;
        } else {
            double alpha = 1.0;
            for (int ls = 0; ls <= S.ls_max; ++ls) {
                if (ls == S.ls_max) alpha = 0.0;
                OpTrial<T> op{W.u, W.ut, W.d, W.dt, W.wb, W.Rw, alpha, T(0), T(0)};
                project_pass(tm, P, op, psd, PsdCheck{&W.st->psd_resid, &W.st->psd_redo, S.psd_tol, W.psd_v, P.v_off, W.psd_vok});
                double red[2] = {(double)op.acc0, (double)op.acc1};
                tm.reduce(red);
                const double nRw = sqrt(red[0]);
                const double rho = red[1];
                if ((nRu <= r_safe && nRw <= S.c1 * nRu) || nRw == 0.0) {
                    // K1: u <- w, reuse w~, w_, Rw
                    r_safe = nRw + pow(S.q, (double)(nu + nu_q)) * eta0;
                    const T ta = (T)alpha;
                    T zz = 0;
                    for (int i = tm.rank(); i < nm; i += tm.size()) {
                        const T di = ta * W.d.v[i];
                        W.u.v[i] += di;
                        W.ut.v[i] += ta * W.dt.v[i];
                        W.ub.v[i] = W.wb.v[i];
                        W.zp.v[i] = di;
                        W.xip.v[i] = W.Rw.v[i] - W.Ru.v[i];
                        W.Ru.v[i] = W.Rw.v[i];
                        zz += di * di;
                    }
                    double red2[1] = {(double)zz};
                    if (tm.leader()) {
                        const double di = alpha * *W.d.t;
                        *W.u.t += di;
                        *W.ut.t += alpha * *W.dt.t;
                        *W.ub.t = *W.wb.t;
                        *W.zp.t = di;
                        *W.xip.t = *W.Rw.t - *W.Ru.t;
                        *W.Ru.t = *W.Rw.t;
                        red2[0] += di * di;
                    }
                    tm.reduce(red2);
                    nz2 = red2[0];
                    nRu = nRw;
                    ++k1;
                    break;
                } else if (rho >= S.sigma * nRu * nRw) {
                    // K2: u <- u - lambda rho / ||Rw||^2 Rw, then a fresh u~ solve
                    const double coef = S.lambda * rho / (nRw * nRw);
                    const T ta = (T)alpha, tc = (T)coef;
                    T zz = 0;
                    for (int i = tm.rank(); i < nm; i += tm.size()) {
                        const T di = ta * W.d.v[i];
                        W.zp.v[i] = di;
                        W.xip.v[i] = W.Rw.v[i] - W.Ru.v[i];
                        W.u.v[i] -= tc * W.Rw.v[i];
                        zz += di * di;
                    }
                    double red2[1] = {(double)zz};
                    if (tm.leader()) {
                        const double di = alpha * *W.d.t;
                        *W.zp.t = di;
                        *W.xip.t = *W.Rw.t - *W.Ru.t;
                        *W.u.t -= coef * *W.Rw.t;
                        red2[0] += di * di;
                    }
                    tm.reduce(red2);
                    nz2 = red2[0];
                    cg_total += linsys(tm, P, W, W.u, W.ut, 0, S.cg_rtol, S.cg_max, hg, atol, S.refine != 0);
                    OpResidual<T> opr{W.u, W.ut, W.ub, W.Ru, T(0)};
                    project_pass(tm, P, opr, psd, PsdCheck{&W.st->psd_resid, &W.st->psd_redo, S.psd_tol, W.psd_v, P.v_off, W.psd_vok});
                    double red3[1] = {(double)opr.acc0};
                    tm.reduce(red3);
                    nRu = sqrt(red3[0]);
                    ++k2;
                    break;
                }
                alpha *= 0.5;
                ++bt;
            }
        }
        have_pair = true;
        // the rest of the step (K0, line search, projections; K2's linear solve timed itself)
        if (tm.leader()) {
            const unsigned long long t = gtimer();
            W.st->part_ns[4] += (double)(t - tp) - (W.st->part_ns[2] - lin0);
        }
    }
    if (need_final_check && !tm.aborted()) {
        const int st = termination(tm, P, W, S.eps, 0.0, to);
        if (st != 0 && status != ST_NUMERICAL) status = st;
    }
    if (S.save_state) {
        // the loop state for a continuation in FP64 (the vectors stay in W)
        Resume* R = W.res;
        if (tm.leader()) {
            R->valid = 1;
            R->count = ds.count;
            R->inserted = ds.inserted;
            R->have_pair = have_pair ? 1 : 0;
            R->nu = nu + nu_q;
            R->eta = eta;
            R->eta0 = eta0;
            R->r_safe = r_safe;
            R->nz2 = nz2;
        }
        if (tm.block() == 0 && (S.direction == 0 || S.direction == 3))
            for (int i = threadIdx.x; i < AAMAX * AAMAX; i += blockDim.x) R->G[i] = G[i];
    }
    write_outputs(tm, P, W, status, to);
    iters_out = iter_base + nu;
    cg_out = cg_total;
    if (tm.leader()) {
        DevState* st = W.st;
        st->status = status;
        st->iters = iter_base + nu;
        st->k0 = k0;
        st->k1 = k1;
        st->k2 = k2;
        st->backtracks = bt;
        st->cg_iters = cg_total;
        st->pr = to.pr;
        st->dr = to.dr;
        st->gap = to.gap;
        st->ic = to.ic;
        st->uc = to.uc;
        st->nRu = nRu;
        if (status == ST_SOLVED || status == ST_MAX_ITERS || status == ST_TIME_LIMIT || status == ST_STALLED) {
            st->pobj = to.pobj;
            st->dobj = to.dobj;
        } else {
            st->pobj = NAN;
            st->dobj = NAN;
        }
    }
    return 0;
}

// ---------------------------------------------------------------------------
// one entry for every mode
// ---------------------------------------------------------------------------
template <typename T, class Team>
__device__ void run_mode(Team& tm, const DevProb<T>& P, const DevWork<T>& W, const DevSettings& S, int mode, int slot,
                         double* G, double* sm_rhs, double* sm_L, double* sm_t, unsigned char* psd)
{
    const int n = P.n, m = P.m, nm = n + m;
    if (mode == MODE_FACTOR) {
        if constexpr (!Team::kGrid) {
            if (W.dinv) direct_setup(tm, P, W, G, sm_L);
        }
        return;
    }
    if (mode == MODE_SETUP) {
        // g = M^{-1}(c, b) from a zero start; ws[0] is zero on entry and left zero
        T* x = W.ws[0];
        double htp;
        const int it = minv(tm, P, W, P.c, P.b, x, S.cg_rtol, S.cg_max, htp);
        for (int i = tm.rank(); i < n; i += tm.size()) {
            W.g[i] = x[i];
            x[i] = T(0);
        }
        for (int i = tm.rank(); i < m; i += tm.size()) W.g[n + i] = W.py[i];
        if (tm.leader()) {
            W.st->hg = htp;
            W.st->setup_cg = it;
        }
        tm.sync();
        return;
    }
    if (mode == MODE_SOLVE) {
        int its = 0;
        long long cgs = 0;
        if (superscs(tm, P, W, S, G, sm_rhs, sm_L, sm_t, psd, S.use_warm != 0, 0, 0, its, cgs)) {
            // the warm start did not beat the cold start's residual: restart cold
            superscs(tm, P, W, S, G, sm_rhs, sm_L, sm_t, psd, false, its, cgs, its, cgs);
            if (tm.leader()) W.st->fallback = 1;
        }
        return;
    }
    if (mode == MODE_RESID) {
        // Sec. 4.3 residuals of a caller's candidate: x = io_in[0,n), y = io_in[n,n+m),
        // s = io_out2[0,m); io_out[0..2] = pr, dr, gap (FP64 data only)
        if constexpr (sizeof(T) == sizeof(double)) {
            const T* xv = W.io_in;
            const T* yv = W.io_in + n;
            const T* sv = W.io_out2;
            T* tmv = W.tm;
            T* tnv = W.tn;
            spmv(tm, P.A, xv, [&](int i, T v) { tmv[i] = v; });
            spmv(tm, P.AT, yv, [&](int j, T v) { tnv[j] = v; });
            tm.sync();
            double a0 = 0, a1 = 0, a2 = 0, a3 = 0;
            for (int i = tm.rank(); i < m; i += tm.size()) {
                const double bi = ro(P.b + i);
                const double e = tmv[i] + sv[i] - bi;
                a0 += e * e;
                a3 += bi * yv[i];
            }
            for (int j = tm.rank(); j < n; j += tm.size()) {
                const double cj = ro(P.c + j);
                const double g = tnv[j] + cj;
                a1 += g * g;
                a2 += cj * xv[j];
            }
            double red[4] = {a0, a1, a2, a3};
            tm.reduce(red);
            if (tm.leader()) {
                W.io_out[0] = sqrt(red[0]) / (1.0 + P.nb);
                W.io_out[1] = sqrt(red[1]) / (1.0 + P.nc);
                W.io_out[2] = fabs(red[2] + red[3]) / (1.0 + fabs(red[2]) + fabs(red[3]));
            }
            tm.sync();
        }
        return;
    }
    if (mode == MODE_SPMV) {
        // sparse products in precision T.  slot 0: io_out = A io_in[0,n);
        // slot 1: io_out = A^T io_in[0,m); slot 2: io_out = A^T io_in[0,m) and
        // io_out2 = A^T io_out2[0,m) in one fused pass.  x is staged at u's
        // start, y at u + n (the offset the solver's psi part has), the second
        // y in tm.
        T* xv = W.u.v;
        T* yv = W.u.v + n;
        T* y2 = W.tm;
        if (slot == 0) {
            for (int j = tm.rank(); j < n; j += tm.size()) xv[j] = (T)W.io_in[j];
        } else {
            for (int i = tm.rank(); i < m; i += tm.size()) {
                yv[i] = (T)W.io_in[i];
                if (slot == 2) y2[i] = (T)W.io_out2[i];
            }
        }
        tm.sync();
        if (slot == 0) {
            spmv(tm, P.A, xv, [&](int i, T v) { W.io_out[i] = (double)v; });
        } else if (slot == 1) {
            spmv(tm, P.AT, yv, [&](int j, T v) { W.io_out[j] = (double)v; });
        } else {
            spmv2(tm, P.AT, yv, y2, [&](int j, T v1, T v2) {
                W.io_out[j] = (double)v1;
                W.io_out2[j] = (double)v2;
            });
        }
        tm.sync();
        return;
    }
    if (mode == MODE_PROFILE) {
        // device-side timing of the solver's building blocks on this problem:
        // io_out[0..4] = ns per A pass, A^T pass, grid barrier, 1-value
        // reduction, and one CG iteration (A pass, barrier, A^T pass with
        // three dots, reduction, update pass, barrier)
        const int reps = slot > 0 ? slot : 10;
        T* xv = W.cp;
        T* yv = W.tm;
        T* zv = W.tn;
        for (int j = tm.rank(); j < n; j += tm.size()) {
            xv[j] = T(1) / T(1 + (j % 7));
            W.cr[j] = xv[j];
        }
        tm.sync();
        double t[6];
        t[0] = (double)gtimer();
        for (int r = 0; r < reps; ++r) {
            spmv(tm, P.A, xv, [&](int i, T s) { yv[i] = s; });
            tm.sync();
        }
        t[1] = (double)gtimer();
        for (int r = 0; r < reps; ++r) {
            spmv(tm, P.AT, yv, [&](int j, T s) { zv[j] = s; });
            tm.sync();
        }
        t[2] = (double)gtimer();
        for (int r = 0; r < reps; ++r) tm.sync();
        t[3] = (double)gtimer();
        for (int r = 0; r < reps; ++r) {
            double v1[1] = {1.0};
            tm.reduce(v1);
        }
        t[4] = (double)gtimer();
        T* q = W.cq;
        T* rr = W.cr;
        for (int r = 0; r < reps; ++r) {
            spmv(tm, P.A, xv, [&](int i, T s) { yv[i] = s; });
            tm.sync();
            T pq = 0, rq = 0, qq = 0;
            spmv(tm, P.AT, yv, [&](int j, T s) {
                const T qj = xv[j] + s;
                q[j] = qj;
                pq += xv[j] * qj;
                rq += rr[j] * qj;
                qq += qj * qj;
            });
            double red[4] = {(double)pq, (double)rq, (double)qq, 0.0};
            tm.reduce(red);
            const T ta = (T)(1e-30 * red[0]);
            for (int j = tm.rank(); j < n; j += tm.size()) {
                const T pj = xv[j];
                W.ws[1][j] += ta * pj;
                const T rj = rr[j] - ta * q[j];
                rr[j] = rj;
                xv[j] = rj + ta * pj;
            }
            tm.sync();
        }
        t[5] = (double)gtimer();
        if (tm.leader())
            for (int k = 0; k < 5; ++k) W.io_out[k] = (t[k + 1] - t[k]) / reps;
        tm.sync();
        return;
    }
    // single operators: io_in (FP64, N) -> u (T), results to io_out / io_out2
    for (int i = tm.rank(); i < nm; i += tm.size()) W.u.v[i] = (T)W.io_in[i];
    if (tm.leader()) {
        *W.u.t = W.io_in[nm];
        W.st->psd_resid = 0.0;
        W.st->psd_redo = 0;
    }
    tm.sync();
    if (mode == MODE_LINSYS) {
        // slot 0 / 1: the CG warm start of u~ / d~; + 2: by iterative refinement (FP64 data only)
        linsys(tm, P, W, W.u, W.ut, slot & 1, S.cg_rtol, S.cg_max, W.st->hg, 0.0, (slot & 2) != 0);
        for (int i = tm.rank(); i < nm; i += tm.size()) W.io_out[i] = (double)W.ut.v[i];
        if (tm.leader()) W.io_out[nm] = *W.ut.t;
    } else if (mode == MODE_PROJECT) {
        OpProject<T> op{W.u.v, W.u.t, W.ub.v, W.ub.t};
        project_pass(tm, P, op, psd, PsdCheck{&W.st->psd_resid, &W.st->psd_redo, S.psd_tol, W.psd_v, P.v_off, W.psd_vok});
        tm.sync();
        for (int i = tm.rank(); i < nm; i += tm.size()) W.io_out[i] = (double)W.ub.v[i];
        if (tm.leader()) W.io_out[nm] = *W.ub.t;
    } else if (mode == MODE_APPLY_T) {
        linsys(tm, P, W, W.u, W.ut, 0, S.cg_rtol, S.cg_max, W.st->hg);
        OpResidual<T> op{W.u, W.ut, W.ub, W.Ru, T(0)};
        project_pass(tm, P, op, psd, PsdCheck{&W.st->psd_resid, &W.st->psd_redo, S.psd_tol, W.psd_v, P.v_off, W.psd_vok});
        tm.sync();
        for (int i = tm.rank(); i < nm; i += tm.size()) {
            W.io_out[i] = (double)W.u.v[i] - (double)W.Ru.v[i];
            W.io_out2[i] = (double)W.Ru.v[i];
        }
        if (tm.leader()) {
            W.io_out[nm] = *W.u.t - *W.Ru.t;
            W.io_out2[nm] = *W.Ru.t;
        }
    }
    tm.sync();
}

}  // namespace sscs
