// Reconstruction of an arbitrary list of states.
//
// §VII-C measures the time to reconstruct one million arbitrary output
// states.  For one state x, Eq. reconstruction is a scalar network: node j
// contributes the 4^{c_j} values T_j[.][x|out_j], and the plan's pairwise
// steps over the cut indices alone (a plan with no free qubits) contract it.
//
// Two forms, chosen from the plan:
//   fused      one persistent kernel runs every step of the single-state plan
//              on chip.  Its leaf operands are rows of per-node tables
//              Tt_j[x][cuts] (node tensors transposed so that the 4^{c_j}
//              values a state needs are one contiguous row, FP32, built by
//              the ingest kernel once per tensor version and small enough
//              to stay in L2); intermediates never leave shared memory.
//              Taken when every intermediate fits (e.g. 4^6 floats).
//   per-state  networks whose single-state intermediates are large (the
//              48-qubit QAOA network: 4^12 floats, GEMMs of 2^24..2^28
//              multiply-adds per state) run the single-state plan once per
//              state through the ordinary step kernels, with the state's
//              bits as the fixed bits.
//
// The fused form is bound by FP32 arithmetic, so it does no step twice for
// equal inputs: the result of a step depends only on the output bits of its
// own subcircuits, which many states of a list share (2^17 values for the
// costliest step of the 30-qubit grid, 10^6 states).  A shared subtree is
// chosen (build_program, below), the list is sorted by that subtree's bits (a
// counting sort), and a CTA walks a contiguous range of the sorted list: the
// shared steps run on all 256 threads when a bit they depend on has changed,
// and every state's remaining steps run on one warp, eight states at a time,
// with no barrier between them.  10^6 states of the 30-qubit
// grid, FP32 results: 45.1 -> 4.7 ms (the kernel 4.5 ms: 2.1 in the shared
// steps, 2.1 in the warps'; the sort 0.07 ms).
//
// A short list is bound by one state's latency, not by arithmetic, and the
// sort's launches alone cost 15 us: it takes a state per CTA, in list order, with
// the leaf operands staged or (where they don't fit, or are small) read from
// the tables.  1, 1000 and 16000 states of the 30-qubit grid: 16, 38 and 400 us,
// with a warp per state 59, 97 and 1094; one state of a network with a step of
// 2^8 x 2^4 results and K = 2^10: 86 us, by one warp 531.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <limits>
#include <string>
#include <vector>

#include "device_common.cuh"
#include "launch.h"

namespace tqc {

namespace {

constexpr int ST_THREADS = 256;
constexpr int ST_WARPS = ST_THREADS / 32;
constexpr int ST_WINDOW = 3 * ST_THREADS;  // a group (up to ST_THREADS states), the next one, and some
constexpr int ST_MAX_LEAVES = 16;
constexpr int ST_MAX_STEPS = ST_MAX_LEAVES - 1;
constexpr int ST_MAX_SMEM_FLOATS = 200 * 1024 / 4;
constexpr int ST_MAX_KEY_BITS = 22;  // counters of the sort: at most 2^22
constexpr int SCAN_PER_CTA = 4096;

struct SLeaf {
    const float *table;  // [2^{n_q}][4^{cuts}]: row x is the leaf operand of states with x|out_j = x
    int32_t row_log2;    // log2 of the row length (2 * cuts)
    int32_t y_off, n_q;  // x is bits y_off .. y_off + n_q of the permuted state y
};

// Where a step's operand is: a leaf's table row in global memory, the CTA's
// shared memory (a staged leaf, or the
// result of a shared step), or the warp's own part of it.
enum SrcKind { SRC_TABLE = 0, SRC_CTA = 1, SRC_WARP = 2 };

struct SStep {
    uint64_t mask;          // bits of y the result depends on
    int32_t a_leaf, b_leaf; // leaf index, or -1
    int32_t a_kind, b_kind; // SrcKind
    int32_t a_off, b_off;   // offsets (floats) of SRC_CTA / SRC_WARP operands
    int32_t mb, nb, kb;     // log2 of M, N, K
    uint32_t maskR, maskC;  // result-layout bits of the row / column index bits
    int32_t c_kb;           // log2 K of the step consuming the result; -1 for the final step
    int32_t c_off;          // the result's place: rows of 2^c_kb, padded
    int32_t lkl;            // log2 of the lanes sharing one output tile's K range (FP32 results)
    int32_t lkc;            // log2 of the multiply-adds in one partial sum (FP64 results)
    int32_t tab_off;        // result offsets of rows (M) then columns (N), in shared memory
};

struct SProgram {
    int32_t n_leaves, n_steps, n_shared;  // steps [0, n_shared) run per CTA, the rest per warp
    int32_t n_qubits;
    int32_t key_bits;       // the list is sorted by this many top bits of y (0: not sorted)
    int32_t one_each;       // states are taken one at a time (every step is a shared one)
    int32_t whole;          // no shared steps, and the CTA's warps work on one state together
    int32_t restage;        // leaf areas are reused: stage a step's leaves every time it runs
    uint64_t group_mask;    // bits of y the last shared step depends on
    int8_t perm[64];        // bit b of y is bit perm[b] of the state
    SLeaf leaf[ST_MAX_LEAVES];
    SStep step[ST_MAX_STEPS];
    int32_t warp_off, warp_floats;  // per-warp regions
    int32_t smem_floats;
};

// Row pitch of a [rows][K] operand in shared memory: K + 4 floats keeps
// 16-byte access and spreads rows over the banks.
__host__ __device__ __forceinline__ int pitch_of(int k) { return k >= 4 ? k + 4 : k; }

// Two FP32 multiply-adds per instruction (even and odd k in the two halves).
__device__ __forceinline__ void fma2(uint64_t &c, uint64_t a, uint64_t b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}
__device__ __forceinline__ float lo32(uint64_t c) { return __uint_as_float((uint32_t)c); }
__device__ __forceinline__ float hi32(uint64_t c) { return __uint_as_float((uint32_t)(c >> 32)); }

// Store the LEFT = TM TN >> lkl results (at least one) of a tile that are
// left in this lane, e0 on, at rows rt + i rs and columns ct + j cs.
template <int TM, int TN, int LEFT>
__device__ __forceinline__ void put_left(const float *acc, int lkl, int e0, int rt, int ct, int rs, int cs, float *res,
                                         const int *tab_r, const int *tab_c) {
    if constexpr (LEFT > 1) {
        if ((TM * TN >> lkl) < LEFT) return put_left<TM, TN, LEFT / 2>(acc, lkl, e0, rt, ct, rs, cs, res, tab_r, tab_c);
    }
    constexpr int LC = LEFT < TN ? LEFT : TN;  // columns of one row
    const int r = rt + (e0 / TN) * rs, c = ct + (e0 % TN) * cs;
    int oc[LC];
#pragma unroll
    for (int j = 0; j < LC; ++j) oc[j] = tab_c[c + j * cs];
#pragma unroll
    for (int i = 0; i < LEFT / LC; ++i) {
        float *o = res + tab_r[r + i * rs];
#pragma unroll
        for (int j = 0; j < LC; ++j) o[oc[j]] = acc[i * LC + j];
    }
}

// FP32 results: K is split over lanes.  Tile t of every nw x (32 >> lkl):
// 2^lkl neighbouring lanes share a tile, lane ks taking the 16-byte pieces ks,
// ks + 2^lkl, ... of K (whole sectors of a row, no bank conflicts).  Their
// partial sums are added by recursive halving, which leaves every lane a part
// of the tile's results to store, (r, c) at res[tab[r] + tab[M + c]].  AG / BG:
// the operand is in global memory.  4 x 4 tiles move 8 16-byte pieces for 64
// multiply-adds, and shared memory delivers 128 bytes a clock, which bounds a
// CTA's step at half the FP32 rate; 8 x 4 and 8 x 8 tiles move less but
// measured slower (10^6 grid30 states 5.5 and 5.8 against 5.0 ms: two CTAs per
// SM, not three, and longer reductions).
template <int TM, int TN, bool AG, bool BG>
__device__ __forceinline__ void step_split(const float *A, int pa, const float *B, int pb, int mb, int nb, int kb,
                                           int lkl, int w, int nw, int lane, float *res, const int *tab) {
    if constexpr (!AG) __builtin_assume(__isShared(A));
    if constexpr (!BG) __builtin_assume(__isShared(B));
    constexpr int E = TM * TN;
    const int rs = (1 << mb) / TM, cs = (1 << nb) / TN;
    const int lc = nb - (TN == 4 ? 2 : 0);
    const int tiles = rs * cs, per = 32 >> lkl;
    const int ks = lane & ((1 << lkl) - 1);
    for (int tb = w * per; tb < tiles; tb += nw * per) {
        const int t0 = tb + (lane >> lkl);
        const bool valid = t0 < tiles;
        const int t = valid ? t0 : 0;
        const int rt = t >> lc, ct = t & (cs - 1);
        float acc[E];
        if (kb >= 2) {
            const float *pA = A + rt * pa + 4 * ks, *pB = B + ct * pb + 4 * ks;
            const int sa = rs * pa, sb = cs * pb, n4 = 1 << (kb - 2 - lkl), inc = 4 << lkl;
            uint64_t acc2[E];
#pragma unroll
            for (int e = 0; e < E; ++e) acc2[e] = 0;
#pragma unroll 1
            for (int k = 0; k < n4; ++k) {
                ulonglong2 b[TN];
#pragma unroll
                for (int j = 0; j < TN; ++j)
                    b[j] = BG ? __ldg((const ulonglong2 *)(pB + j * sb)) : *(const ulonglong2 *)(pB + j * sb);
#pragma unroll
                for (int i = 0; i < TM; ++i) {
                    const ulonglong2 a =
                        AG ? __ldg((const ulonglong2 *)(pA + i * sa)) : *(const ulonglong2 *)(pA + i * sa);
#pragma unroll
                    for (int j = 0; j < TN; ++j) {
                        fma2(acc2[i * TN + j], a.x, b[j].x);
                        fma2(acc2[i * TN + j], a.y, b[j].y);
                    }
                }
                pA += inc;
                pB += inc;
            }
#pragma unroll
            for (int e = 0; e < E; ++e) acc[e] = lo32(acc2[e]) + hi32(acc2[e]);
        } else {  // K = 1
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) acc[i * TN + j] = A[(rt + i * rs) * pa] * B[(ct + j * cs) * pb];
        }
        // halve the results over lane bit 0, then bit 1, ... while more than
        // one is left; further lane bits add the same result
        int e0 = 0;
        bool mine = valid;
#pragma unroll
        for (int s = 0; s < 5; ++s) {
            if (lkl > s) {
                const bool up = (ks >> s) & 1;
                constexpr int H0 = E / 2;
                const int half = H0 >> s;
                if (half > 0) {
#pragma unroll
                    for (int i = 0; i < (H0 >> s); ++i) {
                        const float lo = acc[i], hi = acc[i + (H0 >> s)];
                        acc[i] = (up ? hi : lo) + __shfl_xor_sync(0xffffffffu, up ? lo : hi, 1 << s);
                    }
                    e0 += up ? half : 0;
                } else {
                    acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 1 << s);
                    mine = mine && !up;
                }
            }
        }
        if (mine) put_left<TM, TN, E>(acc, lkl, e0, rt, ct, rs, cs, res, tab, tab + (1 << mb));
    }
}

// FP64 results: every sum in one order.  Output tiles of TM x TN results (rows
// strided by M / TM, columns by N / TN), one per thread; a result is the sum,
// in order, of K / kc partial sums, each one chain of kc multiply-adds,
// whatever the tile, the number of threads or the shared steps: a state's
// value does not depend on its list (10^6 grid30 states: 6.9 ms, 4.7 with
// the split sums).
template <int TM, int TN, bool AG, bool BG>
__device__ __forceinline__ void step_tiles(const float *A, int pa, const float *B, int pb, int mb, int nb, int kb,
                                           int lkc, int t0, int nt, float *res, const int *tab) {
    if constexpr (!AG) __builtin_assume(__isShared(A));
    if constexpr (!BG) __builtin_assume(__isShared(B));
    constexpr int E = TM * TN;
    const int rs = (1 << mb) / TM, cs = (1 << nb) / TN;
    const int lc = nb - (TN == 4 ? 2 : (TN == 2 ? 1 : 0));
    for (int t = t0; t < rs * cs; t += nt) {
        const int rt = t >> lc, ct = t & (cs - 1);
        float acc[E], tot[E];
#pragma unroll
        for (int e = 0; e < E; ++e) acc[e] = tot[e] = 0.f;
        if (kb >= 2) {
            const float *pA = A + rt * pa, *pB = B + ct * pb;
            const int sa = rs * pa, sb = cs * pb, m4 = (1 << (lkc - 2)) - 1;
            const bool one = lkc == kb;
#pragma unroll (E <= 4 ? 4 : 1)
            for (int k4 = 0; k4 < 1 << (kb - 2); ++k4) {
                float4 a[TM], b[TN];
#pragma unroll
                for (int i = 0; i < TM; ++i)
                    a[i] = AG ? __ldg((const float4 *)(pA + i * sa) + k4) : ((const float4 *)(pA + i * sa))[k4];
#pragma unroll
                for (int j = 0; j < TN; ++j)
                    b[j] = BG ? __ldg((const float4 *)(pB + j * sb) + k4) : ((const float4 *)(pB + j * sb))[k4];
#pragma unroll
                for (int i = 0; i < TM; ++i)
#pragma unroll
                    for (int j = 0; j < TN; ++j) {
                        float &c = acc[i * TN + j];
                        c = fmaf(a[i].x, b[j].x, c);
                        c = fmaf(a[i].y, b[j].y, c);
                        c = fmaf(a[i].z, b[j].z, c);
                        c = fmaf(a[i].w, b[j].w, c);
                    }
                if (!one && (k4 & m4) == m4) {
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        tot[e] += acc[e];
                        acc[e] = 0.f;
                    }
                }
            }
            if (!one) {
#pragma unroll
                for (int e = 0; e < E; ++e) acc[e] = tot[e];
            }
        } else {  // K = 1
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j)
                    acc[i * TN + j] = fmaf(A[(rt + i * rs) * pa], B[(ct + j * cs) * pb], 0.f);
        }
        int oc[TN];
#pragma unroll
        for (int j = 0; j < TN; ++j) oc[j] = tab[(1 << mb) + ct + j * cs];
#pragma unroll
        for (int i = 0; i < TM; ++i) {
            float *o = res + tab[rt + i * rs];
#pragma unroll
            for (int j = 0; j < TN; ++j) o[oc[j]] = acc[i * TN + j];
        }
    }
}

// A step by the warps w, ... of nw.
template <bool ORD, bool AG, bool BG>
__device__ __forceinline__ void step_run(const SStep &S, const float *A, const float *B, int w, int nw, int lane,
                                         float *res, const int *tab) {
    __builtin_assume(__isShared(res));
    __builtin_assume(__isShared(tab));
    const int K = 1 << S.kb, pk = pitch_of(K), pa = AG ? K : pk, pb = BG ? K : pk;
    if constexpr (ORD) {
#define TQC_ST_TILE(TM, TN) \
    step_tiles<TM, TN, AG, BG>(A, pa, B, pb, S.mb, S.nb, S.kb, S.lkc, 32 * w + lane, 32 * nw, res, tab)
        // up to 4 x 4, while every thread has a tile
        const int each = (1 << (S.mb + S.nb)) / (32 * nw);
        if (each < 2 || S.mb < 2 || S.nb < 2) TQC_ST_TILE(1, 1);
        else if (each < 4) TQC_ST_TILE(2, 1);
        else if (each < 16) TQC_ST_TILE(2, 2);
        else TQC_ST_TILE(4, 4);
#undef TQC_ST_TILE
    } else {
#define TQC_ST_TILE(TM, TN) \
    step_split<TM, TN, AG, BG>(A, pa, B, pb, S.mb, S.nb, S.kb, S.lkl, w, nw, lane, res, tab)
        if (S.mb >= 2 && S.nb >= 2) TQC_ST_TILE(4, 4);
        else if (S.mb >= 2) TQC_ST_TILE(4, 1);
        else if (S.nb >= 2) TQC_ST_TILE(1, 4);
        else TQC_ST_TILE(1, 1);
#undef TQC_ST_TILE
    }
}

// Copy a leaf operand (2^row_log2 floats, rows of 2^kb, from one table row)
// to padded rows in shared memory with 16-byte asynchronous copies (by
// threads i of n; the caller waits).
__device__ __forceinline__ void copy_rows(const float *row, int row_log2, int kb, float *dst, int i, int n) {
    if (row_log2 < 2) {  // a subcircuit without cuts: one value
        if (i == 0) dst[0] = __ldg(row);
        return;
    }
    const int lq = kb >= 2 ? kb - 2 : 30, skip = kb >= 2 ? 4 : 0;  // pieces per row (K = 1: contiguous)
    for (; i < 1 << (row_log2 - 2); i += n)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                         (uint32_t)__cvta_generic_to_shared(dst + 4 * i + skip * (i >> lq))),
                     "l"(row + 4 * i)
                     : "memory");
}
__device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// The final step on one warp: lane i takes the partial sums i, i + 32, ...
// (2^lkc multiply-adds each), which are added in order.
__device__ __forceinline__ float final_dot(const float *A, const float *B, int kb, int lkc, int lane) {
    if (kb < 2) return fmaf(A[0], B[0], 0.f);
    const int blocks = 1 << (kb - lkc), n4 = 1 << (lkc - 2);
    float v = 0.f;
    for (int b0 = 0; b0 < blocks; b0 += 32) {
        float c = 0.f;
        if (b0 + lane < blocks)
            for (int k = (b0 + lane) * n4; k < (b0 + lane + 1) * n4; ++k) {
                const float4 a = ((const float4 *)A)[k], b = ((const float4 *)B)[k];
                c = fmaf(a.x, b.x, c);
                c = fmaf(a.y, b.y, c);
                c = fmaf(a.z, b.z, c);
                c = fmaf(a.w, b.w, c);
            }
        const int m = blocks - b0 < 32 ? blocks - b0 : 32;
        for (int i = 0; i < m; ++i) v += __shfl_sync(0xffffffffu, c, i);
    }
    return v;
}

// ORD: the results are FP64 (and every sum in one order), else FP32.  WHOLE:
// the program's (no shared steps, a state per CTA); a kernel of its own, so
// that the other one keeps its registers.
template <bool ORD, bool WHOLE>
__global__ void __launch_bounds__(ST_THREADS, 3)
    states_kernel(const __grid_constant__ SProgram P, const uint64_t *__restrict__ list,
                  const uint32_t *__restrict__ place, int64_t n, void *out, const double *zinfo) {
    extern __shared__ __align__(16) float sm[];
    __shared__ uint64_t win_y[ST_WINDOW];
    __shared__ uint32_t win_place[ST_WINDOW];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const double scale = zinfo[1];
    // Every state runs the same program: the place of result row r and column
    // c in the consumer's padded operand is tab[r] + tab[M + c] (the row and
    // column bits are disjoint, so the deposit of (r, c) splits into two
    // parts), computed once per CTA.
    for (int si = 0; si < P.n_steps; ++si) {
        const SStep &S = P.step[si];
        const int M = 1 << S.mb, N = 1 << S.nb;
        int *tab = (int *)(sm + S.tab_off);
        const int ck = S.c_kb < 0 ? 1 : 1 << S.c_kb, pc = pitch_of(ck);
        for (int i = tid; i < M + N; i += ST_THREADS) {
            const uint32_t d = i < M ? pdep32((uint32_t)i, S.maskR) : pdep32((uint32_t)(i - M), S.maskC);
            tab[i] = S.c_kb < 0 ? 0 : (int)(d >> S.c_kb) * pc + (int)(d & (uint32_t)(ck - 1));
        }
    }
    __syncthreads();
    auto store = [&](int64_t at, float v) {
        const double d = (double)v * scale;
        if (ORD) ((double *)out)[at] = d;
        else ((float *)out)[at] = (float)d;
    };
    auto row_of = [&](int leaf, uint64_t y) {
        const SLeaf &L = P.leaf[leaf];
        return L.table + ((int64_t)((y >> L.y_off) & ((1ull << L.n_q) - 1ull)) << L.row_log2);
    };
    // the permuted state at position p of the list (whole warps call this)
    auto state_at = [&](int64_t p) {
        const uint64_t x = list[p];
        if (P.key_bits) return x;  // permuted by the sort
        const uint32_t lo = __ballot_sync(0xffffffffu, lane < P.n_qubits && ((x >> P.perm[lane]) & 1ull));
        const uint32_t hi =
            __ballot_sync(0xffffffffu, lane + 32 < P.n_qubits && ((x >> P.perm[(lane + 32) & 63]) & 1ull));
        return ((uint64_t)hi << 32) | lo;
    };
    // steps [n_shared, n_steps) of one state on one warp (WHOLE: on the CTA's), leaf rows read from the tables (staged copies per warp cost a CTA
    // per SM and measured no faster)
    float *wsm = sm + P.warp_off + (WHOLE ? 0 : warp * P.warp_floats);
    const int w = WHOLE ? warp : 0, nw = WHOLE ? ST_WARPS : 1;
    auto warp_state = [&](uint64_t y, int64_t at) {
        auto sync = [&] {
            if constexpr (WHOLE) __syncthreads();
            else __syncwarp();
        };
        for (int si = P.n_shared; si < P.n_steps; ++si) {
            const SStep &S = P.step[si];
            const bool ag = S.a_kind == SRC_TABLE, bg = S.b_kind == SRC_TABLE;
            const float *A = ag ? row_of(S.a_leaf, y) : (S.a_kind == SRC_CTA ? sm : wsm) + S.a_off;
            const float *B = bg ? row_of(S.b_leaf, y) : (S.b_kind == SRC_CTA ? sm : wsm) + S.b_off;
            if (S.c_kb < 0) {
                if (w == 0) {
                    const float v = final_dot(A, B, S.kb, S.lkc, lane);
                    if (lane == 0) store(at, v);
                }
                sync();
                return;
            }
            const int *tab = (const int *)(sm + S.tab_off);
            float *res = wsm + S.c_off;
            if (ag && bg) step_run<ORD, true, true>(S, A, B, w, nw, lane, res, tab);
            else if (ag) step_run<ORD, true, false>(S, A, B, w, nw, lane, res, tab);
            else if (bg) step_run<ORD, false, true>(S, A, B, w, nw, lane, res, tab);
            else step_run<ORD, false, false>(S, A, B, w, nw, lane, res, tab);
            sync();
        }
    };
    if (P.n_steps == 0) {  // one subcircuit without cuts: a table lookup
        for (int64_t p = (int64_t)blockIdx.x * ST_WARPS + warp; p < n; p += (int64_t)gridDim.x * ST_WARPS) {
            const uint64_t y = state_at(p);
            if (lane == 0) store(p, *row_of(0, y));
        }
        return;
    }
    const int64_t p0 = n * blockIdx.x / gridDim.x, p1 = n * (blockIdx.x + 1) / gridDim.x;
    auto place_of = [&](int64_t p) { return place ? (int64_t)place[p] : p; };
    if (WHOLE || P.n_shared == 0) {
        for (int64_t p = p0 + warp - w; p < p1; p += ST_WARPS / nw) {
            const uint64_t y = state_at(p);
            warp_state(y, place_of(p));
        }
        return;
    }
    // Stage the leaf operands of the shared steps that changed since the last
    // staging (diff: the bits of y that did).
    auto stage = [&](int s0, int s1, uint64_t y, uint64_t diff, bool all) {
        for (int si = s0; si < s1; ++si) {
            const SStep &S = P.step[si];
#pragma unroll
            for (int op = 0; op < 2; ++op) {
                const int leaf = op ? S.b_leaf : S.a_leaf;
                if (leaf < 0) continue;
                const uint64_t lm = ((1ull << P.leaf[leaf].n_q) - 1ull) << P.leaf[leaf].y_off;
                if (!all && !(diff & lm)) continue;
                copy_rows(row_of(leaf, y), P.leaf[leaf].row_log2, S.kb, sm + (op ? S.b_off : S.a_off), tid, ST_THREADS);
            }
        }
    };
    // One shared step on the whole CTA (not the final one).
    auto shared_step = [&](const SStep &S) {
        step_run<ORD, false, false>(S, sm + S.a_off, sm + S.b_off, warp, ST_WARPS, lane, sm + S.c_off,
                                    (const int *)(sm + S.tab_off));
    };
    if (P.one_each) {  // every step on the whole CTA, one state at a time
        uint64_t prev = 0;
        for (int64_t p = p0; p < p1; ++p) {
            const uint64_t y = state_at(p), diff = y ^ prev;
            const bool first = p == p0;
            prev = y;
            for (int si = 0; si < P.n_shared; ++si) {
                const SStep &S = P.step[si];
                // skipped when nothing it depends on has changed
                if (!first && S.c_kb >= 0 && !(diff & S.mask)) continue;
                stage(si, si + 1, y, diff, first || P.restage);
                copies_wait();
                __syncthreads();
                if (S.c_kb >= 0) {
                    shared_step(S);
                } else {
                    if (warp == 0) {
                        const float v = final_dot(sm + S.a_off, sm + S.b_off, S.kb, S.lkc, lane);
                        if (lane == 0) store(place_of(p), v);
                    }
                }
                __syncthreads();
            }
        }
        return;
    }
    // Groups of states that share the subtree's bits (consecutive in the
    // sorted list).  While the warps run the states of one group, the leaf
    // operands of the next group's shared steps are on their way: a group
    // takes two barriers, and one between shared steps.
    auto run_shared = [&](uint64_t diff, bool all) {
        for (int si = 0; si < P.n_shared; ++si) {
            const SStep &S = P.step[si];
            if (!all && !(diff & S.mask)) continue;
            shared_step(S);
            if (si + 1 < P.n_shared) __syncthreads();
        }
    };
    // A window of the sorted list in shared memory: [wb, wb + ST_WINDOW).
    int64_t wb = p0;
    auto load_window = [&](int64_t at) {
        wb = at;
        for (int i = tid; i < ST_WINDOW; i += ST_THREADS)
            if (at + i < p1) {
                win_y[i] = list[at + i];
                win_place[i] = place[at + i];
            }
    };
    auto group_size = [&](int64_t p, uint64_t y) {  // up to one state per thread; a barrier
        const int64_t q = p + tid;
        return __syncthreads_count(q < p1 && ((win_y[q < p1 ? q - wb : 0] ^ y) & P.group_mask) == 0);
    };
    if (p0 >= p1) return;
    int64_t p = p0;
    load_window(p0);
    __syncthreads();
    uint64_t y = win_y[0];
    stage(0, P.n_shared, y, 0, true);
    int cnt = group_size(p0, y);
    copies_wait();
    __syncthreads();
    run_shared(0, true);
    while (true) {
        const int64_t pn = p + cnt;
        if (pn < p1 && pn + ST_THREADS > wb + ST_WINDOW && wb + ST_WINDOW < p1) {
            // the window moves on; the states of this group keep their part of it
            __syncthreads();
            load_window(p);
            __syncthreads();
        }
        const uint64_t yn = pn < p1 ? win_y[pn - wb] : y, diff = yn ^ y;
        const int next = group_size(pn, yn);  // the barrier ends the shared steps' writes
        if (next > 0) stage(0, P.n_shared, yn, diff, false);
        for (int k = warp; k < cnt; k += ST_WARPS) warp_state(win_y[p + k - wb], (int64_t)win_place[p + k - wb]);
        if (next == 0) break;
        p = pn;
        cnt = next;
        y = yn;
        if (!(diff & P.group_mask)) continue;  // a group longer than the CTA's threads goes on
        copies_wait();
        __syncthreads();
        run_shared(diff, false);
    }
}

// ---- counting sort of the list by the top key_bits of the permuted state
// y: count (a state's rank among those counted so far with its key), an
// exclusive scan of the counters, scatter.  Which of two states with equal
// keys comes first does not change any state's value.
__global__ void states_count_kernel(const __grid_constant__ SProgram P, const uint64_t *__restrict__ states, int64_t n,
                                    uint64_t *__restrict__ ys, uint32_t *__restrict__ rank, uint32_t *counters) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t act = __ballot_sync(0xffffffffu, i < n);
    if (i >= n) return;
    const uint64_t x = states[i];
    uint64_t y = 0;
    for (int b = 0; b < P.n_qubits; ++b) y |= ((x >> P.perm[b]) & 1ull) << b;
    ys[i] = y;
    const uint32_t key = (uint32_t)(y >> (P.n_qubits - P.key_bits));
    // one atomic per distinct key of the warp
    const uint32_t peers = __match_any_sync(act, key);
    const int lane = threadIdx.x & 31, lead = __ffs(peers) - 1;
    uint32_t base = 0;
    if (lane == lead) base = atomicAdd(counters + key, (uint32_t)__popc(peers));
    base = __shfl_sync(peers, base, lead);
    rank[i] = base + (uint32_t)__popc(peers & ((1u << lane) - 1u));
}

__device__ __forceinline__ uint32_t block_sum(uint32_t v, uint32_t *red) {
    v = __reduce_add_sync(0xffffffffu, v);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    uint32_t t = 0;
#pragma unroll
    for (int i = 0; i < ST_WARPS; ++i) t += red[i];
    return t;
}

__global__ void __launch_bounds__(ST_THREADS) states_sums_kernel(const uint32_t *counters, int n, uint32_t *sums) {
    __shared__ uint32_t red[ST_WARPS];
    uint32_t v = 0;
    const int base = blockIdx.x * SCAN_PER_CTA;
    for (int i = threadIdx.x; i < SCAN_PER_CTA; i += ST_THREADS)
        if (base + i < n) v += counters[base + i];
    const uint32_t t = block_sum(v, red);
    if (threadIdx.x == 0) sums[blockIdx.x] = t;
}

__global__ void __launch_bounds__(ST_THREADS) states_scan_kernel(uint32_t *counters, int n, const uint32_t *sums) {
    __shared__ uint32_t red[ST_WARPS], wsum[ST_WARPS];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t v = 0;
    for (int i = tid; i < (int)blockIdx.x; i += ST_THREADS) v += sums[i];
    uint32_t run = block_sum(v, red);
    const int base = blockIdx.x * SCAN_PER_CTA;
    for (int c = 0; c < SCAN_PER_CTA; c += ST_THREADS) {
        const int i = base + c + tid;
        const uint32_t x = i < n ? counters[i] : 0;
        uint32_t s = x;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t u = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += u;
        }
        __syncthreads();
        if (lane == 31) wsum[warp] = s;
        __syncthreads();
        uint32_t before = 0, total = 0;
#pragma unroll
        for (int w = 0; w < ST_WARPS; ++w) {
            if (w < warp) before += wsum[w];
            total += wsum[w];
        }
        if (i < n) counters[i] = run + before + s - x;
        run += total;
    }
}

__global__ void states_scatter_kernel(const uint64_t *__restrict__ ys, const uint32_t *__restrict__ rank, int64_t n,
                                      int shift, const uint32_t *__restrict__ offsets, uint64_t *__restrict__ sorted,
                                      uint32_t *__restrict__ place) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint64_t y = ys[i];
    const uint32_t at = offsets[y >> shift] + rank[i];
    sorted[at] = y;
    place[at] = (uint32_t)i;
}

int64_t align4(int64_t x) { return (x + 3) & ~int64_t(3); }

// Distinct values among n uniform draws from 2^q.
double distinct(double n, int q) {
    const double d = std::ldexp(1.0, q);
    return q > 60 ? n : d * -std::expm1(-n / d);
}

// Bits of the sort key of a list of n states, of which `want` would serve: few
// enough that clearing and scanning the counters (16 to 32 per state) costs
// less than the states, and that a short list's buffers are small.
int key_bits_for(double n, int want) {
    return std::min(want, (int)std::ceil(std::log2(std::max(1.0, n))) + 4);
}

// The fused form's program with the subtree of step `top` shared (-1: no
// shared steps, a state per warp; TOP_WHOLE: none, a state per CTA; the last
// step: a state per CTA, its leaf operands staged), the list sorted or (no
// subtree, or the last step's) in its own order, without table pointers (set
// at launch), and its estimated cost; false when it does not fit.
// compact: leaf operands of the shared steps reuse two areas.
constexpr int TOP_WHOLE = -2;
bool layout_program(const Plan &p, double n, int top, bool sort, bool compact, SProgram *P, double *cost,
                    std::string *why) {
    std::memset(P, 0, sizeof(*P));
    P->whole = top == TOP_WHOLE;
    const int ns = (int)p.steps.size();
    P->n_leaves = p.m;
    P->n_steps = ns;
    P->n_qubits = p.net->n_qubits;
    std::vector<int> producer(p.tensors.size(), -1), consumer(p.tensors.size(), -1);
    for (int s = 0; s < ns; ++s) {
        producer[(size_t)p.steps[s].c] = s;
        consumer[(size_t)p.steps[s].a] = consumer[(size_t)p.steps[s].b] = s;
    }
    // output qubits and multiply-adds below every tensor
    std::vector<int> q(p.tensors.size(), 0);
    std::vector<double> macs(p.tensors.size(), 0);
    for (int j = 0; j < p.m; ++j) q[j] = (int)p.net->nodes[j].out_qubits.size();
    for (int s = 0; s < ns; ++s) {
        const StepPlan &st = p.steps[s];
        q[(size_t)st.c] = q[(size_t)st.a] + q[(size_t)st.b];
        macs[(size_t)st.c] = macs[(size_t)st.a] + macs[(size_t)st.b] + std::ldexp(1.0, st.mb + st.nb + st.kb);
    }
    // steps of the shared subtree first
    std::vector<char> shared(p.tensors.size(), 0);
    if (top >= 0) shared[(size_t)p.steps[top].c] = 1;
    for (int s = ns - 1; s >= 0; --s)
        if (shared[(size_t)p.steps[s].c]) shared[(size_t)p.steps[s].a] = shared[(size_t)p.steps[s].b] = 1;
    std::vector<int> order;
    for (int pass = 0; pass < 2; ++pass)
        for (int s = 0; s < ns; ++s)
            if ((shared[(size_t)p.steps[s].c] != 0) == (pass == 0)) order.push_back(s);
    // y: the sort key's leaves on top, the costliest subtree first at every
    // level, so that consecutive states of the sorted list share its bits
    std::vector<int> rank_order;
    std::vector<int> stack;
    auto heavy = [&](int t) {
        const StepPlan &st = p.steps[producer[(size_t)t]];
        return macs[(size_t)st.a] > macs[(size_t)st.b] || (macs[(size_t)st.a] == macs[(size_t)st.b] && q[(size_t)st.a] > q[(size_t)st.b]);
    };
    const int root = ns > 0 ? p.steps[ns - 1].c : 0;
    int key_t = top >= 0 ? p.steps[top].c : -1;  // the tensor whose bits are the sort key
    while (key_t >= 0 && q[(size_t)key_t] > ST_MAX_KEY_BITS) {
        if (producer[(size_t)key_t] < 0) {
            key_t = -1;
            break;
        }
        const StepPlan &st = p.steps[producer[(size_t)key_t]];
        key_t = heavy(key_t) ? st.a : st.b;
    }
    std::vector<char> placed((size_t)p.m, 0);
    auto place_below = [&](int t0) {
        stack.assign(1, t0);
        while (!stack.empty()) {
            const int t = stack.back();
            stack.pop_back();
            if (producer[(size_t)t] < 0) {
                if (!placed[(size_t)t]) rank_order.push_back(t);
                placed[(size_t)t] = 1;
                continue;
            }
            const StepPlan &st = p.steps[producer[(size_t)t]];
            const bool h = heavy(t);
            stack.push_back(h ? st.b : st.a);
            stack.push_back(h ? st.a : st.b);
        }
    };
    if (key_t >= 0) place_below(key_t);
    if (top >= 0) place_below(p.steps[top].c);
    place_below(root);
    int at = P->n_qubits;
    for (int j : rank_order) {
        const Node &nd = p.net->nodes[j];
        at -= (int)nd.out_qubits.size();
        P->leaf[j].row_log2 = p.tensors[j].nbits();
        P->leaf[j].y_off = at;
        P->leaf[j].n_q = (int)nd.out_qubits.size();
        for (size_t k = 0; k < nd.out_qubits.size(); ++k) P->perm[at + (int)k] = (int8_t)nd.out_qubits[k];
        if (P->leaf[j].n_q == 0) P->leaf[j].y_off = 0;
    }
    auto bits_of = [&](uint64_t leaves) {
        uint64_t m = 0;
        for (int j = 0; j < p.m; ++j)
            if (leaves >> j & 1)
                for (int k = 0; k < P->leaf[j].n_q; ++k) m |= 1ull << (P->leaf[j].y_off + k);
        return m;
    };
    P->key_bits = key_t >= 0 ? q[(size_t)key_t] : 0;
    P->one_each = top >= 0 && (top == ns - 1 || key_t != p.steps[top].c || P->key_bits == 0);
    if (!sort) P->key_bits = 0;
    P->restage = compact;
    P->group_mask = top >= 0 ? bits_of(p.tensors[(size_t)p.steps[top].c].leaves) : 0;
    if (P->one_each && top != ns - 1) return *why = "shared subtree has too many output bits", false;
    const int n_shared = (int)std::count_if(order.begin(), order.end(), [&](int s) { return shared[(size_t)p.steps[s].c] != 0; });
    P->n_shared = n_shared;
    // shared memory: leaf operands of the shared steps, intermediates, the
    // warps' own intermediates, the offset tables
    int64_t off = 0, woff = 0, area[2] = {0, 0};
    std::vector<int> place(p.tensors.size(), 0);
    for (int i = 0; i < n_shared; ++i) {
        const StepPlan &st = p.steps[order[(size_t)i]];
        const int64_t pk = pitch_of(1 << st.kb);
        const int64_t need[2] = {((int64_t)1 << st.mb) * pk, ((int64_t)1 << st.nb) * pk};
        const int t[2] = {st.a, st.b};
        for (int k = 0; k < 2; ++k) {
            if (t[k] >= p.m) continue;
            if (compact) area[k] = std::max(area[k], align4(need[k]));
            else {
                place[(size_t)t[k]] = (int)off;
                off += align4(need[k]);
            }
        }
    }
    if (compact) {
        for (int i = 0; i < n_shared; ++i) {
            const StepPlan &st = p.steps[order[(size_t)i]];
            if (st.a < p.m) place[(size_t)st.a] = 0;
            if (st.b < p.m) place[(size_t)st.b] = (int)area[0];
        }
        off = area[0] + area[1];
    }
    for (int i = 0; i < ns; ++i) {
        const StepPlan &st = p.steps[order[(size_t)i]];
        const int c = consumer[(size_t)st.c];
        if (c < 0) {  // the final step: a scalar per state
            if (st.mb != 0 || st.nb != 0) return *why = "final step is not a scalar", false;
            continue;
        }
        const int64_t ck = (int64_t)1 << p.steps[c].kb;
        const int64_t need = align4((((int64_t)1 << (st.mb + st.nb)) / ck) * pitch_of((int)ck));
        int64_t &o = i < n_shared ? off : woff;
        place[(size_t)st.c] = (int)o;
        o += need;
    }
    for (int i = 0; i < ns; ++i) {
        const StepPlan &st = p.steps[order[(size_t)i]];
        SStep &S = P->step[i];
        S.mb = st.mb;
        S.nb = st.nb;
        S.kb = st.kb;
        S.maskR = (uint32_t)st.maskR;
        S.maskC = (uint32_t)st.maskC;
        S.mask = bits_of(p.tensors[(size_t)st.c].leaves);
        const int c = consumer[(size_t)st.c];
        // lanes per output tile: what the tiles leave idle, at most one per 16
        // bytes of K; rows read from global memory always 8 (a whole line)
        const int tiles = std::max(0, st.mb - 2) + std::max(0, st.nb - 2);  // log2
        const bool cta = i < n_shared || P->whole, table = i >= n_shared && (st.a < p.m || st.b < p.m);
        const int lkl = std::max(table ? 3 : 0, std::min(5, (cta ? 8 : 5) - tiles));
        S.lkl = std::max(0, std::min(lkl, st.kb - 2));
        // partial sums: K in as many parts as give 256 threads a tile each, of
        // at least 4 multiply-adds
        S.lkc = st.kb;
        while (st.kb - S.lkc + 1 + tiles <= 8 && S.lkc >= 3) --S.lkc;
        S.c_kb = c < 0 ? -1 : p.steps[c].kb;
        S.c_off = place[(size_t)st.c];
        auto operand = [&](int t, int32_t *leaf, int32_t *kind, int32_t *o) {
            *leaf = t < p.m ? t : -1;
            *kind = i < n_shared ? SRC_CTA : (t < p.m ? SRC_TABLE : (shared[(size_t)t] ? SRC_CTA : SRC_WARP));
            *o = place[(size_t)t];
        };
        operand(st.a, &S.a_leaf, &S.a_kind, &S.a_off);
        operand(st.b, &S.b_leaf, &S.b_kind, &S.b_off);
        S.tab_off = (int32_t)off;
        off += align4(((int64_t)1 << st.mb) + ((int64_t)1 << st.nb));
    }
    P->warp_off = (int32_t)off;
    P->warp_floats = (int32_t)woff;
    off += woff * (P->whole ? 1 : ST_WARPS);
    if (off > ST_MAX_SMEM_FLOATS) return *why = "intermediates exceed shared memory", false;
    P->smem_floats = (int32_t)std::max<int64_t>(off, 4);
    if (!cost) return true;
    // Estimated clocks.  The latencies (of a step on a warp or a CTA of its
    // own, and with every slot of the SM taken), the 64 multiply-adds per clock
    // of a CTA's step and the sort's cost are fitted to every split of nine
    // networks (1348 to 278592 multiply-adds per state) at nine lengths from 1
    // to 10^6, timed against each other.
    const double sms = sm_count();
    const int per_sm = std::max(1, std::min(3, (int)(227 * 1024 / (P->smem_floats * 4 + 10 * 1024))));
    const double warps = ST_WARPS * per_sm;
    std::vector<double> times(p.tensors.size(), n);  // how often every tensor is computed
    if (top >= 0 && P->key_bits) {
        const int t = p.steps[top].c;
        times[(size_t)t] = P->one_each ? n : distinct(n, q[(size_t)t]);
        for (int s = top; s >= 0; --s) {
            const StepPlan &st = p.steps[s];
            if (!shared[(size_t)st.c]) continue;
            const int hv = heavy(st.c) ? st.a : st.b, lt = heavy(st.c) ? st.b : st.a;
            times[(size_t)lt] = times[(size_t)st.c];
            times[(size_t)hv] =
                q[(size_t)hv] <= P->key_bits ? std::min(times[(size_t)st.c], distinct(n, q[(size_t)hv])) : times[(size_t)st.c];
        }
    }
    double warp_alone = 0, warp_full = 0, cta_alone = 0, cta_full = 0, shared_clk = 0, whole_alone = 0, whole_full = 0;
    for (int i = 0; i < ns; ++i) {
        const StepPlan &st = p.steps[order[(size_t)i]];
        const double macs = std::ldexp(1.0, st.mb + st.nb + st.kb);
        if (i >= n_shared) {
            warp_alone += 1500.0 + 0.32 * macs;
            warp_full += 1000.0 + 100.0 * warps + 0.57 * macs;
            whole_alone += 1500.0 + 0.32 / ST_WARPS * macs;
            whole_full += 2800.0 + 0.57 / ST_WARPS * macs;
        } else {
            cta_alone += 1200.0 + macs / 64.0;
            cta_full += 2800.0 + macs / 64.0 * per_sm;
            shared_clk += times[(size_t)st.c] * (macs / 64.0 + (P->one_each ? 2800.0 : 1500.0) / per_sm);
        }
    }
    // s units of work per SM on `slots` slots
    auto rounds = [](double s, double slots, double alone, double full) {
        return std::max(1.0, s / slots) * (alone + (full - alone) * std::min(1.0, s / slots));
    };
    const double sorted = P->key_bits ? 31000.0 + 0.15 * n + 0.005 * std::ldexp(1.0, key_bits_for(n, P->key_bits)) : 0.0;
    if (P->whole) {
        *cost = rounds(n / sms, per_sm, whole_alone, whole_full);
    } else if (n_shared == 0) {
        *cost = rounds(n / sms, warps, warp_alone, warp_full);
    } else if (P->one_each) {
        *cost = P->key_bits ? sorted + std::max(cta_alone, shared_clk / sms) : rounds(n / sms, per_sm, cta_alone, cta_full);
    } else {
        const double groups = std::max(times[(size_t)p.steps[top].c], std::min(n, sms * per_sm)), s = n / groups;
        const double turns = std::max(1.0, s / ST_WARPS + 0.4);  // of a group's states through the warps
        const double turn = (warp_alone + (warp_full - warp_alone) * std::min(1.0, s / turns / ST_WARPS)) / per_sm;
        *cost = sorted + std::max(cta_alone + warp_alone, (shared_clk + groups * (2000.0 / per_sm + turns * turn)) / sms);
    }
    return true;
}

// The program of a single-state plan for a list of n states: the split into
// shared and per-warp steps of least estimated cost (can_sort = false: among
// those that take the list as it is), else (nothing else fits) every state on
// a whole CTA with reused leaf areas.
bool build_program(const Plan &p, int64_t n, bool can_sort, SProgram *P, std::string *why) {
    if (!p.free_qubits.empty()) return *why = "free qubits", false;
    if (p.n_slices() != 1) return *why = "sliced", false;
    if (p.m > ST_MAX_LEAVES) return *why = "more than 16 subcircuits", false;
    if (p.net->n_qubits > 64) return *why = "more than 64 qubits", false;
    for (auto &st : p.steps) {
        if (st.kblk) return *why = "K-blocked operands", false;
        if (st.mb + st.kb > 20 || st.nb + st.kb > 20 || st.mb + st.nb > 20) return *why = "step too large", false;
        if (st.maskR >> 32 || st.maskC >> 32) return *why = "result wider than 32 bits", false;
    }
    const int ns = (int)p.steps.size();
    if (n > (int64_t)1 << 31) can_sort = false;  // positions of the sorted list are 32-bit
    double best = std::numeric_limits<double>::infinity();
    std::string w;
    for (int top = -1; top < ns; ++top)
        for (int sort = 0; sort < 2; ++sort) {
            if (sort ? !can_sort || top < 0 : top >= 0 && top != ns - 1) continue;
            SProgram Q;
            double cost = 0;
            if (!layout_program(p, (double)n, top, sort != 0, false, &Q, &cost, &w)) continue;
            if (Q.key_bits) cost *= 1.08;  // sorted only for a gain beyond the estimates' error
            if (cost < best) {
                best = cost;
                *P = Q;
            }
        }
    if (std::isfinite(best)) {  // short lists: a warp per state would leave most of the SMs idle
        SProgram Q;
        double cost = 0;
        if (layout_program(p, (double)n, TOP_WHOLE, false, false, &Q, &cost, &w) && cost < best) *P = Q;
    } else if (!layout_program(p, (double)n, ns - 1, false, true, P, nullptr, why)) {
        return false;
    }
    if (P->key_bits) P->key_bits = key_bits_for((double)n, P->key_bits);
    return true;
}

tqc_status cuda_fail(cudaError_t e, const char *what) {
    return fail(TQC_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

}  // namespace

// Shared-memory floats of the fused form, or -1 when the plan runs per state.
int states_fused_floats(const Plan &p) {
    SProgram P;
    std::string why;
    return build_program(p, 1, true, &P, &why) ? P.smem_floats : -1;
}

tqc_status exec_contract_states(Plan *p, const uint64_t *states, int64_t n, void *d_out, int out_dtype,
                                double *z_out, void *stream) {
    if (!p->free_qubits.empty())
        return fail(TQC_ERR_INVALID, "state lists need a plan with no free qubits (use_free_mask = 1, masks 0)");
    if (p->n_slices() != 1) return fail(TQC_ERR_UNSUPPORTED, "state lists need an unsliced plan");
    if (p->net->n_qubits > 64) return fail(TQC_ERR_UNSUPPORTED, "state lists support up to 64 qubits");
    if (n < 0) return fail(TQC_ERR_INVALID, "negative state count");
    const uint64_t qmask = p->net->n_qubits == 64 ? ~0ull : ((1ull << p->net->n_qubits) - 1);
    uint64_t any = 0;
    for (int64_t i = 0; i < n; ++i) any |= states[i];
    for (int64_t i = 0; (any & ~qmask) && i < n; ++i)
        if (states[i] & ~qmask) return fail(TQC_ERR_INVALID, "state " + std::to_string(i) + " has bits beyond n_qubits");
    tqc_status st = exec_prepare(p);
    if (st != TQC_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    ExecCtx c;
    c.ws = p->d_ws;
    c.zws = p->d_zws;
    c.zinfo = p->d_zinfo;
    c.kpart = p->d_kpart;
    if (p->z_version != p->net->version) {
        st = exec_total_mass(*p, c, stream);
        if (st != TQC_OK) return st;
        p->z_version = p->net->version;
    }
    // The program for the last list's length is kept: choosing one takes longer
    // on the host (2-7 us) than a short list's kernel.
    SProgram P;
    std::string why;
    auto program = [&] {
        if (p->states_n != n) {
            p->states_prog.clear();
            if (build_program(*p, n, !p->states_no_sort, &P, &why))
                p->states_prog.assign((const char *)&P, (const char *)(&P + 1));
            p->states_n = n;
        } else if (!p->states_prog.empty()) {
            std::memcpy((void *)&P, p->states_prog.data(), sizeof P);
        }
        return !p->states_prog.empty();
    };
    bool fused = n > 0 && program();
    const int esize = out_dtype == TQC_F64 ? 8 : 4;
    if (fused) {
        // per-node tables Tt_j[x][cuts], rebuilt when the tensors changed
        if (p->tab_version != p->net->version || !p->d_tab) {
            int64_t need = 0;
            std::vector<int64_t> toff;
            for (int j = 0; j < p->m; ++j) {
                toff.push_back(need);
                need += ((p->net->nodes[j].elems * 4 + 255) / 256) * 256;
            }
            if (need > p->tab_bytes) {
                if (p->d_tab) cudaFree(p->d_tab);
                p->d_tab = nullptr;
                p->tab_bytes = 0;
                if (cudaMalloc(&p->d_tab, (size_t)need) != cudaSuccess) {
                    cudaGetLastError();
                    return fail(TQC_ERR_OOM, "state-list tables of " + std::to_string(need) + " bytes");
                }
                p->tab_bytes = need;
            }
            p->tab_off = toff;
            std::vector<IngestArgs> leaves;
            for (int j = 0; j < p->m; ++j) {
                const Node &nd = p->net->nodes[j];
                const TensorPlan &t = p->tensors[j];
                IngestArgs g;
                g.src = nd.d_data;
                g.src_dtype = nd.dtype;
                int b = 0;
                for (auto &md : t.layout.modes) {  // the leaf's own layout: its cut bits
                    const int pos = exec_src_pos_cut(nd, md.id);
                    g.srcpos[b++] = (int8_t)pos;
                    g.srcpos[b++] = (int8_t)(pos + 1);
                }
                for (size_t k = 0; k < nd.out_qubits.size(); ++k) g.srcpos[b++] = (int8_t)k;  // then x
                g.nbits = b;
                g.dst = (char *)p->d_tab + toff[(size_t)j];
                g.storage = ST_F32;
                leaves.push_back(g);
            }
            cudaError_t e = launch_ingest(leaves.data(), p->m, s);
            if (e != cudaSuccess) return cuda_fail(e, "state-list table");
            p->tab_version = p->net->version;
        }
        // the list, and for the sort: permuted states, ranks, sorted states,
        // their places in the list, counters and their block sums.  Sized for
        // the widest key of any split, so that a shorter list never grows them;
        // where the device has no room for the sort the list is taken as it is.
        const int64_t n8 = align4(n) * 8, n4 = align4(n) * 4;
        const int64_t max_keys = (int64_t)1 << key_bits_for((double)n, std::min(ST_MAX_KEY_BITS, p->net->n_qubits));
        const int64_t all = 3 * n8 + 2 * n4 + align4(max_keys) * 4 + align4(max_keys / SCAN_PER_CTA + 1) * 4;
        auto reserve = [&](int64_t need) {
            if (need <= p->states_bytes) return cudaSuccess;
            if (p->d_states) cudaFree(p->d_states);
            p->d_states = nullptr;
            p->states_bytes = 0;
            const cudaError_t e = cudaMalloc(&p->d_states, (size_t)need);
            if (e == cudaSuccess) p->states_bytes = need;
            else cudaGetLastError();
            return e;
        };
        cudaError_t e = reserve(p->states_no_sort || n > (int64_t)1 << 31 ? n8 : all);
        if (e == cudaErrorMemoryAllocation && !p->states_no_sort) {
            p->states_no_sort = true;
            p->states_n = -1;
            fused = program();
            e = fused ? reserve(n8) : cudaSuccess;
        }
        if (e != cudaSuccess) return fail(TQC_ERR_OOM, "state list of " + std::to_string(n) + " states");
    }
    if (fused) {
        for (int j = 0; j < p->m; ++j) P.leaf[j].table = (const float *)((char *)p->d_tab + p->tab_off[(size_t)j]);
        const int64_t n8 = align4(n) * 8, n4 = align4(n) * 4, n_keys = P.key_bits ? (int64_t)1 << P.key_bits : 0;
        const int64_t n_sums = (n_keys + SCAN_PER_CTA - 1) / SCAN_PER_CTA;
        uint64_t *d_list = (uint64_t *)p->d_states;
        uint32_t *d_place = nullptr;
        cudaError_t e = cudaMemcpyAsync(d_list, states, (size_t)n * 8, cudaMemcpyHostToDevice, s);
        if (e != cudaSuccess) return cuda_fail(e, "state list upload");
        if (P.key_bits) {
            char *at = (char *)p->d_states + n8;
            auto take = [&](int64_t bytes) { char *r = at; at += bytes; return r; };
            uint64_t *ys = (uint64_t *)take(n8), *sorted = (uint64_t *)take(n8);
            uint32_t *rank = (uint32_t *)take(n4);
            d_place = (uint32_t *)take(n4);
            uint32_t *counters = (uint32_t *)take(align4(n_keys) * 4), *sums = (uint32_t *)take(align4(n_sums) * 4);
            e = cudaMemsetAsync(counters, 0, (size_t)n_keys * 4, s);
            if (e != cudaSuccess) return cuda_fail(e, "state list sort");
            const unsigned blocks = (unsigned)((n + ST_THREADS - 1) / ST_THREADS);
            states_count_kernel<<<blocks, ST_THREADS, 0, s>>>(P, d_list, n, ys, rank, counters);
            states_sums_kernel<<<(unsigned)n_sums, ST_THREADS, 0, s>>>(counters, (int)n_keys, sums);
            states_scan_kernel<<<(unsigned)n_sums, ST_THREADS, 0, s>>>(counters, (int)n_keys, sums);
            states_scatter_kernel<<<blocks, ST_THREADS, 0, s>>>(ys, rank, n, P.n_qubits - P.key_bits, counters, sorted,
                                                                d_place);
            e = cudaGetLastError();
            if (e != cudaSuccess) return cuda_fail(e, "state list sort");
            d_list = sorted;
        }
        const size_t smem = (size_t)P.smem_floats * 4;
        const bool f64 = out_dtype == TQC_F64;
        auto *kernel = P.whole ? (f64 ? states_kernel<true, true> : states_kernel<false, true>)
                               : (f64 ? states_kernel<true, false> : states_kernel<false, false>);
        static size_t attrs[2][2] = {{0, 0}, {0, 0}};
        size_t &attr = attrs[P.whole][f64];
        if (smem > 36 * 1024 && smem > attr) {  // beside 9 KB of static shared memory
            e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return cuda_fail(e, "state-list kernel attribute");
            attr = smem;
        }
        int per_sm = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, ST_THREADS, smem);
        if (e != cudaSuccess || per_sm < 1) return fail(TQC_ERR_UNSUPPORTED, "state-list kernel does not fit an SM");
        const int64_t grid = std::min<int64_t>(n, (int64_t)per_sm * sm_count());
        kernel<<<(unsigned)grid, ST_THREADS, smem, s>>>(P, d_list, d_place, n, d_out, p->d_zinfo);
        e = cudaGetLastError();
        if (e != cudaSuccess) return cuda_fail(e, "state-list kernel");
    } else if (n > 0) {
        // per state: the single-state plan with the state's bits as the fixed bits
        std::vector<uint8_t> fixed((size_t)p->net->n_qubits);
        c.compute_z = false;
        p->reuse_ok = false;  // the workspace now holds other states' intermediates
        for (int64_t i = 0; i < n; ++i) {
            for (int q = 0; q < p->net->n_qubits; ++q) fixed[(size_t)q] = (uint8_t)((states[i] >> q) & 1);
            st = exec_run(*p, c, fixed.data(), (char *)d_out + i * esize, out_dtype, stream, nullptr);
            if (st != TQC_OK) return st;
        }
    }
    if (z_out) {
        double zi[4];
        cudaError_t e = cudaMemcpyAsync(zi, p->d_zinfo, sizeof zi, cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return cuda_fail(e, "z copy");
        *z_out = zi[0];
        if (((int *)(zi + 2))[0] != 0) {
            cudaMemsetAsync(p->d_zinfo + 2, 0, sizeof(int), s);
            return fail(TQC_ERR_TIMEOUT, "a tensor-core step gave up waiting on its pipeline");
        }
    }
    return TQC_OK;
}

}  // namespace tqc
