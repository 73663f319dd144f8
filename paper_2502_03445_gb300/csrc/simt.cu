// CUDA-core kernels: the plain FP32 pairwise step (also used for the small-K
// steps of the tensor-core form), its FP64 twin for the total-mass network,
// tensor ingest (bin restriction, slicing, layout permutation, cast), the
// total-mass reduction and the FP64 slice-sum finalisation.
//
// A pairwise step is the contraction of two subcircuit tensors over their
// shared cut edges (§III-B, Fig. tensor_contraction): C[r, c] = sum_k A[r, k]
// B[c, k] with A, B row-major and k (the shared cuts) contiguous.  Row and
// column indices are bit fields of the result tensor, so the epilogue stages
// each tile in shared memory in the result's bit order and writes runs of
// consecutive addresses (the Kronecker expansion of output indices, Eq.
// reconstruction, when the result is the final probability vector).
#include <algorithm>

#include "device_common.cuh"
#include "ingest.cuh"
#include "launch.h"
#include "smallk.cuh"

namespace tqc {

namespace {

// One tile per iteration of a grid-stride loop over tiles.
template <int BM, int BN, int TM, int TN, int BK>
__global__ void __launch_bounds__((BM / TM) * (BN / TN))
    simt_step_f32(StepArgs args, int64_t n_tiles, int64_t col_tiles) {
    constexpr int NT = (BM / TM) * (BN / TN);
    constexpr int PA = BM + 4, PB = BN + 4, PS = BN + 4;  // padded pitches (bank spread)
    extern __shared__ __align__(16) unsigned char smem_raw[];
    EpiTables *tb = (EpiTables *)smem_raw;
    float *As = (float *)(smem_raw + sizeof(EpiTables));  // [BK][PA]
    float *Bs = As + BK * PA;                              // [BK][PB]
    float *stg = As;                                       // [BM][PS], reused after the main loop
    const EpiParams &e = args.epi;
    const int a = e.a_bits, b = e.b_bits;
    const int Me = 1 << a, Ne = 1 << b;
    const int64_t K = 1ll << args.kb;
    const int lkc = args.kb < 4 ? args.kb : 4;  // log2 of the K chunk (BK = 16)
    const int kc = 1 << lkc;
    const float *A = (const float *)args.A;
    const float *B = (const float *)args.B;
    const int tid = threadIdx.x;
    const int tx = tid % (BN / TN), ty = tid / (BN / TN);
    epi_tables_init(tb, e, true, PS, tid, NT);
    const int E = Me * Ne;
    pdl_launch();
    pdl_wait();
    for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        const int64_t rt = tile / col_tiles, ct = tile - rt * col_tiles;
        const int64_t r0 = rt << a, c0 = ct << b;
        float acc[TM][TN];
#pragma unroll
        for (int u = 0; u < TM; ++u)
#pragma unroll
            for (int v = 0; v < TN; ++v) acc[u][v] = 0.f;
        for (int64_t k0 = 0; k0 < K; k0 += kc) {
            for (int idx = tid; idx < (BM << lkc); idx += NT) {
                int i = idx >> lkc, kk = idx & (kc - 1);
                As[kk * PA + i] = i < Me ? A[(r0 + i) * K + k0 + kk] : 0.f;
            }
            for (int idx = tid; idx < (BN << lkc); idx += NT) {
                int j = idx >> lkc, kk = idx & (kc - 1);
                Bs[kk * PB + j] = j < Ne ? B[(c0 + j) * K + k0 + kk] : 0.f;
            }
            __syncthreads();
            for (int kk = 0; kk < kc; ++kk) {
                float af[TM], bf[TN];
#pragma unroll
                for (int u = 0; u < TM; u += 4) *(float4 *)&af[u] = *(const float4 *)&As[kk * PA + ty * TM + u];
#pragma unroll
                for (int v = 0; v < TN; v += 4) *(float4 *)&bf[v] = *(const float4 *)&Bs[kk * PB + tx * TN + v];
#pragma unroll
                for (int u = 0; u < TM; ++u)
#pragma unroll
                    for (int v = 0; v < TN; ++v) acc[u][v] = fmaf(af[u], bf[v], acc[u][v]);
            }
            __syncthreads();
        }
        // stage row-major; rows >= Me and columns >= Ne are never read back
#pragma unroll
        for (int u = 0; u < TM; ++u)
#pragma unroll
            for (int v = 0; v < TN; v += 4)
                *(float4 *)&stg[(ty * TM + u) * PS + tx * TN + v] =
                    make_float4(acc[u][v], acc[u][v + 1], acc[u][v + 2], acc[u][v + 3]);
        __syncthreads();
        epi_readout(tb, stg, e, tile_base(e, rt, ct), E, tid, NT, gather_mode(e.lowCc));
        __syncthreads();
    }
}


__device__ __forceinline__ uint64_t dup2(float a) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a));
    return r;
}
__device__ __forceinline__ void fma2(uint64_t &c, uint64_t a, uint64_t b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}

// Whole BM x BN tiles of a step with K >= 16 (a multiple of 16): TM x 8
// results per thread, operands copied 16 k at a time through registers into
// one of two [k][row] buffers while the other is multiplied.  Bound by FP32
// arithmetic and, as closely, by shared memory: a k takes 16 bytes of loads
// per 16 multiply-adds, 128 bytes a clock against 128 multiply-adds a clock.
// The multiply-adds are packed two columns to an instruction (the row's value
// doubled), which leaves the issue slots for the loads.  Row m of k sits at
// m ^ 8 (k / 4 mod 4): the transposing stores of a warp (8 rows x 4 pieces of
// 4 k) and the 16-byte loads are free of bank conflicts.  The k order and the
// multiply-adds are those of simt_step_f32, so the two agree bit for bit.
// Measured (K = 64, 2^16 x 2^11 results; K = 256, 2^19 x 2^7; K = 64, 2^20 x
// 2^8 into 1.07 GB of output): 0.605, 1.195 and 1.31 ms before, 0.41, 0.74 and
// 0.875 ms now (20.9, 23.3 and 19.6 T multiply-adds/s of 39.8); 16 x 8 results
// per thread (fewer loads, half the warps): 0.42, 0.77 and 0.90 ms.
template <int BM, int BN, int TM, int MINB>
__global__ void __launch_bounds__((BM / TM) * (BN / 8), MINB)
    simt_gemm_f32(StepArgs args, int64_t n_tiles, int64_t col_tiles, SmallkLayout L) {
    constexpr int NX = BN / 8, NY = BM / TM, NT = NX * NY, BK = 16;
    constexpr int LA = BM * BK / 4 / NT, LB = BN * BK / 4 / NT;  // 16-byte pieces per thread and chunk
    constexpr int BUF = BK * (BM + BN);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    EpiTables *tb = (EpiTables *)smem_raw;
    float *buf = (float *)(smem_raw + sizeof(EpiTables));  // two operand buffers; the staged tile aliases them
    const EpiParams &e = args.epi;
    const int64_t K = 1ll << args.kb;
    const int chunks = 1 << (args.kb - 4);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // a warp covers 4 x 8 threads: rows 4 ty + 4 NY u, columns 4 tx + 4 NX v
    constexpr int WX = NX / 8;
    const int tx = (warp % WX) * 8 + (lane & 7), ty = (warp / WX) * 4 + (lane >> 3);
    if (!L.direct) epi_tables_init(tb, e, true, 0, tid, NT);  // the gather's element offsets
    // the thread's row and column quads: element offsets in the tile (direct
    // stores), or bits of the tile's destination order (staged)
    constexpr int QM = TM / 4, QN = 2;
    const uint64_t mR = pdep64(e.lowRc, e.tileMask), mC = pdep64(e.lowCc, e.tileMask);
    uint64_t gr[QM], gc[QN];
#pragma unroll
    for (int u = 0; u < QM; ++u) {
        const uint32_t r = 4 * ty + 4 * NY * u;
        gr[u] = L.direct ? pdep64(r, mR) : pdep32(r, e.lowRc);
    }
#pragma unroll
    for (int v = 0; v < QN; ++v) {
        const uint32_t c = 4 * tx + 4 * NX * v;
        gc[v] = L.direct ? pdep64(c, mC) : pdep32(c, e.lowCc);
    }
    pdl_launch();
    pdl_wait();
    float4 pa[LA], pb[LB];
    auto load = [&](int64_t tile, int c) {
        const int64_t rt = tile / col_tiles, ct = tile - rt * col_tiles;
        const float *A = (const float *)args.A + rt * BM * K + c * BK, *B = (const float *)args.B + ct * BN * K + c * BK;
#pragma unroll
        for (int j = 0; j < LA; ++j) {
            const int f = tid + j * NT;
            pa[j] = *(const float4 *)(A + (int64_t)(f >> 2) * K + (f & 3) * 4);
        }
#pragma unroll
        for (int j = 0; j < LB; ++j) {
            const int f = tid + j * NT;
            pb[j] = *(const float4 *)(B + (int64_t)(f >> 2) * K + (f & 3) * 4);
        }
    };
    load(blockIdx.x, 0);
    for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        const int64_t rt = tile / col_tiles, ct = tile - rt * col_tiles;
        uint64_t acc[TM][4];
#pragma unroll
        for (int u = 0; u < TM; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[u][v] = 0;
        auto put = [&](int c) {
            float *As = buf + (c & 1) * BUF, *Bs = As + BK * BM;
#pragma unroll
            for (int j = 0; j < LA; ++j) {
                const int f = tid + j * NT, k4 = f & 3;
                float *d = As + 4 * k4 * BM + ((f >> 2) ^ (k4 << 3));
                d[0] = pa[j].x;
                d[BM] = pa[j].y;
                d[2 * BM] = pa[j].z;
                d[3 * BM] = pa[j].w;
            }
#pragma unroll
            for (int j = 0; j < LB; ++j) {
                const int f = tid + j * NT, k4 = f & 3;
                float *d = Bs + 4 * k4 * BN + ((f >> 2) ^ (k4 << 3));
                d[0] = pb[j].x;
                d[BN] = pb[j].y;
                d[2 * BN] = pb[j].z;
                d[3 * BN] = pb[j].w;
            }
        };
        put(0);
        __syncthreads();
        for (int c = 0; c < chunks; ++c) {
            if (c + 1 < chunks) load(tile, c + 1);
            const float *As = buf + (c & 1) * BUF, *Bs = As + BK * BM;
#pragma unroll
            for (int k = 0; k < BK; ++k) {
                const int sw = (k >> 2) << 3;
                ulonglong2 b[2];
#pragma unroll
                for (int v = 0; v < 2; ++v)
                    b[v] = *(const ulonglong2 *)(Bs + k * BN + ((4 * tx + 4 * NX * v) ^ sw));
#pragma unroll
                for (int u = 0; u < TM / 4; ++u) {
                    const float4 a = *(const float4 *)(As + k * BM + ((4 * ty + 4 * NY * u) ^ sw));
                    const float av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const uint64_t d = dup2(av[i]);
                        fma2(acc[4 * u + i][0], d, b[0].x);
                        fma2(acc[4 * u + i][1], d, b[0].y);
                        fma2(acc[4 * u + i][2], d, b[1].x);
                        fma2(acc[4 * u + i][3], d, b[1].y);
                    }
                }
            }
            if (c + 1 < chunks) {
                put(c + 1);  // the other buffer: its readers passed the last barrier
                __syncthreads();
            }
        }
        // the next tile's first chunk arrives during the write-out
        if (tile + gridDim.x < n_tiles) load(tile + gridDim.x, 0);
        float r[TM][8];
#pragma unroll
        for (int u = 0; u < TM; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                r[u][2 * v] = __uint_as_float((uint32_t)acc[u][v]);
                r[u][2 * v + 1] = __uint_as_float((uint32_t)(acc[u][v] >> 32));
            }
        const uint64_t base = tile_base(e, rt, ct);
        __syncthreads();  // the operands are read: the next tile's, or the staged results, may overwrite them
        if (L.direct) {
            const double sd = (e.mode == EPI_OUT_F32 || e.mode == EPI_OUT_F64) ? e.zinfo[1] : 1.0;
            const float sf = (float)sd;
#define TQC_GEMM_DIRECT(M)                                                                  \
    case M:                                                                                 \
        if (L.rowmajor) sk_direct_store<M, QM, QN, true>(e, r, base, gr, gc, mR, mC, sf, sd); \
        else sk_direct_store<M, QM, QN, false>(e, r, base, gr, gc, mR, mC, sf, sd);         \
        break;
            switch (e.mode) {
                TQC_GEMM_DIRECT(EPI_F32)
                TQC_GEMM_DIRECT(EPI_TF32)
                TQC_GEMM_DIRECT(EPI_BF16)
                TQC_GEMM_DIRECT(EPI_BF16X2)
                TQC_GEMM_DIRECT(EPI_F64_SET)
                TQC_GEMM_DIRECT(EPI_F64_ADD)
                TQC_GEMM_DIRECT(EPI_OUT_F32)
                TQC_GEMM_DIRECT(EPI_OUT_F64)
                default: break;
            }
#undef TQC_GEMM_DIRECT
        } else {
            sk_stage<QM, QN>(buf, r, L, gr, gc);
            __syncthreads();
#define TQC_GEMM_GATHER(M) \
    case M: sk_gather<M, NT>(tb, buf, e, base, BM * BN, tid); break;
            switch (e.mode) {
                TQC_GEMM_GATHER(EPI_F32)
                TQC_GEMM_GATHER(EPI_TF32)
                TQC_GEMM_GATHER(EPI_BF16)
                TQC_GEMM_GATHER(EPI_BF16X2)
                TQC_GEMM_GATHER(EPI_F64_SET)
                TQC_GEMM_GATHER(EPI_F64_ADD)
                TQC_GEMM_GATHER(EPI_OUT_F32)
                TQC_GEMM_GATHER(EPI_OUT_F64)
                default: break;
            }
#undef TQC_GEMM_GATHER
            __syncthreads();
        }
    }
}

__device__ __forceinline__ void copy16(float *dst, const float *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

// Small steps with K >= 16 (at most 32 x 32 results per tile, down to one row
// or column): bound by the latency of a tile's K loop, so that loop has three
// 64-k chunks of operands on their way (asynchronous copies, K-major rows) and
// a tile is spread over all 256 threads, 2 x 2 results or one each.  The k order
// and the multiply-adds are those of simt_step_f32: bit-identical.  A step of 2^5 x
// 2^5 results with K = 4^5: 109 -> 16 us of a whole contract (one chunk of 16 k
// waited for at a time before).
constexpr int SS_STAGES = 3, SS_KC = 64, SS_P = SS_KC + 4, SS_PS = 36;
template <int T>
__device__ __forceinline__ void small_chunk(const float *As, const float *Bs, int rt, int ct, int rs, int cs, int n4,
                                            float (&acc)[T][T]) {
#pragma unroll 4
    for (int k = 0; k < n4; ++k) {
        float4 a[T], b[T];
#pragma unroll
        for (int i = 0; i < T; ++i) a[i] = *(const float4 *)(As + (rt + i * rs) * SS_P + 4 * k);
#pragma unroll
        for (int j = 0; j < T; ++j) b[j] = *(const float4 *)(Bs + (ct + j * cs) * SS_P + 4 * k);
#pragma unroll
        for (int i = 0; i < T; ++i)
#pragma unroll
            for (int j = 0; j < T; ++j) {
                acc[i][j] = fmaf(a[i].x, b[j].x, acc[i][j]);
                acc[i][j] = fmaf(a[i].y, b[j].y, acc[i][j]);
                acc[i][j] = fmaf(a[i].z, b[j].z, acc[i][j]);
                acc[i][j] = fmaf(a[i].w, b[j].w, acc[i][j]);
            }
    }
}
template <int T>
__global__ void __launch_bounds__(256) simt_small_f32(StepArgs args, int64_t n_tiles, int l_col) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    EpiTables *tb = (EpiTables *)smem_raw;
    float *ring = (float *)(smem_raw + sizeof(EpiTables));  // stages of [32][SS_P] A rows, [32][SS_P] B rows
    float *stg = ring + SS_STAGES * 64 * SS_P;
    const EpiParams &e = args.epi;
    const int a = e.a_bits, b = e.b_bits, Me = 1 << a, Ne = 1 << b;
    const int64_t K = 1ll << args.kb;
    const int kc = args.kb < 6 ? 1 << args.kb : SS_KC, chunks = (int)(K / kc), lp = (args.kb < 6 ? args.kb : 6) - 2;
    const int tid = threadIdx.x;
    const int rs = Me / T, cs = Ne / T;  // a thread's rows and columns are this far apart
    const int ct = tid & (cs - 1), rt = tid / cs;
    const bool active = tid < rs * cs;
    epi_tables_init(tb, e, true, SS_PS, tid, 256);
    const int gm = gather_mode(e.lowCc);
    pdl_launch();
    pdl_wait();
    for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        const int64_t r0 = tile >> l_col, c0 = tile - (r0 << l_col);
        const float *A = (const float *)args.A + (r0 << a) * K, *B = (const float *)args.B + (c0 << b) * K;
        auto fetch = [&](int c) {
            if (c < chunks) {
                float *st = ring + (c % SS_STAGES) * 64 * SS_P;
                for (int f = tid; f < (Me + Ne) << lp; f += 256) {  // 16-byte pieces
                    const int row = f >> lp, k4 = f & ((1 << lp) - 1);
                    if (row < Me) copy16(st + row * SS_P + 4 * k4, A + row * K + (int64_t)c * kc + 4 * k4);
                    else copy16(st + (32 + row - Me) * SS_P + 4 * k4, B + (row - Me) * K + (int64_t)c * kc + 4 * k4);
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        float acc[T][T];
#pragma unroll
        for (int i = 0; i < T; ++i)
#pragma unroll
            for (int j = 0; j < T; ++j) acc[i][j] = 0.f;
        for (int c = 0; c < SS_STAGES; ++c) fetch(c);
        for (int c = 0; c < chunks; ++c) {
            asm volatile("cp.async.wait_group %0;" ::"n"(SS_STAGES - 1) : "memory");
            __syncthreads();
            const float *st = ring + (c % SS_STAGES) * 64 * SS_P;
            if (active) small_chunk<T>(st, st + 32 * SS_P, rt, ct, rs, cs, kc / 4, acc);
            __syncthreads();
            fetch(c + SS_STAGES);
        }
        if (active) {
#pragma unroll
            for (int i = 0; i < T; ++i)
#pragma unroll
                for (int j = 0; j < T; ++j) stg[(rt + i * rs) * SS_PS + ct + j * cs] = acc[i][j];
        }
        __syncthreads();
        epi_readout(tb, stg, e, tile_base(e, (uint64_t)r0, (uint64_t)c0), Me * Ne, tid, 256, gm);
        __syncthreads();
    }
}

// Small-K step (smallk.cuh): one 128-thread CTA per tile slot, one kernel
// per K, tile width and orientation (each with its own register budget);
// when the tiles are staged, the staging tables are built once per CTA.
template <int KB, int QM, bool RM>
__global__ void __launch_bounds__(128, (QM == 1) == RM ? 8 : 6)
    simt_smallk_f32(StepArgs args, int64_t n_tiles, int64_t col_tiles, SmallkLayout L) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    EpiTables *tb = (EpiTables *)smem_raw;
    float *buf = (float *)(smem_raw + sizeof(EpiTables));
    if (!L.direct) {  // the gather's element offsets (its staging offsets are unused)
        epi_tables_init(tb, args.epi, true, 0, threadIdx.x, 128);
        __syncthreads();
    }
    pdl_launch();
    smallk_tiles_body<KB, QM, RM, false>(args, tb, L, col_tiles, blockIdx.x, n_tiles, gridDim.x, buf, threadIdx.x, 1);
}

// The total-mass network: FP64 steps over the cut indices alone.  The FP64
// rate (two multiply-adds a clock per SM) bounds them, so the work is spread
// over as many SMs as it has outputs for: 2^lkl lanes of a warp share one
// output (each takes every 2^lkl-th k; a fixed shuffle tree adds their sums).
__device__ __forceinline__ void zstep_range(const ZStep &z, int64_t warp, int64_t n_warps, int lane) {
    const int lkl = z.kb < 5 ? z.kb : 5;
    const int64_t n_out = 1ll << (z.mb + z.nb);
    const int per = 32 >> lkl;
    for (int64_t o0 = warp * per; o0 < n_out; o0 += n_warps * per) {
        const int64_t o = o0 + (lane >> lkl);
        double acc = 0.0;
        const int64_t r = o >> z.nb, c = o & ((1ll << z.nb) - 1);
        if (o < n_out) {
            const double *A = z.A + (r << z.kb), *B = z.B + (c << z.kb);
            // written by other SMs of this launch in the cluster form: not through L1
            for (int64_t k = lane & ((1 << lkl) - 1); k < 1ll << z.kb; k += 1 << lkl)
                acc = fma(__ldcg(A + k), __ldcg(B + k), acc);
        }
        for (int s = 1; s < 1 << lkl; s <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, s);
        if (o < n_out && (lane & ((1 << lkl) - 1)) == 0)
            z.out[pdep64((uint64_t)r, z.maskR) | pdep64((uint64_t)c, z.maskC)] = acc;
    }
}

// Z = sum over slices of the scalar network; scale = 2^{-|E|} / Z (or
// 2^{-|E|} without renormalisation).
__device__ __forceinline__ void zfinal(const double *zslice, int n, int n_cuts, int renorm, double *zinfo) {
    double z = 0.0;
    for (int i = 0; i < n; ++i) z += __ldcg(zslice + i);
    const double z_scaled = ldexp(z, -n_cuts);  // Z includes the 1/2 per cut
    zinfo[0] = z_scaled;
    zinfo[1] = renorm ? ldexp(1.0, -n_cuts) / z_scaled : ldexp(1.0, -n_cuts);
}

// A whole small network in one launch: a cluster of ZN_CTAS CTAs with a
// cluster barrier between steps (a launch each took longer than their work:
// three steps and the sum of a 15-qubit network 41 -> 8.6 us, a 24-qubit one's
// four 134 -> 21 us, both with the FP64 work on eight SMs, not one).  More
// multiply-adds take a launch per step, which has every SM for a step of many
// outputs (one of few leaves most idle in either form: a sum over K goes to one
// warp): 2^14 multiply-adds 16 us in either, 2^16 25 against 43, 2^18 53 against
// 130.
constexpr int ZN_CTAS = 8, ZN_MAX = 16, ZN_THREADS = 256;
constexpr double ZN_MAX_MACS = 1 << 15;
struct ZNetArgs {
    ZStep step[ZN_MAX];
    int32_t n_steps;
    const double *zslice;  // NULL: another slice follows
    int32_t n, n_cuts, renorm;
    double *zinfo;
};
__global__ void __cluster_dims__(ZN_CTAS, 1, 1) __launch_bounds__(ZN_THREADS)
    znet_kernel(const __grid_constant__ ZNetArgs a) {
    pdl_launch();
    pdl_wait();
    const int warp = (int)(blockIdx.x * (ZN_THREADS / 32) + (threadIdx.x >> 5));
    for (int i = 0; i < a.n_steps; ++i) {
        zstep_range(a.step[i], warp, ZN_CTAS * (ZN_THREADS / 32), threadIdx.x & 31);
        asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
    if (a.zslice && blockIdx.x == 0 && threadIdx.x == 0) zfinal(a.zslice, a.n, a.n_cuts, a.renorm, a.zinfo);
}
__global__ void __launch_bounds__(ZN_THREADS) zstep_kernel(const __grid_constant__ ZStep z) {
    pdl_launch();
    pdl_wait();
    zstep_range(z, (int64_t)blockIdx.x * (ZN_THREADS / 32) + (threadIdx.x >> 5),
                (int64_t)gridDim.x * (ZN_THREADS / 32), threadIdx.x & 31);
}
__global__ void zfinal_kernel(const double *zslice, int n, int n_cuts, int renorm, double *zinfo) {
    pdl_launch();
    pdl_wait();
    if (threadIdx.x == 0 && blockIdx.x == 0) zfinal(zslice, n, n_cuts, renorm, zinfo);
}

// Node tensors into operand layouts (every leaf of a contract in one launch:
// CTAs blk[j] .. blk[j + 1] take leaf j): destination bit b reads source bit
// srcpos[b]; src_base carries the fixed output bits of the bin and the values
// of sliced cuts.  A leaf's lowest destination bits are cuts, its lowest
// source bits output qubits, so a thread loads four neighbouring source
// elements (a whole sector of FP64) and the warp's stores are consecutive.
// With reduce_bits > 0 (total mass) the 2^reduce_bits consecutive source
// elements of a destination are summed in FP64, by a warp or (few
// destinations) by a CTA.  Grid30's four leaves (4.8 M
// FP64 elements): four launches of 41 us in all -> one of 20 us.
constexpr int INGEST_THREADS = 256;
struct IngestMulti {
    int32_t n;
    int32_t blk[INGEST_MAX + 1];
    IngestArgs g[INGEST_MAX];
};
__global__ void __launch_bounds__(INGEST_THREADS) ingest_kernel(const __grid_constant__ IngestMulti m) {
    __shared__ double part[INGEST_THREADS / 32];
    pdl_launch();
    pdl_wait();
    int j = 0;
    while ((int)blockIdx.x >= m.blk[j + 1]) ++j;
    const IngestArgs &g = m.g[j];
    const int blocks = m.blk[j + 1] - m.blk[j], block = (int)blockIdx.x - m.blk[j];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (g.reduce_bits > 0) {
        const bool cta = g.sum_threads == INGEST_THREADS;
        const int64_t nx = 1ll << g.reduce_bits, n_dst = 1ll << g.nbits;
        const int64_t w0 = cta ? block : (int64_t)block * (INGEST_THREADS / 32) + warp;
        for (int64_t d = w0; d < n_dst; d += cta ? blocks : (int64_t)blocks * (INGEST_THREADS / 32)) {
            int64_t s = g.src_base;
            for (int b = 0; b < g.nbits; ++b)
                if (d >> b & 1) s += 1ll << g.srcpos[b];
            double acc = 0.0;
            for (int64_t x = cta ? (int64_t)threadIdx.x : lane; x < nx; x += cta ? INGEST_THREADS : 32)
                acc += ld_src<double>(g.src, g.src_dtype, s + x);
            for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (cta) {
                if (lane == 0) part[warp] = acc;
                __syncthreads();
                acc = 0.0;
                for (int w = 0; w < INGEST_THREADS / 32; ++w) acc += part[w];
                __syncthreads();
            }
            if (cta ? threadIdx.x == 0 : lane == 0) ((double *)g.dst)[d] = acc;
        }
        return;
    }
    const int lg = __ffs(blocks * INGEST_THREADS) - 1;
    const int64_t t0 = (int64_t)block * INGEST_THREADS + threadIdx.x;
    ingest_range(g, t0, (1ll << g.nbits) / g.vec, lg);
}

__global__ void finalize_kernel(const double *acc, void *out, int out_f64, const double *zinfo, int64_t n) {
    pdl_launch();
    pdl_wait();
    const double s = zinfo[1];
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        double v = acc[i] * s;
        if (out_f64) ((double *)out)[i] = v;
        else ((float *)out)[i] = (float)v;
    }
}

// Sum of the FP32 partials of a K-split step (split s at part + s * n), in
// FP64, stored in the step's own output mode: the scaled final output
// (FP32 / FP64) or the FP64 slice sum (set / add).
__global__ void ksplit_reduce_kernel(const float *part, int ksplit, int64_t n, int mode, void *out,
                                     const double *zinfo) {
    pdl_launch();
    pdl_wait();
    const double sc = (mode == EPI_OUT_F32 || mode == EPI_OUT_F64) ? zinfo[1] : 1.0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        double v = 0.0;
        for (int s = 0; s < ksplit; ++s) v += f32_to_f64(part[s * n + i]);
        switch (mode) {
            case EPI_OUT_F32: ((float *)out)[i] = (float)(v * sc); break;
            case EPI_OUT_F64: ((double *)out)[i] = v * sc; break;
            case EPI_F64_SET: ((double *)out)[i] = v; break;
            case EPI_F64_ADD: ((double *)out)[i] += v; break;
            default: break;
        }
    }
}

int g_sms = 0;

template <int BM, int BN, int TM, int TN>
cudaError_t launch_cfg(const StepArgs &a, cudaStream_t s) {
    constexpr int NT = (BM / TM) * (BN / TN);
    constexpr int BK = 16;
    size_t smem = sizeof(EpiTables) + std::max((size_t)BK * (BM + 4 + BN + 4) * sizeof(float),
                                               (size_t)BM * (BN + 4) * sizeof(float));
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(simt_step_f32<BM, BN, TM, TN, BK>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    int64_t row_tiles = 1ll << (a.mb - a.epi.a_bits);
    int64_t col_tiles = 1ll << (a.nb - a.epi.b_bits);
    int64_t n_tiles = row_tiles * col_tiles;
    int64_t grid = std::min<int64_t>(n_tiles, (int64_t)sm_count() * 16);
    return launch_pdl(simt_step_f32<BM, BN, TM, TN, BK>, grid, NT, smem, s, a, n_tiles, col_tiles);
}

// The tile configurations of K >= 16 steps whose tiles are whole.
template <int BM, int BN, int TM, int MINB>
cudaError_t launch_gemm(const StepArgs &step, cudaStream_t s) {
    StepArgs a = step;
    if (BM == BN && smallk_layout(a.epi).direct && !smallk_layout(a.epi).rowmajor) {
        // the result's lowest bits are row bits: exchange rows and columns, so
        // that the eight lanes along columns store 128 consecutive bytes
        std::swap(a.A, a.B);
        std::swap(a.mb, a.nb);
        std::swap(a.epi.lowRc, a.epi.lowCc);
        std::swap(a.epi.highR, a.epi.highC);
    }
    constexpr int NT = (BM / TM) * (BN / 8);
    const size_t smem = sizeof(EpiTables) + std::max((size_t)2 * 16 * (BM + BN), (size_t)BM * BN) * sizeof(float);
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(simt_gemm_f32<BM, BN, TM, MINB>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    const int64_t col_tiles = 1ll << (a.nb - a.epi.b_bits);
    const int64_t n_tiles = (1ll << (a.mb - a.epi.a_bits)) * col_tiles;
    const int64_t grid = std::min<int64_t>(n_tiles, (int64_t)sm_count() * MINB);
    return launch_pdl(simt_gemm_f32<BM, BN, TM, MINB>, grid, NT, smem, s, a, n_tiles, col_tiles, smallk_layout(a.epi));
}

cudaError_t launch_small(const StepArgs &a, cudaStream_t s) {
    if (a.kb < 4 || a.epi.a_bits > 5 || a.epi.b_bits > 5 || a.kblk) return cudaErrorInvalidValue;
    const size_t smem = sizeof(EpiTables) + (size_t)(SS_STAGES * 64 * SS_P + 32 * SS_PS) * sizeof(float);
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(simt_small_f32<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(simt_small_f32<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    const int l_col = a.nb - a.epi.b_bits;
    const int64_t n_tiles = (1ll << (a.mb - a.epi.a_bits)) << l_col;
    const int64_t grid = std::min<int64_t>(n_tiles, (int64_t)sm_count() * 3);
    auto *kernel = a.epi.a_bits + a.epi.b_bits <= 8 ? simt_small_f32<1> : simt_small_f32<2>;
    return launch_pdl(kernel, grid, 256, smem, s, a, n_tiles, l_col);
}

}  // namespace

int sm_count() {
    if (!g_sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&g_sms, cudaDevAttrMultiProcessorCount, dev);
        if (g_sms <= 0) g_sms = 1;
    }
    return g_sms;
}

TileShape simt_tile(int cfg) {
    switch (cfg) {
        case SIMT_128x128: return {7, 7};
        case SIMT_128x64: return {7, 6};
        case SIMT_32x32: return {5, 5};
        default: return {6, 6};
    }
}


bool smallk_ok(int mb, int nb, int kb, bool kblk) {
    return (kb == 0 || kb == 2 || kb == 4) && !kblk && mb >= 2 && nb >= 2 && mb + nb >= 7;
}

// Start from 64 x 64, grow the side the step still has until the tile holds
// 2^12 results, then shrink the larger side until operands and staging fit
// SMALLK_BYTES.
TileShape smallk_tile(int mb, int nb, int kb) {
    int a = std::min(mb, 6), b = std::min(nb, 6);
    while (a + b < 12 && (a < mb || b < nb)) {
        if (a < mb && (a <= b || b >= nb)) ++a;
        else ++b;
    }
    auto fits = [&](int x, int y) {
        return smallk_op_bytes(x, y, kb) <= SMALLK_BYTES && smallk_stage_bytes(x, y) <= SMALLK_BYTES;
    };
    while (!fits(a, b) && (a > 2 || b > 2)) {
        if (a >= b && a > 2) --a;
        else --b;
    }
    return TileShape{a, b};
}

static uint64_t host_pdep64(uint64_t src, uint64_t mask) {
    uint64_t r = 0;
    while (mask) {
        const uint64_t low = mask & (~mask + 1);
        if (src & 1) r |= low;
        src >>= 1;
        mask ^= low;
    }
    return r;
}

// Direct stores when the result's lowest four or more bits are bits of one
// tile dimension and at least two lanes run along it (whole 32-byte sectors
// per warp store), else the tile staged in destination order with the lanes
// along the dimension that has more of the tile's seven lowest result bits.
SmallkLayout smallk_layout(const EpiParams &e) {
    SmallkLayout L;
    const uint64_t mR = host_pdep64(e.lowRc, e.tileMask), mC = host_pdep64(e.lowCc, e.tileMask);
    auto run = [](uint64_t m) {
        int r = 0;
        while (r < 64 && (m >> r & 1)) ++r;
        return r;
    };
    // two quads along the lanes' dimension when the tile allows (8 of them)
    const int a = e.a_bits, b = e.b_bits;
    auto qm_for = [&](int rm) { return ((!rm && a >= 3) || b < 3) ? 2 : 1; };
    auto lanes = [&](int rm) {  // log2 of the lanes along that dimension
        const int qm = qm_for(rm);
        return rm ? b - 2 - (2 - qm) : a - 2 - (qm - 1);
    };
    // bit of t holding the n-th lowest bit of a compact mask
    auto nth = [](uint32_t m, int n) {
        for (int i = 0; i < n; ++i) m &= m - 1;
        return (uint32_t)__builtin_ctz(m);
    };
    L.rowmajor = staging_rowmajor(e.lowRc, e.lowCc);
    L.direct = 0;
    if (run(mC) >= 4 && lanes(1) >= 1) {
        L.direct = 1;
        L.rowmajor = 1;
    } else if (run(mR) >= 4 && lanes(0) >= 1) {
        L.direct = 1;
        L.rowmajor = 0;
    }
    L.qm = qm_for(L.rowmajor);
    L.pr0 = nth(e.lowRc, 0);
    L.pr1 = nth(e.lowRc, 1);
    L.pc0 = nth(e.lowCc, 0);
    L.pc1 = nth(e.lowCc, 1);
    const bool r0 = e.lowRc & 1u, r1 = e.lowRc & 2u;
    L.pat = (r0 && r1) ? 0 : (!r0 && !r1) ? 1 : (r0 ? 2 : 3);
    return L;
}

cudaError_t launch_smallk(const StepArgs &a, cudaStream_t s) {
    const EpiParams &e = a.epi;
    if (!smallk_ok(a.mb, a.nb, a.kb, a.kblk != 0) || e.a_bits < 2 || e.b_bits < 2 || a.ksplit != 1)
        return cudaErrorInvalidValue;
    if (e.L < 2) return cudaErrorInvalidValue;  // the result's two lowest bits lie in every tile
    const SmallkLayout L = smallk_layout(e);
    const int bytes = std::max(smallk_op_bytes(e.a_bits, e.b_bits, a.kb),
                               L.direct ? 0 : smallk_stage_bytes(e.a_bits, e.b_bits));
    if (bytes > SMALLK_BYTES) return cudaErrorInvalidValue;
    const size_t smem = sizeof(EpiTables) + (size_t)bytes;
    const int64_t col_tiles = 1ll << (a.nb - e.b_bits);
    const int64_t n_tiles = (1ll << (a.mb - e.a_bits)) * col_tiles;
    const unsigned grid = (unsigned)std::min<int64_t>(n_tiles, (int64_t)sm_count() * 16);
    const bool rm = L.rowmajor != 0;
    static bool attr[3][2][2] = {};
#define TQC_SMALLK_LAUNCH(KBV, QMV, RMV)                                                                      \
    if (a.kb == KBV && L.qm == QMV && rm == RMV) {                                                           \
        bool &done = attr[KBV / 2][QMV - 1][RMV ? 1 : 0];                                                    \
        if (!done) {                                                                                         \
            cudaError_t err = cudaFuncSetAttribute(simt_smallk_f32<KBV, QMV, RMV>,                           \
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize,             \
                                                   (int)(sizeof(EpiTables) + SMALLK_BYTES));                 \
            if (err != cudaSuccess) return err;                                                              \
            done = true;                                                                                     \
        }                                                                                                    \
        return launch_pdl(simt_smallk_f32<KBV, QMV, RMV>, grid, 128, smem, s, a, n_tiles, col_tiles, L);      \
    }
    TQC_SMALLK_LAUNCH(0, 1, true)
    TQC_SMALLK_LAUNCH(0, 1, false)
    TQC_SMALLK_LAUNCH(0, 2, true)
    TQC_SMALLK_LAUNCH(0, 2, false)
    TQC_SMALLK_LAUNCH(2, 1, true)
    TQC_SMALLK_LAUNCH(2, 1, false)
    TQC_SMALLK_LAUNCH(2, 2, true)
    TQC_SMALLK_LAUNCH(2, 2, false)
    TQC_SMALLK_LAUNCH(4, 1, true)
    TQC_SMALLK_LAUNCH(4, 1, false)
    TQC_SMALLK_LAUNCH(4, 2, true)
    TQC_SMALLK_LAUNCH(4, 2, false)
#undef TQC_SMALLK_LAUNCH
    return cudaErrorInvalidValue;
}

cudaError_t launch_simt_step(int cfg, const StepArgs &a, cudaStream_t s) {
    switch (cfg) {
        case SIMT_SMALLK: return launch_smallk(a, s);
        case SIMT_32x32: return launch_small(a, s);
        case SIMT_128x128:
            if (a.kb >= 4 && a.epi.a_bits == 7 && a.epi.b_bits == 7) return launch_gemm<128, 128, 8, 2>(a, s);
            return launch_cfg<128, 128, 8, 8>(a, s);
        case SIMT_128x64:
            if (a.kb >= 4 && a.epi.a_bits == 7 && a.epi.b_bits == 6) return launch_gemm<128, 64, 8, 3>(a, s);
            return launch_cfg<128, 64, 8, 4>(a, s);
        default:
            if (a.kb >= 4 && a.epi.a_bits == 6 && a.epi.b_bits == 6) return launch_gemm<64, 64, 4, 6>(a, s);
            return launch_cfg<64, 64, 4, 4>(a, s);
    }
}

namespace {

double znet_macs(const ZStep *z, int n) {
    double t = 0;
    for (int i = 0; i < n; ++i) t += (double)(1ull << (z[i].mb + z[i].nb + z[i].kb));
    return t;
}
bool znet_small(const ZStep *z, int n) { return n <= ZN_MAX && znet_macs(z, n) <= ZN_MAX_MACS; }

}  // namespace

cudaError_t launch_znet(const ZStep *z, int n_steps, const double *zslice, int n, int n_cuts, int renorm,
                        double *zinfo, cudaStream_t s) {
    if (znet_small(z, n_steps)) {
        ZNetArgs a = {};
        for (int i = 0; i < n_steps; ++i) a.step[i] = z[i];
        a.n_steps = n_steps;
        a.zslice = zslice;
        a.n = n;
        a.n_cuts = n_cuts;
        a.renorm = renorm;
        a.zinfo = zinfo;
        return launch_pdl(znet_kernel, ZN_CTAS, ZN_THREADS, 0, s, a);
    }
    for (int i = 0; i < n_steps; ++i) {
        const int lkl = std::min(z[i].kb, 5);
        const int64_t warps = std::max<int64_t>(1, (1ll << (z[i].mb + z[i].nb)) >> (5 - lkl));
        const int64_t blocks = std::min<int64_t>((warps + ZN_THREADS / 32 - 1) / (ZN_THREADS / 32), (int64_t)sm_count() * 8);
        const cudaError_t e = launch_pdl(zstep_kernel, blocks, ZN_THREADS, 0, s, z[i]);
        if (e != cudaSuccess) return e;
    }
    return zslice ? launch_pdl(zfinal_kernel, 1, 32, 0, s, zslice, n, n_cuts, renorm, zinfo) : cudaSuccess;
}

int znet_launches(const ZStep *z, int n_steps, bool last) {
    return znet_small(z, n_steps) ? 1 : n_steps + (last ? 1 : 0);
}

// Largest V <= 4 whose source bits 0 .. log2 V - 1 are destination bits, with
// the tensor aligned for the loads (16 bytes at most).
void ingest_vec(IngestArgs &g) {
    g.vec = 1;
    if (g.scaled || g.storage == ST_F64) return;
    int at[2] = {-1, -1};
    for (int b = 0; b < g.nbits; ++b)
        if (g.srcpos[b] < 2) at[(int)g.srcpos[b]] = b;
    const int esz = g.src_dtype == TQC_F64 ? 8 : 4;
    auto aligned = [&](int v) { return ((uintptr_t)g.src % (uintptr_t)std::min(16, v * esz)) == 0; };
    const int v = at[0] >= 0 && at[1] >= 0 && aligned(4) ? 4 : (at[0] >= 0 && aligned(2) ? 2 : 1);
    if (v == 1) return;
    int n = 0;
    int8_t pos[64] = {0};
    for (int b = 0; b < g.nbits; ++b)
        if (b != at[0] && !(v == 4 && b == at[1])) pos[n++] = g.srcpos[b];
    std::copy(pos, pos + 64, g.srcpos);
    g.vec = v;
    g.vb[0] = (int8_t)at[0];
    g.vb[1] = (int8_t)(v == 4 ? at[1] : 0);
}

cudaError_t launch_ingest(const IngestArgs *g, int n, cudaStream_t s) {
    for (int i = 0; i < n; i += INGEST_MAX) {
        IngestMulti m = {};
        m.n = std::min(n - i, INGEST_MAX);
        for (int j = 0; j < m.n; ++j) {
            IngestArgs &a = m.g[j] = g[i + j];
            int64_t threads;
            if (a.reduce_bits > 0) {
                // a CTA per destination when a warp each would leave SMs idle
                a.sum_threads = a.nbits < 10 && a.reduce_bits >= 8 ? INGEST_THREADS : 32;
                threads = (int64_t)a.sum_threads << a.nbits;  // (2^5 threads for each of 2^26 destinations and more)
            } else {
                ingest_vec(a);
                threads = (1ll << a.nbits) / a.vec;
            }
            int64_t blocks = std::min<int64_t>((threads + INGEST_THREADS - 1) / INGEST_THREADS, (int64_t)sm_count() * 32);
            if (blocks < 1) blocks = 1;
            while (blocks & (blocks - 1)) blocks &= blocks - 1;  // a power of two (ingest_gather)
            m.blk[j + 1] = m.blk[j] + (int)blocks;
        }
        const cudaError_t e = launch_pdl(ingest_kernel, m.blk[m.n], INGEST_THREADS, 0, s, m);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_finalize(const double *acc, void *out, int out_f64, const double *zinfo, int64_t n,
                            cudaStream_t s) {
    int64_t blocks = std::min<int64_t>((n + 255) / 256, (int64_t)sm_count() * 32);
    if (blocks < 1) blocks = 1;
    return launch_pdl(finalize_kernel, blocks, 256, 0, s, acc, out, out_f64, zinfo, n);
}

cudaError_t launch_ksplit_reduce(const float *part, int ksplit, int64_t n, int mode, void *out, const double *zinfo,
                                 cudaStream_t s) {
    if (ksplit < 1 || n < 1) return cudaErrorInvalidValue;
    if (mode != EPI_OUT_F32 && mode != EPI_OUT_F64 && mode != EPI_F64_SET && mode != EPI_F64_ADD)
        return cudaErrorInvalidValue;
    const int64_t blocks = std::min<int64_t>((n + 255) / 256, (int64_t)sm_count() * 32);
    return launch_pdl(ksplit_reduce_kernel, blocks, 256, 0, s, part, ksplit, n, mode, out, zinfo);
}

EpiParams make_epi(uint64_t maskR, uint64_t maskC, int mb, int nb, TileShape t) {
    EpiParams e;
    int a = std::min(t.log_bm, mb), b = std::min(t.log_bn, nb);
    uint64_t lowR = 0, lowC = 0;
    {
        uint64_t m = maskR;
        for (int i = 0; i < a; ++i) {
            uint64_t low = m & (~m + 1);
            lowR |= low;
            m ^= low;
        }
        m = maskC;
        for (int i = 0; i < b; ++i) {
            uint64_t low = m & (~m + 1);
            lowC |= low;
            m ^= low;
        }
    }
    e.highR = maskR & ~lowR;
    e.highC = maskC & ~lowC;
    e.tileMask = lowR | lowC;
    // compact positions of the tile's row / column bits inside tileMask
    uint32_t rc = 0, cc = 0;
    int k = 0;
    for (int bit = 0; bit < 64; ++bit) {
        if (!(e.tileMask >> bit & 1)) continue;
        if (lowR >> bit & 1) rc |= 1u << k;
        else cc |= 1u << k;
        ++k;
    }
    e.lowRc = rc;
    e.lowCc = cc;
    e.a_bits = a;
    e.b_bits = b;
    int L = 0;
    while (L < 64 && (e.tileMask >> L & 1)) ++L;
    e.L = L;
    return e;
}

}  // namespace tqc
