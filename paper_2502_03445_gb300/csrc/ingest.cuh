// Gather of a node tensor into an operand layout, shared by the ingest kernel
// (simt.cu) and the batched launch (batch.cu).
#pragma once

#include "device_common.cuh"

namespace tqc {

template <typename T>
__device__ __forceinline__ T ld_src(const void *p, int dtype, int64_t i) {
    return dtype == TQC_F64 ? (T)((const double *)p)[i] : (T)((const float *)p)[i];
}

// FP64 bits -> nearest FP32 (ties to even), the conversion instruction's
// result, in integer arithmetic for normal results: the instruction runs at
// the FP64 rate, which held grid30's largest leaf (2^22 elements) to 24 us.
__device__ __forceinline__ float f64_to_f32(uint64_t b) {
    const uint32_t hi = (uint32_t)(b >> 32), lo = (uint32_t)b;
    const uint32_t e = (hi >> 20) & 0x7ffu;
    if (e - 897u > 253u) return (float)__longlong_as_double((long long)b);  // zero, subnormal, overflow, inf, NaN
    uint32_t u = __funnelshift_l(lo, hi, 3) - (896u << 23);  // exponent rebased (modulo 512), 23 mantissa bits
    u += ((lo << 3) | (u & 1u)) > 0x80000000u;                // round to nearest even; a carry is right
    return __uint_as_float(u | (hi & 0x80000000u));
}

// V source elements from element s on (V > 1: the address is a multiple of V elements).
template <int V>
__device__ __forceinline__ void ingest_load(const IngestArgs &g, int64_t s, float (&v)[V]) {
    if (g.src_dtype == TQC_F64) {
        const double *p = (const double *)g.src + s;
        if constexpr (V == 1) {
            v[0] = f64_to_f32((uint64_t)__double_as_longlong(__ldg(p)));
        } else {
#pragma unroll
            for (int i = 0; i < V; i += 2) {
                const ulonglong2 q = __ldg((const ulonglong2 *)(p + i));
                v[i] = f64_to_f32(q.x);
                v[i + 1] = f64_to_f32(q.y);
            }
        }
    } else {
        const float *p = (const float *)g.src + s;
        if constexpr (V == 4) {
            const float4 q = __ldg((const float4 *)p);
            v[0] = q.x;
            v[1] = q.y;
            v[2] = q.z;
            v[3] = q.w;
        } else if constexpr (V == 2) {
            const float2 q = __ldg((const float2 *)p);
            v[0] = q.x;
            v[1] = q.y;
        } else {
            v[0] = __ldg(p);
        }
    }
}

// Gather a leaf: index t (of 2^nbits / V) stands for V neighbouring source
// elements, whose destinations differ in bits vb[0] (and vb[1]).  The calling
// thread takes t0, t0 + 2^lg, ... below n: its t share their lg low bits, so
// that part of the source offset is summed once.
template <int V>
__device__ __forceinline__ void ingest_gather(const IngestArgs &g, int64_t t0, int64_t n, int lg) {
    const int nb = g.nbits - (V == 4 ? 2 : (V == 2 ? 1 : 0));  // bits of t: srcpos[0 .. nb)
    const int64_t stride = 1ll << lg;
    int64_t s_lo = g.src_base;
    for (int b = 0; b < nb && b < lg; ++b)
        if (t0 >> b & 1) s_lo += 1ll << g.srcpos[b];
    const int p0 = V == 4 ? (g.vb[0] < g.vb[1] ? g.vb[0] : g.vb[1]) : g.vb[0];
    const int p1 = V == 4 ? (g.vb[0] < g.vb[1] ? g.vb[1] : g.vb[0]) : 0;
    const int64_t d1 = 1ll << g.vb[0], d2 = V == 4 ? 1ll << g.vb[1] : 0;
    for (int64_t t = t0; t < n; t += stride) {
        int64_t s = s_lo;
        for (int b = lg; b < nb; ++b)
            if (t >> b & 1) s += 1ll << g.srcpos[b];
        int64_t d = t;  // destination of the first: zero bits inserted at vb
        if (V >= 2) d = ((d >> p0) << (p0 + 1)) | (d & ((1ll << p0) - 1));
        if (V == 4) d = ((d >> p1) << (p1 + 1)) | (d & ((1ll << p1) - 1));
        auto at = [&](int i) { return d + ((i & 1) ? d1 : 0) + ((i & 2) ? d2 : 0); };
        if (g.scaled || g.storage == ST_F64) {
#pragma unroll
            for (int i = 0; i < V; ++i) {
                const double x = ld_src<double>(g.src, g.src_dtype, s + i);
                if (!g.scaled) ((double *)g.dst)[at(i)] = x;
                else if (g.out_f64) ((double *)g.dst)[at(i)] = x * g.zinfo[1];
                else ((float *)g.dst)[at(i)] = (float)(x * g.zinfo[1]);
            }
            continue;
        }
        float v[V];
        ingest_load<V>(g, s, v);
        switch (g.storage) {
            case ST_F32:
#pragma unroll
                for (int i = 0; i < V; ++i) ((float *)g.dst)[at(i)] = v[i];
                break;
            case ST_TF32:
#pragma unroll
                for (int i = 0; i < V; ++i) ((float *)g.dst)[at(i)] = to_tf32(v[i]);
                break;
            case ST_BF16:
#pragma unroll
                for (int i = 0; i < V; ++i) ((__nv_bfloat16 *)g.dst)[at(i)] = __float2bfloat16_rn(v[i]);
                break;
            case ST_BF16X2:
                // hi = bf16(v), lo = bf16(v - hi) from the FP32 value (v - hi is exact in FP32)
#pragma unroll
                for (int i = 0; i < V; ++i) {
                    const __nv_bfloat16 h = __float2bfloat16_rn(v[i]);
                    ((__nv_bfloat16 *)g.dst)[at(i)] = h;
                    ((__nv_bfloat16 *)g.dst_lo)[at(i)] = __float2bfloat16_rn(v[i] - __bfloat162float(h));
                }
                break;
            default: break;
        }
    }
}

__device__ __forceinline__ void ingest_range(const IngestArgs &g, int64_t t0, int64_t n, int lg) {
    if (g.vec == 4) ingest_gather<4>(g, t0, n, lg);
    else if (g.vec == 2) ingest_gather<2>(g, t0, n, lg);
    else ingest_gather<1>(g, t0, n, lg);
}

}  // namespace tqc
