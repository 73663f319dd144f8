// Heavy state selection (§IV, Alg. heavy_state_selection).
//
// Step 1 runs on the device: for every output state i of subcircuit C_j, the
// L2 norm of its entries over all cut assignments e,
//     ||p_{j,i}|| = sqrt(sum_e T_j[e][i]^2),
// a column reduction of the [4^c][2^o] node tensor (FP64 sums in a fixed
// order, so equal tensors give bit-identical norms and ties resolve the same
// way on every call).  Step 2 (seed each subcircuit
// with its heaviest state, then add states in descending norm until the
// product of the per-subcircuit counts reaches s_max) orders a few thousand
// numbers and runs on the host.  The selected states become a new network
// whose subcircuit j keeps only those rows (gathered on the device, padded
// with zero rows to a power of two); its outputs are the per-subcircuit
// selection indices, subcircuit 0's bits lowest, so the ordinary plan /
// contract path reconstructs the product set.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "launch.h"
#include "tqc_internal.h"

struct tqc_net {
    tqc::Net n;
};

namespace tqc {
namespace {

// norm[x] = sqrt(sum_e T[e][x]^2).  A CTA takes 2^lx states per warp (32, or
// all of fewer) and, in its eight warps, wr row groups times 8 / wr groups of
// states; the rows are further split over a cluster of gridDim.y CTAs, whose
// sums the first one reads through distributed shared memory, and (large
// tensors of few states) over gridDim.z clusters, whose sums hss_root_kernel
// adds.  Every sum is formed in a fixed order: lane, row group, cluster rank,
// cluster.  Bound by latency: a lane waits for one batch of 16 loads at a time
// (2-4 us with few warps on an SM).  The four tensors of the 30-qubit grid (38
// MB: 5.7 us of HBM, 7.8 us at the FP64 rate of two multiply-adds a clock per
// SM) in four calls: 151 us with up to 586 partial sums per state added in one
// thread of a second kernel, 55 with clusters, 48 with fewer states per warp
// where few CTAs would run (32 for the 128-state tensor, now 128); 35 when the
// tensors are still in L2.
template <typename V>
__global__ void __launch_bounds__(256)
    hss_norms_kernel(const V *__restrict__ T, int64_t n_x, int64_t n_e, int lx, int wr, double *out) {
    __shared__ double part[8][32];
    __shared__ double tot[256];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = warp & (wr - 1), wx = warp / wr;               // row group; group of states
    const int64_t x0 = ((int64_t)blockIdx.x * (8 / wr) + wx) << lx;
    const int64_t x = x0 + (lane & ((1 << lx) - 1));
    const int64_t rows = (int64_t)gridDim.z * gridDim.y * wr << (5 - lx);  // rows apart
    double acc = 0.0;
    if (x < n_x) {
        const V *p = T + x;
        const int64_t e0 = ((((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * wr + g) << (5 - lx)) + (lane >> lx);
        int64_t e = e0;
        for (; e + 15 * rows < n_e; e += 16 * rows) {  // sixteen loads in flight
            V v[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = __ldg(p + (e + i * rows) * n_x);
#pragma unroll
            for (int i = 0; i < 16; ++i) acc += (double)v[i] * (double)v[i];
        }
        for (; e < n_e; e += rows) {
            const double v = (double)__ldg(p + e * n_x);
            acc += v * v;
        }
    }
    for (int o = 1 << lx; o < 32; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    part[warp][lane] = acc;
    __syncthreads();
    if (g == 0) {
        double t = 0.0;
        for (int w = 0; w < wr; ++w) t += part[wx * wr + w][lane];
        tot[wx * 32 + lane] = t;
    }
    if (gridDim.y > 1)
        asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (blockIdx.y == 0 && g == 0 && x < n_x && lane < 1 << lx) {
        double t = tot[wx * 32 + lane];
        const uint32_t mine = (uint32_t)__cvta_generic_to_shared(&tot[wx * 32 + lane]);
        for (uint32_t r = 1; r < gridDim.y; ++r) {
            uint32_t at;
            double v;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"(mine), "r"(r));
            asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(at) : "memory");
            t += v;
        }
        if (gridDim.z > 1) out[blockIdx.z * n_x + x] = t;
        else out[x] = sqrt(t);
    }
    if (gridDim.y > 1)  // the other CTAs' shared memory stays until it has been read
        asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// norm[x] = sqrt of the sum of the n clusters' part[z][x]: a warp per state.
__global__ void __launch_bounds__(256) hss_root_kernel(const double *part, int n, int64_t n_x, double *norm) {
    const int lane = threadIdx.x & 31;
    const int64_t x = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (x >= n_x) return;
    double t = 0.0;
    for (int z = lane; z < n; z += 32) t += part[z * n_x + x];
    for (int o = 1; o < 32; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) norm[x] = sqrt(t);
}

// out[e][r] = r < count ? T[e][states[r]] : 0   (r < 2^k)
template <typename V>
__global__ void hss_gather_kernel(const V *T, int64_t n_x, int64_t n_e, const int32_t *states, int32_t count, int k,
                                  V *out) {
    const int64_t n_r = (int64_t)1 << k;
    const int64_t total = n_e * n_r;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = i >> k, r = i & (n_r - 1);
        out[i] = r < count ? T[e * n_x + states[r]] : (V)0;
    }
}

template <typename V>
cudaError_t launch_norms(const Node &nd, double *d_norms, cudaStream_t s) {
    const int64_t n_x = (int64_t)1 << nd.out_qubits.size(), n_e = (int64_t)1 << (2 * nd.cut_ids.size());
    int lx = (int)std::min<size_t>(5, nd.out_qubits.size());
    const int wr = (int)std::min<int64_t>(8, n_e);  // 1, 4 or 8
    // up to eight CTAs share the rows, while a lane has at least eight of them
    int ys = 1;
    while (ys < 8 && n_e >= ((int64_t)16 * wr * ys << (5 - lx))) ys *= 2;
    // Few states leave SMs idle even so: a warp then takes more rows of fewer
    // states, down to eight (a whole 32-byte sector of FP32), while a lane
    // keeps the 16 rows that it loads at once.
    while (lx > 3 && (n_x >> lx) * wr * ys < 8 * (int64_t)sm_count() && n_e >= ((int64_t)32 * wr * ys << (5 - lx))) --lx;
    const int64_t per = (int64_t)(8 / wr) << lx;  // states of a CTA
    const int64_t xs = (n_x + per - 1) / per;
    // Fewer CTAs than SMs, or (tensors beyond L2) than twice as many, with 128
    // rows or more per lane: the rows are split over up to 14 CTAs per SM, with
    // at least 32 rows per lane left.  The second launch and its scratch
    // (stream-ordered, some ten KB) cost 9 us of host time, what 128 rows take.
    // FP64, 4^9 rows of 8 states: 92 -> 20 us; 4^10 of 16: 812 -> 50; 4^7 of 2^10:
    // 66 -> 47; FP32, 4^10 of 16: 582 -> 87.
    const int64_t sms = sm_count(), ctas = xs * ys;
    const int64_t r = n_e / ((int64_t)wr * ys << (5 - lx));  // rows per lane
    int64_t zs = 1;
    if (r >= 128 && (ctas < sms || (ctas < 2 * sms && n_x * n_e * (int64_t)sizeof(V) >= (int64_t)128 << 20)))
        while (2 * zs * ctas <= 14 * sms && r >= 64 * zs) zs *= 2;
    double *part = d_norms;
    if (zs > 1) {
        const cudaError_t e = cudaMallocAsync((void **)&part, sizeof(double) * (size_t)(zs * n_x), s);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)xs, (unsigned)ys, (unsigned)zs);
    cfg.blockDim = dim3(256);
    cfg.stream = s;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = 1;
    at.val.clusterDim.y = (unsigned)ys;
    at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, hss_norms_kernel<V>, (const V *)nd.d_data, n_x, n_e, lx, wr, part);
    if (zs > 1) {
        if (e == cudaSuccess) {
            hss_root_kernel<<<(unsigned)((n_x + 7) / 8), 256, 0, s>>>(part, (int)zs, n_x, d_norms);
            e = cudaGetLastError();
        }
        cudaFreeAsync(part, s);
    }
    return e;
}

tqc_status node_norms(const Node &nd, double *d_norms, cudaStream_t s) {
    if (nd.out_qubits.size() > 35) return fail(TQC_ERR_UNSUPPORTED, "hss: too many output states");
    const cudaError_t e = nd.dtype == TQC_F64 ? launch_norms<double>(nd, d_norms, s) : launch_norms<float>(nd, d_norms, s);
    if (e != cudaSuccess) return fail(TQC_ERR_CUDA, "hss: norm kernels");
    return TQC_OK;
}

}  // namespace
}  // namespace tqc

using namespace tqc;

extern "C" {

tqc_status tqc_hss_norms(tqc_net_t net, int32_t sub, double *d_norms, void *cuda_stream) {
    if (!net || !d_norms) return fail(TQC_ERR_INVALID, "NULL argument");
    Net &n = net->n;
    if (!n.has_data) return fail(TQC_ERR_INVALID, "shape-only network has no device tensors");
    if (sub < 0 || sub >= (int)n.nodes.size()) return fail(TQC_ERR_INVALID, "subcircuit index out of range");
    return node_norms(n.nodes[(size_t)sub], d_norms, (cudaStream_t)cuda_stream);
}

tqc_status tqc_hss_select(tqc_net_t net, int64_t s_max, int32_t *counts, int32_t *states, int64_t states_cap,
                          int64_t *n_states_out) {
    if (!net || !counts || !states || !n_states_out) return fail(TQC_ERR_INVALID, "NULL argument");
    if (s_max < 1) return fail(TQC_ERR_INVALID, "s_max must be at least 1");
    Net &n = net->n;
    if (!n.has_data) return fail(TQC_ERR_INVALID, "shape-only network has no device tensors");
    const int m = (int)n.nodes.size();
    // step 1 on the device: every subcircuit's state norms
    std::vector<std::vector<double>> norms(m);
    size_t biggest = 0;
    for (auto &nd : n.nodes) biggest = std::max(biggest, (size_t)1 << nd.out_qubits.size());
    double *d = nullptr;
    if (cudaMalloc(&d, sizeof(double) * biggest) != cudaSuccess) {
        cudaGetLastError();
        return fail(TQC_ERR_OOM, "hss: norm buffer");
    }
    for (int j = 0; j < m; ++j) {
        const size_t nx = (size_t)1 << n.nodes[j].out_qubits.size();
        tqc_status st = node_norms(n.nodes[j], d, 0);
        if (st != TQC_OK) {
            cudaFree(d);
            return st;
        }
        norms[j].resize(nx);
        if (cudaMemcpy(norms[j].data(), d, sizeof(double) * nx, cudaMemcpyDeviceToHost) != cudaSuccess) {
            cudaFree(d);
            return fail(TQC_ERR_CUDA, "hss: norm copy");
        }
    }
    cudaFree(d);
    // step 2: seed every subcircuit with its heaviest state (ties: lowest
    // index), then take states in descending norm (ties: lowest subcircuit,
    // then lowest index) while the product of the counts is below s_max
    std::vector<std::vector<int32_t>> sel(m);
    struct Cand {
        double v;
        int32_t j, i;
    };
    std::vector<Cand> pool;
    for (int j = 0; j < m; ++j) {
        const auto &v = norms[j];
        const int32_t best = (int32_t)(std::max_element(v.begin(), v.end()) - v.begin());
        sel[j].push_back(best);
        for (int32_t i = 0; i < (int32_t)v.size(); ++i)
            if (i != best) pool.push_back({v[i], j, i});
    }
    std::stable_sort(pool.begin(), pool.end(), [](const Cand &a, const Cand &b) {
        if (a.v != b.v) return a.v > b.v;
        if (a.j != b.j) return a.j < b.j;
        return a.i < b.i;
    });
    auto product = [&]() {
        double p = 1.0;
        for (auto &x : sel) p *= (double)x.size();
        return p;
    };
    for (size_t k = 0; k < pool.size() && product() < (double)s_max; ++k) sel[pool[k].j].push_back(pool[k].i);
    int64_t total = 0;
    for (int j = 0; j < m; ++j) total += (int64_t)sel[j].size();
    if (total > states_cap) return fail(TQC_ERR_INVALID, "hss: states buffer too small (" + std::to_string(total) + ")");
    int64_t off = 0;
    for (int j = 0; j < m; ++j) {
        std::sort(sel[j].begin(), sel[j].end());
        counts[j] = (int32_t)sel[j].size();
        std::copy(sel[j].begin(), sel[j].end(), states + off);
        off += (int64_t)sel[j].size();
    }
    *n_states_out = (int64_t)product();
    return TQC_OK;
}

tqc_status tqc_network_select(tqc_net_t net, const int32_t *counts, const int32_t *states, tqc_net_t *out) {
    if (!net || !counts || !states || !out) return fail(TQC_ERR_INVALID, "NULL argument");
    *out = nullptr;
    const Net &src = net->n;
    if (!src.has_data) return fail(TQC_ERR_INVALID, "shape-only network has no device tensors");
    const int m = (int)src.nodes.size();
    Net dst;
    dst.n_cuts = src.n_cuts;
    dst.cut_nodes = src.cut_nodes;
    dst.has_data = true;
    dst.device = src.device;
    std::vector<int> kbits(m);
    int nq = 0, off = 0;
    for (int j = 0; j < m; ++j) {
        const int64_t nx = (int64_t)1 << src.nodes[j].out_qubits.size();
        if (counts[j] < 1 || counts[j] > nx)
            return fail(TQC_ERR_INVALID, "subcircuit " + std::to_string(j) + ": count must be in 1.." + std::to_string(nx));
        for (int r = 0; r < counts[j]; ++r) {
            const int32_t st = states[off + r];
            if (st < 0 || st >= nx || (r > 0 && st <= states[off + r - 1]))
                return fail(TQC_ERR_INVALID, "subcircuit " + std::to_string(j) + ": states must be increasing and in range");
        }
        int k = 0;
        while (((int64_t)1 << k) < counts[j]) ++k;
        kbits[j] = k;
        nq += k;
        off += counts[j];
    }
    if (nq == 0) kbits[0] = nq = 1;  // one padding bit: the network needs at least one output
    if (nq > 128) return fail(TQC_ERR_UNSUPPORTED, "selection has more than 128 index bits");
    dst.n_qubits = nq;
    int q = 0;
    off = 0;
    for (int j = 0; j < m; ++j) {
        const Node &sn = src.nodes[j];
        Node nd;
        nd.cut_ids = sn.cut_ids;
        nd.cut_role = sn.cut_role;
        nd.dtype = sn.dtype;
        for (int b = 0; b < kbits[j]; ++b) nd.out_qubits.push_back(q++);
        const int64_t n_e = (int64_t)1 << (2 * sn.cut_ids.size());
        nd.elems = n_e << kbits[j];
        const size_t esz = sn.dtype == TQC_F64 ? 8 : 4;
        int32_t *d_states = nullptr;
        cudaError_t e = cudaMalloc(&nd.d_data, (size_t)nd.elems * esz);
        if (e == cudaSuccess) e = cudaMalloc(&d_states, sizeof(int32_t) * counts[j]);
        if (e == cudaSuccess)
            e = cudaMemcpy(d_states, states + off, sizeof(int32_t) * counts[j], cudaMemcpyHostToDevice);
        if (e == cudaSuccess) {
            const int64_t nx = (int64_t)1 << sn.out_qubits.size();
            const int64_t blocks = std::min<int64_t>((nd.elems + 255) / 256, 16ll * sm_count());
            if (sn.dtype == TQC_F64)
                hss_gather_kernel<double><<<(unsigned)blocks, 256>>>((const double *)sn.d_data, nx, n_e, d_states,
                                                                     counts[j], kbits[j], (double *)nd.d_data);
            else
                hss_gather_kernel<float><<<(unsigned)blocks, 256>>>((const float *)sn.d_data, nx, n_e, d_states,
                                                                    counts[j], kbits[j], (float *)nd.d_data);
            e = cudaGetLastError();
            if (e == cudaSuccess) e = cudaDeviceSynchronize();
        }
        cudaFree(d_states);
        if (e != cudaSuccess) {
            cudaGetLastError();
            cudaFree(nd.d_data);
            for (auto &x : dst.nodes) cudaFree(x.d_data);
            return fail(TQC_ERR_CUDA, std::string("network_select: ") + cudaGetErrorString(e));
        }
        dst.nodes.push_back(std::move(nd));
        off += counts[j];
    }
    struct tqc_net *h = new (std::nothrow) struct tqc_net;
    if (!h) {
        for (auto &x : dst.nodes) cudaFree(x.d_data);
        return fail(TQC_ERR_OOM, "host allocation failed");
    }
    h->n = std::move(dst);
    *out = h;
    return TQC_OK;
}

}  // extern "C"
