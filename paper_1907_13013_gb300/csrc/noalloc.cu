// fpsa_sweep_noalloc: one LD transport sweep for callers that cannot allocate
// device memory (declaration and contract in include/fpsa.h).
//
// The context-based path keeps the sweep coefficients of every cell and ordinate
// and the segment maps of its two-kernel sweep in buffers owned by the context.
// Some callers cannot allocate: code running inside another framework's memory pool
// or under its allocator lock, or a process whose device memory is fully reserved up
// front. For them this entry point runs the whole sweep as ONE kernel without any
// scratch in global memory: the coefficients are formed in registers from h and
// sigma_t, and the maps of the cell chunks meet by shuffles, in shared memory and
// across the blocks of a thread-block cluster.
//
// The Gauss-Legendre ordinates of every even N up to the maximum are written into a
// __device__ table once per device (the first call's set-up); per call nothing is
// copied from host memory.
#include <cooperative_groups.h>

#include <mutex>
#include <vector>

#include "fpsa_internal.h"
#include "kernels.cuh"

namespace {

constexpr int kNoallocMaxN = 256;
constexpr long long kMaxCellAngles = FPSA_SWEEP_NOALLOC_MAX_CELL_ANGLES;
// mu of order N (even) starts at (N/2 - 1)(N/2) in the ordinate table
constexpr int mu_offset(int N) { return (N / 2 - 1) * (N / 2); }
constexpr int kMuTable = mu_offset(kNoallocMaxN) + kNoallocMaxN;

// Ordinates of every even N <= kNoallocMaxN, ascending within each order.
static __device__ __align__(256) double g_noalloc_mu[kMuTable];

// Device address of the table, looked up once per device with that device current
// (in host code the name of a __device__ array is only a stand-in, never a usable
// device address).
struct DeviceSymbols {
    bool ready = false;
    double *mu = nullptr;
};
constexpr int kMaxDevices = 64;
std::mutex g_symbols_mutex;
DeviceSymbols g_symbols[kMaxDevices];

// First use on a device: the symbol address, then the ordinate table (one
// synchronous copy of host-built tables; later calls copy nothing).
int symbols_for_current_device(DeviceSymbols **out) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return FPSA_ECUDA;
    std::lock_guard<std::mutex> lock(g_symbols_mutex);
    DeviceSymbols &s = g_symbols[dev];
    if (!s.ready) {
        DeviceSymbols t;
        if (cudaGetSymbolAddress((void **)&t.mu, g_noalloc_mu) != cudaSuccess) return FPSA_ECUDA;
        std::vector<double> mu(kMuTable, 0.0);
        for (int N = 2; N <= kNoallocMaxN; N += 2) {
            fpsa::Tables tab;
            fpsa::build_tables(N, 1, FPSA_LAPLACIAN_WFD, tab);  // only mu is used
            std::copy(tab.mu.begin(), tab.mu.end(), mu.begin() + mu_offset(N));
        }
        if (cudaMemcpy(t.mu, mu.data(), mu.size() * sizeof(double), cudaMemcpyHostToDevice) != cudaSuccess)
            return FPSA_ECUDA;
        t.ready = true;
        s = t;
    }
    *out = &s;
    return FPSA_OK;
}

// ---------------------------------------------------------------------------
// The sweep of one slab. A warp holds kOrd ordinates of one direction (consecutive n)
// times kSub chunks of `per` consecutive cells in sweep order; a block holds kWarps warps
// along the slab, a cluster of C blocks the whole slab. The chunk maps (x -> a x + b, the
// LD cell algebra of kernels.cuh) are scanned within the warp by shuffles, then over the
// block's warps in shared memory, then over the cluster's blocks in distributed shared
// memory, and every lane sweeps its chunk from its exact inflow. With per <= kBatch
// (kCached) a lane keeps its cells' maps in registers, so every input is read once.
//
// What bounds it: FP64 arithmetic (about 40 operations per cell and ordinate, the
// reciprocal's among them, on cores that issue two FP64 FMAs a clock and SM) and, for
// small slabs, the launch. Hence few ordinates per block and not 32: N = 64, K = 2000
// then spreads over the whole chip. Measured on the device, back to back, with kOrd
// ordinates, kWarps warps, cluster C: N = 64, K = 2000: 16.4 us (2, 4, 8), 18.4 (2, 8, 8),
// 26.6 (4, 8, 8: the cluster's blocks share SMs), 38.9 (8, 8, 8); N = 16, K = 200: 6.2 us
// (2, 4, 4), 8.2 (4, 8, 4), 9.2 (2, 4, 1). The three kernels before it (geometry,
// coefficients, a sweep of one block per ordinate) took 39 and 14 us.
// ---------------------------------------------------------------------------
constexpr int kOrd = 2, kSub = 32 / kOrd, kWarps = 4, kBatch = 4, kMaxCluster = 8;
constexpr int kChunksPerBlock = kWarps * kSub;
constexpr int kEnoughBlocks = 128;  // blocks that give nearly every SM work

struct CellMaps {  // outflow = a x + b, upwind node value = au x + bu
    double a, b, au, bu;
};

__device__ __forceinline__ CellMaps cell_maps(double nu, double h, double st, double qu, double qd) {
    const double s6 = st * h * (1.0 / 6.0), half = 0.5 * nu;
    const double t00 = fma(2.0, s6, half), t01 = half + s6, t10 = s6 - half;
    const double id = 1.0 / fma(t00, t00, -t01 * t10);
    const double m1 = h * (1.0 / 6.0);
    const double ru = m1 * fma(2.0, qu, qd), rd = m1 * fma(2.0, qd, qu);
    const double i00 = t00 * id, i01 = t01 * id, i10 = t10 * id;
    return {-i10 * nu, fma(i00, rd, -i10 * ru), i00 * nu, fma(i00, ru, -i01 * rd)};
}

template <bool kCached>
__global__ void __launch_bounds__(kWarps * 32) k_sweep_noalloc(const double *__restrict__ mu,
                                                               const double *__restrict__ h,
                                                               const double *__restrict__ sigma_t, const double *q,
                                                               double *psi, int N, int K, int per, int C) {
    namespace cg = cooperative_groups;
    using fpsa::Affine;
    using fpsa::compose;
    __shared__ Affine<double> s_warp[kWarps][kOrd];
    __shared__ Affine<double> s_block[kOrd];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, ord = lane & (kOrd - 1), sub = lane / kOrd;
    const int rank = blockIdx.x % C, group = blockIdx.x / C, gpd = (N / 2 + kOrd - 1) / kOrd;
    const bool fwd = group >= gpd;  // ordinates n >= N/2 have mu > 0: swept left to right
    const int idx = (fwd ? group - gpd : group) * kOrd + ord;
    const bool valid = idx < N / 2;
    const int n = (fwd ? N / 2 : 0) + (valid ? idx : 0);
    const int iu = fwd ? 0 : N, id = N - iu;  // offsets of the upwind and downwind node
    const double nu = fabs(mu[n]);
    const int p0 = min(((rank * kWarps + w) * kSub + sub) * per, K), p1 = min(p0 + per, K);
    const double *qn = q + n;
    double *pn = psi + n;

    auto load = [&](int pb, double (&hh)[kBatch], double (&st)[kBatch], double (&qu)[kBatch], double (&qd)[kBatch]) {
#pragma unroll
        for (int t = 0; t < kBatch; ++t) {
            const int p = pb + t, c = fwd ? p : K - 1 - p;
            if (p < p1) {
                hh[t] = h[c];
                st[t] = sigma_t[c];
                qu[t] = qn[(size_t)2 * c * N + iu];
                qd[t] = qn[(size_t)2 * c * N + id];
            }
        }
    };

    // the chunk's map
    Affine<double> m{1.0, 0.0};
    CellMaps keep[kCached ? kBatch : 1];
    for (int pb = p0; pb < p1; pb += kBatch) {
        double hh[kBatch], st[kBatch], qu[kBatch], qd[kBatch];
        load(pb, hh, st, qu, qd);
#pragma unroll
        for (int t = 0; t < kBatch; ++t)
            if (pb + t < p1) {
                const CellMaps cm = cell_maps(nu, hh[t], st[t], qu[t], qd[t]);
                if constexpr (kCached) keep[t] = cm;
                m = compose(m, Affine<double>{cm.a, cm.b});
            }
    }
    // inclusive scan over the warp's chunks, then the maps of the warps and blocks before
    Affine<double> inc = m;
#pragma unroll
    for (int d = kOrd; d < 32; d *= 2) {
        const Affine<double> prev{__shfl_up_sync(0xffffffffu, inc.a, d), __shfl_up_sync(0xffffffffu, inc.b, d)};
        if (lane >= d) inc = compose(prev, inc);
    }
    if (sub == kSub - 1) s_warp[w][ord] = inc;
    __syncthreads();
    double x = 0.0;  // vacuum edge
    if (C > 1) {
        cg::cluster_group cl = cg::this_cluster();
        if (w == 0 && sub == 0) {
            Affine<double> t = s_warp[0][ord];
            for (int v = 1; v < kWarps; ++v) t = compose(t, s_warp[v][ord]);
            s_block[ord] = t;
        }
        cl.sync();
        Affine<double> t[kMaxCluster - 1];  // all requested together
#pragma unroll
        for (int v = 0; v < kMaxCluster - 1; ++v)
            t[v] = v < rank ? *cl.map_shared_rank(&s_block[ord], v) : Affine<double>{1.0, 0.0};
#pragma unroll
        for (int v = 0; v < kMaxCluster - 1; ++v)
            if (v < rank) x = fma(t[v].a, x, t[v].b);
        cl.barrier_arrive();  // the other blocks' maps have been read (waited for before exit)
    }
#pragma unroll
    for (int v = 0; v < kWarps - 1; ++v)
        if (v < w) x = fma(s_warp[v][ord].a, x, s_warp[v][ord].b);
    {
        const double ea = __shfl_up_sync(0xffffffffu, inc.a, kOrd), eb = __shfl_up_sync(0xffffffffu, inc.b, kOrd);
        if (sub > 0) x = fma(ea, x, eb);
    }
    // the chunk from its inflow
    for (int pb = p0; pb < p1; pb += kBatch) {
        double hh[kBatch], st[kBatch], qu[kBatch], qd[kBatch];
        if constexpr (!kCached) load(pb, hh, st, qu, qd);
#pragma unroll
        for (int t = 0; t < kBatch; ++t) {
            const int p = pb + t, c = fwd ? p : K - 1 - p;
            if (p < p1) {
                CellMaps cm;
                if constexpr (kCached) cm = keep[t];
                else cm = cell_maps(nu, hh[t], st[t], qu[t], qd[t]);
                if (valid) pn[(size_t)2 * c * N + iu] = fma(cm.au, x, cm.bu);
                x = fma(cm.a, x, cm.b);
                if (valid) pn[(size_t)2 * c * N + id] = x;
            }
        }
    }
    if (C > 1) cg::this_cluster().barrier_wait();
}

}  // namespace

extern "C" int fpsa_sweep_noalloc(int32_t n_ordinates, int32_t n_cells, const double *h, const double *sigma_t,
                                  const double *q, double *psi, void *stream) {
    const int N = n_ordinates, K = n_cells;
    if (N < 2 || N % 2 || K < 1 || !h || !sigma_t || !q || !psi) return FPSA_EINVAL;
    if (N > kNoallocMaxN || (long long)K * N > kMaxCellAngles) return FPSA_ENOTSUP;
    DeviceSymbols *sym = nullptr;
    int rc = symbols_for_current_device(&sym);
    if (rc != FPSA_OK) return rc;
    // Larger clusters (at most 8 blocks, the portable limit) while lanes have more than one
    // cell, but once the lanes' cells fit registers and the blocks fill the chip, splitting
    // further only adds blocks (N = 128, K = 1000: 16.4 us with C = 4, 18.4 with C = 8).
    const int groups = 2 * ((N / 2 + kOrd - 1) / kOrd);
    auto cells_per_lane = [&](int c) { return (K + c * kChunksPerBlock - 1) / (c * kChunksPerBlock); };
    int C = 1;
    while (C < kMaxCluster && cells_per_lane(C) > 1 && (cells_per_lane(C) > kBatch || C * groups < kEnoughBlocks)) C *= 2;
    const int per = cells_per_lane(C);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(C * groups));
    cfg.blockDim = dim3(kWarps * 32);
    cfg.stream = static_cast<cudaStream_t>(stream);
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)C;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = C > 1 ? 1 : 0;
    // The launch's own status is checked (cudaLaunchKernelEx returns it), so an error
    // left pending by unrelated earlier work is neither reported nor cleared here
    // unless it has made the context unusable.
    const double *mu = sym->mu + mu_offset(N);
    const cudaError_t e = per <= kBatch
                              ? cudaLaunchKernelEx(&cfg, k_sweep_noalloc<true>, mu, h, sigma_t, q, psi, N, K, per, C)
                              : cudaLaunchKernelEx(&cfg, k_sweep_noalloc<false>, mu, h, sigma_t, q, psi, N, K, per, C);
    return e == cudaSuccess ? FPSA_OK : FPSA_ECUDA;
}
