// Block cyclic reduction solve with many right-hand sides on tensor cores (the
// FP32 factors of the mixed-precision path; 2N a multiple of 128 up to 512, at
// least 16 right-hand sides).
//
// The dataflow solve k_bcr_solve_flow applies an eliminated cell's A^{-1} to at
// most 8 right-hand sides per unit, so with R of them every factor is read R / 8
// times per solve. Here a unit is one (cell, phase, tile of RT <= 64 right-hand
// sides, slice of 128 rows), and its products are GEMMs on the tensor cores
// (M = 128 rows, N = RT, accumulated in FP32 in tensor memory):
//   forward  Y_i = A_i^{-1} r_i, rows of the slice; the slice holding R+ (L-) then forms
//            B_right Y_i[R+] (C_left Y_i[L-]) and subtracts it from the neighbour's r
//   backward u_i = Y_i - P_i [u_left[R+] ; u_right[L-]], rows of the slice,
//            P_i = [A_i^{-1}[:, L+] B_i , A_i^{-1}[:, R-] C_i]
// (the reduction of k_bcr_solve_flow, with the couplings multiplied into the backward
// operator once per factorization: a backward unit is then one product instead of two
// dependent ones of which every slice repeated the first). Precision: the factors and the
// vectors they multiply in split BF16 with three products, as the contractions,
//   A x ~= A_hi x_hi + A_hi x_lo + A_lo x_hi;
// the couplings in three BF16 parts with six products (all pairs of weight 2^-16 and
// more), which keeps FP32's 24 bits. Both are stored a second time for this solve,
// already split and in the K-major core-matrix layout, one bulk copy (the TMA engine) per
// chunk: A^{-1} and P by (slice, 32 columns), 16 KB (k_bcr_factor_split,
// k_bcr_backward_split), a coupling block by 16 columns (k_bcr_coupling_split).
// With P in two parts a solve is as far from the exact solution of the stored factors as with
// the couplings multiplied by u in 24 bits first and the result split before A^{-1}: emulated
// over ten slabs (N = 64 to 256, HG 0.8 to 0.99, 50 to 1000 per cm, cells of 1/200 to 1/3000
// cm), three draws each, relative 2-norms of 2.3e-6 to 5.1e-6, 0.96 to 1.01 times the other
// form's and 0.99 of them on average.
//
// A CTA is four worker warps, a copying and an issuing thread that share a ring of kStages
// stages, a chunk of the operand A and one of the operand B each. The copying thread takes
// the units and copies A chunks as many stages ahead as are free, across units; the issuing
// thread issues the products of a stage once its copy has landed and the workers have
// written its B chunk; the workers load the vectors four chunks ahead, split them, and run
// the epilogues. (One thread for copies and products, with descriptors built for each, took
// 1 us a chunk, half of the time of a unit.) What bounds it: at the wide levels the
// factors' stream through the stages (with the conversion of the vectors behind it), at
// the narrow ones the chain of hops, each a unit's length. Hence slices of 128 rows (four
// CTAs share a cell at 2N = 512) and a pipeline without a block barrier per chunk: one CTA
// for all rows, 16-column chunks with a barrier, a wait for the products and a copy issued
// only then, and the couplings on the FP32 cores took 3.43 ms at 2N = 512, 1250 cells and
// 64 right-hand sides, 1.72 ms with 16; with one thread for copies and products 1.68 and
// 1.25 ms, with the couplings multiplied in every backward unit 1.20 and 0.70 ms, now 0.89
// and 0.53 ms.
//
// Units are taken from a work queue in phase order (forward levels, roots, backward
// levels), within a phase the slices others wait for first: a unit depends only on units
// with lower indices, every one of which is held by a running CTA, so every wait ends and
// an ordinary launch suffices (two CTAs per SM: the shared-memory request admits no third,
// so their 2 x 256 tensor-memory columns always fit). Every wait is bounded; on a timeout
// the error is recorded, the CTA lets its copies and products land (bounded), frees its
// tensor memory and stops, and the other CTAs' waits give up as soon as they see the flag.
#pragma once

#include "kernels.cuh"
#include "tc_contract.cuh"

namespace fpsa {
namespace tcs {

constexpr int kWorkers = 128, kThreads = kWorkers + 64;  // a copying and an issuing warp
constexpr int kK = 32;                     // factor columns per chunk
constexpr int kKc = 16;                    // coupling columns per chunk
constexpr int kStages = 4;
constexpr unsigned kFlagTries = 1u << 28;
constexpr int kAhead = 4;                  // chunks of the vectors in flight per worker
constexpr int kUnitRing = 8;               // units the driver may have taken ahead of the workers
constexpr int kMaxRT = 64;                 // right-hand sides per unit
constexpr int kMaxN2 = 512;
constexpr uint32_t kMinSmem = 80u * 1024u;  // > 228 KB / 3: at most two CTAs per SM
constexpr uint32_t kChunkA = 128u * kK * 4u;  // hi and lo, 128 x 32 BF16 each

__host__ __device__ constexpr int rhs_tile(int R) { return R >= kMaxRT ? kMaxRT : (R + 15) / 16 * 16; }
__host__ __device__ constexpr bool applies(int n2, int R) { return n2 % 128 == 0 && n2 <= kMaxN2 && R >= 16; }
__host__ __device__ constexpr size_t cell_bytes(int n2) { return (size_t)n2 * n2 * 4u; }
__host__ __device__ constexpr size_t backward_bytes(int n2) { return cell_bytes(n2) / 2; }
// one coupling block: N/2 x N/2 in three BF16 parts; a chunk of its columns
__host__ __device__ constexpr size_t coupling_bytes(int n2) { return (size_t)(n2 / 4) * (n2 / 4) * 6u; }
__host__ __device__ constexpr uint32_t coupling_chunk(int n2) { return (uint32_t)(n2 / 4) * kKc * 6u; }
// one chunk of the vectors: RT x 32 in two parts (or RT x 16 in three)
__host__ __device__ constexpr uint32_t chunk_b(int RT) { return (uint32_t)RT * kK * 4u; }

// Shared memory: the stages (A chunk, B chunk), the ring of units, the mbarriers and the
// tensor-memory slot.
struct Plan {
    uint32_t stage, units, bars, total;
    __host__ __device__ static Plan make(int RT) {
        Plan p;
        p.stage = kChunkA + chunk_b(RT);
        p.units = kStages * p.stage;
        p.bars = p.units + kUnitRing * 64u;
        p.total = p.bars + 8u * (3 * kStages + kUnitRing + 2) + 64u;
        if (p.total < kMinSmem) p.total = kMinSmem;
        return p;
    }
};

// The split copy of the stored inverses (FP32, transposed: Mt[col][row] = A^{-1}[row][col]):
// block (cell, kc) writes columns 32 kc .. 32 kc + 31; chunk (cell, slice m, kc) holds rows
// 128 m .. as hi and lo, element (row, k) of a part at kmajor_offset(row, k, 32).
// Consecutive threads take consecutive rows, so every column is read coalesced.
__global__ void __launch_bounds__(256) k_bcr_factor_split(const float *__restrict__ A, unsigned char *__restrict__ out,
                                                          int n2) {
    const int nkc = n2 / kK;
    const int cell = blockIdx.x / nkc, kc = blockIdx.x - cell * nkc;
    const float *Mt = A + (size_t)cell * n2 * n2 + (size_t)kc * kK * n2;
    unsigned char *o = out + (size_t)cell * cell_bytes(n2);
    for (int i = threadIdx.x; i < (kK / 8) * n2; i += blockDim.x) {
        const int row = i % n2, g = i / n2;
        uint32_t hi[4], lo[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            __nv_bfloat16 h0, l0, h1, l1;
            tc::split_bf16(Mt[(size_t)(8 * g + 2 * j) * n2 + row], h0, l0);
            tc::split_bf16(Mt[(size_t)(8 * g + 2 * j + 1) * n2 + row], h1, l1);
            hi[j] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
            lo[j] = (uint32_t)__bfloat16_as_ushort(l0) | ((uint32_t)__bfloat16_as_ushort(l1) << 16);
        }
        unsigned char *c = o + ((size_t)(row / 128) * nkc + kc) * kChunkA + tc::kmajor_offset(row % 128, 8 * g, kK);
        *reinterpret_cast<uint4 *>(c) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
        *reinterpret_cast<uint4 *>(c + kChunkA / 2) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
    }
}

// The backward operators P_i (2N x N, FP32 sums, split as the inverses): block (item, side,
// slice m) forms A_i^{-1}[128 m .., L+] B_i (side 0) or A_i^{-1}[128 m .., R-] C_i, 2 h2
// threads with 8 x 8 outputs each, both operands through shared memory in k-chunks of 16
// (contiguous in memory along their other index). Bounded by FP32 arithmetic: 2 N^3 / 2
// FMAs a cell, 1.41 ms for 1250 cells at 2N = 512, once per factorization.
__global__ void __launch_bounds__(256) k_bcr_backward_split(const float *__restrict__ A, const float *__restrict__ Bc,
                                                            const float *__restrict__ Cc,
                                                            const BcrItem *__restrict__ items,
                                                            unsigned char *__restrict__ out, int n2) {
    constexpr int KC = 16;
    const BcrItem it = items[blockIdx.x];
    const int side = blockIdx.y, m = blockIdx.z, N = n2 / 2, h2 = n2 / 4;
    if ((side ? it.right : it.left) < 0) return;  // (a root has neither)
    __shared__ __align__(16) float Ls[KC][128], Rs[KC][kMaxN2 / 4];
    const float *L = A + (size_t)it.cell * n2 * n2 + (size_t)(side ? N : h2) * n2 + 128 * m;
    const float *W = (side ? Cc : Bc) + (size_t)it.s_cell * h2 * h2;
    const int t = threadIdx.x, rg = t & 15, cg = t >> 4;  // rows 4 rg .. + 3 and 64 more, columns 8 cg .. + 7
    float acc[8][8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
    for (int k0 = 0; k0 < h2; k0 += KC) {
        for (int i = t; i < KC * 32; i += blockDim.x)
            *reinterpret_cast<float4 *>(&Ls[i >> 5][4 * (i & 31)]) =
                __ldg(reinterpret_cast<const float4 *>(L + (size_t)(k0 + (i >> 5)) * n2) + (i & 31));
        for (int i = t; i < KC * (h2 / 4); i += blockDim.x) {
            const int k = i / (h2 / 4), c = i - k * (h2 / 4);
            *reinterpret_cast<float4 *>(&Rs[k][4 * c]) =
                __ldg(reinterpret_cast<const float4 *>(W + (size_t)(k0 + k) * h2) + c);
        }
        __syncthreads();
#pragma unroll 4
        for (int k = 0; k < KC; ++k) {
            float l[8], r[8];
            *reinterpret_cast<float4 *>(l) = *reinterpret_cast<const float4 *>(&Ls[k][4 * rg]);
            *reinterpret_cast<float4 *>(l + 4) = *reinterpret_cast<const float4 *>(&Ls[k][64 + 4 * rg]);
            *reinterpret_cast<float4 *>(r) = *reinterpret_cast<const float4 *>(&Rs[k][8 * cg]);
            *reinterpret_cast<float4 *>(r + 4) = *reinterpret_cast<const float4 *>(&Rs[k][8 * cg + 4]);
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(l[i], r[j], acc[i][j]);
        }
        __syncthreads();
    }
    const int col = side * h2 + 8 * cg;
    unsigned char *c = out + (size_t)it.cell * backward_bytes(n2) + ((size_t)m * (N / kK) + col / kK) * kChunkA;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        uint32_t hi[4], lo[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            __nv_bfloat16 h0, l0, h1, l1;
            tc::split_bf16(acc[i][2 * j], h0, l0);
            tc::split_bf16(acc[i][2 * j + 1], h1, l1);
            hi[j] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
            lo[j] = (uint32_t)__bfloat16_as_ushort(l0) | ((uint32_t)__bfloat16_as_ushort(l1) << 16);
        }
        unsigned char *o = c + tc::kmajor_offset(4 * rg + (i & 3) + 64 * (i >> 2), col % kK, kK);
        *reinterpret_cast<uint4 *>(o) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
        *reinterpret_cast<uint4 *>(o + kChunkA / 2) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
    }
}

// x = p[0] + p[1] + p[2] in BF16 parts (24 bits)
__device__ __forceinline__ void split3(float x, __nv_bfloat16 (&p)[3]) {
    p[0] = __float2bfloat16_rn(x);
    const float r = x - __bfloat162float(p[0]);
    p[1] = __float2bfloat16_rn(r);
    p[2] = __float2bfloat16_rn(r - __bfloat162float(p[1]));
}
// eight values as one 16-byte core-matrix row per part
__device__ __forceinline__ void store_split3(unsigned char *dst, uint32_t part, const float *x) {
    uint32_t w[3][4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        __nv_bfloat16 a[3], b[3];
        split3(x[2 * j], a);
        split3(x[2 * j + 1], b);
#pragma unroll
        for (int k = 0; k < 3; ++k)
            w[k][j] = (uint32_t)__bfloat16_as_ushort(a[k]) | ((uint32_t)__bfloat16_as_ushort(b[k]) << 16);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) *reinterpret_cast<uint4 *>(dst + k * part) = make_uint4(w[k][0], w[k][1], w[k][2], w[k][3]);
}

// The split copy of the coupling blocks (row-major h2 x h2): block (slot, kc) writes columns
// 16 kc .. 16 kc + 15 of the three parts, element (row, k) at kmajor_offset(row, k, 16).
__global__ void __launch_bounds__(256) k_bcr_coupling_split(const float *__restrict__ M, unsigned char *__restrict__ out,
                                                            int n2) {
    const int h2 = n2 / 4, nkc = h2 / kKc;
    const int slot = blockIdx.x / nkc, kc = blockIdx.x - slot * nkc;
    const float *m = M + (size_t)slot * h2 * h2 + kc * kKc;
    unsigned char *o = out + (size_t)slot * coupling_bytes(n2) + (size_t)kc * coupling_chunk(n2);
    for (int i = threadIdx.x; i < 2 * h2; i += blockDim.x) {
        const int row = i >> 1, half = i & 1;
        float x[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) x[j] = m[(size_t)row * h2 + 8 * half + j];
        store_split3(o + tc::kmajor_offset(row, 8 * half, kKc), (uint32_t)h2 * kKc * 2u, x);
    }
}

// A unit as the driver hands it to the workers (id < 0: no more units).
struct Unit {
    int id, m, ch, bwd;
    int cell, left, right, s_left, s_right, local, K_inst, level;
    int pad[4];
};
static_assert(sizeof(Unit) == 64, "one slot of the unit ring");

__device__ __forceinline__ void worker_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kWorkers) : "memory"); }
// Did any worker fail? (a barrier of the workers: they stop together)
__device__ __forceinline__ bool worker_any(bool v) { return gbar_or(1, kWorkers, v); }
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(bar)) : "memory");
}

template <int V>
struct Const {
    static constexpr int value = V;
};

// One counter of a unit's dataflow wait (bounded), giving up at once when an error has been recorded.
__device__ __forceinline__ void poll(const int *c, int want, int *err, unsigned limit) {
    unsigned spins = 0;
    while (ld_acquire_gpu(c) < want) {
        if (++spins > limit || *(volatile int *)err != 0) {
            atomicExch(err, 1);
            break;
        }
        if (spins > 256) __nanosleep(32);
    }
}

}  // namespace tcs

// The solve: units as above over the concatenated item array of lv. Counters per (tile of
// RT right-hand sides, cell), n of each, zero at launch: flow[0 .. n) edge slices (the ones
// that push, first and last) of eliminated neighbours done, [n .. 2n) forward slices written
// (for the cell's own backward slices), then two per cell, the L- and the R+ rows of u final.
// An edge slice counts for BOTH neighbours of its cell, whichever it pushes into: a cell at
// distance 2^l of another then starts, and pushes into the cells between which it lies, only
// after both pushes of every cell of a lower level between them have landed, so the pushes
// into a row are added in level order and a solve gives the same bits each time. (Counted
// for the pushed-to neighbour alone, the push of a further cell could come before that of a
// nearer one, made by another CTA.) queue: this launch's unit counter (zero at launch).
// zero_next / queue_next: the other parity's counters, zeroed for the following solve.
template <int RT>
__global__ void __launch_bounds__(tcs::kThreads, 2) k_bcr_solve_tc(
    const unsigned char *__restrict__ Atc, const unsigned char *__restrict__ Ptc, const unsigned char *__restrict__ Btc, const unsigned char *__restrict__ Ctc,
    const BcrItem *__restrict__ items, LevelTable lv, float *rhs, float *Y, int N, int sumK, int R,
    int *flow, int *queue, int *err, int *zero_next, long long nzero, int *queue_next, const int *stop) {
    using namespace tcs;
    for (long long i = (long long)blockIdx.x * kThreads + threadIdx.x; i < nzero; i += (long long)gridDim.x * kThreads)
        zero_next[i] = 0;
    if (blockIdx.x == 0 && threadIdx.x == 0) *queue_next = 0;
    tc::grid_dependency_wait();
    if (stopped(stop)) return;
    extern __shared__ __align__(128) unsigned char smem_tcs[];
    __shared__ int s_fail;  // a wait of this CTA gave up
    const int n2 = 2 * N, h2 = N / 2, MT = n2 / 128, t = threadIdx.x;
    const Plan pl = Plan::make(RT);
    Unit *ring = reinterpret_cast<Unit *>(smem_tcs + pl.units);
    uint64_t *full_a = reinterpret_cast<uint64_t *>(smem_tcs + pl.bars), *full_b = full_a + kStages,
             *empty = full_b + kStages, *unit_bar = empty + kStages, *seg_bar = unit_bar + kUnitRing,
             *drain = seg_bar + 1;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(drain + 1);
    constexpr uint32_t kCols = 3 * RT <= 64 ? 64u : (3 * RT <= 128 ? 128u : 256u);
    if (t == 0) {
        for (int i = 0; i < kStages; ++i) {
            tc::mbar_init(full_a + i, 1);
            tc::mbar_init(full_b + i, kWorkers);
            tc::mbar_init(empty + i, 1);
        }
        for (int i = 0; i < kUnitRing; ++i) tc::mbar_init(unit_bar + i, 1);
        tc::mbar_init(seg_bar, 1);
        tc::mbar_init(drain, 1);
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (t < 32) {
        tc::tmem_alloc(tslot, kCols);
        tc::tmem_relinquish();
    }
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = *tslot;

    const int nch = (R + RT - 1) / RT, nl = lv.n_levels, P = 2 * nl;
    const size_t rstride = (size_t)sumK * n2, n = (size_t)nch * sumK;
    const int nc = h2 / kKc;  // chunks of a coupling product
    auto failed = [&]() { return *(volatile int *)&s_fail != 0; };
    auto fail = [&]() {
        *(volatile int *)&s_fail = 1;
        atomicExch(err, 1);
    };
    // A unit's chunks, in order: forward, n2 / 32 of A^{-1}, then the couplings of its pushes;
    // backward, those of P (only its left half without a right neighbour).
    auto push_right = [&](const Unit &u) { return !u.bwd && u.right >= 0 && u.m == MT - 1; };
    auto push_left = [&](const Unit &u) { return !u.bwd && u.left >= 0 && u.m == 0; };
    auto n_main = [&](const Unit &u) { return (u.bwd ? (u.right >= 0 ? N : h2) : n2) / kK; };

    // Waits of the copying and the issuing thread: the workers may be waiting for other
    // units, with their own limit, so these end by the flag (kFlagTries is far beyond it).
    auto wait_flag = [&](uint64_t *bar, uint32_t par) {
        for (unsigned i = 0; !tc::mbar_test(bar, par); ++i)
            if (failed() || i > kFlagTries) return false;
        return true;
    };
    if (t == kWorkers) {
        // ---- copies: takes the units and streams their chunks of A through the stages
        int total = 0;
        auto phase_items = [&](int ph) {
            const int l = ph <= nl ? ph : 2 * nl - ph;
            return l < nl ? lv.off[l + 1] - lv.off[l] : lv.n_roots;
        };
        for (int ph = 0; ph <= P; ++ph) total += phase_items(ph) * nch * MT;
        int popped = atomicAdd(queue, 1);
        uint32_t issued = 0;
        bool ok = true;
        for (uint32_t taken = 0; ok; ++taken) {
            // the next unit into the ring (at most kStages + 1 units beyond the workers')
            Unit u{};
            u.id = popped < total ? popped : -1;
            if (u.id >= 0) {
                popped = atomicAdd(queue, 1);
                int ph = 0, w = u.id;
                for (int k = phase_items(0) * nch * MT; w >= k; k = phase_items(ph) * nch * MT) {
                    w -= k;
                    ++ph;
                }
                const int per = phase_items(ph) * nch, si = w / per, x = w - si * per;
                const BcrItem it = items[lv.off[ph <= nl ? ph : 2 * nl - ph] + x / nch];
                u.m = si == 0 ? MT - 1 : si - 1;  // the slices others wait for (R+, then L-) first
                u.ch = x % nch;
                u.bwd = ph > nl;
                u.cell = it.cell;
                u.left = it.left;
                u.right = it.right;
                u.s_left = it.s_left;
                u.s_right = it.s_right;
                u.local = it.local;
                u.K_inst = it.K_inst;
                u.level = it.level;
            }
            ring[taken % kUnitRing] = u;
            mbar_arrive(&unit_bar[taken % kUnitRing]);  // (release)
            if (u.id < 0) break;
            auto copy = [&](const unsigned char *src, int chunks, uint32_t bytes) {
                for (int c = 0; c < chunks && ok; ++c, src += bytes, ++issued) {
                    const int s = issued % kStages;
                    if (issued >= (uint32_t)kStages) ok = wait_flag(&empty[s], (issued / kStages - 1u) & 1u);
                    if (!ok) break;
                    tc::mbar_arrive_expect_tx(&full_a[s], bytes);
                    tc::bulk_copy_g2s(smem_tcs + s * pl.stage, src, bytes, &full_a[s]);
                }
            };
            const size_t slice = (size_t)u.m * ((u.bwd ? N : n2) / kK) * kChunkA;
            copy((u.bwd ? Ptc + (size_t)u.cell * backward_bytes(n2) : Atc + (size_t)u.cell * cell_bytes(n2)) + slice,
                 n_main(u), kChunkA);
            const size_t cbytes = coupling_bytes(n2);
            if (push_right(u)) copy(Btc + (size_t)u.s_right * cbytes, nc, coupling_chunk(n2));
            if (push_left(u)) copy(Ctc + (size_t)u.s_left * cbytes, nc, coupling_chunk(n2));
        }
        if (!ok) fail();
        // every copy has landed before the CTA ends (bounded)
        for (uint32_t j = issued > (uint32_t)kStages ? issued - kStages : 0; j < issued; ++j)
            if (!tc::mbar_wait(&full_a[j % kStages], (j / kStages) & 1u)) break;
    } else if (t == kWorkers + 32) {
        // ---- products, in the order of the copies. The descriptors differ from stage to
        // stage and part to part by constants only.
        const uint32_t idesc = tc::idesc_bf16(128, RT);
        const uint64_t am = tc::smem_desc(tc::smem_u32(smem_tcs), 128, kK * 16),
                       bm = tc::smem_desc(tc::smem_u32(smem_tcs) + kChunkA, 128, kK * 16),
                       ac = tc::smem_desc(tc::smem_u32(smem_tcs), 128, kKc * 16),
                       bc = tc::smem_desc(tc::smem_u32(smem_tcs) + kChunkA, 128, kKc * 16);
        const uint32_t ap = (uint32_t)h2 * kKc * 2u / 16u;  // between the parts of a coupling chunk
        const uint32_t step = pl.stage / 16u;
        int s = 0;
        uint32_t par = 0;
        bool ok = true;
        auto begin = [&]() {  // the stage's chunks of both operands are there
            ok = wait_flag(&full_b[s], par) && tc::mbar_wait(&full_a[s], par);
            tc::tc_fence_after();
            return ok;
        };
        auto end = [&]() {
            tc::mma_commit(&empty[s]);
            if (++s == kStages) {
                s = 0;
                par ^= 1u;
            }
        };
        auto main_chunks = [&](int chunks) {
            for (int i = 0; i < chunks && begin(); ++i) {
                const uint64_t a0 = am + (uint64_t)(s * step), b0 = bm + (uint64_t)(s * step);
#pragma unroll
                for (int j = 0; j < kK / 16; ++j) {
                    const uint64_t ah = a0 + 16u * j, al = ah + kChunkA / 32u, bh = b0 + 16u * j, bl = bh + RT * kK / 8u;
                    tc::mma_bf16(tmem, ah, bh, idesc, (j > 0 || i > 0) ? 1u : 0u);
                    tc::mma_bf16(tmem, ah, bl, idesc, 1u);
                    tc::mma_bf16(tmem, al, bh, idesc, 1u);
                }
                end();
            }
        };
        // (rows from N/2 up read what follows in the stage; their accumulator lanes are ignored)
        auto coupling_chunks = [&](uint32_t acc) {
            for (int i = 0; i < nc && begin(); ++i) {
                const uint64_t a0 = ac + (uint64_t)(s * step), a1 = a0 + ap, a2 = a1 + ap;
                const uint64_t b0 = bc + (uint64_t)(s * step), b1 = b0 + RT * kKc / 8u, b2 = b1 + RT * kKc / 8u;
                tc::mma_bf16(acc, a0, b0, idesc, i > 0 ? 1u : 0u);
                tc::mma_bf16(acc, a0, b1, idesc, 1u);
                tc::mma_bf16(acc, a1, b0, idesc, 1u);
                tc::mma_bf16(acc, a0, b2, idesc, 1u);
                tc::mma_bf16(acc, a2, b0, idesc, 1u);
                tc::mma_bf16(acc, a1, b1, idesc, 1u);
                end();
            }
        };
        for (uint32_t j = 0; ok; ++j) {
            if (!(ok = wait_flag(&unit_bar[j % kUnitRing], (j / kUnitRing) & 1u))) break;
            const Unit u = ring[j % kUnitRing];
            if (u.id < 0) break;
            // after each group of chunks the workers read its accumulators
            main_chunks(n_main(u));
            tc::mma_commit(seg_bar);
            const bool pr = push_right(u), plf = push_left(u);
            if (pr) coupling_chunks(tmem + RT);
            if (plf) coupling_chunks(tmem + 2u * RT);
            if (pr || plf) tc::mma_commit(seg_bar);
        }
        if (!ok) fail();
        tc::mma_commit(drain);  // every product has been done before the CTA ends (bounded)
        (void)tc::mbar_wait(drain, 0);
    } else if (t < kWorkers) {
        // ---- workers
        const uint32_t lane_base = (uint32_t)(t & ~31) << 16;
        const unsigned limit = flow_spin_limit(err);
        uint32_t q = 0, segs = 0;
        bool ok = true;
        // wait (bounded by time, and by the flag) for a phase of bar
        auto wait_bar = [&](uint64_t *bar, uint32_t par) {
            if (!tc::mbar_wait(bar, par)) fail();
            return !failed();
        };
        // The unit's next `chunks` chunks of KC columns of the vectors v_r[k] = src[r stride + k]
        // (r < nrc, else 0; from chunk `first` on of src2) in P parts, kAhead of them in flight.
        auto feed = [&](auto KCt, auto Pt, const float *src, size_t stride, int chunks, int nrc, int first,
                        const float *src2) {
            constexpr int KC = decltype(KCt)::value, PARTS = decltype(Pt)::value, GR = KC / 8;
            constexpr int NG = (RT * GR + kWorkers - 1) / kWorkers;  // groups of 8 values per worker and chunk
            float4 v[kAhead][NG][2];
            auto load = [&](int c, float4 (&x)[NG][2]) {
#pragma unroll
                for (int g = 0; g < NG; ++g) {
                    const int id = t + g * kWorkers, r = id / GR, k = 8 * (id % GR);
                    x[g][0] = x[g][1] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (r < nrc && c < chunks) {
                        const float4 *p = reinterpret_cast<const float4 *>(
                            (c < first ? src + c * KC : src2 + (c - first) * KC) + (size_t)r * stride + k);
                        x[g][0] = __ldcg(p);
                        x[g][1] = __ldcg(p + 1);
                    }
                }
            };
#pragma unroll
            for (int a = 0; a < kAhead; ++a) load(a, v[a]);
            for (int c0 = 0; c0 < chunks && ok; c0 += kAhead) {
#pragma unroll
                for (int a = 0; a < kAhead; ++a) {
                    if (c0 + a >= chunks || !ok) break;
                    const int s = q % kStages;
                    if (q >= (uint32_t)kStages) ok = wait_bar(&empty[s], (q / kStages - 1u) & 1u);
                    unsigned char *bs = smem_tcs + s * pl.stage + kChunkA;
#pragma unroll
                    for (int g = 0; g < NG; ++g) {
                        const int id = t + g * kWorkers, r = id / GR, k = 8 * (id % GR);
                        if (r < RT) {
                            const float4 lo4 = v[a][g][0], hi4 = v[a][g][1];
                            const float x[8] = {lo4.x, lo4.y, lo4.z, lo4.w, hi4.x, hi4.y, hi4.z, hi4.w};
                            unsigned char *d = bs + tc::kmajor_offset(r, k, KC);
                            if constexpr (PARTS == 3) {
                                store_split3(d, (uint32_t)RT * KC * 2u, x);
                            } else {
                                uint32_t hi[4], lo[4];
#pragma unroll
                                for (int j = 0; j < 4; ++j) {
                                    __nv_bfloat16 h0, l0, h1, l1;
                                    tc::split_bf16(x[2 * j], h0, l0);
                                    tc::split_bf16(x[2 * j + 1], h1, l1);
                                    hi[j] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
                                    lo[j] = (uint32_t)__bfloat16_as_ushort(l0) | ((uint32_t)__bfloat16_as_ushort(l1) << 16);
                                }
                                *reinterpret_cast<uint4 *>(d) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                                *reinterpret_cast<uint4 *>(d + (uint32_t)RT * KC * 2u) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                            }
                        }
                    }
                    load(c0 + kAhead + a, v[a]);
                    tc::fence_async_smem();  // the st.shared above, before the tensor core reads them
                    tc::tc_fence_before();   // and the accumulator reads before it, before the next products
                    mbar_arrive(&full_b[s]);
                    ++q;
                }
            }
        };
        auto wait_seg = [&]() {  // the group of chunks just fed has been multiplied
            if (ok) ok = wait_bar(seg_bar, segs & 1u);
            ++segs;
            tc::tc_fence_after();
        };
        for (uint32_t j = 0;; ++j) {
            // (units are taken as their chunks are copied: a few chunks ahead of the products)
            ok = wait_bar(&unit_bar[j % kUnitRing], (j / kUnitRing) & 1u);
            if (worker_any(!ok)) break;
            const Unit u = ring[j % kUnitRing];
            if (u.id < 0) break;
            const int r0 = u.ch * RT, nrc = min(RT, R - r0), row = 128 * u.m + t;
            int *cnt = flow + (size_t)u.ch * sumK, *written = cnt + n, *fin = flow + 2 * n + (size_t)u.ch * sumK * 2;
            float *Yc = Y + (size_t)r0 * rstride + (size_t)u.cell * n2;
            if (!u.bwd) {
                int want = 0;
                for (int lp = 0; lp < u.level; ++lp)
                    want += (u.local >= (1 << lp)) + (u.local + (1 << lp) < u.K_inst);
                want *= min(MT, 2);  // edge slices of a neighbour
                if (t == 0 && want) poll(cnt + u.cell, want, err, limit);
            } else {  // three warps, so that the polls overlap
                if (t == 0) poll(fin + 2 * u.left + 1, 1, err, limit);
                if (t == 32 && u.right >= 0) poll(fin + 2 * u.right, 1, err, limit);
                if (t == 64) poll(written + u.cell, MT, err, limit);
            }
            worker_sync();
            if (!u.bwd) {
                feed(Const<kK>{}, Const<2>{}, rhs + (size_t)r0 * rstride + (size_t)u.cell * n2, rstride, n2 / kK, nrc, n2 / kK, nullptr);
                wait_seg();
                if (worker_any(!ok)) break;
#pragma unroll
                for (int c = 0; c < RT; c += 16) {
                    float v[16];
                    tc::tmem_ld16(tmem + lane_base + c, v);
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        if (c + i < nrc) Yc[(size_t)(c + i) * rstride + row] = v[i];
                }
                const bool pr = push_right(u), plf = push_left(u);
                if (pr || plf) {
                    worker_sync();  // the rows this CTA just wrote are read back below
                    // y[R+], then y[L-]
                    feed(Const<kKc>{}, Const<3>{}, pr ? Yc + N + h2 : Yc, rstride, pr && plf ? 2 * nc : nc, nrc, nc, Yc);
                    wait_seg();
                    if (worker_any(!ok)) break;
#pragma unroll
                    for (int side = 0; side < 2; ++side) {
                        if (!(side ? plf : pr)) continue;
                        float *o = rhs + (size_t)r0 * rstride + (size_t)(side ? u.left : u.right) * n2 + (side ? N : h2) + t;
#pragma unroll
                        for (int c = 0; c < RT; c += 16) {
                            float v[16];
                            tc::tmem_ld16(tmem + lane_base + (uint32_t)((1 + side) * RT + c), v);
#pragma unroll
                            for (int i = 0; i < 16; ++i)
                                if (t < h2 && c + i < nrc) atomicAdd(o + (size_t)(c + i) * rstride, -v[i]);
                        }
                    }
                }
                worker_sync();
                if (t == 0) {
                    __threadfence();
                    if (u.left < 0) {  // a root: its solution is final
                        if (u.m == 0) atomicAdd(fin + 2 * u.cell, 1);
                        if (u.m == MT - 1) atomicAdd(fin + 2 * u.cell + 1, 1);
                    } else {
                        atomicAdd(written + u.cell, 1);
                        if (u.m == 0 || u.m == MT - 1) {
                            atomicAdd(cnt + u.left, 1);
                            if (u.right >= 0) atomicAdd(cnt + u.right, 1);
                        }
                    }
                }
            } else {
                feed(Const<kK>{}, Const<2>{}, Y + (size_t)r0 * rstride + (size_t)u.left * n2 + N + h2, rstride, n_main(u), nrc,
                     h2 / kK, u.right >= 0 ? Y + (size_t)r0 * rstride + (size_t)u.right * n2 : nullptr);
                float y[RT];
#pragma unroll
                for (int c = 0; c < RT; ++c) y[c] = c < nrc ? __ldcg(Yc + (size_t)c * rstride + row) : 0.f;
                wait_seg();
                if (worker_any(!ok)) break;
#pragma unroll
                for (int c = 0; c < RT; c += 16) {
                    float v[16];
                    tc::tmem_ld16(tmem + lane_base + c, v);
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        if (c + i < nrc) Yc[(size_t)(c + i) * rstride + row] = y[c + i] - v[i];
                }
                worker_sync();
                if (t == 0) {
                    __threadfence();
                    if (u.m == 0) atomicAdd(fin + 2 * u.cell, 1);
                    if (u.m == MT - 1) atomicAdd(fin + 2 * u.cell + 1, 1);
                }
            }
        }
    }
    __syncwarp();
    tc::tc_fence_before();
    __syncthreads();
    if (t < 32) tc::tmem_dealloc(tmem, kCols);
}

}  // namespace fpsa
