// Tensor-core (tcgen05) angular contractions for the FP32 inner solves of the
// mixed-precision path (sm_100a / sm_103a, inline PTX).
//
// A contraction over a tile of 128 columns (64 cells x 2 LD nodes) is the GEMM
//   Out[c][o] = sum_k X[c][k] Op[o][k],   c < 128, o, k < N,
// with Op = D (phi = D psi, Eq. phi-mom) or Op = M (q = M src, Eq. treq).
// Precision: split BF16 with three products. x = x_hi + x_lo with
// x_hi = bf16(x), x_lo = bf16(x - x_hi) (likewise for Op), and
//   x Op ~= x_hi Op_hi + x_hi Op_lo + x_lo Op_hi
// accumulated in FP32 in tensor memory (the dropped x_lo Op_lo term is ~2^-16
// relative). One elected thread issues tcgen05.mma (M = 128, N = N, K = 16 per
// instruction, cta_group::1, kind::f16, A and B both BF16); completion is
// signalled through an mbarrier by tcgen05.commit; the four warps read their 32
// accumulator lanes back with tcgen05.ld.
//
// Shared-memory operand layout (no swizzle, K-major): an R x K BF16 operand is a
// grid of 8 x 8 "core matrices" (8 rows of 16 bytes, 128 contiguous bytes);
// element (row, k) sits at byte
//   ((row / 8) * (K / 8) + k / 8) * 128 + (row % 8) * 16 + (k % 8) * 2,
// so core matrices adjacent in K are 128 B apart (leading byte offset) and
// adjacent 8-row groups K * 16 B apart (stride byte offset). A K-step of 16
// starts 256 B further. The constant operands (D, M) are stored in global memory
// already split and in this layout and are staged with one bulk asynchronous
// copy (cp.async.bulk, the TMA engine) per CTA.
//
// Every wait on an mbarrier is bounded; on timeout the kernel records an error
// flag, releases its tensor memory and returns.
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

#include "bulk_copy.cuh"

namespace fpsa {
namespace tc {

__device__ __forceinline__ void tmem_alloc(uint32_t *dst, uint32_t ncols) {  // whole warp
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst)), "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {  // whole warp
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor: start address, leading / stride byte offsets,
// descriptor version 1, no swizzle.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

// Instruction descriptor of kind::f16 with BF16 A and B, FP32 accumulator,
// both operands K-major, shape M x N.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                         uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

// 16 consecutive FP32 accumulator columns of this thread's lane.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float *v) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// byte offset of element (row, k) in the K-major no-swizzle layout with K columns
__host__ __device__ __forceinline__ uint32_t kmajor_offset(int row, int k, int K) {
    return (uint32_t)((((row >> 3) * (K >> 3) + (k >> 3)) << 7) + ((row & 7) << 4) + ((k & 7) << 1));
}

__device__ __forceinline__ void split_bf16(float x, __nv_bfloat16 &hi, __nv_bfloat16 &lo) {
    hi = __float2bfloat16_rn(x);
    lo = __float2bfloat16_rn(x - __bfloat162float(hi));
}

// Staged global I/O: a tile's 128 columns are 128 contiguous rows of N floats in
// global memory; they move through padded shared buffers [128][kStageLd] in
// k-chunks of kStageK with coalesced 16-byte accesses, and each thread then reads
// or writes its own row (the accumulator lane layout) without bank conflicts.
constexpr int kStageK = 16;
constexpr int kStageLd = kStageK + 4;
constexpr uint32_t kStageBytes = 128u * kStageLd * 4;

// Shared-memory plan of one contraction CTA for N (multiple of 16, <= 128):
//   opD_hi, opD_lo, opM_hi, opM_lo: N x N BF16 each (constant operands)
//   x_hi, x_lo:                     128 x N BF16 each (the column tile)
//   stage[3]:                       [128][kStageLd] FP32 each (staged I/O)
//   bars: 2 mbarriers (bulk copy, MMA), tmem slot
struct Plan {
    uint32_t op_bytes, x_bytes, stage_bytes, total;
    bool full;  // whole-tile staging ([128][N + 4] FP32 per buffer, N <= 64)
    __host__ __device__ static Plan make(int N) {
        Plan p;
        p.op_bytes = (uint32_t)N * N * 2;
        p.x_bytes = 128u * N * 2;
        p.full = N <= 64;
        p.stage_bytes = p.full ? 128u * (N + 4) * 4 : kStageBytes;
        p.total = 4 * p.op_bytes + 2 * p.x_bytes + 3 * p.stage_bytes + 64;
        return p;
    }
};

// Whole-tile staging: asynchronous 16-byte copies of rows [0, nrows) of src (row
// length N floats, N a multiple of 4) into st[row][0..N) with row stride N + 4
// (conflict-free row reads); rows >= nrows are zero-filled. Not committed here.
__device__ __forceinline__ void tile_load_async(float *st, const float *src, int N, int nrows) {
    const int Q = N / 4, ld = N + 4;
    for (int f = threadIdx.x; f < 128 * Q; f += 128) {
        const int row = f / Q, q = f - row * Q;
        float *dst = st + row * ld + 4 * q;
        if (row < nrows)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)),
                         "l"(src + (size_t)row * N + 4 * q)
                         : "memory");
        else
            *reinterpret_cast<float4 *>(dst) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}
__device__ __forceinline__ void async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int NPending>
__device__ __forceinline__ void async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(NPending) : "memory"); }

// dst[row * N + k] = st[row][k] for rows < nrows, coalesced 16-byte stores.
__device__ __forceinline__ void tile_store(const float *st, float *dst, int N, int nrows) {
    const int Q = N / 4, ld = N + 4;
    for (int f = threadIdx.x; f < 128 * Q; f += 128) {
        const int row = f / Q, q = f - row * Q;
        if (row < nrows)
            reinterpret_cast<float4 *>(dst + (size_t)row * N)[q] =
                *reinterpret_cast<const float4 *>(st + row * ld + 4 * q);
    }
}

// st[row][0..kStageK) = src[row * N + k0 ..] for rows < nrows, 0 above (all 128 threads).
__device__ __forceinline__ void stage_in(float *st, const float *src, int N, int nrows, int k0) {
    constexpr int Q = kStageK / 4;  // float4 per row chunk
    for (int f = threadIdx.x; f < 128 * Q; f += 128) {
        const int row = f / Q, q = f - row * Q;
        const float4 v = row < nrows ? __ldg(reinterpret_cast<const float4 *>(src + (size_t)row * N + k0) + q)
                                     : make_float4(0.f, 0.f, 0.f, 0.f);
        *reinterpret_cast<float4 *>(st + row * kStageLd + 4 * q) = v;
    }
}

// dst[row * N + k0 ..] = st[row][0..kStageK) for rows < nrows (all 128 threads).
__device__ __forceinline__ void stage_out(const float *st, float *dst, int N, int nrows, int k0) {
    constexpr int Q = kStageK / 4;
    for (int f = threadIdx.x; f < 128 * Q; f += 128) {
        const int row = f / Q, q = f - row * Q;
        if (row < nrows)
            reinterpret_cast<float4 *>(dst + (size_t)row * N + k0)[q] =
                *reinterpret_cast<const float4 *>(st + row * kStageLd + 4 * q);
    }
}

// 16 floats of row `row` from k0 in a padded buffer of row stride ld (16-byte aligned rows).
__device__ __forceinline__ void row_get16_ld(const float *st, int ld, int row, int k0, float *v) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float4 x = *reinterpret_cast<const float4 *>(st + row * ld + k0 + 4 * q);
        v[4 * q] = x.x; v[4 * q + 1] = x.y; v[4 * q + 2] = x.z; v[4 * q + 3] = x.w;
    }
}
__device__ __forceinline__ void row_put16_ld(float *st, int ld, int row, int k0, const float *v) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
        *reinterpret_cast<float4 *>(st + row * ld + k0 + 4 * q) = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2],
                                                                            v[4 * q + 3]);
}

__device__ __forceinline__ void row_get16(const float *st, int row, float *v) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float4 x = *reinterpret_cast<const float4 *>(st + row * kStageLd + 4 * q);
        v[4 * q] = x.x; v[4 * q + 1] = x.y; v[4 * q + 2] = x.z; v[4 * q + 3] = x.w;
    }
}

__device__ __forceinline__ void row_put16(float *st, int row, const float *v) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
        *reinterpret_cast<float4 *>(st + row * kStageLd + 4 * q) = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2],
                                                                              v[4 * q + 3]);
}

__host__ __device__ constexpr uint32_t tmem_cols_for(int N) { return N <= 32 ? 32u : (N <= 64 ? 64u : (N <= 128 ? 128u : 256u)); }

// Issue Out = X Op over K = N for the tile in x_hi / x_lo against op_hi / op_lo
// (three products per K-step), then commit to bar. Called by one thread.
__device__ __forceinline__ void issue_split_gemm(uint32_t tmem, const unsigned char *x_hi, const unsigned char *x_lo,
                                                 const unsigned char *op_hi, const unsigned char *op_lo, int N,
                                                 uint64_t *bar) {
    const uint32_t idesc = idesc_bf16(128, N);
    const uint32_t sbo = (uint32_t)N * 16;  // (K / 8) core matrices of 128 B per 8-row group
    const uint32_t xh = smem_u32(x_hi), xl = smem_u32(x_lo), oh = smem_u32(op_hi), ol = smem_u32(op_lo);
    for (int s = 0; s < N / 16; ++s) {
        const uint32_t ko = 256u * s;
        const uint64_t a_hi = smem_desc(xh + ko, 128, sbo), a_lo = smem_desc(xl + ko, 128, sbo);
        const uint64_t b_hi = smem_desc(oh + ko, 128, sbo), b_lo = smem_desc(ol + ko, 128, sbo);
        mma_bf16(tmem, a_hi, b_hi, idesc, s > 0 ? 1u : 0u);
        mma_bf16(tmem, a_hi, b_lo, idesc, 1u);
        mma_bf16(tmem, a_lo, b_hi, idesc, 1u);
    }
    mma_commit(bar);
}

// Write 16 FP32 values of tile row c, columns k0..k0+15 (k0 a multiple of 8), into
// x_hi / x_lo: two 16-byte stores per half (one core-matrix row each).
__device__ __forceinline__ void store_split_row16(unsigned char *x_hi, unsigned char *x_lo, int c, int k0,
                                                  const float *v, int N) {
#pragma unroll
    for (int half = 0; half < 2; ++half) {
        __align__(16) __nv_bfloat16 h[8], l[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) split_bf16(v[8 * half + i], h[i], l[i]);
        const uint32_t off = kmajor_offset(c, k0 + 8 * half, N);
        *reinterpret_cast<uint4 *>(x_hi + off) = *reinterpret_cast<const uint4 *>(h);
        *reinterpret_cast<uint4 *>(x_lo + off) = *reinterpret_cast<const uint4 *>(l);
    }
}

}  // namespace tc

// ---------------------------------------------------------------------------
// Fused FPSA contraction kernels on tensor cores (FP32 data), persistent over
// 128-column tiles. Columns are (cell, node) pairs of one rhs: column index
// j = 2 g + a within rhs r. 128 threads: thread t owns tile row t (accumulator
// lane t); global reads and writes go through the staged, coalesced k-chunks.
//   k_tc_fp_rhs:        phi_half = D psi;  rhs = m (x) M Sigma (phi_half - phi)
//   k_tc_update_scatter: phi = phi_base + D v;  q = M (Sigma phi) + q_ang
// err is set to 1 if an mbarrier wait ran out (the kernel then stops).
// ---------------------------------------------------------------------------
struct TcOps {
    const unsigned char *D;  // D_hi then D_lo, N x N BF16 each, K-major core-matrix layout
    const unsigned char *M;  // M_hi then M_lo
};

// Common prologue: smem carve-up, TMEM allocation, operand staging. Returns false on timeout.
struct TcCta {
    unsigned char *opD_hi, *opD_lo, *opM_hi, *opM_lo, *x_hi, *x_lo;
    float *stA, *stB, *stC;
    uint64_t *bar_copy, *bar_mma;
    uint32_t *tmem_slot;
    uint32_t tmem;
    uint32_t mma_phase;
};

__device__ __forceinline__ bool tc_cta_setup(TcCta &s, unsigned char *smem, const TcOps &ops, int N, int *err,
                                             bool wait_ops = true) {
    const tc::Plan pl = tc::Plan::make(N);
    s.opD_hi = smem;
    s.opD_lo = smem + pl.op_bytes;
    s.opM_hi = smem + 2 * pl.op_bytes;
    s.opM_lo = smem + 3 * pl.op_bytes;
    s.x_hi = smem + 4 * pl.op_bytes;
    s.x_lo = s.x_hi + pl.x_bytes;
    s.stA = reinterpret_cast<float *>(s.x_lo + pl.x_bytes);
    s.stB = reinterpret_cast<float *>(reinterpret_cast<unsigned char *>(s.stA) + pl.stage_bytes);
    s.stC = reinterpret_cast<float *>(reinterpret_cast<unsigned char *>(s.stB) + pl.stage_bytes);
    unsigned char *tail = reinterpret_cast<unsigned char *>(s.stC) + pl.stage_bytes;
    s.bar_copy = reinterpret_cast<uint64_t *>(tail);
    s.bar_mma = s.bar_copy + 1;
    s.tmem_slot = reinterpret_cast<uint32_t *>(s.bar_mma + 1);
    s.mma_phase = 0;
    if (threadIdx.x == 0) {
        tc::mbar_init(s.bar_copy, 1);
        tc::mbar_init(s.bar_mma, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (threadIdx.x < 32) {
        tc::tmem_alloc(s.tmem_slot, tc::tmem_cols_for(N));
        tc::tmem_relinquish();
    }
    __syncthreads();
    tc::tc_fence_after();
    s.tmem = *s.tmem_slot;
    if (threadIdx.x == 0) {
        tc::mbar_arrive_expect_tx(s.bar_copy, 4 * pl.op_bytes);
        tc::bulk_copy_g2s(s.opD_hi, ops.D, 2 * pl.op_bytes, s.bar_copy);
        tc::bulk_copy_g2s(s.opM_hi, ops.M, 2 * pl.op_bytes, s.bar_copy);
    }
    if (!wait_ops) return true;
    const bool ok = tc::mbar_wait(s.bar_copy, 0);
    if (!ok && threadIdx.x == 0) atomicExch(err, 1);
    return ok;
}

// Wait for the operator copy started by tc_cta_setup(..., wait_ops = false).
__device__ __forceinline__ bool tc_wait_ops(TcCta &s, int *err) {
    const bool ok = tc::mbar_wait(s.bar_copy, 0);
    if (!ok && threadIdx.x == 0) atomicExch(err, 1);
    return ok;
}

__device__ __forceinline__ void tc_cta_teardown(TcCta &s, int N) {
    tc::tc_fence_before();
    __syncthreads();
    if (threadIdx.x < 32) tc::tmem_dealloc(s.tmem, tc::tmem_cols_for(N));
}

// Run one split GEMM on the tile already in x_hi / x_lo against (op_hi, op_lo);
// afterwards the accumulator lanes are ready for tcgen05.ld. Returns false on timeout.
__device__ __forceinline__ bool tc_gemm(TcCta &s, const unsigned char *op_hi, const unsigned char *op_lo, int N,
                                        int *err) {
    tc::fence_async_smem();  // the tile's st.shared must be visible to the tensor core
    tc::tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0) {
        tc::tc_fence_after();
        tc::issue_split_gemm(s.tmem, s.x_hi, s.x_lo, op_hi, op_lo, N, s.bar_mma);
    }
    const bool ok = tc::mbar_wait(s.bar_mma, s.mma_phase);
    s.mma_phase ^= 1u;
    tc::tc_fence_after();
    if (!ok && threadIdx.x == 0) atomicExch(err, 1);
    return ok;
}

__global__ void __launch_bounds__(128) k_tc_fp_rhs(const float *__restrict__ psi_half, const float *__restrict__ phi,
                                                   float *__restrict__ phi_half, const float *__restrict__ sigma_s,
                                                   const double *__restrict__ h, TcOps ops,
                                                   float *__restrict__ rhs, int N, int sumK, int R, int *err) {
    extern __shared__ __align__(128) unsigned char smem_tc[];
    TcCta s;
    const bool ok0 = tc_cta_setup(s, smem_tc, ops, N, err);
    tc::grid_dependency_wait();  // the inputs come from the previous kernel
    const int t = threadIdx.x;
    const uint32_t lane_base = (uint32_t)(t & ~31) << 16;
    const int tiles_per_r = (2 * sumK + 127) / 128;
    const int ntiles = tiles_per_r * R;
    bool ok = ok0;
    for (int tile = blockIdx.x; ok && tile < ntiles; tile += gridDim.x) {
        const int r = tile / tiles_per_r, j0 = (tile % tiles_per_r) * 128;
        const int ncols = min(128, 2 * sumK - j0), ncell = (ncols + 1) >> 1;
        const bool live = t < ncols;
        const int g = (j0 + t) >> 1;
        const size_t cb = ((size_t)r * sumK * 2 + j0) * N;  // the tile's first element
        const float *sig = sigma_s + (size_t)(j0 >> 1) * N;
        // A = psi columns
        for (int k0 = 0; k0 < N; k0 += tc::kStageK) {
            tc::stage_in(s.stA, psi_half + cb, N, ncols, k0);
            __syncthreads();
            float v[16];
            tc::row_get16(s.stA, t, v);
            tc::store_split_row16(s.x_hi, s.x_lo, t, k0, v, N);
            __syncthreads();
        }
        if (!(ok = tc_gemm(s, s.opD_hi, s.opD_lo, N, err))) break;
        // phi_half = D psi; next A = Sigma (phi_half - phi)
        for (int k0 = 0; k0 < N; k0 += tc::kStageK) {
            tc::stage_in(s.stA, phi + cb, N, ncols, k0);
            tc::stage_in(s.stB, sig, N, ncell, k0);
            float a[16];
            tc::tmem_ld16(s.tmem + lane_base + k0, a);
            __syncthreads();
            float ph[16], sg[16], v[16];
            tc::row_get16(s.stA, t, ph);
            tc::row_get16(s.stB, t >> 1, sg);
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = live ? sg[i] * (a[i] - ph[i]) : 0.f;
            tc::row_put16(s.stC, t, a);
            tc::store_split_row16(s.x_hi, s.x_lo, t, k0, v, N);
            __syncthreads();
            tc::stage_out(s.stC, phi_half + cb, N, ncols, k0);
        }
        if (!(ok = tc_gemm(s, s.opM_hi, s.opM_lo, N, err))) break;
        // rhs = m (x) r: node partner is the adjacent lane (column j ^ 1)
        const float w = live ? (float)(h[g] / 6.0) : 0.f;
        for (int k0 = 0; k0 < N; k0 += tc::kStageK) {
            float a[16], o[16];
            tc::tmem_ld16(s.tmem + lane_base + k0, a);
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const float other = __shfl_xor_sync(0xffffffffu, a[i], 1);  // r at the other node
                o[i] = w * (2.f * a[i] + other);
            }
            __syncthreads();  // stC of the previous chunk has been written out
            tc::row_put16(s.stC, t, o);
            __syncthreads();
            tc::stage_out(s.stC, rhs + cb, N, ncols, k0);
        }
    }
    tc_cta_teardown(s, N);
}

__global__ void __launch_bounds__(128) k_tc_update_scatter(const float *__restrict__ v_in,
                                                           const float *__restrict__ phi_base,
                                                           float *__restrict__ phi, const float *__restrict__ sigma_s,
                                                           TcOps ops, float *__restrict__ q,
                                                           const float *__restrict__ qang, int N, int sumK, int R,
                                                           int *err) {
    extern __shared__ __align__(128) unsigned char smem_tc[];
    TcCta s;
    const bool ok0 = tc_cta_setup(s, smem_tc, ops, N, err);
    tc::grid_dependency_wait();  // the inputs come from the previous kernel
    const int t = threadIdx.x;
    const uint32_t lane_base = (uint32_t)(t & ~31) << 16;
    const int tiles_per_r = (2 * sumK + 127) / 128;
    const int ntiles = tiles_per_r * R;
    bool ok = ok0;
    for (int tile = blockIdx.x; ok && tile < ntiles; tile += gridDim.x) {
        const int r = tile / tiles_per_r, j0 = (tile % tiles_per_r) * 128;
        const int ncols = min(128, 2 * sumK - j0), ncell = (ncols + 1) >> 1;
        const bool live = t < ncols;
        const size_t cb = ((size_t)r * sumK * 2 + j0) * N;
        const float *sig = sigma_s + (size_t)(j0 >> 1) * N;
        for (int k0 = 0; k0 < N; k0 += tc::kStageK) {
            tc::stage_in(s.stA, v_in + cb, N, ncols, k0);
            __syncthreads();
            float v[16];
            tc::row_get16(s.stA, t, v);
            tc::store_split_row16(s.x_hi, s.x_lo, t, k0, v, N);
            __syncthreads();
        }
        if (!(ok = tc_gemm(s, s.opD_hi, s.opD_lo, N, err))) break;
        // phi = phi_base + D v; next A = Sigma phi
        for (int k0 = 0; k0 < N; k0 += tc::kStageK) {
            if (phi_base) tc::stage_in(s.stA, phi_base + cb, N, ncols, k0);
            tc::stage_in(s.stB, sig, N, ncell, k0);
            float a[16];
            tc::tmem_ld16(s.tmem + lane_base + k0, a);
            __syncthreads();
            float pb[16], sg[16], v[16];
            if (phi_base) tc::row_get16(s.stA, t, pb);
            tc::row_get16(s.stB, t >> 1, sg);
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                a[i] += phi_base ? pb[i] : 0.f;
                v[i] = live ? sg[i] * a[i] : 0.f;
            }
            tc::row_put16(s.stC, t, a);
            tc::store_split_row16(s.x_hi, s.x_lo, t, k0, v, N);
            __syncthreads();
            tc::stage_out(s.stC, phi + cb, N, ncols, k0);
        }
        if (!(ok = tc_gemm(s, s.opM_hi, s.opM_lo, N, err))) break;
        // q = M (Sigma phi) + q_ang
        for (int k0 = 0; k0 < N; k0 += tc::kStageK) {
            if (qang) tc::stage_in(s.stA, qang + cb, N, ncols, k0);
            float a[16];
            tc::tmem_ld16(s.tmem + lane_base + k0, a);
            __syncthreads();
            if (qang) {
                float qa[16];
                tc::row_get16(s.stA, t, qa);
#pragma unroll
                for (int i = 0; i < 16; ++i) a[i] += qa[i];
            }
            tc::row_put16(s.stC, t, a);
            __syncthreads();
            tc::stage_out(s.stC, q + cb, N, ncols, k0);
        }
    }
    tc_cta_teardown(s, N);
}

// Whole-tile variants for N <= 64: every global input of a tile is requested by
// asynchronous copies as soon as its buffer is free (the psi / v tile and the phi and
// sigma tiles at the start, overlapping the operator copy and the first GEMM), and
// outputs leave through the staging buffers with coalesced 16-byte stores.
//   stA: psi / v tile, then the outputs;  stB: phi / phi_base, then q_ang;  stC: sigma rows
__global__ void __launch_bounds__(128) k_tc_fp_rhs_tile(const float *__restrict__ psi_half,
                                                        const float *__restrict__ phi, float *__restrict__ phi_half,
                                                        const float *__restrict__ sigma_s, const double *__restrict__ h,
                                                        TcOps ops, float *__restrict__ rhs, int N, int sumK, int R,
                                                        int *err) {
    extern __shared__ __align__(128) unsigned char smem_tc[];
    TcCta s;
    const int t = threadIdx.x, ld = N + 4;
    const uint32_t lane_base = (uint32_t)(t & ~31) << 16;
    const int tiles_per_r = (2 * sumK + 127) / 128;
    const int ntiles = tiles_per_r * R;
    bool ok = tc_cta_setup(s, smem_tc, ops, N, err, false);
    tc::grid_dependency_wait();  // the inputs come from the previous kernel
    bool first = true;
    for (int tile = blockIdx.x; ok && tile < ntiles; tile += gridDim.x) {
        const int r = tile / tiles_per_r, j0 = (tile % tiles_per_r) * 128;
        const int ncols = min(128, 2 * sumK - j0), ncell = (ncols + 1) >> 1;
        const bool live = t < ncols;
        const int g = (j0 + t) >> 1;
        const size_t cb = ((size_t)r * sumK * 2 + j0) * N;
        tc::tile_load_async(s.stA, psi_half + cb, N, ncols);
        tc::async_commit();
        tc::tile_load_async(s.stB, phi + cb, N, ncols);
        tc::tile_load_async(s.stC, sigma_s + (size_t)(j0 >> 1) * N, N, ncell);
        tc::async_commit();
        if (first && !(ok = tc_wait_ops(s, err))) break;
        first = false;
        tc::async_wait<1>();
        __syncthreads();
        for (int k0 = 0; k0 < N; k0 += 16) {
            float v[16];
            tc::row_get16_ld(s.stA, ld, t, k0, v);
            tc::store_split_row16(s.x_hi, s.x_lo, t, k0, v, N);
        }
        if (!(ok = tc_gemm(s, s.opD_hi, s.opD_lo, N, err))) break;
        tc::async_wait<0>();
        __syncthreads();
        // phi_half = D psi -> stA; next A = Sigma (phi_half - phi)
        for (int k0 = 0; k0 < N; k0 += 16) {
            float a[16], ph[16], sg[16], v[16];
            tc::tmem_ld16(s.tmem + lane_base + k0, a);
            tc::row_get16_ld(s.stB, ld, t, k0, ph);
            tc::row_get16_ld(s.stC, ld, t >> 1, k0, sg);
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = live ? sg[i] * (a[i] - ph[i]) : 0.f;
            tc::row_put16_ld(s.stA, ld, t, k0, a);
            tc::store_split_row16(s.x_hi, s.x_lo, t, k0, v, N);
        }
        __syncthreads();
        tc::tile_store(s.stA, phi_half + cb, N, ncols);
        if (!(ok = tc_gemm(s, s.opM_hi, s.opM_lo, N, err))) break;
        // rhs = m (x) r: node partner is the adjacent lane (column j ^ 1)
        const float w = live ? (float)(h[g] / 6.0) : 0.f;
        for (int k0 = 0; k0 < N; k0 += 16) {
            float a[16], o[16];
            tc::tmem_ld16(s.tmem + lane_base + k0, a);
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const float other = __shfl_xor_sync(0xffffffffu, a[i], 1);
                o[i] = w * (2.f * a[i] + other);
            }
            tc::row_put16_ld(s.stA, ld, t, k0, o);
        }
        __syncthreads();
        tc::tile_store(s.stA, rhs + cb, N, ncols);
        __syncthreads();  // stA / stB / stC free for the next tile's copies
    }
    if (first) tc_wait_ops(s, err);  // no copy may land after the CTA has gone
    tc::async_wait<0>();
    tc_cta_teardown(s, N);
}

__global__ void __launch_bounds__(128) k_tc_update_scatter_tile(const float *__restrict__ v_in,
                                                                const float *__restrict__ phi_base,
                                                                float *__restrict__ phi,
                                                                const float *__restrict__ sigma_s, TcOps ops,
                                                                float *__restrict__ q, const float *__restrict__ qang,
                                                                int N, int sumK, int R, int *err) {
    extern __shared__ __align__(128) unsigned char smem_tc[];
    TcCta s;
    const int t = threadIdx.x, ld = N + 4;
    const uint32_t lane_base = (uint32_t)(t & ~31) << 16;
    const int tiles_per_r = (2 * sumK + 127) / 128;
    const int ntiles = tiles_per_r * R;
    bool ok = tc_cta_setup(s, smem_tc, ops, N, err, false);
    tc::grid_dependency_wait();  // the inputs come from the previous kernel
    bool first = true;
    for (int tile = blockIdx.x; ok && tile < ntiles; tile += gridDim.x) {
        const int r = tile / tiles_per_r, j0 = (tile % tiles_per_r) * 128;
        const int ncols = min(128, 2 * sumK - j0), ncell = (ncols + 1) >> 1;
        const bool live = t < ncols;
        const size_t cb = ((size_t)r * sumK * 2 + j0) * N;
        tc::tile_load_async(s.stA, v_in + cb, N, ncols);
        tc::async_commit();
        if (phi_base) tc::tile_load_async(s.stB, phi_base + cb, N, ncols);
        tc::tile_load_async(s.stC, sigma_s + (size_t)(j0 >> 1) * N, N, ncell);
        tc::async_commit();
        if (first && !(ok = tc_wait_ops(s, err))) break;
        first = false;
        tc::async_wait<1>();
        __syncthreads();
        for (int k0 = 0; k0 < N; k0 += 16) {
            float v[16];
            tc::row_get16_ld(s.stA, ld, t, k0, v);
            tc::store_split_row16(s.x_hi, s.x_lo, t, k0, v, N);
        }
        if (!(ok = tc_gemm(s, s.opD_hi, s.opD_lo, N, err))) break;
        tc::async_wait<0>();
        __syncthreads();
        // phi = phi_base + D v -> stA; next A = Sigma phi
        for (int k0 = 0; k0 < N; k0 += 16) {
            float a[16], pb[16], sg[16], v[16];
            tc::tmem_ld16(s.tmem + lane_base + k0, a);
            if (phi_base) tc::row_get16_ld(s.stB, ld, t, k0, pb);
            tc::row_get16_ld(s.stC, ld, t >> 1, k0, sg);
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                a[i] += phi_base ? pb[i] : 0.f;
                v[i] = live ? sg[i] * a[i] : 0.f;
            }
            tc::row_put16_ld(s.stA, ld, t, k0, a);
            tc::store_split_row16(s.x_hi, s.x_lo, t, k0, v, N);
        }
        __syncthreads();
        if (qang) {  // stB is free now: the q_ang tile arrives during the second GEMM
            tc::tile_load_async(s.stB, qang + cb, N, ncols);
        }
        tc::async_commit();
        tc::tile_store(s.stA, phi + cb, N, ncols);
        if (!(ok = tc_gemm(s, s.opM_hi, s.opM_lo, N, err))) break;
        tc::async_wait<0>();
        __syncthreads();
        // q = M (Sigma phi) + q_ang
        for (int k0 = 0; k0 < N; k0 += 16) {
            float a[16];
            tc::tmem_ld16(s.tmem + lane_base + k0, a);
            if (qang) {
                float qa[16];
                tc::row_get16_ld(s.stB, ld, t, k0, qa);
#pragma unroll
                for (int i = 0; i < 16; ++i) a[i] += qa[i];
            }
            tc::row_put16_ld(s.stA, ld, t, k0, a);
        }
        __syncthreads();
        tc::tile_store(s.stA, q + cb, N, ncols);
        __syncthreads();
    }
    if (first) tc_wait_ops(s, err);  // no copy may land after the CTA has gone
    tc::async_wait<0>();
    tc_cta_teardown(s, N);
}

// ---------------------------------------------------------------------------
// Few-column variants of the same two kernels (N <= 128) for problems whose 128-column
// tiles leave most SMs without one. The roles are exchanged: the operator is the A operand
// (M = 128 rows, row o = output o; rows from N up read whatever follows in shared memory
// and are ignored, the accumulator's lanes being independent) and a tile of CT columns
// the B operand (N = CT), so a tile is as small as 16 columns. Thread t < N owns output t
// of every column: its global accesses are whole rows across the threads, all requested
// at the start, and both nodes of a cell meet in one thread. What bounds it is latency
// (one pass of loads, two short chains of MMAs, one of stores per block), and from CT = 32 on
// the registers that hold a thread's outputs (CT = 64: 255, 208 bytes of spills in the
// update). Used where col_tile says (fpsa_internal.h), with the figures there.
// ---------------------------------------------------------------------------
namespace tc {
// Shared memory: the operators as in Plan, x_hi and x_lo (CT x N BF16 each), 2 mbarriers,
// tmem slot; at least what 128 rows of the last operator span.
struct ColPlan {
    uint32_t op_bytes, x_bytes, bars, total;
    __host__ __device__ static ColPlan make(int N, int CT) {
        ColPlan p;
        p.op_bytes = (uint32_t)N * N * 2;
        p.x_bytes = (uint32_t)CT * N * 2;
        p.bars = 4 * p.op_bytes + 2 * p.x_bytes;
        p.total = p.bars + 64;
        const uint32_t span = 3 * p.op_bytes + 256u * (uint32_t)N;
        if (p.total < span) p.total = span;
        return p;
    }
};
}  // namespace tc

template <int CT>
struct TcCols {
    unsigned char *op[4], *x_hi, *x_lo;  // D_hi, D_lo, M_hi, M_lo
    uint64_t *bars;                      // operator copy, MMAs
    uint32_t tmem;
    static constexpr uint32_t kCols = 2 * CT < 32 ? 32u : 2u * CT;

    // barriers, tensor memory and the operators' copy: nothing of the previous kernel's
    __device__ __forceinline__ void setup(unsigned char *smem, const TcOps &ops, int N) {
        const tc::ColPlan pl = tc::ColPlan::make(N, CT);
        for (int i = 0; i < 4; ++i) op[i] = smem + i * pl.op_bytes;
        x_hi = smem + 4 * pl.op_bytes;
        x_lo = x_hi + pl.x_bytes;
        bars = reinterpret_cast<uint64_t *>(smem + pl.bars);
        uint32_t *slot = reinterpret_cast<uint32_t *>(bars + 2);
        if (threadIdx.x == 0) {
            tc::mbar_init(bars, 1);
            tc::mbar_init(bars + 1, 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        if (threadIdx.x < 32) {
            tc::tmem_alloc(slot, kCols);
            tc::tmem_relinquish();
        }
        __syncthreads();
        tc::tc_fence_after();
        tmem = *slot;
        if (threadIdx.x == 0) {
            tc::mbar_arrive_expect_tx(bars, 4 * pl.op_bytes);
            tc::bulk_copy_g2s(op[0], ops.D, 2 * pl.op_bytes, bars);
            tc::bulk_copy_g2s(op[2], ops.M, 2 * pl.op_bytes, bars);
        }
    }
    // v[c] = element k = threadIdx.x of column c, into x_hi / x_lo (row c). Adjacent threads
    // exchange values so that each stores two adjacent k of one column.
    __device__ __forceinline__ void store_x(const float (&v)[CT], int N) {
        const int t = threadIdx.x, odd = t & 1;
#pragma unroll
        for (int c = 0; c < CT; c += 2) {
            const float other = __shfl_xor_sync(0xffffffffu, odd ? v[c] : v[c + 1], 1);
            const float k0 = odd ? other : v[c], k1 = odd ? v[c + 1] : other;
            __nv_bfloat16 h0, l0, h1, l1;
            tc::split_bf16(k0, h0, l0);
            tc::split_bf16(k1, h1, l1);
            if (t < N) {
                const uint32_t off = tc::kmajor_offset(c + odd, t & ~1, N);
                *reinterpret_cast<uint32_t *>(x_hi + off) =
                    (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
                *reinterpret_cast<uint32_t *>(x_lo + off) =
                    (uint32_t)__bfloat16_as_ushort(l0) | ((uint32_t)__bfloat16_as_ushort(l1) << 16);
            }
        }
    }
    // GEMM `which` (0: D, 1: M) of the tile in x_hi / x_lo; a[c] = output threadIdx.x of column c.
    __device__ __forceinline__ bool gemm(int which, int N, float (&a)[CT]) {
        const uint32_t acc = tmem + (uint32_t)(which * CT);
        tc::fence_async_smem();  // the tile's st.shared must be visible to the tensor core
        tc::tc_fence_before();
        __syncthreads();
        bool ok = true;
        if (threadIdx.x == 0) {
            ok = tc::mbar_wait(bars, 0);
            tc::tc_fence_after();
            if (ok) {
                const uint32_t idesc = tc::idesc_bf16(128, CT), sbo = (uint32_t)N * 16;
                const uint32_t oh = tc::smem_u32(op[2 * which]), ol = tc::smem_u32(op[2 * which + 1]);
                const uint32_t xh = tc::smem_u32(x_hi), xl = tc::smem_u32(x_lo);
                for (int s = 0; s < N / 16; ++s) {
                    const uint32_t ko = 256u * s;
                    const uint64_t a_hi = tc::smem_desc(oh + ko, 128, sbo), a_lo = tc::smem_desc(ol + ko, 128, sbo);
                    const uint64_t b_hi = tc::smem_desc(xh + ko, 128, sbo), b_lo = tc::smem_desc(xl + ko, 128, sbo);
                    tc::mma_bf16(acc, a_hi, b_hi, idesc, s > 0 ? 1u : 0u);
                    tc::mma_bf16(acc, a_hi, b_lo, idesc, 1u);
                    tc::mma_bf16(acc, a_lo, b_hi, idesc, 1u);
                }
            }
            tc::mma_commit(bars + 1);
        }
        ok = tc::mbar_wait(bars + 1, (uint32_t)which) && ok;
        tc::tc_fence_after();
        const uint32_t lane_base = (uint32_t)(threadIdx.x & ~31) << 16;
#pragma unroll
        for (int c = 0; c < CT; c += 16) tc::tmem_ld16(acc + lane_base + c, a + c);
        return __syncthreads_and(ok) != 0;  // x_hi / x_lo may be rewritten
    }
    __device__ __forceinline__ void teardown(bool ok, int *err) {
        if (threadIdx.x == 0) {
            if (!tc::mbar_wait(bars, 0)) ok = false;  // no copy may land after the block has gone (bounded)
            if (!ok) atomicExch(err, 1);
        }
        tc::tc_fence_before();
        __syncthreads();
        if (threadIdx.x < 32) tc::tmem_dealloc(tmem, kCols);
    }
};

// v[c] = src[(j0 + c) N + t] for live columns and t < N, else 0
template <int CT>
__device__ __forceinline__ void load_cols(const float *src, size_t cb, int ncols, int N, float (&v)[CT]) {
    const int t = threadIdx.x;
#pragma unroll
    for (int c = 0; c < CT; ++c) v[c] = (src && t < N && c < ncols) ? __ldcg(src + cb + (size_t)c * N + t) : 0.f;
}
template <int CT>
__device__ __forceinline__ void store_cols(float *dst, size_t cb, int ncols, int N, const float (&v)[CT]) {
    const int t = threadIdx.x;
#pragma unroll
    for (int c = 0; c < CT; ++c)
        if (t < N && c < ncols) dst[cb + (size_t)c * N + t] = v[c];
}

template <int CT>
__global__ void __launch_bounds__(128) k_tc_fp_rhs_cols(const float *psi_half, const float *phi, float *phi_half,
                                                        const float *sigma_s, const double *h, TcOps ops, float *rhs,
                                                        int N, int sumK, int *err) {
    extern __shared__ __align__(128) unsigned char smem_tc[];
    __shared__ float w[CT / 2];  // h / 6 of the cells (an FP64 divide: once per cell, not per thread)
    TcCols<CT> s;
    const int j0 = blockIdx.x * CT, ncols = min(CT, 2 * sumK - j0), g0 = j0 >> 1, t = threadIdx.x;
    if (t < CT / 2) w[t] = 2 * t < ncols ? (float)(h[g0 + t] / 6.0) : 0.f;
    s.setup(smem_tc, ops, N);
    tc::grid_dependency_wait();  // the inputs come from the previous kernel
    const size_t cb = ((size_t)blockIdx.y * sumK * 2 + j0) * N;
    float v[CT], ph[CT], sg[CT / 2], a[CT];
    load_cols<CT>(psi_half, cb, ncols, N, v);
    load_cols<CT>(phi, cb, ncols, N, ph);
    load_cols<CT / 2>(sigma_s, (size_t)g0 * N, ncols / 2, N, sg);
    s.store_x(v, N);
    bool ok = s.gemm(0, N, a);
    if (ok) {  // phi_half = D psi; next x = Sigma (phi_half - phi)
        store_cols<CT>(phi_half, cb, ncols, N, a);
#pragma unroll
        for (int c = 0; c < CT; ++c) v[c] = sg[c / 2] * (a[c] - ph[c]);
        s.store_x(v, N);
        ok = s.gemm(1, N, a);
    }
    if (ok) {  // rhs = m (x) r
#pragma unroll
        for (int c = 0; c < CT; c += 2) {
            const float wc = w[c / 2], r0 = a[c], r1 = a[c + 1];
            a[c] = wc * (2.f * r0 + r1);
            a[c + 1] = wc * (r0 + 2.f * r1);
        }
        store_cols<CT>(rhs, cb, ncols, N, a);
    }
    s.teardown(ok, err);
}

template <int CT>
__global__ void __launch_bounds__(128) k_tc_update_scatter_cols(const float *v_in, const float *phi_base, float *phi,
                                                                const float *sigma_s, TcOps ops, float *q,
                                                                const float *qang, int N, int sumK, int *err) {
    extern __shared__ __align__(128) unsigned char smem_tc[];
    TcCols<CT> s;
    s.setup(smem_tc, ops, N);
    tc::grid_dependency_wait();  // the inputs come from the previous kernel
    const int j0 = blockIdx.x * CT, ncols = min(CT, 2 * sumK - j0);
    const size_t cb = ((size_t)blockIdx.y * sumK * 2 + j0) * N;
    float v[CT], pb[CT], sg[CT / 2], qa[CT], a[CT];
    load_cols<CT>(v_in, cb, ncols, N, v);
    load_cols<CT>(phi_base, cb, ncols, N, pb);
    load_cols<CT / 2>(sigma_s, (size_t)(j0 >> 1) * N, ncols / 2, N, sg);
    load_cols<CT>(qang, cb, ncols, N, qa);
    s.store_x(v, N);
    bool ok = s.gemm(0, N, a);
    if (ok) {  // phi = phi_base + D v; next x = Sigma phi
#pragma unroll
        for (int c = 0; c < CT; ++c) {
            a[c] += pb[c];
            v[c] = sg[c / 2] * a[c];
        }
        store_cols<CT>(phi, cb, ncols, N, a);
        s.store_x(v, N);
        ok = s.gemm(1, N, a);
    }
    if (ok) {  // q = M (Sigma phi) + q_ang
#pragma unroll
        for (int c = 0; c < CT; ++c) a[c] += qa[c];
        store_cols<CT>(q, cb, ncols, N, a);
    }
    s.teardown(ok, err);
}

// ---------------------------------------------------------------------------
// Contractions for N > 128 (N a multiple of 32, at most 256): the operators (2 N^2 BF16
// values each, split hi / lo) no longer fit shared memory. As in the few-column kernels the
// operator is the A operand (rows = outputs, two M = 128 tiles) and a tile of CT = 64
// columns the B operand, so that a warp's global accesses are 128 contiguous bytes of a
// column and both nodes of a cell meet in one thread. A CTA is eight worker warps (thread t
// owns output t of every column), an issuing thread and one that streams the operators through
// kStages stages, 16 columns of hi and lo each (stored chunk-major in global memory, [N / 16
// chunks][N rows][16] in the K-major core-matrix layout; shared by every tile, so they stay
// in L2), across GEMMs and tiles: what it copies next never depends on the data. Two CTAs
// per SM, so that one's loads and stores run during the other's products.
// What bounds it: the operators' stream from L2 (0.5 MB a tile of 64 columns) and the
// tile's own 0.26 MB of global traffic. A tile of 128 columns whose thread t owned COLUMN t
// (rows of 1 KB read 16 bytes per lane and instruction, one CTA per SM) took 0.62 and 0.71
// ms for 160000 columns at N = 256, with one thread for copies and products 0.44
// and 0.50, now 0.26 and 0.29.
//   k_tc_wide<FpRhs>         phi_half = D psi;  rhs = m (x) M Sigma (phi_half - phi)
//   k_tc_wide<UpdateScatter> phi = phi_base + D v;  q = M (Sigma phi) + q_ang
//   k_tc_wide<RhsMoments>    rhs = m (x) M Sigma v                 (GMRES; v: moments)
//   k_tc_wide<MomentsAxpy>   out = base + sign D psi               (GMRES)
// err is set to 1 if an mbarrier wait ran out (the CTA then stops).
// ---------------------------------------------------------------------------
namespace tc {
constexpr int kChunkK = 16;
// byte offset of element (row, k) of an N x N operator in the chunk-major layout
__host__ __device__ __forceinline__ uint32_t chunk_offset(int row, int k, int N) {
    return (uint32_t)(k / kChunkK) * (uint32_t)N * kChunkK * 2u + kmajor_offset(row, k % kChunkK, kChunkK);
}
}  // namespace tc

namespace tcw {
constexpr int kWorkers = 256, kThreads = kWorkers + 64, kCT = 64, kStages = 3;
constexpr unsigned kFlagTries = 1u << 28;  // of a wait that ends with the workers' bounded ones
constexpr uint32_t kPart = 256u * tc::kChunkK * 2u, kStage = 2 * kPart;  // hi and lo of a chunk, 256 rows of room
constexpr uint32_t kTmem = 256;                                          // two GEMMs x two row tiles x kCT
struct Plan {
    uint32_t x_bytes, stages, bars, total;
    __host__ __device__ static Plan make(int N) {
        Plan p;
        p.x_bytes = (uint32_t)kCT * N * 2;
        p.stages = 2 * p.x_bytes;
        p.bars = p.stages + kStages * kStage;
        p.total = p.bars + 128;
        return p;
    }
};
enum Kind { FpRhs, UpdateScatter, RhsMoments, MomentsAxpy };
struct Args {
    const float *in, *base, *sigma, *qang;  // psi / v, phi / phi_base / base, Sigma, q_ang (base, qang: may be NULL)
    const double *h;
    float *mid, *out;  // phi_half / phi; rhs / q / out (base may alias mid or out)
    float sign;
};
}  // namespace tcw

template <int KIND>
__global__ void __launch_bounds__(tcw::kThreads, 2) k_tc_wide(tcw::Args g, TcOps ops, int N, int sumK, int R, int *err) {
    using namespace tcw;
    constexpr bool kMass = KIND == FpRhs || KIND == RhsMoments, kTwo = KIND == FpRhs || KIND == UpdateScatter;
    constexpr int kGemms = kTwo ? 2 : 1;
    extern __shared__ __align__(128) unsigned char smem_tc[];
    __shared__ int s_fail;                // a wait of this CTA gave up
    __shared__ float s_w[2][kCT / 2];     // h / 6 of a tile's cells
    const Plan pl = Plan::make(N);
    unsigned char *x_hi = smem_tc, *x_lo = smem_tc + pl.x_bytes, *stg = smem_tc + pl.stages;
    uint64_t *full = reinterpret_cast<uint64_t *>(smem_tc + pl.bars), *empty = full + kStages, *full_x = empty + kStages,
             *acc_bar = full_x + 1, *drain = acc_bar + 1;
    uint32_t *slot = reinterpret_cast<uint32_t *>(drain + 1);
    const int t = threadIdx.x;
    if (t == 0) {
        for (int i = 0; i < 2 * kStages; ++i) tc::mbar_init(full + i, 1);
        tc::mbar_init(full_x, kWorkers);
        tc::mbar_init(acc_bar, 1);
        tc::mbar_init(drain, 1);
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (t < 32) {
        tc::tmem_alloc(slot, kTmem);
        tc::tmem_relinquish();
    }
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = *slot;
    const int tiles_per_r = (2 * sumK + kCT - 1) / kCT, ntiles = tiles_per_r * R;
    auto failed = [&]() { return *(volatile int *)&s_fail != 0; };
    auto fail = [&]() {
        *(volatile int *)&s_fail = 1;
        atomicExch(err, 1);
    };
    const int nch = N / tc::kChunkK, mine = blockIdx.x < ntiles ? (ntiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    auto wait_flag = [&](uint64_t *bar, uint32_t par) {
        for (unsigned i = 0; !tc::mbar_test(bar, par); ++i)
            if (failed() || i > kFlagTries) return false;
        return true;
    };
    if (t == kWorkers) {
        // ---- copies: this CTA's tiles x GEMMs x chunks, in order, as stages become free
        const uint32_t part = (uint32_t)N * tc::kChunkK * 2;  // bytes of hi (or lo) of a chunk
        const size_t lo = (size_t)N * N * 2;
        uint32_t issued = 0, par = 1;
        int s = 0;
        bool ok = true;
        for (int i = 0; i < mine && ok; ++i)
            for (int gm = 0; gm < kGemms && ok; ++gm) {
                const unsigned char *src = (KIND == RhsMoments || gm == 1) ? ops.M : ops.D;
                for (int kc = 0; kc < nch; ++kc, src += part) {
                    if (issued >= (uint32_t)kStages && !(ok = wait_flag(&empty[s], par))) break;
                    tc::mbar_arrive_expect_tx(&full[s], 2 * part);
                    tc::bulk_copy_g2s(stg + s * kStage, src, part, &full[s]);
                    tc::bulk_copy_g2s(stg + s * kStage + kPart, src + lo, part, &full[s]);
                    ++issued;
                    if (++s == kStages) {
                        s = 0;
                        par ^= 1u;
                    }
                }
            }
        if (!ok) fail();
        // nothing may land after the CTA has gone (bounded)
        for (uint32_t j = issued > (uint32_t)kStages ? issued - kStages : 0; j < issued; ++j)
            if (!tc::mbar_wait(&full[j % kStages], (j / kStages) & 1u)) break;
    } else if (t == kWorkers + 32) {
        // ---- products, in the order of the copies; descriptors that differ by constants
        const uint32_t idesc = tc::idesc_bf16(128, kCT), sbo_x = (uint32_t)N * 16;
        const uint64_t bh0 = tc::smem_desc(tc::smem_u32(x_hi), 128, sbo_x), bl0 = tc::smem_desc(tc::smem_u32(x_lo), 128, sbo_x);
        const uint64_t a0 = tc::smem_desc(tc::smem_u32(stg), 128, tc::kChunkK * 16);
        uint32_t xs = 0, par = 0;
        int s = 0;
        bool ok = true;
        for (int i = 0; i < mine && ok; ++i)
            for (int gm = 0; gm < kGemms && ok; ++gm) {
                if (!(ok = wait_flag(full_x, xs & 1u))) break;  // the workers' tile
                ++xs;
                const uint32_t acc = tmem + (uint32_t)(2 * gm * kCT);
                for (int kc = 0; kc < nch; ++kc) {
                    if (!(ok = tc::mbar_wait(&full[s], par))) break;
                    tc::tc_fence_after();
                    const uint64_t ah = a0 + (uint64_t)(s * (kStage / 16)), al = ah + (uint64_t)(kPart / 16);
                    const uint64_t bh = bh0 + (uint64_t)(16 * kc), bl = bl0 + (uint64_t)(16 * kc);
                    const uint32_t more = kc > 0 ? 1u : 0u;
#pragma unroll
                    for (int m = 0; m < 2; ++m) {
                        tc::mma_bf16(acc + m * kCT, ah + m * 256u, bh, idesc, more);
                        tc::mma_bf16(acc + m * kCT, ah + m * 256u, bl, idesc, 1u);
                        tc::mma_bf16(acc + m * kCT, al + m * 256u, bh, idesc, 1u);
                    }
                    tc::mma_commit(&empty[s]);
                    if (++s == kStages) {
                        s = 0;
                        par ^= 1u;
                    }
                }
                if (ok) tc::mma_commit(acc_bar);
            }
        if (!ok) fail();
        tc::mma_commit(drain);
        (void)tc::mbar_wait(drain, 0);
    } else if (t < kWorkers) {
        // ---- workers
        tc::grid_dependency_wait();  // the inputs come from the previous kernel
        const bool live = t < N;     // (N is a multiple of 32: whole warps)
        const uint32_t at = tmem + ((uint32_t)(t & 96) << 16) + (uint32_t)((t >> 7) * kCT);
        uint32_t accs = 0;
        // 16 columns from column c0 into x_hi / x_lo (row = column, k = t; adjacent threads exchange
        // values so that each stores two adjacent k of one column)
        auto store16 = [&](int c0, const float (&v)[16]) {
            const int odd = t & 1;
#pragma unroll
            for (int c = 0; c < 16; c += 2) {
                const float other = __shfl_xor_sync(0xffffffffu, odd ? v[c] : v[c + 1], 1);
                const float k0 = odd ? other : v[c], k1 = odd ? v[c + 1] : other;
                __nv_bfloat16 h0, l0, h1, l1;
                tc::split_bf16(k0, h0, l0);
                tc::split_bf16(k1, h1, l1);
                const uint32_t off = tc::kmajor_offset(c0 + c + odd, t & ~1, N);
                *reinterpret_cast<uint32_t *>(x_hi + off) =
                    (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
                *reinterpret_cast<uint32_t *>(x_lo + off) =
                    (uint32_t)__bfloat16_as_ushort(l0) | ((uint32_t)__bfloat16_as_ushort(l1) << 16);
            }
        };
        auto hand_over = [&]() {  // the tile in x_hi / x_lo to the driver
            tc::fence_async_smem();
            tc::tc_fence_before();
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(full_x)) : "memory");
        };
        auto wait_acc = [&]() {  // a GEMM's accumulators are ready; all workers agree whether to go on
            if (!tc::mbar_wait(acc_bar, accs & 1u)) fail();
            ++accs;
            const bool stop = gbar_or(1, kWorkers, failed());
            tc::tc_fence_after();
            return !stop;
        };
        int par = 0;
        for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, par ^= 1) {
            const int r = tile / tiles_per_r, j0 = (tile % tiles_per_r) * kCT, nc = min(kCT, 2 * sumK - j0);
            const size_t cb = ((size_t)r * sumK * 2 + j0) * N + t;
            const float *sg = g.sigma + (size_t)(j0 >> 1) * N + t;
            if (kMass && t < kCT / 2) s_w[par][t] = 2 * t < nc ? (float)(g.h[(j0 >> 1) + t] / 6.0) : 0.f;
            if (live) {
#pragma unroll 1
                for (int c0 = 0; c0 < kCT; c0 += 16) {
                    float v[16];
#pragma unroll
                    for (int c = 0; c < 16; ++c) v[c] = c0 + c < nc ? __ldcg(g.in + cb + (size_t)(c0 + c) * N) : 0.f;
                    if constexpr (KIND == RhsMoments) {
#pragma unroll
                        for (int c = 0; c < 16; ++c)
                            v[c] *= c0 + c < nc ? __ldg(sg + (size_t)((c0 + c) >> 1) * N) : 0.f;
                    }
                    store16(c0, v);
                }
            }
            hand_over();
            if constexpr (kTwo) {
                if (!wait_acc()) break;
                if (live) {
#pragma unroll 1
                    for (int c0 = 0; c0 < kCT; c0 += 16) {
                        float a[16], b[16], s[8];
#pragma unroll
                        for (int c = 0; c < 16; ++c)
                            b[c] = (g.base && c0 + c < nc) ? __ldcg(g.base + cb + (size_t)(c0 + c) * N) : 0.f;
#pragma unroll
                        for (int c = 0; c < 8; ++c)
                            s[c] = c0 + 2 * c < nc ? __ldg(sg + (size_t)((c0 >> 1) + c) * N) : 0.f;
                        tc::tmem_ld16(at + (uint32_t)c0, a);
#pragma unroll
                        for (int c = 0; c < 16; ++c) {
                            if (KIND == UpdateScatter) a[c] += b[c];
                            if (c0 + c < nc) g.mid[cb + (size_t)(c0 + c) * N] = a[c];
                            a[c] = KIND == FpRhs ? s[c / 2] * (a[c] - b[c]) : s[c / 2] * a[c];
                        }
                        store16(c0, a);
                    }
                }
                hand_over();
            }
            if (!wait_acc()) break;
            if (live) {
#pragma unroll 1
                for (int c0 = 0; c0 < kCT; c0 += 16) {
                    float a[16], b[16];
                    const float *add = KIND == UpdateScatter ? g.qang : (KIND == MomentsAxpy ? g.base : nullptr);
#pragma unroll
                    for (int c = 0; c < 16; ++c)
                        b[c] = (!kMass && add && c0 + c < nc) ? __ldcg(add + cb + (size_t)(c0 + c) * N) : 0.f;
                    tc::tmem_ld16(at + (uint32_t)((kGemms - 1) * 2 * kCT + c0), a);
#pragma unroll
                    for (int c = 0; c < 16; c += 2) {
                        float y0, y1;
                        if constexpr (kMass) {
                            const float w = s_w[par][(c0 + c) >> 1];
                            y0 = w * (2.f * a[c] + a[c + 1]);
                            y1 = w * (a[c] + 2.f * a[c + 1]);
                        } else if constexpr (KIND == MomentsAxpy) {
                            y0 = b[c] + g.sign * a[c];
                            y1 = b[c + 1] + g.sign * a[c + 1];
                        } else {
                            y0 = a[c] + b[c];
                            y1 = a[c + 1] + b[c + 1];
                        }
                        if (c0 + c < nc) {  // (columns come in pairs)
                            g.out[cb + (size_t)(c0 + c) * N] = y0;
                            g.out[cb + (size_t)(c0 + c + 1) * N] = y1;
                        }
                    }
                }
            }
        }
    }
    __syncwarp();
    tc::tc_fence_before();
    __syncthreads();
    if (t < 32) tc::tmem_dealloc(tmem, kTmem);
}

// ---------------------------------------------------------------------------
// Tensor-core contractions of the GMRES operator (the FP32 inner solve of GMRES-IR), one
// GEMM each, N <= 128 (above: k_tc_wide).
//   k_tc_fp_rhs_moments:  rhs = m (x) M Sigma v      (v: moments)
//   k_tc_moments_axpy:    out = base + sign D psi   (base may be NULL or alias out)
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(128) k_tc_fp_rhs_moments(const float *__restrict__ v,
                                                           const float *__restrict__ sigma_s,
                                                           const double *__restrict__ h, TcOps ops,
                                                           float *__restrict__ rhs, int N, int sumK, int R, int *err) {
    extern __shared__ __align__(128) unsigned char smem_tc[];
    TcCta e;
    bool ok = tc_cta_setup(e, smem_tc, ops, N, err);
    tc::grid_dependency_wait();  // the inputs come from the previous kernel
    const int t = threadIdx.x;
    const uint32_t lane_base = (uint32_t)(t & ~31) << 16;
    const int tiles_per_r = (2 * sumK + 127) / 128;
    const int ntiles = tiles_per_r * R;
    for (int tile = blockIdx.x; ok && tile < ntiles; tile += gridDim.x) {
        const int r = tile / tiles_per_r, j0 = (tile % tiles_per_r) * 128;
        const int ncols = min(128, 2 * sumK - j0), ncell = (ncols + 1) >> 1;
        const bool live = t < ncols;
        const int g = (j0 + t) >> 1;
        const size_t cb = ((size_t)r * sumK * 2 + j0) * N;
        const float *sig = sigma_s + (size_t)(j0 >> 1) * N;
        // A = Sigma v
        for (int k0 = 0; k0 < N; k0 += tc::kStageK) {
            tc::stage_in(e.stA, v + cb, N, ncols, k0);
            tc::stage_in(e.stB, sig, N, ncell, k0);
            __syncthreads();
            float vv[16], sg[16], a[16];
            tc::row_get16(e.stA, t, vv);
            tc::row_get16(e.stB, t >> 1, sg);
#pragma unroll
            for (int i = 0; i < 16; ++i) a[i] = live ? sg[i] * vv[i] : 0.f;
            tc::store_split_row16(e.x_hi, e.x_lo, t, k0, a, N);
            __syncthreads();
        }
        if (!(ok = tc_gemm(e, e.opM_hi, e.opM_lo, N, err))) break;
        // rhs = m (x) r: node partner is the adjacent lane (column j ^ 1)
        const float w = live ? (float)(h[g] / 6.0) : 0.f;
        for (int k0 = 0; k0 < N; k0 += tc::kStageK) {
            float a[16], o[16];
            tc::tmem_ld16(e.tmem + lane_base + k0, a);
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const float other = __shfl_xor_sync(0xffffffffu, a[i], 1);
                o[i] = w * (2.f * a[i] + other);
            }
            __syncthreads();  // stC of the previous chunk has been written out
            tc::row_put16(e.stC, t, o);
            __syncthreads();
            tc::stage_out(e.stC, rhs + cb, N, ncols, k0);
        }
    }
    tc_cta_teardown(e, N);
}

__global__ void __launch_bounds__(128) k_tc_moments_axpy(const float *__restrict__ psi, const float *base, float sign,
                                                         TcOps ops, float *out, int N, int sumK, int R, int *err) {
    extern __shared__ __align__(128) unsigned char smem_tc[];
    TcCta e;
    bool ok = tc_cta_setup(e, smem_tc, ops, N, err);
    tc::grid_dependency_wait();  // the inputs come from the previous kernel
    const int t = threadIdx.x;
    const uint32_t lane_base = (uint32_t)(t & ~31) << 16;
    const int tiles_per_r = (2 * sumK + 127) / 128;
    const int ntiles = tiles_per_r * R;
    for (int tile = blockIdx.x; ok && tile < ntiles; tile += gridDim.x) {
        const int r = tile / tiles_per_r, j0 = (tile % tiles_per_r) * 128;
        const int ncols = min(128, 2 * sumK - j0);
        const size_t cb = ((size_t)r * sumK * 2 + j0) * N;
        for (int k0 = 0; k0 < N; k0 += tc::kStageK) {
            tc::stage_in(e.stA, psi + cb, N, ncols, k0);
            __syncthreads();
            float vv[16];
            tc::row_get16(e.stA, t, vv);
            tc::store_split_row16(e.x_hi, e.x_lo, t, k0, vv, N);
            __syncthreads();
        }
        if (!(ok = tc_gemm(e, e.opD_hi, e.opD_lo, N, err))) break;
        // out = base + sign D psi (base read chunk by chunk before out is written: it may alias)
        for (int k0 = 0; k0 < N; k0 += tc::kStageK) {
            if (base) tc::stage_in(e.stA, base + cb, N, ncols, k0);
            float a[16];
            tc::tmem_ld16(e.tmem + lane_base + k0, a);
            __syncthreads();
            float bs[16];
            if (base) tc::row_get16(e.stA, t, bs);
#pragma unroll
            for (int i = 0; i < 16; ++i) a[i] = (base ? bs[i] : 0.f) + sign * a[i];
            tc::row_put16(e.stC, t, a);
            __syncthreads();
            tc::stage_out(e.stC, out + cb, N, ncols, k0);
        }
    }
    tc_cta_teardown(e, N);
}

}  // namespace fpsa
