// Block cyclic reduction factorization for FP blocks larger than one CTA can
// invert in registers / shared memory (2N > 128): in-place recursive block-Schur
// inversion of each eliminated cell's 2N x 2N block,
//   [[A11, A12], [A21, A22]]^{-1}: P = A11^{-1}, X = P A12, Y = A21 P,
//   S = A22 - A21 X, Q = S^{-1},
//   A12 <- -X Q,  A21 <- -Q Y,  A11 <- P - X A21,  A22 <- Q,
// recursing on A11 and S until blocks are <= 128 (then Gauss-Jordan with partial
// pivoting, `gj_reg_body` / `gj_smem_body`). No pivoting crosses the halves; the
// FP blocks are well conditioned (the L-node half is |H|/2 + (h/3) K with
// K = sigma_a I - sigma_tr/2 A_FP), and the FP64 growth check of the whole block
// (max|A| max|A^{-1}|) guards every case. The inverse is finally transposed in
// place to the layout the BCR solve reads. All operations are batched over the
// eliminated cells of one level (a chunk of at most kLargeChunk at a time).
#pragma once

#include "kernels.cuh"

namespace fpsa {

constexpr int kLargeChunk = 1024;

// Matrix e of a batch: base + idx(e) * stride, row-major with leading dimension ld;
// idx(e) = items[e].cell (by_cell) or e.
template <typename T>
struct BMat {
    T *base;
    long long stride;
    int ld;
    int by_cell;
    __host__ __device__ BMat sub(int r0, int c0) const { return BMat{base + (long long)r0 * ld + c0, stride, ld, by_cell}; }
};

template <typename T>
__device__ __forceinline__ T *bmat_ptr(const BMat<T> &m, const BcrItem *items, int e) {
    return m.base + (long long)(m.by_cell ? items[e].cell : e) * m.stride;
}

template <typename T, int N2>
__global__ void __launch_bounds__(512) k_binv_reg_rm(BMat<T> M, const BcrItem *__restrict__ items,
                                                     int *__restrict__ status) {
    T *p = bmat_ptr(M, items, blockIdx.x);
    if constexpr (sizeof(T) == 4) gj_panel_body<N2>(p, M.ld, p, M.ld, false, nullptr, status);
    else gj_reg_body<T, N2>(p, M.ld, p, M.ld, false, nullptr, status);
}

template <typename T>
__global__ void k_binv_smem_rm(BMat<T> M, int n, const BcrItem *__restrict__ items, int *__restrict__ status) {
    T *p = bmat_ptr(M, items, blockIdx.x);
    gj_smem_body(p, M.ld, p, M.ld, false, n, nullptr, status);
}

// C = alpha A B + beta C for n x n blocks of a batch (blockIdx.z = batch element),
// 64 x 64 output tiles, 256 threads with 4 x 4 outputs each, k-steps of 16 through
// shared memory. C never aliases A or B.
template <typename T>
__global__ void __launch_bounds__(256) k_bgemm(int n, T alpha, BMat<T> A, BMat<T> B, T beta, BMat<T> C,
                                               const BcrItem *__restrict__ items) {
    __shared__ T As[16][64 + 1], Bs[16][64 + 1];
    const T *a = bmat_ptr(A, items, blockIdx.z);
    const T *b = bmat_ptr(B, items, blockIdx.z);
    T *c = bmat_ptr(C, items, blockIdx.z);
    const int r0 = blockIdx.y * 64, c0 = blockIdx.x * 64;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    T acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = T(0);
    for (int k0 = 0; k0 < n; k0 += 16) {
        for (int idx = threadIdx.x; idx < 16 * 64; idx += 256) {
            const int kk = idx & 15, rr = idx >> 4;  // A tile: rows r0.., cols k0..
            const int gr = r0 + rr, gk = k0 + kk;
            As[kk][rr] = (gr < n && gk < n) ? a[(size_t)gr * A.ld + gk] : T(0);
            const int cc = idx & 63, kb = idx >> 6;  // B tile: rows k0.., cols c0..
            const int gk2 = k0 + kb, gc = c0 + cc;
            Bs[kb][cc] = (gk2 < n && gc < n) ? b[(size_t)gk2 * B.ld + gc] : T(0);
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < 16; ++kk) {
            T av[4], bv[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) av[i] = As[kk][ty + 16 * i];
#pragma unroll
            for (int j = 0; j < 4; ++j) bv[j] = Bs[kk][tx + 16 * j];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fma(av[i], bv[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int gr = r0 + ty + 16 * i, gc = c0 + tx + 16 * j;
            if (gr < n && gc < n) {
                T *dst = c + (size_t)gr * C.ld + gc;
                *dst = alpha * acc[i][j] + (beta != T(0) ? beta * *dst : T(0));
            }
        }
}

// Block-wide maximum of |v| (valid in thread 0), for blocks of up to 1024 threads.
__device__ __forceinline__ double block_max(double m) {
    __shared__ double red[32];
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0)
        for (int i = 1; i < (int)(blockDim.x >> 5); ++i) m = fmax(m, red[i]);
    return m;
}

// max|A| of each block of the batch (contiguous, n even; before inversion), for
// the growth check, into the zeroed amax[e] (as the bits of a non-negative double, whose
// order is that of the values). Bound by the read of the blocks (131 MB at n = 256 and 500
// items): kMaxSplit thread blocks per item, 16-byte loads eight deep (one block of single
// loads per item took 144 us there, 561 us at n = 512).
constexpr int kMaxSplit = 8;
template <typename T>
__global__ void __launch_bounds__(256) k_bamax(BMat<T> M, int n, const BcrItem *__restrict__ items,
                                               unsigned long long *__restrict__ amax) {
    using VT = typename VecOf<T>::type;
    const VT *p = reinterpret_cast<const VT *>(bmat_ptr(M, items, blockIdx.x));
    const int words = n * n / VecOf<T>::V, per = (words + kMaxSplit - 1) / kMaxSplit;
    const int w0 = blockIdx.y * per, w1 = min(words, w0 + per);
    T m = T(0);
    for (int i = w0 + threadIdx.x; i < w1; i += 8 * 256) {
        VT v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (i + 256 * u < w1) v[u] = __ldcg(p + i + 256 * u);
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (i + 256 * u < w1) {
                m = fmax(m, fmax(fabs(v[u].x), fabs(v[u].y)));
                if constexpr (VecOf<T>::V == 4) m = fmax(m, fmax(fabs(v[u].z), fabs(v[u].w)));
            }
    }
    const double b = block_max((double)m);
    if (threadIdx.x == 0) atomicMax(amax + blockIdx.x, dkey(b));
}

// In-place transpose of each n x n inverse (row-major -> the transposed layout of
// the BCR solve) with the growth check max|A| max|A^{-1}| and a finiteness check. One
// block per item and pair of mirrored 32 x 32 tiles (blockIdx.y counts the tiles on and
// above the diagonal), both read and written by whole rows: one pass over the blocks at
// memory rate (element by element, one block per item: 113 us at n = 256 and 500 items).
template <typename T>
__global__ void __launch_bounds__(256) k_btranspose(BMat<T> M, int n, const BcrItem *__restrict__ items,
                                                    const unsigned long long *__restrict__ amax,
                                                    unsigned long long *__restrict__ growth, int *__restrict__ status) {
    __shared__ T ta[32][33], tb[32][33];
    T *p = bmat_ptr(M, items, blockIdx.x);
    int bi = 0, rest = blockIdx.y;
    for (int row = (n + 31) / 32; rest >= row; --row) {
        rest -= row;
        ++bi;
    }
    const int i0 = 32 * bi, j0 = 32 * (bi + rest), x = threadIdx.x & 31, y0 = threadIdx.x >> 5;
    T m = T(0);
    bool bad = false;
    auto take = [&](T v) {
        m = fmax(m, fabs(v));
        if (!isfinite(v)) bad = true;
        return v;
    };
#pragma unroll
    for (int y = y0; y < 32; y += 8) {
        if (i0 + y < n && j0 + x < n) ta[y][x] = take(p[(size_t)(i0 + y) * M.ld + j0 + x]);
        if (j0 + y < n && i0 + x < n) tb[y][x] = take(p[(size_t)(j0 + y) * M.ld + i0 + x]);
    }
    __syncthreads();
#pragma unroll
    for (int y = y0; y < 32; y += 8) {
        if (i0 + y < n && j0 + x < n) p[(size_t)(i0 + y) * M.ld + j0 + x] = tb[x][y];
        if (j0 + y < n && i0 + x < n) p[(size_t)(j0 + y) * M.ld + i0 + x] = ta[x][y];
    }
    const double b = block_max((double)m);
    if (threadIdx.x == 0) atomicMax(growth, dkey(b * __longlong_as_double((long long)amax[blockIdx.x])));
    if (bad) atomicExch(status, 1);
}

}  // namespace fpsa
