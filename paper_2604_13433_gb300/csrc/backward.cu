// Backward products of PackSELL matrices in slices of 32 rows: dx = A^T dy
// and dval = alpha dy_i x_j on the pattern (CSR order), each alone or both in
// one pass over the words. The CSR-order (C = 1) form is in split.cu; other
// slice heights run the thread-per-row kernels of spmv.cu.
#include <cuda_fp16.h>

#include <algorithm>

#include "device.cuh"
#include "internal.h"

namespace packsell {
namespace {

constexpr int BW = 8;       // warps per block, one slice each
constexpr int BR = 16;      // words of a row per round
constexpr int BS = BR + 1;  // staging row stride: lanes writing one column hit 32 banks

// Where a row's values of the current round go.
struct __align__(16) RowRun {
    long long q;  // first position in CSR order
    int cnt;
    int pad;
};

// One warp per slice, one lane per row, BR words per round: the round's words
// are loaded together, then its x gathers, then dx takes one reduction
// (atomic add) per value. What bounded the two separate thread-per-row
// kernels was the write of dval: consecutive lanes write consecutive rows, a
// row length apart, so a store of 32 values touched 32 sectors (199 us of
// the 250 us that dx and dval took on the 27-point 113 x 112 x 111 matrix,
// 37.7M values). Here a round's values go to shared memory, row by row, and
// half a warp writes each row's run of up to 16 consecutive values. With both
// results in one pass the words are read and decoded once: 85 us (302 MB of
// words and dval, 3.6 TB/s, beside 37.7M reductions into dx).
template <int FMT, bool DX, bool DV>
__global__ void __launch_bounds__(BW * 32, 4)
    k_back_slices(int n, int sigma, int sig_shift, long long k_left,
                  const int64_t *__restrict__ offset, const uint32_t *__restrict__ pack,
                  const void *__restrict__ perm, int perm_bytes, bool dy_storage, Decode dc,
                  const int64_t *__restrict__ rowptr, float alpha, const float *__restrict__ dy,
                  const float *__restrict__ x, float *__restrict__ dx, float *__restrict__ out) {
    __shared__ float s_val[DV ? BW : 1][DV ? 32 * BS : 1];
    __shared__ RowRun s_run[DV ? BW : 1][DV ? 32 : 1];
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
    const int i = (blockIdx.x * BW + wl) * 32 + lane;
    if (i - lane >= n) return;  // warp-uniform
    const bool live = i < n;
    const int64_t s = offset[i >> 5];
    const int w = (int)((offset[(i >> 5) + 1] - s) >> 5);
    const uint32_t *__restrict__ pp = pack + s + lane;
    const int blk = sig_shift >= 0 ? (i >> sig_shift) << sig_shift : (i / sigma) * sigma;
    int c = (k_left < blk) ? (int)(blk - k_left) : 0;
    int io = i;
    if (live && perm_bytes)
        io = blk + (perm_bytes == 1 ? (int)((const uint8_t *)perm)[i] : (int)((const uint16_t *)perm)[i]);
    // dval's dy is in original order; dx's follows the matrix's output order
    const float g = DX && live ? dy[dy_storage ? i : io] : 0.f;
    const float a = DV && live ? alpha * dy[io] : 0.f;
    long long q = DV && live ? rowptr[io] : 0;
    const long long qend = DV && live ? rowptr[io + 1] : 0;  // (the bounds-check build's)
    for (int j0 = 0; j0 < w; j0 += BR) {
        uint32_t wd[BR];
#pragma unroll
        for (int u = 0; u < BR; ++u) wd[u] = (j0 + u < w) ? ldg_stream(pp + (j0 + u) * 32) : 0u;
        float xv[BR];
#pragma unroll
        for (int u = 0; u < BR; ++u) {
            const bool f = (wd[u] & 1u) != 0u;
            c += (int)((wd[u] >> 1) & (f ? dc.dmask : 0x7fffffffu));
            xv[u] = 0.f;
            if (f && PS_IN_RANGE(c, dc.xlen)) {
                if (DV) xv[u] = __ldg(x + c);
                if (DX && g != 0.f) atomicAdd(dx + c, word_value<FMT>(wd[u], dc) * g);
            }
        }
        if (DV) {
            int t = 0;
#pragma unroll
            for (int u = 0; u < BR; ++u)
                if ((wd[u] & 1u) && PS_IN_RANGE(q + t, qend)) s_val[wl][lane * BS + t++] = a * xv[u];
            s_run[wl][lane] = RowRun{q, t, 0};
            q += t;
            __syncwarp();
            const int sub = lane & 15;
#pragma unroll 4
            for (int k = 0; k < 16; ++k) {
                const int r = 2 * k + (lane >> 4);
                const RowRun run = s_run[wl][r];
                if (sub < run.cnt) __stcs(out + run.q + sub, s_val[wl][r * BS + sub]);
            }
            __syncwarp();
        }
    }
}

template <int FMT, bool DX, bool DV>
void launch_back(const Matrix &A, float alpha, const float *dy, const float *x, float *dx, float *out,
                 cudaStream_t s) {
    const int sg = A.p.sigma;
    const int sh = (sg & (sg - 1)) == 0 ? __builtin_ctz((unsigned)sg) : -1;
    const unsigned g = (unsigned)((A.n_slices + BW - 1) / BW);
    k_back_slices<FMT, DX, DV><<<g, BW * 32, 0, s>>>((int)A.n, sg, sh, A.p.k_left, A.offset, A.pack,
                                                     A.perm, A.perm_bytes, A.p.explicit_perm != 0,
                                                     make_decode(A), A.rowptr, alpha, dy, x, dx, out);
}

template <int FMT>
void launch_back_fmt(const Matrix &A, float alpha, const float *dy, const float *x, float *dx,
                     float *out, cudaStream_t s) {
    if (dx && out) launch_back<FMT, true, true>(A, alpha, dy, x, dx, out, s);
    else if (dx) launch_back<FMT, true, false>(A, alpha, dy, x, dx, out, s);
    else launch_back<FMT, false, true>(A, alpha, dy, x, dx, out, s);
}

}  // namespace

bool backward_fused(const Matrix &A) {
    return is_packed(A.p.format) && A.n > 0 &&
           (A.p.C == 32 || (A.p.C == 1 && A.perm_bytes == 0 && A.split_items));
}

packsell_status backward_impl(const Matrix &A, float alpha, const float *dy, const float *x, float *dx,
                              float *out, cudaStream_t s) {
    if (dx && A.m > 0) PS_CUDA(cudaMemsetAsync(dx, 0, sizeof(float) * A.m, s));
    if (A.nnz == 0 || (!dx && !out)) return PACKSELL_OK;
    if (A.p.C == 1) return launch_split_backward(A, alpha, dy, x, dx, out, s);
    if (A.p.format == PACKSELL_FMT_FP16)
        launch_back_fmt<PACKSELL_FMT_FP16>(A, alpha, dy, x, dx, out, s);
    else
        launch_back_fmt<PACKSELL_FMT_E8MY>(A, alpha, dy, x, dx, out, s);
    PS_LAUNCH_CHECK("packsell backward product");
    return PACKSELL_OK;
}

}  // namespace packsell
