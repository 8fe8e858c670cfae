// Work items of the CSR-order (C = 1) kernels, cut on the device.
//
// Three kernels each take a list of items: tiles of consecutive rows and single
// long rows, long rows first and the longest of them early (they are the
// longest serial paths), tiles in row order. The rule is one (struct
// CutRule): from row r0 a tile takes the most rows that hold at most `words`
// words and are at most `rows`; a row of more words is an item of its own. So
// a tile starts behind every long row whatever was cut before it, and the rows
// are cut in parallel, one warp per chunk of kCutChunk rows: from behind the
// first long row of its chunk to behind the first of the next. Where a chunk
// has no long row a tile starts at its first row instead. (A tile started at
// every chunk gave 0.5 to 1 % more items, which cost variant 14 up to 4.5 %
// where the last round of its warps became one longer: 28.7 -> 30.0 us on a
// power-law matrix of 1M rows. On the host, from a copy of the row offsets, the
// three lists of a 1.4M-row matrix took about 20 ms of its encoding.)
#include <cuda_runtime.h>

#include <algorithm>

#include "device.cuh"
#include "internal.h"

namespace packsell {
namespace {

constexpr int IW = 8;          // warps per block, one chunk each
constexpr int kBuckets = 256;  // of long rows: eight per power of two, longest first
constexpr int kPlans = 3;

struct CutArgs {
    CutRule rule[kPlans];
    int *tiles[kPlans];    // per chunk: tiles, then (after the scan) those before it
    int *bucket[kPlans];   // long rows per bucket, then the bucket's next place
    int *totals;           // per plan: long rows, items; then whether a row has INT32_MAX words or more
    void *items[kPlans];
    int n, chunks;
};

__device__ __forceinline__ int bucket_of(long long w) {  // w >= 1
    const int e = 63 - __clzll(w);
    const int frac = e >= 3 ? (int)((w >> (e - 3)) & 7) : (int)((w << (3 - e)) & 7);
    return kBuckets - 1 - min(kBuckets - 1, 8 * e + frac);
}

__device__ __forceinline__ void put(const CutArgs &a, int plan, int at, long long base, int r0, int rows,
                                    long long w) {
    const int meta = rows > 0 ? (rows << 16) | (int)w : -(int)min(w, (long long)INT32_MAX);
    if (a.rule[plan].kind == CUT_CSR)
        ((int2 *)a.items[plan])[at] = make_int2(r0, r0 + max(rows, 1));
    else if (a.rule[plan].kind == CUT_SPLIT)
        ((SplitItem *)a.items[plan])[at] = SplitItem{base, r0, meta};
    else
        ((MultiItem *)a.items[plan])[at] = MultiItem{base, r0, meta, 0, 0, 0, 0};
}

// The first row that a chunk's warp cuts: behind the chunk's first long row, or
// the chunk's first row where it has none (n past the last chunk).
__device__ int cut_start(const CutArgs &a, int words, int chunk, const int64_t *__restrict__ off) {
    if (chunk == 0) return 0;
    if (chunk >= a.chunks) return a.n;
    const int lane = threadIdx.x & 31, r0 = chunk * kCutChunk, len = min(a.n - r0, kCutChunk);
    for (int t0 = 0; t0 < len; t0 += 128) {
        int64_t w[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int t = t0 + 32 * q + lane;
            w[q] = t < len ? off[r0 + t + 1] - off[r0 + t] : 0;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const unsigned hit = __ballot_sync(0xffffffffu, w[q] > words);
            if (hit) return r0 + t0 + 32 * q + __ffs(hit);
        }
    }
    return r0;
}

// One warp per chunk of rows: the number of rows of the next tile by two
// rounds of 32 offset reads (eight rows apart, then one).
template <bool FILL>
__global__ void __launch_bounds__(IW * 32) k_cut_items(CutArgs a, const int64_t *__restrict__ off) {
    const int plan = blockIdx.y, lane = threadIdx.x & 31;
    const int chunk = blockIdx.x * IW + (threadIdx.x >> 5);
    if (chunk >= a.chunks) return;
    const CutRule rule = a.rule[plan];
    int r = cut_start(a, rule.words, chunk, off);
    const int end = cut_start(a, rule.words, chunk + 1, off);
    int tiles = FILL ? a.tiles[plan][chunk] : 0;
    while (r < end) {
        const long long o = off[r];
        const int most = min(rule.rows, end - r);
        // rows r .. r + t hold off[r + t] - o words
        const int step = (most + 31) / 32;
        int t = min((lane + 1) * step, most);
        const int full = __popc(__ballot_sync(0xffffffffu, off[r + t] - o <= rule.words)) * step;
        const int base = min(full, most);
        t = min(base + lane + 1, most);
        const bool fits = lane < step && base + lane + 1 <= most && off[r + t] - o <= rule.words;
        const int rows = base + __popc(__ballot_sync(0xffffffffu, fits));
        if (rows == 0) {  // a long row
            const long long w = off[r + 1] - o;
            if (lane == 0) {
                const int at = atomicAdd(a.bucket[plan] + bucket_of(w), 1);
                if (FILL) put(a, plan, at, o, r, 0, w);
                else if (w >= INT32_MAX) a.totals[2 * kPlans] = 1;
            }
            r += 1;
        } else {
            if (FILL && lane == 0) put(a, plan, tiles, o, r, rows, off[r + rows] - o);
            ++tiles;
            r += rows;
        }
    }
    if (!FILL && lane == 0) a.tiles[plan][chunk] = tiles;
}

// One block per plan: places of the buckets (from 0), of the chunks' tiles
// (after the long rows), and the totals.
__global__ void __launch_bounds__(1024) k_cut_scan(CutArgs a) {
    __shared__ int s[32];
    const int plan = blockIdx.x, lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
    auto scan = [&](int v, int *sum) {  // exclusive over the block
        int inc = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += u;
        }
        __syncthreads();
        if (lane == 31) s[wl] = inc;
        __syncthreads();
        int before = 0, all = 0;
        for (int q = 0; q < 32; ++q) {
            if (q < wl) before += s[q];
            all += s[q];
        }
        *sum = all;
        return before + inc - v;
    };
    int nlong;
    const int b = threadIdx.x < kBuckets ? a.bucket[plan][threadIdx.x] : 0;
    const int pb = scan(b, &nlong);
    if (threadIdx.x < kBuckets) a.bucket[plan][threadIdx.x] = pb;
    int at = nlong;
    for (int c0 = 0; c0 < a.chunks; c0 += 1024) {
        const int c = c0 + threadIdx.x, v = c < a.chunks ? a.tiles[plan][c] : 0;
        int sum;
        const int p = scan(v, &sum);
        if (c < a.chunks) a.tiles[plan][c] = at + p;
        at += sum;
    }
    if (threadIdx.x == 0) {
        a.totals[2 * plan] = nlong;
        a.totals[2 * plan + 1] = at;
    }
}

}  // namespace

packsell_status plan_items(Matrix &A, cudaStream_t s) {
    if (!is_packed(A.p.format) || A.p.C != 1 || A.n == 0) return PACKSELL_OK;
    // every item holds a row of its own, and items are counted in 32 bits
    if (A.n >= INT32_MAX) return fail(PACKSELL_ERR_RANGE, "plan of the CSR-order kernels: too many rows");
    const CutRule rules[kPlans] = {csr_rule(), split_rule(), multi_rule()};
    const size_t item_bytes[kPlans] = {sizeof(int2), sizeof(SplitItem), sizeof(MultiItem)};
    void **out[kPlans] = {&A.csr_items, &A.split_items, &A.multi_items};
    int *count[kPlans] = {&A.csr_nitems, &A.split_nitems, &A.multi_nitems};
    CutArgs a{};
    a.n = (int)A.n;
    a.chunks = (int)((A.n + kCutChunk - 1) / kCutChunk);
    const size_t ints = kPlans * ((size_t)a.chunks + kBuckets + 2) + 1;
    int *mem = nullptr, h[2 * kPlans + 1] = {};
    PS_CUDA(pool_get(&mem, sizeof(int) * ints, s));
    a.totals = mem;
    int *at = mem + 2 * kPlans + 1;
    for (int p = 0; p < kPlans; ++p) {
        a.rule[p] = rules[p];
        a.bucket[p] = at;
        at += kBuckets;
    }
    for (int p = 0; p < kPlans; ++p) {
        a.tiles[p] = at;
        at += a.chunks;
    }
    const dim3 grid((a.chunks + IW - 1) / IW, kPlans);
    cudaError_t e = cudaMemsetAsync(mem, 0, sizeof(int) * ((2 + kBuckets) * kPlans + 1), s);
    if (e == cudaSuccess) {
        k_cut_items<false><<<grid, IW * 32, 0, s>>>(a, A.offset);
        k_cut_scan<<<kPlans, 1024, 0, s>>>(a);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(h, a.totals, sizeof(h), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e == cudaSuccess && h[2 * kPlans]) {
        pool_put(mem, s);
        return fail(PACKSELL_ERR_RANGE, "split-row plan: row too long");
    }
    for (int p = 0; p < kPlans && e == cudaSuccess; ++p) {
        e = pool_get(out[p], item_bytes[p] * (size_t)h[2 * p + 1], s);
        a.items[p] = *out[p];
    }
    if (e == cudaSuccess) {
        k_cut_items<true><<<grid, IW * 32, 0, s>>>(a, A.offset);
        e = cudaGetLastError();
    }
    pool_put(mem, s);
    if (e != cudaSuccess) return cuda_fail(e, "plan of the CSR-order kernels");
    for (int p = 0; p < kPlans; ++p) *count[p] = h[2 * p + 1];
    return PACKSELL_OK;
}

}  // namespace packsell
