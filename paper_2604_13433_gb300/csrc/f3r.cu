// F3R: the nested Krylov solver of §5.2.1 (FGMRES, FGMRES, FGMRES and an
// innermost preconditioned Richardson), with the FP16 SpMV of the two inner
// layers as PackSELL FP16 or FP16 SELL, or every layer in FP64.
//
// Layer 1 is restarted flexible GMRES in double precision on the FP64
// operator; its preconditioner is layer 2, m2 iterations of flexible GMRES
// from zero on the FP32 (or FP64) operator; layer 2's preconditioner is layer
// 3, m3 iterations of flexible GMRES from zero on the FP16 operator; layer 3's
// preconditioner is layer 4, m4 steps of Richardson z <- z + omega (r - A z)
// from z = 0 on the FP16 operator (Jacobi preconditioning is the identity on
// the symmetrically scaled matrices of §5.2). Every layer builds its Krylov
// basis with classical Gram-Schmidt: the dot products of a step are one
// deterministic reduction (block partials summed in block order, in double
// precision), the update of the new vector is done in the layer's arithmetic
// (double for the FP64 layers; FP32 for the FP32 layers of FP16-F3R, whose
// per-thread partial sums are FP32 as well, since on GB300 the FP64 pipe
// and not memory would bound those kernels), and the Hessenberg matrix, its
// Givens rotations and the small least-squares solve stay on the device in
// double precision.
// Layers 2-4 run a fixed number of steps (no convergence test); layer 1
// reads its residual estimate |g_{j+1}| after every step and confirms
// convergence on the true residual b - A x in FP64.
//
// The two inner SpMVs of the FP16 layers are the only kernels that differ
// between PackSELL-F3R and FP16-SELL-F3R, and both sum every row as the
// same chain of fused multiply-adds over the same FP16 values: the two
// solvers produce the same iterates, bit for bit (the paper's observation
// that they converge identically).
#include <cuda_fp16.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <string>
#include <type_traits>
#include <vector>

#include "device.cuh"
#include "f3r_plan.h"
#include "internal.h"
#include "meet.cuh"

namespace packsell {

int device_sms();

namespace {

constexpr int FT = 256;  // threads per block of the vector kernels

inline int fgrid(int64_t n) {
    return (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)device_sms() * 4, (n + FT - 1) / FT));
}

// sum of the block's FT values in shared memory by one warp (every lane has
// it): 13 FP64 additions where a shuffle tree in all eight warps takes 40 (an
// FP64 warp instruction takes about 16 cycles of an SM). With `err`, the
// values' rounding errors are added too, a lane's in FP32 first (a second
// rounding of 2^-24 of them): one more FP64 addition.
template <typename T>
__device__ __forceinline__ double warp_total(const T *v, int lane, const float *err = nullptr) {
    double x[FT / 32], t = 0.0;
    if (err) {
        float e = 0.f;
#pragma unroll
        for (int q = 0; q < FT / 32; ++q) e += err[32 * q + lane];
        t = (double)e;
    }
#pragma unroll
    for (int q = 0; q < FT / 32; ++q) x[q] = (double)v[32 * q + lane];
#pragma unroll
    for (int q = 0; q < FT / 32; ++q) t += x[q];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;
}

// block-wide sum of a double (fixed order), result in thread 0; sh: FT values
__device__ __forceinline__ double block_sum(double v, double *sh) {
    sh[threadIdx.x] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x < 32) t = warp_total(sh, threadIdx.x);
    __syncthreads();
    return t;
}

// Arnoldi state of one layer (double, device): H column-major (m+1) x m,
// Givens cosines and sines, right-hand side g (m+1), solution y (m), and
// scal = {beta = ||rhs||, 1 / (last norm), |g_{j+1}|}
struct Hess {
    double *H, *cs, *sn, *g, *y, *scal;
    int m;
};

// The reducing kernels below end with the step that needs the whole
// reduction: each block writes its partial, and the block that arrives last
// (an atomic counter, back at 0 when it is done) adds the partials in block
// order and finishes, so no one-block kernel follows. Called by every thread
// after thread 0 has written the block's partial; true in the last block
// once every partial is visible.
__device__ __forceinline__ bool last_block(unsigned *counter) {
    __shared__ bool last;
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(counter, 1u) == gridDim.x * gridDim.y - 1u;
        if (last) *counter = 0u;
    }
    __syncthreads();
    if (last) __threadfence();
    return last;
}

// sum of the G partials at p, in block order (the whole block; thread 0 has it)
__device__ __forceinline__ double partial_sum(const double *p, int G, double *sh) {
    double s = 0.0;
    for (int b0 = threadIdx.x; b0 < G; b0 += 4 * FT) {  // the loads together, then the additions
        double v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = b0 + q * FT < G ? ((const volatile double *)p)[b0 + q * FT] : 0.0;
#pragma unroll
        for (int q = 0; q < 4; ++q) s += v[q];
    }
    return block_sum(s, sh);
}

// beta = ||rhs|| from the partials; g = beta e_1; scal[1] = 1 / beta
__device__ __forceinline__ void begin_finish(int G, const double *part, Hess h, double *sh) {
    const double s = partial_sum(part, G, sh);
    if (threadIdx.x == 0) {
        const double beta = sqrt(s);
        h.scal[0] = beta;
        h.scal[1] = beta > 0.0 ? 1.0 / beta : 0.0;
        h.scal[2] = beta;
        for (int i = 0; i <= h.m; ++i) h.g[i] = 0.0;
        h.g[0] = beta;
    }
}

// partial sums of v.v per block; the last block sets up the layer (begin_finish)
template <typename T>
__global__ void __launch_bounds__(FT) k_norm2_begin(int64_t n, const T *__restrict__ v,
                                                    double *__restrict__ part, unsigned *counter,
                                                    Hess h) {
    __shared__ double sh[FT];
    double s = 0.0;
    if constexpr (std::is_same<T, float>::value) {  // an FP32 layer: FP32 thread partials
        float sf = 0.f;
        for (int64_t i = blockIdx.x * (int64_t)FT + threadIdx.x; i < n; i += (int64_t)gridDim.x * FT)
            sf = fmaf(v[i], v[i], sf);
        s = (double)sf;
    } else {
        for (int64_t i = blockIdx.x * (int64_t)FT + threadIdx.x; i < n; i += (int64_t)gridDim.x * FT) {
            const double a = (double)v[i];
            s = fma(a, a, s);
        }
    }
    s = block_sum(s, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
    if (last_block(counter)) begin_finish(gridDim.x, part, h, sh);
}

// partial sums of w.v_i for the cnt basis vectors v_i (blockIdx.y = i); the
// last block sets h[i][j] = the sum of the partials of w.v_i, in block order
template <typename T>
__global__ void __launch_bounds__(FT) k_mdot(int64_t n, const T *__restrict__ V,
                                             const T *__restrict__ w, double *__restrict__ part,
                                             unsigned *counter, Hess h, int j) {
    __shared__ double sh[FT];
    const T *__restrict__ v = V + (int64_t)blockIdx.y * n;
    double s = 0.0;
    if constexpr (std::is_same<T, float>::value) {
        float sf = 0.f;
        for (int64_t i = blockIdx.x * (int64_t)FT + threadIdx.x; i < n; i += (int64_t)gridDim.x * FT)
            sf = fmaf(w[i], v[i], sf);
        s = (double)sf;
    } else {
        for (int64_t i = blockIdx.x * (int64_t)FT + threadIdx.x; i < n; i += (int64_t)gridDim.x * FT)
            s = fma((double)w[i], (double)v[i], s);
    }
    s = block_sum(s, sh);
    if (threadIdx.x == 0) part[(int64_t)blockIdx.y * gridDim.x + blockIdx.x] = s;
    if (!last_block(counter)) return;
    const int G = gridDim.x;
    for (int i = 0; i < (int)gridDim.y; ++i) {
        const double t = partial_sum(part + (int64_t)i * G, G, sh);
        if (threadIdx.x == 0) h.H[i + (int64_t)j * (h.m + 1)] = t;
    }
}

// out = (TO)(in * scal[k])
template <typename TI, typename TO>
__global__ void __launch_bounds__(FT) k_scale(int64_t n, const TI *__restrict__ in, TO *__restrict__ out,
                                              const double *__restrict__ scal) {
    const double s = *scal;
    if constexpr (std::is_same<TI, float>::value && std::is_same<TO, float>::value) {
        const float sf = (float)s;
        for (int64_t i = blockIdx.x * (int64_t)FT + threadIdx.x; i < n; i += (int64_t)gridDim.x * FT)
            out[i] = in[i] * sf;
    } else {
        for (int64_t i = blockIdx.x * (int64_t)FT + threadIdx.x; i < n; i += (int64_t)gridDim.x * FT)
            out[i] = (TO)((double)in[i] * s);
    }
}

// h[j+1][j] = ||w||; the earlier Givens rotations on column j, a new one
// that zeroes h[j+1][j]; g updated; scal[1] = 1 / h[j+1][j], scal[2] = |g[j+1]|
__device__ __forceinline__ void givens_column(double s, Hess h, int j) {  // s = w.w
    const int ld = h.m + 1;
    double *col = h.H + (int64_t)j * ld;
    const double hn = sqrt(s);
    col[j + 1] = hn;
    for (int k = 0; k < j; ++k) {
        const double a = col[k], b = col[k + 1];
        col[k] = h.cs[k] * a + h.sn[k] * b;
        col[k + 1] = -h.sn[k] * a + h.cs[k] * b;
    }
    const double a = col[j], b = col[j + 1];
    const double r = hypot(a, b);
    const double c = r > 0.0 ? a / r : 1.0, sn = r > 0.0 ? b / r : 0.0;
    h.cs[j] = c;
    h.sn[j] = sn;
    col[j] = r;
    col[j + 1] = 0.0;
    h.g[j + 1] = -sn * h.g[j];
    h.g[j] = c * h.g[j];
    h.scal[1] = hn > 0.0 ? 1.0 / hn : 0.0;
    h.scal[2] = fabs(h.g[j + 1]);
}

__device__ __forceinline__ void arnoldi_finish(int G, const double *part, Hess h, int j, double *sh) {
    const double s = partial_sum(part, G, sh);
    if (threadIdx.x == 0) givens_column(s, h, j);
}

// w = w - sum_i h[i][j] v_i (in double, rounded once to T); partials of w.w;
// the last block closes the Arnoldi step (arnoldi_finish)
template <typename T>
__global__ void __launch_bounds__(FT) k_orth(int64_t n, const T *__restrict__ V, int cnt, Hess h, int j,
                                             T *__restrict__ w, double *__restrict__ part,
                                             unsigned *counter) {
    __shared__ double sh[FT];
    __shared__ double hc[64];
    __shared__ float hf[64];
    for (int i = threadIdx.x; i < cnt; i += FT) {
        hc[i] = h.H[i + (int64_t)j * (h.m + 1)];
        hf[i] = (float)hc[i];
    }
    __syncthreads();
    double s = 0.0;
    if constexpr (std::is_same<T, float>::value) {
        float sf = 0.f;
        for (int64_t e = blockIdx.x * (int64_t)FT + threadIdx.x; e < n; e += (int64_t)gridDim.x * FT) {
            float a = w[e];
            for (int i = 0; i < cnt; ++i) a = fmaf(-hf[i], V[(int64_t)i * n + e], a);
            w[e] = a;
            sf = fmaf(a, a, sf);
        }
        s = (double)sf;
    } else {
        for (int64_t e = blockIdx.x * (int64_t)FT + threadIdx.x; e < n; e += (int64_t)gridDim.x * FT) {
            double a = (double)w[e];
            for (int i = 0; i < cnt; ++i) a -= hc[i] * (double)V[(int64_t)i * n + e];
            const T r = (T)a;
            w[e] = r;
            s = fma((double)r, (double)r, s);
        }
    }
    s = block_sum(s, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
    if (last_block(counter)) arnoldi_finish(gridDim.x, part, h, j, sh);
}

// ---- an Arnoldi step's vector work in one kernel (FP32 layers) ----
// The three kernels above read the new vector w three times and write it
// twice, and each ends in a reduction that the next one waits for: on the
// 27-point 128^3 matrix (8.4 MB vectors, all in L2) a step of layer 3 spent
// about 50 us in them (F3R 64.5 ms; 62.4 ms with this kernel, 56.4 ms with the
// Richardson steps in the products' epilogues as well). Here every thread keeps its E elements of w in
// registers through the dot products, the update and the scaling, and the
// blocks (all resident: a cooperative launch) meet twice. Every block adds
// all partials itself, in block order, so all have the same sums.
// A thread's vectors are four elements wide, so it holds more products than a
// thread of the separate kernels does, which add no two in FP32 up to 155,648
// unknowns. Its products form four FP32 chains, one per place in the vector,
// and the chains are added with their rounding error (two_sum): where a thread
// has one vector (up to 622,592 unknowns) sum and error both enter the FP64
// sums, and beyond that a chain is a quarter as long as a thread's chain in
// the separate kernels. (One FP32 chain per thread: 64^3 unknowns 7.93 ms
// instead of 8.03, 128^3 55.88 instead of 55.94.)
__device__ __forceinline__ float two_sum(float a, float b, float &err) {  // Knuth: a + b = sum + err
    const float s = a + b, t = s - a;
    err = (a - (s - t)) + (b - t);
    return s;
}

template <int E>
__global__ void __launch_bounds__(FT, 4)
    k_arnoldi(int64_t n, const float *__restrict__ V, int cnt, Hess h, int j, float *__restrict__ w,
              double *__restrict__ part, Meet m) {
    constexpr int PB = 8;  // quantities reduced together, one per warp
    __shared__ float sh[PB][FT], sh_err[PB][FT];
    __shared__ float hf[64];
    __shared__ double s_norm;
    // (one answer for the block: another one may be setting the flag)
    if (__syncthreads_or(*(volatile int *)m.timeout != 0)) return;
    const int G = gridDim.x, wl = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t tid = blockIdx.x * (int64_t)FT + threadIdx.x, st = (int64_t)G * FT, nv = n / 4;
    const bool one = nv <= st;  // at most one vector per thread
    float4 a[E / 4];
#pragma unroll
    for (int k = 0; k < E / 4; ++k) {
        const int64_t v = tid + k * st;
        a[k] = v < nv ? reinterpret_cast<const float4 *>(w)[v] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    // the n % 4 elements after the last whole vector, one thread each
    const int64_t te = nv * 4 + tid;
    const bool tail = te < n;
    float at = tail ? w[te] : 0.f;
    // the grid's sum of one quantity, every lane of the warp (partials in block order)
    auto total = [&](const double *p) {
        double s = 0.0;
        for (int b0 = 0; b0 < G; b0 += 8 * 32) {  // eight loads in flight, added in order
            double v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int b = b0 + 32 * q + lane;
                v[q] = b < G ? ((const volatile double *)p)[b] : 0.0;
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) s += v[q];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        return s;
    };
    // this thread's part of a quantity: its four chains and the tail's product
    auto put = [&](int slot, float4 f, float ft) {
        float e0, e1, e2, e3;
        const float s = two_sum(two_sum(two_sum(f.x, f.y, e0), two_sum(f.z, f.w, e1), e2), ft, e3);
        sh[slot][threadIdx.x] = s;
        if (one) sh_err[slot][threadIdx.x] = (e0 + e1) + (e2 + e3);
    };
    // the block's sums of the quantities [i0, i0 + count) in sh, one partial each
    auto block_parts = [&](int i0, int count, double *out) {
        __syncthreads();
        if (wl < count) {
            const double s = warp_total(sh[wl], lane, one ? sh_err[wl] : nullptr);
            if (lane == 0) out[(int64_t)(i0 + wl) * G + blockIdx.x] = s;
        }
        __syncthreads();
    };
    for (int i = 0; i < cnt; ++i) {
        const float *__restrict__ v = V + (int64_t)i * n;
        const bool al = ((uintptr_t)v & 15u) == 0;
        float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int k = 0; k < E / 4; ++k) {
            const int64_t q = tid + k * st;
            if (q < nv) {
                const float4 b = al ? reinterpret_cast<const float4 *>(v)[q]
                                    : make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
                f.x = fmaf(a[k].x, b.x, f.x);
                f.y = fmaf(a[k].y, b.y, f.y);
                f.z = fmaf(a[k].z, b.z, f.z);
                f.w = fmaf(a[k].w, b.w, f.w);
            }
        }
        put(i % PB, f, tail ? at * v[te] : 0.f);
        if (i % PB == PB - 1 || i + 1 == cnt) block_parts(i / PB * PB, i % PB + 1, part);
    }
    if (!meet(m, 1)) return;
    for (int i = wl; i < cnt; i += FT / 32) {
        const double s = total(part + (int64_t)i * G);
        if (lane == 0) {
            hf[i] = (float)s;
            if (blockIdx.x == 0) h.H[i + (int64_t)j * (h.m + 1)] = s;
        }
    }
    __syncthreads();
    for (int i = 0; i < cnt; ++i) {
        const float *__restrict__ v = V + (int64_t)i * n;
        const bool al = ((uintptr_t)v & 15u) == 0;
        const float c = -hf[i];
        if (tail) at = fmaf(c, v[te], at);
#pragma unroll
        for (int k = 0; k < E / 4; ++k) {
            const int64_t q = tid + k * st;
            if (q < nv) {
                const float4 b = al ? reinterpret_cast<const float4 *>(v)[q]
                                    : make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
                a[k].x = fmaf(c, b.x, a[k].x);
                a[k].y = fmaf(c, b.y, a[k].y);
                a[k].z = fmaf(c, b.z, a[k].z);
                a[k].w = fmaf(c, b.w, a[k].w);
            }
        }
    }
    float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int k = 0; k < E / 4; ++k) {
        f.x = fmaf(a[k].x, a[k].x, f.x);
        f.y = fmaf(a[k].y, a[k].y, f.y);
        f.z = fmaf(a[k].z, a[k].z, f.z);
        f.w = fmaf(a[k].w, a[k].w, f.w);
    }
    put(0, f, at * at);
    double *np = part + (int64_t)cnt * G;  // behind the dot products' partials
    block_parts(0, 1, np);
    if (!meet(m, 2)) return;
    meet_done(m);
    if (wl == 0) {
        const double s = total(np);
        if (lane == 0) s_norm = s;
    }
    __syncthreads();
    const double hn = sqrt(s_norm);
    const float sf = (float)(hn > 0.0 ? 1.0 / hn : 0.0);
#pragma unroll
    for (int k = 0; k < E / 4; ++k) {
        const int64_t q = tid + k * st;
        if (q < nv)
            reinterpret_cast<float4 *>(w)[q] = make_float4(a[k].x * sf, a[k].y * sf, a[k].z * sf, a[k].w * sf);
    }
    if (tail) w[te] = at * sf;
    if (blockIdx.x == 0 && threadIdx.x == 0) givens_column(s_norm, h, j);
}

// y = R^-1 g over the first k columns (R the rotated Hessenberg matrix)
__global__ void k_backsolve(Hess h, int k) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    const int ld = h.m + 1;
    for (int i = k - 1; i >= 0; --i) {
        double t = h.g[i];
        for (int c = i + 1; c < k; ++c) t -= h.H[i + (int64_t)c * ld] * h.y[c];
        const double d = h.H[i + (int64_t)i * ld];
        h.y[i] = d != 0.0 ? t / d : 0.0;
    }
}

// out = (ACC ? out : 0) + sum_{j<k} y_j z_j (in double, rounded once)
template <typename TZ, typename TO, bool ACC>
__global__ void __launch_bounds__(FT) k_combine(int64_t n, const TZ *__restrict__ Z, int k,
                                                const double *__restrict__ y, TO *__restrict__ out) {
    __shared__ double ys[64];
    __shared__ float yf[64];
    for (int i = threadIdx.x; i < k; i += FT) {
        ys[i] = y[i];
        yf[i] = (float)y[i];
    }
    __syncthreads();
    if constexpr (std::is_same<TZ, float>::value && std::is_same<TO, float>::value) {
        for (int64_t e = blockIdx.x * (int64_t)FT + threadIdx.x; e < n; e += (int64_t)gridDim.x * FT) {
            float a = ACC ? out[e] : 0.f;
            for (int j = 0; j < k; ++j) a = fmaf(yf[j], Z[(int64_t)j * n + e], a);
            out[e] = a;
        }
    } else {
        for (int64_t e = blockIdx.x * (int64_t)FT + threadIdx.x; e < n; e += (int64_t)gridDim.x * FT) {
            double a = ACC ? (double)out[e] : 0.0;
            for (int j = 0; j < k; ++j) a += ys[j] * (double)Z[(int64_t)j * n + e];
            out[e] = (TO)a;
        }
    }
}

// Richardson: z = omega r (first step) or z = z + omega (r - t)
template <typename T>
__global__ void __launch_bounds__(FT) k_rich(int64_t n, T *__restrict__ z, const T *__restrict__ r,
                                             const T *__restrict__ t, float omega, int first) {
    for (int64_t e = blockIdx.x * (int64_t)FT + threadIdx.x; e < n; e += (int64_t)gridDim.x * FT)
        z[e] = first ? (T)(omega * r[e]) : (T)fma((T)omega, r[e] - t[e], z[e]);
}

// r = b - A x (x, r, b double) and the partials of r.r; the last block sets
// up layer 1 from r (begin_finish: beta = ||r||, v_0 scale)
__global__ void __launch_bounds__(FT) k_resid(int64_t n, const double *__restrict__ b,
                                              const double *__restrict__ ax, double *__restrict__ r,
                                              double *__restrict__ part, unsigned *counter, Hess h) {
    __shared__ double sh[FT];
    double s = 0.0;
    for (int64_t e = blockIdx.x * (int64_t)FT + threadIdx.x; e < n; e += (int64_t)gridDim.x * FT) {
        const double v = b[e] - ax[e];
        r[e] = v;
        s = fma(v, v, s);
    }
    s = block_sum(s, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
    if (last_block(counter)) begin_finish(gridDim.x, part, h, sh);
}

// one product of a layer: double vectors on the FP64 formats (SELL_F64,
// 64-bit words), float vectors on the others
packsell_status layer_spmv(const Matrix &A, const double *x, double *y, cudaStream_t s) {
    return spmv_f64_impl(A, x, y, s);
}
packsell_status layer_spmv(const Matrix &A, const float *x, float *y, cudaStream_t s) {
    return spmv_impl(A, x, y, s);
}

// device memory of the solve, in one allocation
struct Pool {
    char *base = nullptr, *cur = nullptr;
    size_t left = 0;
    template <typename T>
    T *take(size_t count) {
        size_t b = (count * sizeof(T) + 255) & ~(size_t)255;
        if (b > left) return nullptr;
        T *p = reinterpret_cast<T *>(cur);
        cur += b;
        left -= b;
        return p;
    }
};

template <typename T>
struct Layer {
    int m = 0;
    T *V = nullptr;  // (m + 1) basis vectors
    T *Z = nullptr;  // m preconditioned vectors
    Hess h{};
};

template <typename T>
bool make_layer(Pool &P, Layer<T> &L, int m, int64_t n) {
    L.m = m;
    L.V = P.take<T>((size_t)(m + 1) * n);
    L.Z = P.take<T>((size_t)m * n);
    L.h.m = m;
    L.h.H = P.take<double>((size_t)(m + 1) * m);
    L.h.cs = P.take<double>(m);
    L.h.sn = P.take<double>(m);
    L.h.g = P.take<double>(m + 1);
    L.h.y = P.take<double>(m);
    L.h.scal = P.take<double>(4);
    return L.V && L.Z && L.h.H && L.h.cs && L.h.sn && L.h.g && L.h.y && L.h.scal;
}

template <typename TI>
struct F3R {
    const Matrix *A1, *A2, *A3;
    int64_t n;
    int G;
    double *part;  // G * 64 partials
    unsigned *counter;  // blocks of the running reduction that have finished (0 between launches)
    Meet meet{};        // of k_arnoldi
    StepPlan step;      // of the FP32 layers
    Layer<double> L1;
    Layer<TI> L2, L3;
    TI *rt = nullptr;  // the product of a Richardson step (the iterate is layer 3's z_j)
    int m4;
    float omega;
    cudaStream_t s;

    // layer 4: z = Richardson(r), m4 steps from z = 0. A product whose kernel
    // takes the step as its epilogue reads one buffer and writes the other
    // (z and rt in turn, the last step into z); the first iterate omega r is
    // r itself when omega = 1.
    packsell_status richardson(const TI *r, TI *z) {
        if constexpr (std::is_same<TI, float>::value) {
            const TI *cur = r;
            int steps = m4 - 1;
            if (steps > 0) {
                if (omega != 1.f) {
                    TI *first = steps % 2 == 0 ? z : rt;
                    k_rich<TI><<<G, FT, 0, s>>>(n, first, r, (const TI *)nullptr, omega, 1);
                    cur = first;
                }
                bool done = true;
                for (; steps > 0 && done; --steps) {
                    TI *next = steps % 2 == 1 ? z : rt;
                    packsell_status st = spmv_rich(*A3, cur, r, omega, next, &done, s);
                    if (st != PACKSELL_OK) return st;
                    if (!done) break;  // (before the first step: another kernel serves this matrix)
                    cur = next;
                }
                if (done) {
                    PS_LAUNCH_CHECK("f3r: Richardson");
                    return PACKSELL_OK;
                }
            }
        }
        k_rich<TI><<<G, FT, 0, s>>>(n, z, r, (const TI *)nullptr, omega, 1);
        for (int k = 1; k < m4; ++k) {
            packsell_status st = layer_spmv(*A3, z, rt, s);
            if (st != PACKSELL_OK) return st;
            k_rich<TI><<<G, FT, 0, s>>>(n, z, r, rt, omega, 0);
        }
        PS_LAUNCH_CHECK("f3r: Richardson");
        return PACKSELL_OK;
    }

    // whether k_arnoldi runs, and on how many blocks; the trial launch finds
    // the timeout flag set and returns at once
    void plan_arnoldi() {
        auto per_sm = [](int e) {
            int per = 0;
            const cudaError_t r = e == 16 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_arnoldi<16>, FT, 0)
                                          : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_arnoldi<32>, FT, 0);
            if (r != cudaSuccess) cudaGetLastError();
            return r == cudaSuccess ? per : 0;
        };
        auto fits = [&](int e, int blocks) {
            step.blocks = blocks;
            cudaError_t r = cudaMemsetAsync(meet.timeout, 0xff, sizeof(int), s);
            if (r == cudaSuccess) {
                Layer<float> none;
                r = e == 16 ? launch_step<16>(none, nullptr, 0, 0) : launch_step<32>(none, nullptr, 0, 0);
            }
            if (r != cudaSuccess) cudaGetLastError();
            return r == cudaSuccess;
        };
        step = plan_step(n, device_sms(), FT, per_sm, fits);
    }

    template <int E>
    cudaError_t launch_step(Layer<float> &L, float *w, int cnt, int j) {
        return launch_coop(k_arnoldi<E>, (unsigned)step.blocks, FT, 0, s, n, (const float *)L.V, cnt, L.h,
                           j, w, part, meet);
    }

    // one Arnoldi step j of layer L on operator A: w = A z_j, orthogonalise
    // against v_0..v_j, normalise into v_{j+1}
    template <typename T>
    packsell_status arnoldi(Layer<T> &L, const Matrix &A, int j) {
        T *w = L.V + (int64_t)(j + 1) * n;
        packsell_status st = layer_spmv(A, L.Z + (int64_t)j * n, w, s);
        if (st != PACKSELL_OK) return st;
        const int cnt = j + 1;
        if constexpr (std::is_same<T, float>::value) {
            if (step.elems && ((uintptr_t)w & 15u) == 0) {
                const cudaError_t e = step.elems == 16 ? launch_step<16>(L, w, cnt, j) : launch_step<32>(L, w, cnt, j);
                if (e != cudaSuccess) return cuda_fail(e, "f3r: Arnoldi step");
                return PACKSELL_OK;
            }
        }
        k_mdot<T><<<dim3(G, cnt), FT, 0, s>>>(n, L.V, w, part, counter, L.h, j);
        k_orth<T><<<G, FT, 0, s>>>(n, L.V, cnt, L.h, j, w, part, counter);
        k_scale<T, T><<<G, FT, 0, s>>>(n, w, w, L.h.scal + 1);
        PS_LAUNCH_CHECK("f3r: Arnoldi step");
        return PACKSELL_OK;
    }

    // v_0 = rhs / ||rhs|| (converted to T), g = ||rhs|| e_1
    template <typename T, typename TR>
    void begin(Layer<T> &L, const TR *rhs) {
        k_norm2_begin<TR><<<G, FT, 0, s>>>(n, rhs, part, counter, L.h);
        k_scale<TR, T><<<G, FT, 0, s>>>(n, rhs, L.V, L.h.scal + 1);
    }

    // layer 3: m3 steps of FGMRES from zero on A3, preconditioned by layer 4
    packsell_status layer3(const TI *rhs, TI *out) {
        begin(L3, rhs);
        for (int j = 0; j < L3.m; ++j) {
            packsell_status st = richardson(L3.V + (int64_t)j * n, L3.Z + (int64_t)j * n);
            if (st == PACKSELL_OK) st = arnoldi(L3, *A3, j);
            if (st != PACKSELL_OK) return st;
        }
        k_backsolve<<<1, 32, 0, s>>>(L3.h, L3.m);
        k_combine<TI, TI, false><<<G, FT, 0, s>>>(n, L3.Z, L3.m, L3.h.y, out);
        PS_LAUNCH_CHECK("f3r: layer 3");
        return PACKSELL_OK;
    }

    // layer 2: m2 steps of FGMRES from zero on A2, preconditioned by layer 3
    packsell_status layer2(const double *rhs, double *out) {
        begin(L2, rhs);
        for (int j = 0; j < L2.m; ++j) {
            packsell_status st = layer3(L2.V + (int64_t)j * n, L2.Z + (int64_t)j * n);
            if (st == PACKSELL_OK) st = arnoldi(L2, *A2, j);
            if (st != PACKSELL_OK) return st;
        }
        k_backsolve<<<1, 32, 0, s>>>(L2.h, L2.m);
        k_combine<TI, double, false><<<G, FT, 0, s>>>(n, L2.Z, L2.m, L2.h.y, out);
        PS_LAUNCH_CHECK("f3r: layer 2");
        return PACKSELL_OK;
    }
};

template <typename TI>
packsell_status run_f3r(const Matrix &A1, const Matrix &A2, const Matrix &A3, const double *b,
                        double *x, const packsell_f3r_opts &o, packsell_solve_result *res,
                        cudaStream_t caller) {
    const int64_t n = A1.n;
    cudaStream_t s = nullptr;
    PS_CUDA(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    void *mem = nullptr;
    packsell_status st = PACKSELL_OK;
    int iters = 0, steps = 0;
    double relres = 1.0, relres_true = -1.0;
    bool converged = false;
    const int G = fgrid(n);
    F3R<TI> F{};
    Pool P;
    {
        cudaEventCreateWithFlags(&ev0, cudaEventDisableTiming);
        cudaEventRecord(ev0, caller);
        cudaStreamWaitEvent(s, ev0, 0);  // the caller's pending work first
        cudaEventDestroy(ev0);
        ev0 = nullptr;
        cudaEventCreate(&ev0);
        cudaEventCreate(&ev1);
    }
    const size_t need =
        sizeof(double) * ((size_t)(2 * o.m1 + 1) * n + 5 * (size_t)n + 64 * (size_t)G +
                          (size_t)(o.m1 + 1) * o.m1 + 8 * (size_t)o.m1 + 16) +
        sizeof(TI) * ((size_t)(2 * o.m2 + 1) * n + (size_t)(2 * o.m3 + 1) * n + 2 * (size_t)n) +
        sizeof(double) * ((size_t)(o.m2 + 1) * o.m2 + (size_t)(o.m3 + 1) * o.m3 + 8 * (size_t)(o.m2 + o.m3) + 32) +
        256 * 40;
    double *r = nullptr, *ax = nullptr, *zt = nullptr, *prhs = nullptr, *pout = nullptr;
    double nb = 0.0;
    if (pool_get(&mem, need, s) != cudaSuccess) {
        st = fail(PACKSELL_ERR_NO_MEMORY, "packsell_f3r: workspace allocation");
        goto out;
    }
    P.base = P.cur = (char *)mem;
    P.left = need;
    F.A1 = &A1;
    F.A2 = &A2;
    F.A3 = &A3;
    F.n = n;
    F.G = G;
    F.m4 = o.m4;
    F.omega = (float)o.omega;
    F.s = s;
    F.part = P.take<double>(64 * (size_t)G);
    F.counter = P.take<unsigned>(4);  // the reductions' counter; k_arnoldi's two and its flag
    F.meet = Meet{F.counter + 1, F.counter + 2, (int *)(F.counter + 3)};
    r = P.take<double>(n);
    ax = P.take<double>(n);
    zt = P.take<double>(n);
    prhs = P.take<double>(n);
    pout = P.take<double>(n);
    F.rt = P.take<TI>(n);
    if (!F.part || !F.counter || !r || !ax || !zt || !prhs || !pout || !F.rt || !make_layer(P, F.L1, o.m1, n) ||
        !make_layer(P, F.L2, o.m2, n) || !make_layer(P, F.L3, o.m3, n)) {
        st = fail(PACKSELL_ERR_NO_MEMORY, "packsell_f3r: workspace carving");
        goto out;
    }
    if (std::is_same<TI, float>::value) F.plan_arnoldi();
    {
        auto ck = [&](cudaError_t e) {
            if (e != cudaSuccess) st = cuda_fail(e, "packsell_f3r");
            return e == cudaSuccess;
        };
        auto true_residual = [&](double *rr) -> packsell_status {
            packsell_status e = spmv_f64_impl(A1, x, ax, s);
            if (e != PACKSELL_OK) return e;
            k_resid<<<G, FT, 0, s>>>(n, b, ax, r, F.part, F.counter, F.L1.h);  // beta = ||r||, v_0 scale
            PS_LAUNCH_CHECK("f3r: residual");
            double sc[3];
            if (!ck(cudaMemcpyAsync(sc, F.L1.h.scal, sizeof(sc), cudaMemcpyDeviceToHost, s)) ||
                !ck(cudaStreamSynchronize(s)))
                return st;
            *rr = sc[0];
            return PACKSELL_OK;
        };
        // ||b||
        if (!ck(cudaMemsetAsync(F.counter, 0, 4 * sizeof(unsigned), s))) goto out;
        k_norm2_begin<double><<<G, FT, 0, s>>>(n, b, F.part, F.counter, F.L1.h);
        double sc[3];
        if (!ck(cudaMemcpyAsync(sc, F.L1.h.scal, sizeof(sc), cudaMemcpyDeviceToHost, s)) ||
            !ck(cudaStreamSynchronize(s)))
            goto out;
        nb = sc[0];
        // layers 2-4 (the preconditioner of an outer step) as one CUDA graph:
        // a fixed sequence of some hundreds of kernels with no host step,
        // replayed on the fixed buffers prhs -> pout
        if (cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
            st = fail(PACKSELL_ERR_CUDA, "packsell_f3r: stream capture failed to start");
            goto out;
        }
        {
            const packsell_status cst = F.layer2(prhs, pout);
            const cudaError_t ce = cudaStreamEndCapture(s, &graph);
            if (cst != PACKSELL_OK) {
                st = cst;
                goto out;
            }
            if (ce != cudaSuccess || cudaGraphInstantiate(&exec, graph, 0) != cudaSuccess) {
                st = fail(PACKSELL_ERR_CUDA, "packsell_f3r: graph capture failed");
                goto out;
            }
        }
        if (nb == 0.0) {
            if (!ck(cudaMemsetAsync(x, 0, sizeof(double) * n, s))) goto out;
            relres = relres_true = 0.0;
            converged = true;
            goto done;
        }
        cudaEventRecord(ev0, s);
        while (iters < o.max_iters && !converged) {
            // restart cycle: r = b - A x, v_0 = r / ||r||
            double rn = 0.0;
            st = true_residual(&rn);
            if (st != PACKSELL_OK) goto out;
            relres = rn / nb;
            if (relres < o.rtol) {
                relres_true = relres;
                converged = true;
                break;
            }
            k_scale<double, double><<<G, FT, 0, s>>>(n, r, F.L1.V, F.L1.h.scal + 1);
            int k = 0;
            for (; k < o.m1 && iters < o.max_iters; ++k) {
                if (!ck(cudaMemcpyAsync(prhs, F.L1.V + (int64_t)k * n, sizeof(double) * n,
                                        cudaMemcpyDeviceToDevice, s)) ||
                    !ck(cudaGraphLaunch(exec, s)) ||
                    !ck(cudaMemcpyAsync(F.L1.Z + (int64_t)k * n, pout, sizeof(double) * n,
                                        cudaMemcpyDeviceToDevice, s)))
                    goto out;
                st = F.arnoldi(F.L1, A1, k);
                if (st != PACKSELL_OK) goto out;
                ++iters;
                int timeout = 0;
                if (!ck(cudaMemcpyAsync(sc, F.L1.h.scal, sizeof(sc), cudaMemcpyDeviceToHost, s)) ||
                    !ck(cudaMemcpyAsync(&timeout, F.meet.timeout, sizeof(int), cudaMemcpyDeviceToHost, s)) ||
                    !ck(cudaStreamSynchronize(s)))
                    goto out;
                if (timeout) {
                    st = fail(PACKSELL_ERR_TIMEOUT, "packsell_f3r: a grid-wide wait ran out");
                    goto out;
                }
                relres = sc[2] / nb;
                if (!std::isfinite(relres)) {
                    st = fail(PACKSELL_ERR_BREAKDOWN, "packsell_f3r: non-finite residual");
                    goto out;
                }
                if (relres < o.rtol) {
                    ++k;
                    break;
                }
            }
            // x += sum_j y_j z_j over the cycle's k steps
            k_backsolve<<<1, 32, 0, s>>>(F.L1.h, k);
            k_combine<double, double, true><<<G, FT, 0, s>>>(n, F.L1.Z, k, F.L1.h.y, x);
            PS_LAUNCH_CHECK("f3r: update");
            ++steps;
            if (relres < o.rtol) {
                double rt = 0.0;
                st = true_residual(&rt);
                if (st != PACKSELL_OK) goto out;
                relres_true = rt / nb;
                if (relres_true < o.rtol) converged = true;
                // otherwise the next cycle restarts from the true residual
            }
        }
        cudaEventRecord(ev1, s);
        if (!ck(cudaStreamSynchronize(s))) goto out;
        if (relres_true < 0.0) {
            double rt = 0.0;
            st = true_residual(&rt);
            if (st != PACKSELL_OK) goto out;
            relres_true = rt / nb;
        }
    }
done:
    if (res) {
        float ms = 0.f;
        if (ev0 && ev1 && cudaEventElapsedTime(&ms, ev0, ev1) != cudaSuccess) ms = 0.f;
        res->iters = iters;
        res->inner_iters = iters * o.m2 * o.m3;
        res->relres = relres;
        res->relres_true = relres_true;
        res->seconds = ms * 1e-3;
    }
    if (!converged)
        st = fail(PACKSELL_ERR_NOT_CONVERGED,
                  "packsell_f3r: no convergence in " + std::to_string(o.max_iters) + " outer iterations");
out:
    if (exec) cudaGraphExecDestroy(exec);
    if (graph) cudaGraphDestroy(graph);
    if (mem) pool_put(mem, s);
    cudaStreamSynchronize(s);
    if (ev0) cudaEventDestroy(ev0);
    if (ev1) cudaEventDestroy(ev1);
    cudaStreamDestroy(s);
    (void)steps;
    (void)zt;
    return st;
}

}  // namespace

packsell_status f3r_impl(const Matrix *A1, const Matrix *A2, const Matrix *A3, const double *b,
                         double *x, const packsell_f3r_opts &o, packsell_solve_result *res,
                         cudaStream_t s) {
    if (!A1 || !A2 || !A3) return fail(PACKSELL_ERR_INVALID_ARG, "packsell_f3r: NULL matrix");
    const int64_t n = A1->n;
    auto square = [&](const Matrix *A) { return A->n == n && A->m == n && !A->p.explicit_perm; };
    if (!is_f64_op(A1->p.format) || !square(A1) || !square(A2) || !square(A3))
        return fail(PACKSELL_ERR_INVALID_ARG,
                    "packsell_f3r: A_outer must be SELL_F64 or W64_E11MY; all three square, of "
                    "one size, rows in original order");
    const bool all64 = is_f64_op(A2->p.format) && is_f64_op(A3->p.format);
    const bool mixed = A2->p.format == PACKSELL_FMT_SELL_F32 &&
                       (A3->p.format == PACKSELL_FMT_FP16 || A3->p.format == PACKSELL_FMT_SELL_F16 ||
                        A3->p.format == PACKSELL_FMT_E8MY);
    if (!all64 && !mixed)
        return fail(PACKSELL_ERR_INVALID_ARG,
                    "packsell_f3r: layers 2-4 need FP64 matrices (FP64-F3R) or SELL_F32 and a "
                    "PackSELL / FP16 SELL matrix (FP16-F3R)");
    if (o.m1 < 1 || o.m1 > 60 || o.m2 < 1 || o.m2 > 60 || o.m3 < 1 || o.m3 > 60 || o.m4 < 1 ||
        o.max_iters < 1 || !(o.rtol > 0.0) || !(o.omega > 0.0))
        return fail(PACKSELL_ERR_INVALID_ARG, "packsell_f3r: bad options");
    if (n == 0) {
        if (res) *res = packsell_solve_result{};
        return PACKSELL_OK;
    }
    if (!b || !x) return fail(PACKSELL_ERR_INVALID_ARG, "packsell_f3r: NULL vector");
    return all64 ? run_f3r<double>(*A1, *A2, *A3, b, x, o, res, s)
                 : run_f3r<float>(*A1, *A2, *A3, b, x, o, res, s);
}

}  // namespace packsell
