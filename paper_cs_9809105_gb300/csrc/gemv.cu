// gemv.cu -- matrix-vector products y <- alpha*op(A)*x + beta*y (column-major A).
//
// The paper names the matrix-vector form as a capability of the same alignment
// (Sections 1 and 8) without printing an algorithm; these kernels compute the
// BLAS definition and are bound by HBM bandwidth (one pass over A).
//
//  op = N: y_i = sum_j A(i,j) x_j.  Rows are contiguous, so each thread owns a
//          few consecutive rows and streams down the columns with 128-bit loads.
//          The columns are split over CTAs to put enough bytes in flight; every
//          split writes its partial sums to the workspace and a second kernel,
//          launched as a programmatic dependent (it starts while the splits finish),
//          adds the splits in a fixed order (deterministic results).
//  op = T: y_j = sum_i A(i,j) x_i.  Column j is contiguous: one warp per column, up to eight where
//          there are few columns, 128-bit loads, a fixed shuffle tree for the reduction.
//  INT8:   exact INT32 accumulation with dp4a; for op = N the 16-row x 4-column
//          byte tiles are transposed in registers (byte permutes) so that dp4a
//          multiplies four columns of one row by four packed entries of x.
//
// The 128-bit paths need aligned columns (A and lda), not whole vectors of rows: op = T ends a
// column element by element, and op = N reads whole vectors into the padding rows of every column
// but the last, whose tail it reads element by element (nothing after A(m-1, n-1) is read).
// Before -> now, us in a row in a CUDA graph (N / T): INT8 2100 x 5300 with padded columns 9.2 / 7.8
// -> 5.9 / 3.2, FP32 2101 x 5300 unaligned 16.9 / 29.8 -> 11.9 / 10.5, 16384 x 500 13.6 / 29.7 ->
// 10.0 / 7.4, 1000^2 6.8 / 3.1 -> 3.6 / 2.0, 6654 x 8018 45.5 / 80.2 -> 34.4 / 39.2, 16384^2 150.3 /
// 166.7 -> 150.1 / 156.9.
#include <cstdint>
#include <cuda_runtime.h>

#include "common.cuh"
#include "internal.h"

namespace hsmm {

static __device__ uint32_t g_status_gemv;

uint32_t status_take_gemv() {
    uint32_t v = 0, z = 0;
    cudaMemcpyFromSymbol(&v, g_status_gemv, sizeof(v));
    cudaMemcpyToSymbol(g_status_gemv, &z, sizeof(z));
    return v;
}

namespace {

constexpr int kThreads = 256;

// Every kernel of this file is launched as a programmatic dependent: its CTAs are placed while the
// kernel before it drains, wait on the device for its end (pdl_wait, the first instruction, before
// any access to memory) and only then let the next one be placed.  The only exception is the PLAIN
// form of op = N, where a wait costs more than the gap it hides (16384 x 16384 FP32: 155.8 us with
// it, 150.0 without).  Between others the gap is 0.3 to 2.4 us: FP32 1000 x 1000 N 3.96 -> 3.58 us and
// T 2.40 -> 2.02, INT8 2100 x 5300 N then T 14.35 -> 9.58.
// They are resident while that kernel still writes what they read, so nothing is loaded as read-only
// data: no __ldg, no const __restrict__ (which the compiler turns into the same non-coherent loads and
// may move above the wait), but load() (INT8 14580 x 24 T 3.1 us, 4.4 with plain dereferences).
template <typename K, typename... Q>
cudaError_t launch(K kern, dim3 grid, cudaStream_t st, const Q&... args) {
    return pdl_launch(kern, grid, kThreads, 0, 1, st, args...);
}

// ---------------------------------------------------------------------------
// FP32, op = N
// ---------------------------------------------------------------------------
// Vector path: 4 rows per thread (float4), grid (row blocks, column splits).  2^rt threads of a CTA
// take rows; where that is fewer than all (small m), the CTA's column split is cut again into
// groups of cols_per_group columns, one per 2^rt threads, added in order through shared memory:
// a thread then has fewer columns to walk one latency after the other.  PLAIN: no groups and m % 4
// == 0 (34 registers instead of 60: 22.0 against 22.9 us at 8192 x 4096).
template <bool PLAIN>
__global__ void __launch_bounds__(kThreads) gemv_f32_n_vec(int64_t m, int64_t n, const float* A,
                                                           int64_t lda, const float* x, int64_t incx,
                                                           float* part, int64_t cols_per_split,
                                                           int rt, int64_t cols_per_group) {
    if (!PLAIN) pdl_wait();   // see launch
    pdl_trigger();   // the reduction may be scheduled; it waits for this grid to finish
    if (PLAIN) rt = 8;
    const int tr = int(threadIdx.x) & ((1 << rt) - 1), group = PLAIN ? 0 : int(threadIdx.x) >> rt;
    const int64_t r0 = ((int64_t(blockIdx.x) << rt) + tr) * 4;
    const int64_t js = int64_t(blockIdx.y) * cols_per_split, j0 = PLAIN ? js : js + group * cols_per_group;
    int64_t j1 = min(n, js + cols_per_split);
    if (PLAIN) {
        if (r0 >= m) return;
    } else {
        j1 = r0 < m ? min(j1, j0 + cols_per_group) : 0;      // no rows: no columns
    }
    // columns read as whole vectors (a split may be empty)
    const int64_t jv = (!PLAIN && r0 + 4 > m && j1 == n && j0 < j1) ? j1 - 1 : j1;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    const float* a = A + r0;
    int64_t j = j0;
    // 8 columns in flight per thread
    for (; j + 8 <= jv; j += 8) {
        float4 v[8];
        float xs[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = __ldcs(reinterpret_cast<const float4*>(a + (j + u) * lda));
#pragma unroll
        for (int u = 0; u < 8; ++u) xs[u] = load(x + (j + u) * incx);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            acc.x = fmaf(v[u].x, xs[u], acc.x);
            acc.y = fmaf(v[u].y, xs[u], acc.y);
            acc.z = fmaf(v[u].z, xs[u], acc.z);
            acc.w = fmaf(v[u].w, xs[u], acc.w);
        }
    }
    for (; j < jv; ++j) {
        float4 v = __ldcs(reinterpret_cast<const float4*>(a + j * lda));
        float xv = load(x + j * incx);
        acc.x = fmaf(v.x, xv, acc.x);
        acc.y = fmaf(v.y, xv, acc.y);
        acc.z = fmaf(v.z, xv, acc.z);
        acc.w = fmaf(v.w, xv, acc.w);
    }
    if (!PLAIN && jv < j1) {      // the last column of a matrix whose rows end inside this vector
        const float xv = load(x + jv * incx);
        const float* c = a + jv * lda;
        acc.x = fmaf(load(c), xv, acc.x);
        if (r0 + 1 < m) acc.y = fmaf(load(c + 1), xv, acc.y);
        if (r0 + 2 < m) acc.z = fmaf(load(c + 2), xv, acc.z);
    }
    if constexpr (!PLAIN) {
        __shared__ float4 red[kThreads];
        red[threadIdx.x] = acc;
        __syncthreads();
        if (group != 0) return;
        for (int g = 1; g < kThreads >> rt; ++g) {
            const float4 v = red[(g << rt) + tr];
            acc.x += v.x;
            acc.y += v.y;
            acc.z += v.z;
            acc.w += v.w;
        }
    }
    if (!PLAIN && r0 >= m) return;
    float* p = part + int64_t(blockIdx.y) * m + r0;
    if (PLAIN || m % 4 == 0) {
        *reinterpret_cast<float4*>(p) = acc;
    } else {
        p[0] = acc.x;
        if (r0 + 1 < m) p[1] = acc.y;
        if (r0 + 2 < m) p[2] = acc.z;
        if (r0 + 3 < m) p[3] = acc.w;
    }
}

// Scalar path (unaligned columns): 1 row per thread.
__global__ void __launch_bounds__(kThreads) gemv_f32_n_scalar(int64_t m, int64_t n, const float* A,
                                                              int64_t lda, const float* x,
                                                              int64_t incx, float* part,
                                                              int64_t cols_per_split) {
    pdl_wait();
    pdl_trigger();   // the reduction may be scheduled; it waits for this grid to finish
    const int64_t r = int64_t(blockIdx.x) * kThreads + threadIdx.x;
    const int64_t j0 = int64_t(blockIdx.y) * cols_per_split;
    const int64_t j1 = min(n, j0 + cols_per_split);
    if (r >= m) return;
    float acc = 0.f;
    int64_t j = j0;
    for (; j + 8 <= j1; j += 8) {      // eight columns in flight
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = __ldcs(A + r + (j + u) * lda);
#pragma unroll
        for (int u = 0; u < 8; ++u) acc = fmaf(v[u], load(x + (j + u) * incx), acc);
    }
    for (; j < j1; ++j) acc = fmaf(A[r + j * lda], load(x + j * incx), acc);
    part[int64_t(blockIdx.y) * m + r] = acc;
}

// y_i = alpha * sum_s part[s][i] + beta*y_i.  A CTA takes 32 rows; its 8 warps add the
// splits s = g, g + 8, ... (warp g) and the 8 sums are added in the order g = 0..7: a fixed
// order, so the result is deterministic.  Launched as a programmatic dependent of the split
// kernel: the CTAs start while the splits finish and wait for them on the device.
template <typename T, typename Acc>
__global__ void __launch_bounds__(kThreads) gemv_reduce(int64_t m, int nsplit, const T* part, T alpha,
                                                        T beta, T* y, int64_t incy) {
    pdl_wait();
    pdl_trigger();
    const int r = int(lane_id()), g = int(warp_id());
    const int64_t i = int64_t(blockIdx.x) * 32 + r;
    Acc sum = Acc(0);
    if (i < m)
#pragma unroll 4
        for (int q = g; q < nsplit; q += kThreads / 32) sum += Acc(part[int64_t(q) * m + i]);
    __shared__ Acc red[kThreads / 32][32];
    red[g][r] = sum;
    __syncthreads();
    if (g != 0 || i >= m) return;
    Acc t = red[0][r];
#pragma unroll
    for (int k = 1; k < kThreads / 32; ++k) t += red[k][r];
    if constexpr (sizeof(Acc) == 4 && Acc(-1) > Acc(0)) {
        // INT32 BLAS arithmetic: two's-complement wrap-around
        uint32_t v = uint32_t(alpha) * t;
        if (beta != 0) v += uint32_t(beta) * uint32_t(y[i * incy]);
        y[i * incy] = T(v);
    } else {
        T v = alpha * t;
        if (beta != T(0)) v = fmaf(beta, y[i * incy], v);
        y[i * incy] = v;
    }
}

template <typename T, typename Acc>
cudaError_t launch_reduce(int64_t m, int nsplit, const T* part, T alpha, T beta, T* y, int64_t incy,
                          cudaStream_t st) {
    return launch(gemv_reduce<T, Acc>, dim3(unsigned((m + 31) / 32)), st, m, nsplit, part, alpha, beta, y, incy);
}

// ---------------------------------------------------------------------------
// op = T
// ---------------------------------------------------------------------------
// A CTA of eight warps takes 8, 4, 2 or 1 columns, 1 to 8 warps per column, each a contiguous part
// of the rows; the warps' sums are added in order.  16 bytes a lane and load, four loads of A in
// flight per lane.  (Two columns per warp, x loaded once for both, ran at 5.4 against 6.4 TB/s at
// 16384^2.)
struct GemvT {
    int64_t m, n, lda, incx, incy;
    int64_t rows;                  // rows of a warp, a multiple of 32 vectors
    int shift;                     // 2^shift warps per column
};
__device__ __forceinline__ void t_store(const GemvT& g, float alpha, float beta, float* y, int64_t col, float acc) {
    float v = alpha * acc;
    if (beta != 0.f) v = fmaf(beta, y[col * g.incy], v);
    y[col * g.incy] = v;
}
__device__ __forceinline__ void t_store(const GemvT& g, int32_t alpha, int32_t beta, int32_t* y, int64_t col, int acc) {
    uint32_t v = uint32_t(alpha) * uint32_t(acc);          // INT32 BLAS arithmetic: wrap-around
    if (beta != 0) v += uint32_t(beta) * uint32_t(y[col * g.incy]);
    y[col * g.incy] = int32_t(v);
}
__device__ __forceinline__ void t_fma(const float4& a, const float4& x, float& acc) {
    acc = fmaf(a.x, x.x, acc); acc = fmaf(a.y, x.y, acc); acc = fmaf(a.z, x.z, acc); acc = fmaf(a.w, x.w, acc);
}
__device__ __forceinline__ void t_fma(const int4& a, const int4& x, int& acc) {
    acc = __dp4a(a.x, x.x, acc); acc = __dp4a(a.y, x.y, acc); acc = __dp4a(a.z, x.z, acc); acc = __dp4a(a.w, x.w, acc);
}

// 16-byte streaming loads that stay together in program order: all of a round are in flight before
// the first is used
__device__ __forceinline__ float4 load_stream(const float4* p) {
    float4 v;
    asm volatile("ld.global.cs.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}

// this warp's column, part of it and rows
__device__ __forceinline__ void t_place(const GemvT& g, int64_t& col, int& part, int64_t& i0, int64_t& i1) {
    const int warp = int(warp_id());
    col = int64_t(blockIdx.x) * (kThreads / 32 >> g.shift) + (warp >> g.shift);
    part = warp & ((1 << g.shift) - 1);
    i0 = min(g.m, part * g.rows);
    i1 = min(g.m, i0 + g.rows);
}
// sums of the lanes, then of the warps of a column, in order; the first warp stores y
template <typename S>
__device__ __forceinline__ void t_finish(const GemvT& g, S acc, int64_t col, int part, S alpha, S beta, S* y) {
    const int warp = int(warp_id()), lane = int(lane_id());
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if (g.shift > 0) {
        __shared__ S red[kThreads / 32];
        if (lane == 0) red[warp] = acc;
        __syncthreads();
        if (part != 0) return;
        for (int i = 1; i < 1 << g.shift; ++i) acc += red[warp + i];
    }
    if (lane == 0 && col < g.n) t_store(g, alpha, beta, y, col, acc);
}

// FP32, aligned columns of a whole number of vectors and aligned x, incx == 1, one warp per column:
// all loads of a round are in flight before the first is used (166 -> 157.5 us at 16384^2, 6.8
// TB/s).  The same loop was slower for INT8 (44.3 us at 16384^2 against 40.5 for the general one).
__global__ void __launch_bounds__(kThreads) gemv_f32_t_plain(GemvT g, const float* A,
                                                             const float* x, float alpha, float beta,
                                                             float* y) {
    pdl_wait();
    pdl_trigger();
    const int lane = int(lane_id());
    const int64_t col = int64_t(blockIdx.x) * (kThreads / 32) + warp_id();
    if (col >= g.n) return;
    const int64_t mv = g.m / 4;
    const float4* a = reinterpret_cast<const float4*>(A + col * g.lda);
    const float4* xp = reinterpret_cast<const float4*>(x);
    float acc = 0.f;
    int64_t i = lane;
    for (; i + 96 < mv; i += 128) {
        float4 v[4], w[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = load_stream(a + i + 32 * u);
#pragma unroll
        for (int u = 0; u < 4; ++u) w[u] = load(xp + i + 32 * u);
#pragma unroll
        for (int u = 0; u < 4; ++u) t_fma(v[u], w[u], acc);
    }
    for (; i < mv; i += 32) t_fma(__ldcs(a + i), load(xp + i), acc);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if (lane == 0) t_store(g, alpha, beta, y, col, acc);
}

// The general form: m any, 2^g.shift warps per column.  T: element (float, int8_t), V: 16-byte
// vector of it, S: sum.  Held to five CTAs an SM (INT8 at 16384^2 43.2 -> 40.5 us).
template <typename T, typename V, typename S>
__global__ void __launch_bounds__(kThreads, 5) gemv_t_vec(GemvT g, const T* A, const T* x,
                                                          S alpha, S beta, S* y) {
    constexpr int E = 16 / int(sizeof(T));                 // elements of a vector
    const int lane = int(lane_id());
    pdl_wait();
    pdl_trigger();
    int64_t col, i0, i1;
    int part;
    t_place(g, col, part, i0, i1);
    S acc = S(0);
    if (col < g.n) {
        const T* a = A + col * g.lda;
        const int64_t iv = i0 + (i1 - i0) / E * E;     // rows in whole vectors
        int64_t i = i0;
        for (; i + 128 * E <= iv; i += 128 * E) {
            V v[4], w[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = __ldcs(reinterpret_cast<const V*>(a + i + (32 * u + lane) * E));
#pragma unroll
            for (int u = 0; u < 4; ++u) w[u] = load(reinterpret_cast<const V*>(x + i + (32 * u + lane) * E));
#pragma unroll
            for (int u = 0; u < 4; ++u) t_fma(v[u], w[u], acc);
        }
        if (i < iv) {                                  // what is left of a round
            V v[4], w[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int64_t r = i + (32 * u + lane) * E;
                const bool in = r < iv;
                v[u] = in ? __ldcs(reinterpret_cast<const V*>(a + r)) : V{};
                w[u] = in ? load(reinterpret_cast<const V*>(x + r)) : V{};
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (i + (32 * u + lane) * E < iv) t_fma(v[u], w[u], acc);
        }
        i = iv + lane;                                 // the last m % E rows
        if (i < i1) acc += S(load(a + i)) * S(load(x + i));
    }
    t_finish(g, acc, col, part, alpha, beta, y);
}

// Unaligned columns: one element per lane and load.  UNIT: incx == 1.
template <typename T, typename S, bool UNIT>
__global__ void __launch_bounds__(kThreads) gemv_t_scalar(GemvT g, const T* A, const T* x,
                                                          S alpha, S beta, S* y) {
    const int lane = int(lane_id());
    pdl_wait();
    pdl_trigger();
    int64_t col, i0, i1;
    int part;
    t_place(g, col, part, i0, i1);
    const int64_t incx = UNIT ? 1 : g.incx;
    S acc = S(0);
    if (col < g.n) {
        const T* a = A + col * g.lda + i0 + lane;
        const T* xp = x + (i0 + lane) * incx;
        int64_t left = (i1 - i0 - lane + 31) >> 5;         // elements of this lane
        for (; left >= 8; left -= 8, a += 256, xp += 256 * incx) {
            T v[8], w[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = load(a + 32 * u);
#pragma unroll
            for (int u = 0; u < 8; ++u) w[u] = load(xp + 32 * u * incx);
#pragma unroll
            for (int u = 0; u < 8; ++u) acc += S(v[u]) * S(w[u]);
        }
        for (; left > 0; --left, a += 32, xp += 32 * incx) acc += S(load(a)) * S(load(xp));
    }
    t_finish(g, acc, col, part, alpha, beta, y);
}

// One warp per column where that is 16 warps an SM and more, else up to eight for about as many.
template <typename T, typename V, typename S>
cudaError_t launch_t(int64_t m, int64_t n, S alpha, const T* A, int64_t lda, const T* x, int64_t incx, S beta, S* y,
              int64_t incy, bool vec, cudaStream_t st) {
    const int64_t want = int64_t(num_sms()) * 16, unit = 32 * (16 / int64_t(sizeof(T)));   // one vector per lane
    GemvT g{m, n, lda, incx, incy, 0, 0};
    while ((1 << g.shift) < kThreads / 32 && (n << g.shift) < want && m > (4 * unit << g.shift)) ++g.shift;
    const int64_t parts = int64_t(1) << g.shift;
    g.rows = ((m + unit - 1) / unit + parts - 1) / parts * unit;
    const int cols = kThreads / 32 >> g.shift;
    const unsigned grid = unsigned((n + cols - 1) / cols);
    if constexpr (sizeof(T) == 4) {
        if (vec && g.shift == 0 && m % 4 == 0)
            return launch(gemv_f32_t_plain, dim3(grid), st, g, A, x, alpha, beta, y);
    }
    if (vec) return launch(gemv_t_vec<T, V, S>, dim3(grid), st, g, A, x, alpha, beta, y);
    if (incx == 1) return launch(gemv_t_scalar<T, S, true>, dim3(grid), st, g, A, x, alpha, beta, y);
    return launch(gemv_t_scalar<T, S, false>, dim3(grid), st, g, A, x, alpha, beta, y);
}

// ---------------------------------------------------------------------------
// INT8, op = N: 16 rows per thread, 4 columns per dp4a group
// ---------------------------------------------------------------------------
__device__ __forceinline__ void transpose4x4_bytes(uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3, uint32_t& t0,
                                                   uint32_t& t1, uint32_t& t2, uint32_t& t3) {
    // w_c holds rows r..r+3 of column c; t_r holds columns c0..c3 of row r
    const uint32_t u0 = __byte_perm(w0, w1, 0x5140);
    const uint32_t u1 = __byte_perm(w0, w1, 0x7362);
    const uint32_t u2 = __byte_perm(w2, w3, 0x5140);
    const uint32_t u3 = __byte_perm(w2, w3, 0x7362);
    t0 = __byte_perm(u0, u2, 0x5410);
    t1 = __byte_perm(u0, u2, 0x7632);
    t2 = __byte_perm(u1, u3, 0x5410);
    t3 = __byte_perm(u1, u3, 0x7632);
}

__device__ __forceinline__ uint32_t pack_x4(const int8_t* x, int64_t j, int64_t incx) {
    const uint32_t b0 = uint8_t(load(x + (j + 0) * incx));
    const uint32_t b1 = uint8_t(load(x + (j + 1) * incx));
    const uint32_t b2 = uint8_t(load(x + (j + 2) * incx));
    const uint32_t b3 = uint8_t(load(x + (j + 3) * incx));
    return b0 | (b1 << 8) | (b2 << 16) | (b3 << 24);
}

template <bool PLAIN>
__global__ void __launch_bounds__(kThreads) gemv_i8_n_vec(int64_t m, int64_t n, const int8_t* A,
                                                          int64_t lda, const int8_t* x, int64_t incx,
                                                          int32_t* part, int64_t cols_per_split,
                                                          int rt, int64_t cols_per_group) {
    if (!PLAIN) pdl_wait();   // see launch
    pdl_trigger();   // the reduction may be scheduled; it waits for this grid to finish
    if (PLAIN) rt = 8;                                       // see gemv_f32_n_vec; m % 16 == 0
    const int tr = int(threadIdx.x) & ((1 << rt) - 1), group = PLAIN ? 0 : int(threadIdx.x) >> rt;
    const int64_t r0 = ((int64_t(blockIdx.x) << rt) + tr) * 16;
    const int64_t js = int64_t(blockIdx.y) * cols_per_split, j0 = PLAIN ? js : js + group * cols_per_group;
    int64_t j1 = min(n, js + cols_per_split);
    if (PLAIN) {
        if (r0 >= m) return;
    } else {
        j1 = r0 < m ? min(j1, j0 + cols_per_group) : 0;      // no rows: no columns
    }
    // columns read as whole vectors (a split may be empty)
    const int64_t jv = (!PLAIN && r0 + 16 > m && j1 == n && j0 < j1) ? j1 - 1 : j1;
    int acc[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) acc[r] = 0;
    const int8_t* a = A + r0;
    int64_t j = j0;
    // two groups of four columns (eight 16-byte loads) in flight per thread
    for (; j + 8 <= jv; j += 8) {
        uint4 c[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) c[u] = __ldcs(reinterpret_cast<const uint4*>(a + (j + u) * lda));
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int xp = int(pack_x4(x, j + 4 * h, incx));
            const uint4* cc = c + 4 * h;
            uint32_t t[4];
            transpose4x4_bytes(cc[0].x, cc[1].x, cc[2].x, cc[3].x, t[0], t[1], t[2], t[3]);
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[r] = __dp4a(int(t[r]), xp, acc[r]);
            transpose4x4_bytes(cc[0].y, cc[1].y, cc[2].y, cc[3].y, t[0], t[1], t[2], t[3]);
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[4 + r] = __dp4a(int(t[r]), xp, acc[4 + r]);
            transpose4x4_bytes(cc[0].z, cc[1].z, cc[2].z, cc[3].z, t[0], t[1], t[2], t[3]);
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[8 + r] = __dp4a(int(t[r]), xp, acc[8 + r]);
            transpose4x4_bytes(cc[0].w, cc[1].w, cc[2].w, cc[3].w, t[0], t[1], t[2], t[3]);
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[12 + r] = __dp4a(int(t[r]), xp, acc[12 + r]);
        }
    }
    for (; j + 4 <= jv; j += 4) {
        uint4 c[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) c[u] = __ldcs(reinterpret_cast<const uint4*>(a + (j + u) * lda));
        const int xp = int(pack_x4(x, j, incx));
        uint32_t t[4];
        transpose4x4_bytes(c[0].x, c[1].x, c[2].x, c[3].x, t[0], t[1], t[2], t[3]);
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[r] = __dp4a(int(t[r]), xp, acc[r]);
        transpose4x4_bytes(c[0].y, c[1].y, c[2].y, c[3].y, t[0], t[1], t[2], t[3]);
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[4 + r] = __dp4a(int(t[r]), xp, acc[4 + r]);
        transpose4x4_bytes(c[0].z, c[1].z, c[2].z, c[3].z, t[0], t[1], t[2], t[3]);
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[8 + r] = __dp4a(int(t[r]), xp, acc[8 + r]);
        transpose4x4_bytes(c[0].w, c[1].w, c[2].w, c[3].w, t[0], t[1], t[2], t[3]);
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[12 + r] = __dp4a(int(t[r]), xp, acc[12 + r]);
    }
    for (; j < jv; ++j) {
        const uint4 c = __ldcs(reinterpret_cast<const uint4*>(a + j * lda));
        const int xv = int(load(x + j * incx));
        const uint32_t w[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int b = 0; b < 4; ++b) acc[4 * q + b] += int(int8_t((w[q] >> (8 * b)) & 0xffu)) * xv;
    }
    if (!PLAIN && jv < j1) {      // the last column of a matrix whose rows end inside this vector
        const int xv = int(load(x + jv * incx));
#pragma unroll
        for (int r = 0; r < 16; ++r)
            if (r0 + r < m) acc[r] += int(load(a + r + jv * lda)) * xv;
    }
    if constexpr (!PLAIN) {
        __shared__ int4 red[4][kThreads];
#pragma unroll
        for (int q = 0; q < 4; ++q) red[q][threadIdx.x] = make_int4(acc[4 * q], acc[4 * q + 1], acc[4 * q + 2], acc[4 * q + 3]);
        __syncthreads();
        if (group != 0) return;
        for (int g = 1; g < kThreads >> rt; ++g) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int4 v = red[q][(g << rt) + tr];
                acc[4 * q] += v.x;
                acc[4 * q + 1] += v.y;
                acc[4 * q + 2] += v.z;
                acc[4 * q + 3] += v.w;
            }
        }
    }
    if (!PLAIN && r0 >= m) return;
    int32_t* p = part + int64_t(blockIdx.y) * m + r0;
    if (PLAIN || m % 4 == 0) {   // every split's sums start 16-byte aligned
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (PLAIN || r0 + 4 * q < m)
                reinterpret_cast<int4*>(p)[q] = make_int4(acc[4 * q], acc[4 * q + 1], acc[4 * q + 2], acc[4 * q + 3]);
    } else {
#pragma unroll
        for (int r = 0; r < 16; ++r)
            if (r0 + r < m) p[r] = acc[r];
    }
}

__global__ void __launch_bounds__(kThreads) gemv_i8_n_scalar(int64_t m, int64_t n, const int8_t* A,
                                                             int64_t lda, const int8_t* x, int64_t incx,
                                                             int32_t* part, int64_t cols_per_split) {
    pdl_wait();
    pdl_trigger();   // the reduction may be scheduled; it waits for this grid to finish
    const int64_t r = int64_t(blockIdx.x) * kThreads + threadIdx.x;
    const int64_t j0 = int64_t(blockIdx.y) * cols_per_split;
    const int64_t j1 = min(n, j0 + cols_per_split);
    if (r >= m) return;
    int acc = 0;
    int64_t j = j0;
    for (; j + 8 <= j1; j += 8) {      // eight columns in flight
        int8_t v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = __ldcs(A + r + (j + u) * lda);
#pragma unroll
        for (int u = 0; u < 8; ++u) acc += int(v[u]) * int(load(x + (j + u) * incx));
    }
    for (; j < j1; ++j) acc += int(A[r + j * lda]) * int(load(x + j * incx));
    part[int64_t(blockIdx.y) * m + r] = acc;
}

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

}  // namespace

// Column splits for op = N: enough CTAs for about 4 waves of 256-thread blocks on every SM
// (CTAs of 256 threads with rows_per_thread rows each).
int gemv_splits_rows(int64_t m, int64_t n, int rows_per_thread) {
    const int64_t rows_per_cta = int64_t(kThreads) * rows_per_thread;
    const int64_t rb = (m + rows_per_cta - 1) / rows_per_cta;
    int64_t target = int64_t(num_sms()) * 4;
    int64_t s = (target + rb - 1) / rb;
    if (s < 1) s = 1;
    if (s > 256) s = 256;
    const int64_t min_cols = 64;
    if (n / s < min_cols) s = (n + min_cols - 1) / min_cols;
    if (s < 1) s = 1;
    return int(s);
}

int gemv_splits(int64_t m, int64_t n) { return gemv_splits_rows(m, n, 4); }

// rows per thread of the op = N kernels: 4 (FP32, float4) or 16 (INT8, 16-byte loads)
static int rows_per_thread(hsmm_dtype_t a) { return a == HSMM_R_8I ? 16 : 4; }

size_t gemv_workspace_bytes(hsmm_dtype_t a, hsmm_op_t trans, int64_t m, int64_t n) {
    if (trans != HSMM_OP_N) return 0;
    return size_t(gemv_splits_rows(m, n, rows_per_thread(a))) * size_t(m) * 4u;
}

// Row threads of a CTA of the op = N vector kernels: all 256, or fewer (at least 32) while there
// are under two CTAs an SM (8192 x 4096 FP32, 3.4 CTAs an SM: 22.0 us with 256, 23.3 with 128)
struct NSplit {
    int rt;
    int64_t cols_per_group;
    dim3 grid;
};
static NSplit n_split(int64_t m, int ns, int64_t cps, int rows_per_thread) {
    NSplit s{8, cps, dim3()};
    const int64_t vecs = (m + rows_per_thread - 1) / rows_per_thread;
    auto blocks = [&] { return (vecs + (int64_t(1) << s.rt) - 1) >> s.rt; };
    while (s.rt > 5 && blocks() * ns < int64_t(num_sms()) * 2) --s.rt;
    const int groups = kThreads >> s.rt;
    s.cols_per_group = (cps + groups - 1) / groups;
    s.grid = dim3(unsigned(blocks()), unsigned(ns));
    return s;
}

hsmm_status_t gemv_f32(hsmm_op_t trans, int64_t m, int64_t n, float alpha, const float* A, int64_t lda,
                       const float* x, int64_t incx, float beta, float* y, int64_t incy, void* ws, size_t ws_bytes,
                       cudaStream_t st) {
    if (trans == HSMM_OP_N) {
        const int ns = gemv_splits(m, n);
        if (ws_bytes < size_t(ns) * size_t(m) * 4u || ws == nullptr) return HSMM_STATUS_WORKSPACE_TOO_SMALL;
        const int64_t cps = (n + ns - 1) / ns;
        float* part = static_cast<float*>(ws);
        const bool vec = (lda % 4 == 0) && aligned16(A) && aligned16(ws);
        cudaError_t e = cudaSuccess;
        if (vec) {
            const NSplit sp = n_split(m, ns, cps, 4);
            if (sp.rt == 8 && m % 4 == 0)
                gemv_f32_n_vec<true><<<sp.grid, kThreads, 0, st>>>(m, n, A, lda, x, incx, part, cps, 8, cps);
            else
                e = launch(gemv_f32_n_vec<false>, sp.grid, st, m, n, A, lda, x, incx, part, cps, sp.rt,
                               sp.cols_per_group);
        } else {
            dim3 grid(unsigned((m + kThreads - 1) / kThreads), unsigned(ns));
            e = launch(gemv_f32_n_scalar, grid, st, m, n, A, lda, x, incx, part, cps);
        }
        if (e == cudaSuccess) e = launch_reduce<float, float>(m, ns, part, alpha, beta, y, incy, st);
        count_launches(2);
        if (e != cudaSuccess) return record_cuda(e);
    } else {
        const bool vec = (lda % 4 == 0) && aligned16(A) && aligned16(x) && incx == 1;
        const cudaError_t e = launch_t<float, float4, float>(m, n, alpha, A, lda, x, incx, beta, y, incy, vec, st);
        count_launches(1);
        if (e != cudaSuccess) return record_cuda(e);
    }
    return check_launch();
}

hsmm_status_t gemv_i8(hsmm_op_t trans, int64_t m, int64_t n, int32_t alpha, const int8_t* A, int64_t lda,
                      const int8_t* x, int64_t incx, int32_t beta, int32_t* y, int64_t incy, void* ws,
                      size_t ws_bytes, cudaStream_t st) {
    if (trans == HSMM_OP_N) {
        const int ns = gemv_splits_rows(m, n, rows_per_thread(HSMM_R_8I));
        if (ws_bytes < size_t(ns) * size_t(m) * 4u || ws == nullptr) return HSMM_STATUS_WORKSPACE_TOO_SMALL;
        const int64_t cps = (n + ns - 1) / ns;
        int32_t* part = static_cast<int32_t*>(ws);
        const bool vec = (lda % 16 == 0) && aligned16(A) && aligned16(ws);
        cudaError_t e = cudaSuccess;
        if (vec) {
            const NSplit sp = n_split(m, ns, cps, 16);
            if (sp.rt == 8 && m % 16 == 0)
                gemv_i8_n_vec<true><<<sp.grid, kThreads, 0, st>>>(m, n, A, lda, x, incx, part, cps, 8, cps);
            else
                e = launch(gemv_i8_n_vec<false>, sp.grid, st, m, n, A, lda, x, incx, part, cps, sp.rt,
                               sp.cols_per_group);
        } else {
            dim3 grid(unsigned((m + kThreads - 1) / kThreads), unsigned(ns));
            e = launch(gemv_i8_n_scalar, grid, st, m, n, A, lda, x, incx, part, cps);
        }
        if (e == cudaSuccess) e = launch_reduce<int32_t, uint32_t>(m, ns, part, alpha, beta, y, incy, st);
        count_launches(2);
        if (e != cudaSuccess) return record_cuda(e);
    } else {
        const bool vec = (lda % 16 == 0) && aligned16(A) && aligned16(x) && incx == 1;
        const cudaError_t e = launch_t<int8_t, int4, int>(m, n, alpha, A, lda, x, incx, beta, y, incy, vec, st);
        count_launches(1);
        if (e != cudaSuccess) return record_cuda(e);
    }
    return check_launch();
}

}  // namespace hsmm
