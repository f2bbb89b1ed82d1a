// gemm_f64.cu -- native FP64 product C <- alpha*op(A)*op(B) + beta*C on the FP64 pipe.
//
// Eq. PRODUCT (Section 3.1) computed with FP64 fused multiply-adds.  This is the
// baseline the FP64-accurate slice form is measured against.  The FP64 pipe of a
// GB300 is narrow (two FMAs per clock and SM), so the kernels only have to keep it busy on
// every SM: T x T tiles per CTA, T = 64, 32, 16 or 8 by the size of C, k-slabs of 16 staged
// through shared memory (loads follow whichever index is contiguous for op = N / T).
#include <cstdint>
#include <type_traits>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "common.cuh"
#include "internal.h"

namespace hsmm {

static __device__ uint32_t g_status_gemm_f64;

uint32_t status_take_gemm_f64() {
    uint32_t v = 0, z = 0;
    cudaMemcpyFromSymbol(&v, g_status_gemm_f64, sizeof(v));
    cudaMemcpyToSymbol(g_status_gemm_f64, &z, sizeof(z));
    return v;
}

namespace {

constexpr int BK = 16;

// The product kernels are launched as programmatic dependents: resident while the kernel before still
// writes what they read, so their operands are not const __restrict__ (read-only data).

// T x T tiles on TH x TH threads, a (T / TH)^2 register block each
template <int T>
struct Tile {
    static constexpr int TH = T == 64 || T == 32 ? 16 : 8, NT = TH * TH, RB = T / TH;
    // CTAs per SM the registers are limited for: with few resident ones the small tiles end unevenly
    // (700 x 601 x 1000 at T = 16: 903 us with eight, 745 with fourteen)
    static constexpr int OCC = T == 64 ? 2 : T == 32 ? 4 : 14;
};

// Load the T x BK tile of op(M) at (r0, k0) into s[k][r] (zero outside); along_k: op(M)(r, kk) =
// M[kk + r ld] (kk contiguous), else M[r + kk ld].
template <int T>
__device__ __forceinline__ void load_tile(double (*s)[T + 1], const double* M, int64_t ld, bool along_k,
                                          int64_t rows, int64_t kdim, int64_t r0, int64_t k0) {
    constexpr int NT = Tile<T>::NT;
    const int t = threadIdx.x;
#pragma unroll
    for (int q = 0; q < (T * BK) / NT; ++q) {
        const int idx = t + q * NT;
        const int r = along_k ? idx / BK : idx % T, kk = along_k ? idx % BK : idx / T;
        const int64_t gr = r0 + r, gk = k0 + kk;
        s[kk][r] = (gr < rows && gk < kdim) ? (along_k ? M[gk + gr * ld] : M[gr + gk * ld]) : 0.0;
    }
}

template <int T>
__global__ void __launch_bounds__(Tile<T>::NT, Tile<T>::OCC)
    gemm_f64_kernel(int64_t m, int64_t n, int64_t k, double alpha, const double* A, int64_t lda, bool ta,
                    const double* B, int64_t ldb, bool tb, double beta, double* C,
                    int64_t ldc) {
    constexpr int TH = Tile<T>::TH, RB = Tile<T>::RB;
    __shared__ double As[BK][T + 1];
    __shared__ double Bs[BK][T + 1];
    pdl_wait();
    const int64_t m0 = int64_t(blockIdx.x) * T, n0 = int64_t(blockIdx.y) * T;
    const int tx = threadIdx.x % TH, ty = threadIdx.x / TH;
    double acc[RB][RB];
#pragma unroll
    for (int i = 0; i < RB; ++i)
#pragma unroll
        for (int j = 0; j < RB; ++j) acc[i][j] = 0.0;

    for (int64_t k0 = 0; k0 < k; k0 += BK) {
        load_tile<T>(As, A, lda, ta, m, k, m0, k0);
        load_tile<T>(Bs, B, ldb, !tb, n, k, n0, k0);     // op(B)(kk, c): along k for op = N
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            double a[RB], b[RB];
#pragma unroll
            for (int i = 0; i < RB; ++i) a[i] = As[kk][ty + TH * i];
#pragma unroll
            for (int j = 0; j < RB; ++j) b[j] = Bs[kk][tx + TH * j];
#pragma unroll
            for (int i = 0; i < RB; ++i)
#pragma unroll
                for (int j = 0; j < RB; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < RB; ++j) {
        const int64_t c = n0 + tx + TH * j;
        if (c >= n) continue;
#pragma unroll
        for (int i = 0; i < RB; ++i) {
            const int64_t r = m0 + ty + TH * i;
            if (r >= m) continue;
            double v = alpha * acc[i][j];
            if (beta != 0.0) v = fma(beta, C[r + c * ldc], v);
            C[r + c * ldc] = v;
        }
    }
}

// Tile edge with the least work on the busiest SM.  The pipe is kept busy by any of them, so what
// counts is how evenly the tiles cover the SMs and the matrix's edges; smaller tiles load more
// and are taken for a gain of a few percent and more.  64 -> chosen, us: 700 x 601 x 1000 1034 ->
// 745 (16), 100 x 1498 x 327 348 -> 98 (16), 300^3 315 -> 53 (8), 1024^3 2057 -> 1805 (32), 64 x 64
// x 1000 1032 -> 69 (8); 4096 x 4096 x 1024 keeps 64 (27.6 ms, 1.25 TFLOP/s).  Complex, 32 ->
// chosen: 300 x 200 x 300 320 -> 160 (8), 700 x 500 x 600 1869 -> 1580 (16).
int pick_tile(int64_t m, int64_t n, int largest) {
    const int sms = num_sms();
    int best = largest;
    double best_cost = 0.0;
    for (int t = largest; t >= 8; t /= 2) {
        const int64_t tn = (n + t - 1) / t, tiles = ((m + t - 1) / t) * tn;
        if (tn > 65535 && t != largest) break;
        const double cost = double((tiles + sms - 1) / sms) * t * t * (1.0 + 0.5 / t);
        if (t == largest || cost < 0.97 * best_cost) {
            best = t;
            best_cost = cost;
        }
    }
    return best;
}

// ---------------------------------------------------------------------------
// Complex product (Section 7: the method measured on complex data) on the FP64
// pipe: interleaved (re, im) doubles, op = N, T or C (conjugate transpose).  A
// 32 x 32 complex tile per CTA, k-slabs of 16, a 2 x 2 complex register block per
// thread; each complex multiply-add is four FP64 FMAs.
// ---------------------------------------------------------------------------
constexpr int ZK = 16;

// Load the T x ZK tile of op(M) at (r0, k0) into s[k][r] (zero outside, conjugated for conj)
template <int T>
__device__ __forceinline__ void load_ztile(double2 (*s)[T + 1], const double2* M, int64_t ld, bool along_k,
                                           bool conj, int64_t rows, int64_t kdim, int64_t r0, int64_t k0) {
    constexpr int NT = Tile<T>::NT;
    const int t = threadIdx.x;
#pragma unroll
    for (int q = 0; q < (T * ZK) / NT; ++q) {
        const int idx = t + q * NT;
        const int r = along_k ? idx / ZK : idx % T, kk = along_k ? idx % ZK : idx / T;
        const int64_t gr = r0 + r, gk = k0 + kk;
        double2 v = make_double2(0.0, 0.0);
        if (gr < rows && gk < kdim) {
            v = along_k ? M[gk + gr * ld] : M[gr + gk * ld];
            if (conj) v.y = -v.y;
        }
        s[kk][r] = v;
    }
}

template <int T>
__global__ void __launch_bounds__(Tile<T>::NT) gemm_z64_kernel(int64_t m, int64_t n, int64_t k, double2 alpha,
                                                              const double2* A, int64_t lda, char ta,
                                                              const double2* B, int64_t ldb, char tb,
                                                              double2 beta, double2* C, int64_t ldc) {
    constexpr int TH = Tile<T>::TH, RB = Tile<T>::RB;
    __shared__ double2 As[ZK][T + 1];
    __shared__ double2 Bs[ZK][T + 1];     // Bs[kk][c] = op(B)(k0 + kk, n0 + c)
    pdl_wait();
    const int64_t m0 = int64_t(blockIdx.x) * T, n0 = int64_t(blockIdx.y) * T;
    const int tx = threadIdx.x % TH, ty = threadIdx.x / TH;
    double accr[RB][RB], acci[RB][RB];
#pragma unroll
    for (int i = 0; i < RB; ++i)
#pragma unroll
        for (int j = 0; j < RB; ++j) accr[i][j] = acci[i][j] = 0.0;
    for (int64_t k0 = 0; k0 < k; k0 += ZK) {
        load_ztile<T>(As, A, lda, ta != 'N', ta == 'C', m, k, m0, k0);
        load_ztile<T>(Bs, B, ldb, tb == 'N', tb == 'C', n, k, n0, k0);
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < ZK; ++kk) {
            double2 a[RB], b[RB];
#pragma unroll
            for (int i = 0; i < RB; ++i) a[i] = As[kk][ty + TH * i];
#pragma unroll
            for (int j = 0; j < RB; ++j) b[j] = Bs[kk][tx + TH * j];
#pragma unroll
            for (int i = 0; i < RB; ++i)
#pragma unroll
                for (int j = 0; j < RB; ++j) {
                    accr[i][j] = fma(a[i].x, b[j].x, accr[i][j]);
                    accr[i][j] = fma(-a[i].y, b[j].y, accr[i][j]);
                    acci[i][j] = fma(a[i].x, b[j].y, acci[i][j]);
                    acci[i][j] = fma(a[i].y, b[j].x, acci[i][j]);
                }
        }
        __syncthreads();
    }
    const bool read_c = beta.x != 0.0 || beta.y != 0.0;
#pragma unroll
    for (int j = 0; j < RB; ++j) {
        const int64_t c = n0 + tx + TH * j;
        if (c >= n) continue;
#pragma unroll
        for (int i = 0; i < RB; ++i) {
            const int64_t r = m0 + ty + TH * i;
            if (r >= m) continue;
            double vr = alpha.x * accr[i][j] - alpha.y * acci[i][j];
            double vi = alpha.x * acci[i][j] + alpha.y * accr[i][j];
            if (read_c) {
                const double2 c0 = C[r + c * ldc];
                vr = fma(beta.x, c0.x, fma(-beta.y, c0.y, vr));
                vi = fma(beta.x, c0.y, fma(beta.y, c0.x, vi));
            }
            C[r + c * ldc] = make_double2(vr, vi);
        }
    }
}

__global__ void scale_z64_kernel(int64_t m, int64_t n, double2 beta, double2* __restrict__ C, int64_t ldc) {
    const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    for (int64_t jj = blockIdx.y; jj < n; jj += gridDim.y) {
        if (i >= m) continue;
        double2 v = make_double2(0.0, 0.0);
        if (beta.x != 0.0 || beta.y != 0.0) {
            const double2 c = C[i + jj * ldc];
            v = make_double2(beta.x * c.x - beta.y * c.y, beta.x * c.y + beta.y * c.x);
        }
        C[i + jj * ldc] = v;
    }
}

template <typename T>
__global__ void scale_kernel(int64_t m, int64_t n, T beta, T* __restrict__ C, int64_t ldc) {
    const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    const int64_t j = blockIdx.y;
    for (int64_t jj = j; jj < n; jj += gridDim.y) {
        if (i < m) C[i + jj * ldc] = (beta == T(0)) ? T(0) : T(beta * C[i + jj * ldc]);
    }
}

__global__ void scale_bf16_kernel(int64_t m, int64_t n, float beta, __nv_bfloat16* __restrict__ C, int64_t ldc) {
    const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    for (int64_t jj = blockIdx.y; jj < n; jj += gridDim.y) {
        if (i < m)
            C[i + jj * ldc] = (beta == 0.f) ? __float2bfloat16_rn(0.f)
                                            : __float2bfloat16_rn(beta * __bfloat162float(C[i + jj * ldc]));
    }
}

}  // namespace

hsmm_status_t gemm_f64_native(hsmm_op_t ta, hsmm_op_t tb, int64_t m, int64_t n, int64_t k, double alpha,
                              const double* A, int64_t lda, const double* B, int64_t ldb, double beta, double* C,
                              int64_t ldc, cudaStream_t st) {
    const int t = pick_tile(m, n, 64);
    const dim3 grid(unsigned((m + t - 1) / t), unsigned((n + t - 1) / t));
    if (grid.y > 65535u) return HSMM_STATUS_NOT_SUPPORTED;
    cudaError_t e = cudaSuccess;
    auto launch = [&](auto tile) {
        constexpr int T = decltype(tile)::value;
        e = pdl_launch(gemm_f64_kernel<T>, grid, Tile<T>::NT, 0, 1, st, m, n, k, alpha, A, lda, ta == HSMM_OP_T, B, ldb,
                       tb == HSMM_OP_T, beta, C, ldc);
    };
    if (t == 64) launch(std::integral_constant<int, 64>{});
    else if (t == 32) launch(std::integral_constant<int, 32>{});
    else if (t == 16) launch(std::integral_constant<int, 16>{});
    else launch(std::integral_constant<int, 8>{});
    count_launches(1);
    if (e != cudaSuccess) return record_cuda(e);
    return check_launch();
}

hsmm_status_t gemm_z64_native(hsmm_op_t ta, hsmm_op_t tb, int64_t m, int64_t n, int64_t k, const double* alpha,
                              const void* A, int64_t lda, const void* B, int64_t ldb, const double* beta, void* C,
                              int64_t ldc, cudaStream_t st) {
    const int t = pick_tile(m, n, 32);
    const dim3 grid(unsigned((m + t - 1) / t), unsigned((n + t - 1) / t));
    if (grid.y > 65535u) return HSMM_STATUS_NOT_SUPPORTED;
    cudaError_t e = cudaSuccess;
    auto launch = [&](auto tile) {
        constexpr int T = decltype(tile)::value;
        e = pdl_launch(gemm_z64_kernel<T>, grid, Tile<T>::NT, 0, 1, st, m, n, k, make_double2(alpha[0], alpha[1]),
                       static_cast<const double2*>(A), lda, char(ta), static_cast<const double2*>(B), ldb, char(tb),
                       make_double2(beta[0], beta[1]), static_cast<double2*>(C), ldc);
    };
    if (t == 32) launch(std::integral_constant<int, 32>{});
    else if (t == 16) launch(std::integral_constant<int, 16>{});
    else launch(std::integral_constant<int, 8>{});
    count_launches(1);
    if (e != cudaSuccess) return record_cuda(e);
    return check_launch();
}

hsmm_status_t scale_matrix(hsmm_dtype_t c, int64_t m, int64_t n, const void* beta, void* C, int64_t ldc,
                           cudaStream_t st) {
    dim3 grid(unsigned((m + 255) / 256), unsigned(n < 65535 ? n : 65535));
    switch (c) {
        case HSMM_R_64F:
            scale_kernel<double><<<grid, 256, 0, st>>>(m, n, *static_cast<const double*>(beta),
                                                       static_cast<double*>(C), ldc);
            break;
        case HSMM_R_32F:
            scale_kernel<float><<<grid, 256, 0, st>>>(m, n, *static_cast<const float*>(beta), static_cast<float*>(C),
                                                      ldc);
            break;
        case HSMM_R_32I:
            scale_kernel<int32_t><<<grid, 256, 0, st>>>(m, n, *static_cast<const int32_t*>(beta),
                                                        static_cast<int32_t*>(C), ldc);
            break;
        case HSMM_C_64F: {
            const double* b = static_cast<const double*>(beta);
            scale_z64_kernel<<<grid, 256, 0, st>>>(m, n, make_double2(b[0], b[1]), static_cast<double2*>(C), ldc);
            break;
        }
        case HSMM_R_16BF:
            scale_bf16_kernel<<<grid, 256, 0, st>>>(m, n, *static_cast<const float*>(beta),
                                                    static_cast<__nv_bfloat16*>(C), ldc);
            break;
        default:
            return HSMM_STATUS_NOT_SUPPORTED;
    }
    count_launches(1);
    return check_launch();
}

}  // namespace hsmm
