// internal.h -- host-side declarations shared by the translation units of libhsmm.
#pragma once

#include <atomic>
#include <cstddef>
#include <cstdint>
#include <cuda.h>
#include <cuda_runtime.h>

#include "hsmm.h"

namespace hsmm {

// ---- library state (api.cu) ----
uint64_t wait_timeout_ns();
void count_launches(int64_t n);
int num_sms();
hsmm_status_t record_cuda(cudaError_t e);           // SUCCESS or CUDA_ERROR (remembers the code)
// Remember a human-readable reason for a failing status (per host thread) and return the status.
hsmm_status_t fail(hsmm_status_t st, const char* fmt, ...);
const char* last_detail();
inline hsmm_status_t check_launch() { return record_cuda(cudaGetLastError()); }
inline bool aligned_to(const void* p, uintptr_t bytes) { return reinterpret_cast<uintptr_t>(p) % bytes == 0; }

// Kernel function attributes (dynamic shared memory, non-portable cluster sizes) apply per
// device: `set` runs once for each device the calling thread uses (one bit per device in
// `done`; two threads may both run it, which is harmless).
template <typename F>
inline hsmm_status_t attrs_once_per_device(std::atomic<uint64_t>& done, F&& set) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return record_cuda(e);
    const uint64_t bit = (dev >= 0 && dev < 64) ? (uint64_t(1) << dev) : 0;
    if (bit && (done.load(std::memory_order_acquire) & bit)) return HSMM_STATUS_SUCCESS;
    e = set();
    if (e != cudaSuccess) return record_cuda(e);
    if (bit) done.fetch_or(bit, std::memory_order_release);
    return HSMM_STATUS_SUCCESS;
}

// ---- per translation unit device status words (read and cleared) ----
uint32_t status_take_gemv();
uint32_t status_take_gemm_tc();
uint32_t status_take_grouped();
uint32_t status_take_ozaki_tc();
uint32_t status_take_gemm_f64();
uint32_t status_take_ozaki();
uint32_t status_take_ring();
uint32_t status_take_selftest();

// ---- gemv.cu ----
int gemv_splits(int64_t m, int64_t n);
int gemv_splits_rows(int64_t m, int64_t n, int rows_per_thread);
size_t gemv_workspace_bytes(hsmm_dtype_t a, hsmm_op_t trans, int64_t m, int64_t n);
hsmm_status_t gemv_f32(hsmm_op_t trans, int64_t m, int64_t n, float alpha, const float* A, int64_t lda,
                       const float* x, int64_t incx, float beta, float* y, int64_t incy, void* ws, size_t ws_bytes,
                       cudaStream_t st);
hsmm_status_t gemv_i8(hsmm_op_t trans, int64_t m, int64_t n, int32_t alpha, const int8_t* A, int64_t lda,
                      const int8_t* x, int64_t incx, int32_t beta, int32_t* y, int64_t incy, void* ws,
                      size_t ws_bytes, cudaStream_t st);

// ---- gemm_f64.cu ----
hsmm_status_t gemm_f64_native(hsmm_op_t ta, hsmm_op_t tb, int64_t m, int64_t n, int64_t k, double alpha,
                              const double* A, int64_t lda, const double* B, int64_t ldb, double beta, double* C,
                              int64_t ldc, cudaStream_t st);
// complex FP64 product on the FP64 pipe; A, B, C interleaved (re, im), alpha and beta (re, im)
hsmm_status_t gemm_z64_native(hsmm_op_t ta, hsmm_op_t tb, int64_t m, int64_t n, int64_t k, const double* alpha,
                              const void* A, int64_t lda, const void* B, int64_t ldb, const double* beta, void* C,
                              int64_t ldc, cudaStream_t st);
// C = beta*C (beta == 0 writes zeros), for the BLAS early-outs; element type by size (4 or 8) or bf16 (2)
hsmm_status_t scale_matrix(hsmm_dtype_t c, int64_t m, int64_t n, const void* beta, void* C, int64_t ldc,
                           cudaStream_t st);

// ---- gemm_tc.cu ----
struct TcOperand {
    const void* ptr;
    int64_t ld;
    bool mn_major;   // true: the M (or N) index is contiguous in memory
};
hsmm_status_t gemm_tc(hsmm_dtype_t ab, hsmm_dtype_t c, hsmm_op_t ta, hsmm_op_t tb, int64_t m, int64_t n, int64_t k,
                      float alpha, const void* A, int64_t lda, const void* B, int64_t ldb, float beta, void* C,
                      int64_t ldc, int tile_n, cudaStream_t st);
bool tma_operand_ok(const void* p, int64_t ld, size_t esize);
// 2D (or 3D with a batch dimension) TMA map with 128-byte swizzle; false if encoding failed
// (last_encode_result() then holds the CUresult)
bool encode_map(CUtensorMap* map, CUtensorMapDataType dt, int esize, const void* base, uint64_t inner, uint64_t outer,
                uint64_t ld, uint32_t box_inner, uint32_t box_outer, uint64_t batch = 0,
                uint64_t batch_stride_elems = 0, CUtensorMapSwizzle swizzle = CU_TENSOR_MAP_SWIZZLE_128B,
                uint32_t box_batch = 1,
                uint64_t blocks = 0, uint64_t block_stride_elems = 0);
int last_encode_result();

// ---- gemm_split_tc.cu ----
struct SplitArgs {
    int M, N, K;
    int a_mn, b_mn;         // operand majorness
    int a_mn3, b_mn3;       // MN-major operand described as a 3D tensor of chunks (see gemm_tc)
    float alpha, beta;
    void* C;
    int64_t ldc;
    uint64_t timeout_ns;
    int c_vec;              // four rows of a column of C can be stored at once (beta == 0)
    int bn, stages;         // tile width; stages are set by the launch
};
// 128 x bn tiles, k split over a cluster of `split` CTAs; cost: estimated microseconds (bn = 0: no plan)
struct SplitPlan {
    int bn, split;
    double cost;
};
SplitPlan split_plan(int64_t m, int64_t n, int64_t k, bool tf32, bool b_mn);
hsmm_status_t gemm_tc_split(bool tf32, bool out_bf16, const CUtensorMap& ta, const CUtensorMap& tb, const SplitArgs& g,
                            const SplitPlan& plan, cudaStream_t st);
uint32_t status_take_split();

// Slices of an operand, from row `row0` of its planes on.  block_rows = 0: [t][v][w], row pitch ldq.
// Otherwise a plane holds its columns in blocks of 64, [t][w / 64][v][w % 64] with block_rows rows v
// (the last block ldq % 64 wide): the same bytes, but every 64 columns of a row are one 128-byte line,
// which is what a TMA box reads of it.
struct Slices {
    void* q;
    int64_t ldq, plane;            // elements; plane >= rows * ldq
    int64_t block_rows, row0;
};

// ---- gemm_ozaki_tc.cu ----
// Slice products of the FP64-accurate form: S_d = sum_{t+u=d} Q^A_t (Q^B_u)^T, d = 2..s+1, exact INT32,
// stored as [d-2][n][m].
hsmm_status_t gemm_ozaki_slices(int64_t m, int64_t n, int64_t k, int slices, int bits, const Slices& qa,
                                const Slices& qb, int32_t* sd, int64_t sd_plane, cudaStream_t st);

// ---- ozaki.cu ----
// One operand to split: nv lines of nw entries, entry (v, w) at M[v + w ld] (v_contig) or
// M[w + v ld]; the slices of line v are row row0 + v of q.  Complex operands go into the real form of the complex product (A' =
// [Re, Im] rows for role_b = false; B'' = [[Re, Im], [-Im, Re]] columns for role_b = true, 2 nv
// lines); conj: op = C.
struct SplitOperand {
    const void* M;
    int64_t ld, nv, nw;
    bool v_contig, conj, role_b;
    int32_t* expo;
    Slices q;
};
// Lines of one operand that ozaki_split takes (2097120); more are refused.
constexpr int64_t SPLIT_MAX_LINES = int64_t(65535) * 32;
// Splits one or two operands (count), in one launch if their lines run the same way in memory.
hsmm_status_t ozaki_split(bool cplx, const SplitOperand* ops, int count, int bits, int slices, cudaStream_t st);
// C = alpha 2^(ea_i + eb_j) sum_d 2^(-bits d) S_d + beta C
hsmm_status_t ozaki_recombine(int64_t m, int64_t n, int slices, int bits, const int32_t* sd, int64_t sd_plane,
                              const int32_t* ea, const int32_t* eb, double alpha, double beta, double* C, int64_t ldc,
                              cudaStream_t st);
// C = alpha (Re + i Im) + beta C from the real form's S_d (m x 2n), complex alpha, beta (re, im)
hsmm_status_t ozaki_zrecombine(int64_t m, int64_t n, int slices, int bits, const int32_t* sd, int64_t sd_plane,
                               const int32_t* ea, const int32_t* eb, const double* alpha, const double* beta, void* C,
                               int64_t ldc, cudaStream_t st);
// The workspace carve-up of the FP64-accurate form (documented in hsmm.h)
struct OzakiLayout {
    int64_t ldq, qa_plane, qb_plane, sd_plane;   // pitches in elements
    size_t qa, qb, ea, eb, sd, total;            // byte offsets
};
OzakiLayout ozaki_layout(int64_t m, int64_t n, int64_t k, int slices);
int default_slices(const hsmm_config_t* c);   // cfg->ozaki_slices, or 7
int default_bits(const hsmm_config_t* c);     // cfg->ozaki_bits, or 7
// Rows of op(A) (m x k) / columns of op(B) (k x n) as operands to split; cplx: complex operands
SplitOperand split_operand_a(bool cplx, hsmm_op_t ta, int64_t m, int64_t k, const void* A, int64_t lda, int32_t* ea,
                             const Slices& qa);
SplitOperand split_operand_b(bool cplx, hsmm_op_t tb, int64_t k, int64_t n, const void* B, int64_t ldb, int32_t* eb,
                             const Slices& qb);
// The slices at `q` of a workspace: `rows` rows in a plane, the operand's from row0 on.  Rows of whole
// 128-byte lines are kept as they are, others in blocks of 64 columns.
inline Slices workspace_slices(void* q, int64_t ldq, int64_t plane, int64_t rows, int64_t row0 = 0) {
    return Slices{q, ldq, plane, ldq % 64 == 0 ? 0 : rows, row0};
}
// Plane pitch (elements) of the workspace planes of hsmm_gemm's FP64-accurate form: the
// plane size rounded up to 256 bytes plus 1 KiB, so that the s planes one thread touches
// are not a power of two apart (such strides land on the same DRAM channels).
int64_t ozaki_plane_pitch(int64_t elems, int64_t elem_bytes);
int64_t ozaki_ldq(int64_t k);

// ---- gemm_ring_tc.cu ----
// C = alpha op(A) op(B) + beta C (BF16 in, FP32 out) in the ring order of Algorithm 2 on
// clusters of p CTAs with K auxiliary accumulators
hsmm_status_t gemm_tc_ring(hsmm_op_t ta, hsmm_op_t tb, int64_t m, int64_t n, int64_t k, float alpha, const void* A,
                           int64_t lda, const void* B, int64_t ldb, float beta, float* C, int64_t ldc, int p, int K,
                           cudaStream_t st);
uint32_t status_take_ring_tc();

// ---- nbody.cu ----
// F_i = sum_j f(x_i, z_j) (gravitational f), float4 bodies; ring_p = 0: tiled, else the
// hyper-systolic recipe on clusters of ring_p CTAs with ring_k replicas
hsmm_status_t nbody_forces(int64_t nx, int64_t nz, const float* x, const float* z, float eps2, float* out,
                           int ring_p, int ring_k, cudaStream_t st);

// ---- ring.cu ----
size_t ring_workspace_bytes(int p, int K, int64_t n);
hsmm_status_t ring_gemm_f64(int p, int K, int64_t n, const double* A, int64_t lda, const double* B, int64_t ldb,
                            double* C, int64_t ldc, void* workspace, size_t workspace_bytes, cudaStream_t st);

// ---- gemm_grouped.cu ----
struct GroupedPlan;
hsmm_status_t grouped_plan_create(hsmm_dtype_t ab, hsmm_dtype_t c, int64_t count, const hsmm_gemm_desc_t* descs,
                                  int tile_n, GroupedPlan** out);
// tile_n_per_problem: per problem 128/256 or 0 = automatic (NULL: all automatic);
// schedule 0: problems in the given order, 1: longest k first
hsmm_status_t grouped_plan_create_ex(hsmm_dtype_t ab, hsmm_dtype_t c, int64_t count, const hsmm_gemm_desc_t* descs,
                                     int tile_n, const int* tile_n_per_problem, int schedule, GroupedPlan** out);
hsmm_status_t grouped_plan_launch(GroupedPlan* plan, float alpha, float beta, cudaStream_t st);
hsmm_status_t grouped_plan_info(GroupedPlan* plan, int64_t* tiles, int* tile_n);
void grouped_plan_destroy(GroupedPlan* plan);
// Without a plan: bytes of workspace the launch of these problems needs (0 and *st set on an
// error), and the launch itself with its descriptors and tile table written into the
// workspace by kernels on the stream (nothing allocated; capturable)
size_t grouped_workspace_bytes(hsmm_dtype_t ab, hsmm_dtype_t c, int64_t count, const hsmm_gemm_desc_t* descs,
                               int tile_n, hsmm_status_t* st);
hsmm_status_t grouped_run_in_workspace(hsmm_dtype_t ab, hsmm_dtype_t c, int64_t count, const hsmm_gemm_desc_t* descs,
                                       int tile_n, void* ws, size_t ws_bytes, float alpha, float beta,
                                       cudaStream_t st);

// ---- selftest (api.cu) ----
hsmm_status_t selftest_timeout_launch(uint64_t timeout_ns, cudaStream_t st);

}  // namespace hsmm
