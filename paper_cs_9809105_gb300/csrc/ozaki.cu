// ozaki.cu -- the splitting step of the FP64-accurate product.
//
// Error-free splitting of Ozaki, Ogita, Oishi and Rump (Numer. Algorithms 59,
// 2012) in its fixed-point integer form: for every row of op(A) (every column of
// op(B)) with exponent e (the smallest integer with |m| < 2^e over that line),
//   x = m 2^-e,  for t = 1..s:  y = x 2^bits,  q_t = trunc(y),  x = y - q_t.
// The digits q_t are read from the IEEE-754 significand with integer shifts (the
// values the exact FP64 steps give); |q_t| <= 2^bits - 1 <= 127, so the slices are
// stored exactly as BF16.  Output layout [t][v][w]: v = row of op(A) (column of
// op(B)), w = the contraction index, contiguous, row pitch ldq (a multiple of 8 so
// that the TMA row stride is a multiple of 16 bytes).
//
// One or two launches split both operands of a product (or one).
#include <algorithm>
#include <atomic>
#include <climits>
#include <cstdint>
#include <type_traits>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "common.cuh"
#include "internal.h"

namespace hsmm {

static __device__ uint32_t g_status_ozaki;

uint32_t status_take_ozaki() {
    uint32_t v = 0, z = 0;
    cudaMemcpyFromSymbol(&v, g_status_ozaki, sizeof(v));
    cudaMemcpyToSymbol(g_status_ozaki, &z, sizeof(z));
    return v;
}

int64_t ozaki_ldq(int64_t k) { return (k + 7) / 8 * 8; }

int64_t ozaki_plane_pitch(int64_t elems, int64_t elem_bytes) {
    const int64_t bytes = (elems * elem_bytes + 255) / 256 * 256 + 1024;
    return bytes / elem_bytes;
}

namespace {

__device__ __forceinline__ int line_exponent(double mx) {
    if (mx == 0.0) return INT_MIN;
    int e;
    frexp(mx, &e);       // mx = f 2^e with f in [0.5, 1): mx < 2^e, and 2^(e-1) <= mx
    return e;
}

// |x| as its IEEE-754 bit pattern without the sign.  For finite values the unsigned order of
// these patterns is the order of the magnitudes.  A line's exponent needs only the largest
// high word (sign cleared) while any is non-zero, and the largest low word when all high
// words are zero (tiny subnormals), so the running "maximum" keeps the two 32-bit halves'
// maxima apart: 32-bit integer operations only (64-bit compares went to the narrow FP64 pipe).
__device__ __forceinline__ uint64_t mag_bits(double x) {
    return uint64_t(__double_as_longlong(x)) & 0x7FFFFFFFFFFFFFFFull;
}
__device__ __forceinline__ uint64_t mag_max(uint64_t a, uint64_t b) {
    const uint32_t hi = max(uint32_t(a >> 32), uint32_t(b >> 32)), lo = max(uint32_t(a), uint32_t(b));
    return (uint64_t(hi) << 32) | lo;
}
// exponent of a line from its halfwise maximum (INT_MIN for an all-zero line)
__device__ __forceinline__ int line_exponent_bits(uint64_t mb) {
    const uint64_t top = (mb >> 32) ? (mb & 0xFFFFFFFF00000000ull) : mb;   // the low word matters only alone
    return top == 0 ? INT_MIN : line_exponent(__longlong_as_double(int64_t(top)));
}

// One value prepared for digit extraction.  With |v| = M 2^(E-1075) (M the 53-bit significand),
// digit t of |v| 2^(-e) is floor(M 2^(E - 1075 - e + bits t)) mod 2^bits, read from the
// significand with integer shifts: the same digits the FP64 steps y = x 2^bits, q = trunc(y),
// x = y - q produce, without FP64 arithmetic (the FP64 pipe of this GPU is narrow).  Each digit
// carries the sign of v.  Here |v| = mag 2^(base + e).
struct Digits {
    uint64_t mag;
    int base;
    uint32_t neg;
};

__device__ __forceinline__ Digits prepare_digits(double val, int e) {
    const uint64_t u = uint64_t(__double_as_longlong(val));
    Digits r;
    r.neg = uint32_t(u >> 63);
    int E = int((u >> 52) & 0x7FF);
    r.mag = u & ((uint64_t(1) << 52) - 1);
    if (E != 0) r.mag |= uint64_t(1) << 52; else E = 1;
    if (e == INT_MIN) r.mag = 0;
    r.base = E - 1075 - (e == INT_MIN ? 0 : e);
    return r;
}

__device__ __forceinline__ uint32_t digit_bits(const Digits& x, int bits, int t) {
    const uint32_t mask = (1u << bits) - 1u;
    const int sh = x.base + bits * t;
    if (sh < 0) return (-sh >= 64) ? 0u : uint32_t(x.mag >> -sh) & mask;
    return (sh >= bits) ? 0u : uint32_t(x.mag << sh) & mask;
}

// BF16 patterns of two digits d in [0, 255], each with the sign n of its value (none for d = 0):
// the FP32 number (-1)^n (2^23 + d) holds d in its low significand bits, and minus (-1)^n 2^23
// it is exactly (-1)^n d (+0 for d = 0); one packed subtraction makes both, and the upper halves
// of the two results, gathered by one byte permutation, are the two BF16 patterns (float(d)
// has at most 8 significant bits).  Full-rate FP32 and integer operations only.
__device__ __forceinline__ uint32_t bf16x2_of_digits(uint32_t d0, uint32_t d1, uint64_t bias) {
    const uint64_t a = (uint64_t(uint32_t(bias >> 32) | d1) << 32) | (uint32_t(bias) | d0);
    uint64_t y;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(y) : "l"(a), "l"(bias));
    return __byte_perm(uint32_t(y), uint32_t(y >> 32), 0x7632);
}
// (-1)^n 2^23 of two values, n their signs
__device__ __forceinline__ uint64_t signed_bias(uint32_t n0, uint32_t n1) {
    return (uint64_t(0x4B000000u | (n1 << 31)) << 32) | (0x4B000000u | (n0 << 31));
}

// four BF16 digits of consecutive entries: one 8-byte store (full), or 2-byte ones for the first `valid`
__device__ __forceinline__ void put4(uint16_t* o, uint32_t w01, uint32_t w23, bool full, int valid) {
    if (full) {
        *reinterpret_cast<uint2*>(o) = make_uint2(w01, w23);
    } else {
        o[0] = uint16_t(w01);
        if (valid > 1) o[1] = uint16_t(w01 >> 16);
        if (valid > 2) o[2] = uint16_t(w23);
        if (valid > 3) o[3] = uint16_t(w23 >> 16);
    }
}

// Four consecutive values of one line -> four BF16 digits for each slice t.
__device__ __forceinline__ void slice_store4(const double (&x)[4], int e, int bits, int s, uint16_t* out,
                                             int64_t slice_stride, bool full, int valid) {
    Digits dg[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) dg[c] = prepare_digits(x[c], e);
    const uint64_t b01 = signed_bias(dg[0].neg, dg[1].neg), b23 = signed_bias(dg[2].neg, dg[3].neg);
    for (int t = 1; t <= s; ++t) {
        uint32_t d[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) d[c] = digit_bits(dg[c], bits, t);
        put4(out, bf16x2_of_digits(d[0], d[1], b01), bf16x2_of_digits(d[2], d[3], b23), full, valid);
        out += slice_stride;
    }
}

// Fixed digit width and count known at compile time with BITS * S <= 63: the integer
// F = floor(|v| 2^(BITS S - e)) < 2^(BITS S) holds all S digits (digit t is bits
// BITS (S - t) .. BITS (S - t + 1) - 1 of F), the same digits as digit_bits gives.
template <int BITS, int S>
__device__ __forceinline__ uint64_t digits_word(double val, int e, uint32_t& neg) {
    static_assert(BITS * S <= 63, "all digits must fit one 64-bit word");
    const uint64_t u = uint64_t(__double_as_longlong(val));
    neg = uint32_t(u >> 63);
    int E = int((u >> 52) & 0x7FF);
    uint64_t mag = u & ((uint64_t(1) << 52) - 1);
    if (E != 0) mag |= uint64_t(1) << 52; else E = 1;
    if (e == INT_MIN) return 0;
    const int sh = E - 1075 - e + BITS * S;
    if (sh >= 0) return sh >= 64 ? 0 : (mag << sh);
    return -sh >= 64 ? 0 : (mag >> -sh);
}

template <int BITS, int S>
__device__ __forceinline__ void slice_store4_fixed(const double (&x)[4], int e, uint16_t* out, int64_t slice_stride,
                                                   bool full, int valid) {
    constexpr uint32_t MASK = (1u << BITS) - 1u;
    uint64_t F[4];
    uint32_t ng[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) F[c] = digits_word<BITS, S>(x[c], e, ng[c]);
    const uint64_t b01 = signed_bias(ng[0], ng[1]), b23 = signed_bias(ng[2], ng[3]);
#pragma unroll
    for (int t = 1; t <= S; ++t) {
        uint32_t d[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) d[c] = uint32_t(F[c] >> (BITS * (S - t))) & MASK;
        put4(out + int64_t(t - 1) * slice_stride, bf16x2_of_digits(d[0], d[1], b01), bf16x2_of_digits(d[2], d[3], b23),
             full, valid);
    }
}

// BITS = 0: digit width and count from the arguments; else the compile-time form
template <int BITS, int S>
__device__ __forceinline__ void slice_store4_as(const double (&x)[4], int e, int bits, int s, uint16_t* out,
                                                int64_t slice_stride, bool full, int valid) {
    if constexpr (BITS > 0) slice_store4_fixed<BITS, S>(x, e, out, slice_stride, full, valid);
    else slice_store4(x, e, bits, s, out, slice_stride, full, valid);
}
// The choice of stores made once for all digits: inside the digit loop it cost 4 to 8% of a v-contiguous
// real split (in the complex one, with its four groups of places, two unrolled forms cost more, 3%)
template <int BITS, int S>
__device__ __forceinline__ void slice_store4_any(const double (&x)[4], int e, int bits, int s, uint16_t* out,
                                                 int64_t slice_stride, bool vec) {
    if (vec) slice_store4_as<BITS, S>(x, e, bits, s, out, slice_stride, true, 4);
    else slice_store4_as<BITS, S>(x, e, bits, s, out, slice_stride, false, 4);
}

// ---------------------------------------------------------------------------
// The split of one operand.  nv lines of nw entries; `v_contig`: entry (v, w) at M[v + w ld],
// else at M[w + v ld].  Real: slices of line v in row v (SliceRow), entries nw..ldq-1 zero.
//
// Complex (Section 7: the method on complex data): the complex product op(A) op(B) is the real
// product A' B'' of
//   A'  = [Re op(A), Im op(A)]                              m x 2k
//   B'' = [[Re op(B), Im op(B)], [-Im op(B), Re op(B)]]     2k x 2n
// whose first n columns are Re(op(A) op(B)) and last n are Im(op(A) op(B)).  Each line (row of
// op(A), column of op(B)) gets one exponent from the largest real or imaginary part.  A line of
// nw entries fills row v with [Re, Im] (A') or row v with [Re, -Im] and row nv + v with [Im, Re]
// (B''), 2 nw values and zeros up to ldq.
//
// Three schedules:
//  * w contiguous, one pass: one to eight warps hold a line in registers (real, seven digits of seven
//    bits, up to 8 x 4 values a thread), or a CTA in shared memory (complex, three CTAs an SM), take
//    its exponent and slice it.
//  * w contiguous, two passes (scan_w, slice_w): other digits, and longer lines.  In one pass the
//    shifts of general digits ran at two CTAs an SM, and a line that did not fit was read again in one
//    serial chain: us, one pass -> two: 8192^2, eight digits of six bits 739 -> 448, 12000^2 964 -> 638,
//    1024^2 six bits 23.9 -> 11.5; complex 16 x 4096 x 8000 (whole product) 1880 -> 1520.
//  * v contiguous: a cluster of 1 to 8 CTAs shares 32 or 128 lines and scans a part of w each; the
//    maxima meet in distributed shared memory.  A second kernel slices tiles of 64 w x 32 lines,
//    transposed through shared memory.  (As a programmatic dependent it was slower, 14.2 against 10.4 us
//    at 1000 x 900.  Slicing in the scanning cluster, the lines read again from L2, was slower from
//    2048 x 4096 on: 339 against 323 us at 8192^2.)
// All kernels of the form but the slicing ones and long products are programmatic dependents of the one
// before them (pdl_launch), and the products let theirs start only at their end (from the start on:
// 2 us more at 300 x 400 x 500).  Us a call, eager, before -> now: 128^3 23.2 -> 17.4 (op(A) = T) and 37.4 -> 25.7
// (N), 300 x 400 x 500 33.3 -> 25.4 and 46.0 -> 34, 1000 x 1200 x 900 77.6 -> 69.5 and 89.8 -> 79.
// Bound by DRAM at large sizes (8 bytes in, 2 s bytes out for each value) and by launches at small
// ones: an operand took four launches before (initialise the exponents, scan, slice, fix up), the
// scan read everything once more, and complex rows of odd length were stored two bytes at a
// time.  Before -> now, seven slices of seven bits, us in a row in a CUDA graph: w contiguous
// 8192^2 300 -> 247 (6.0 TB/s), 4096^2 81 -> 68, 1000 x 900 8.9 -> 5.3; v contiguous 1000 x 900
// 15.6 -> 9.9, 5000 x 300 14.2 -> 12.3, 4096^2 91 -> 93, 8192^2 326 -> 333, 20000 x 2000 197 -> 206
// (1256 scanning CTAs are two waves and a bit); both operands of a complex 1500 x 1100 x 2301
// product 190 -> 76.
// ---------------------------------------------------------------------------
constexpr int SPLIT_CLUSTER = 8;   // most CTAs that share 32 or 128 v-contiguous lines, or a w-contiguous one
constexpr int SPLIT_HELD = 8;      // chunks of four values a thread holds (real, w contiguous)

struct SplitJob {
    const double* M;               // complex: pairs of doubles
    int64_t ld, nv, nw;
    int32_t* expo;
    uint16_t* q;                   // of line 0
    int64_t ldq, plane;
    int64_t wt, block, tail;       // columns in blocks of 64, pitch of those, pitch of rows in the rest
    int64_t tail_at;               // the rest from here
    bool blocked;                  // else row-major, pitch ldq
    int v_contig, conj, role_b;
    int vec_in, vec_out;           // 16-byte loads (real, w contiguous); 8-byte stores
    int warps;                     // w contiguous, real: warps per line (1, 2, 4 or 8)
    int two_pass, group;           // w contiguous, real: scan and slice (scan_w, slice_w), threads of a line there
    unsigned pieces;               // slicing kernels: CTAs along w (a block index divides in 32 bits: with 64 the
                                   // slicing took 4 to 8% longer)
    unsigned blocks;
};

// Row v of slice 1 (see Slices; BLOCKED: in blocks of 64 columns), whose entries up to the next
// multiple of 64 are consecutive.  A kernel of its own for each: the address arithmetic of the blocks
// cost 2 to 7% (complex 4096^2, v contiguous, 481 -> 510 us with the product by 16 columns).
template <bool BLOCKED>
struct SliceRow {
    uint16_t *blocks, *tail;       // tail: where entry 0 would be if the row had the tail's pitch throughout
    int64_t block;
    int wt;
    __device__ __forceinline__ SliceRow(const SplitJob& j, int64_t v)
        : blocks(j.q + v * (BLOCKED ? 64 : j.ldq)), tail(j.q + j.tail_at + v * j.tail - j.wt), block(j.block),
          wt(int(j.wt)) {}
    __device__ __forceinline__ uint16_t* at(int64_t w) const {
        if constexpr (BLOCKED) return int(w) < wt ? blocks + (int(w) >> 6) * block + (int(w) & 63) : tail + int(w);
        else return blocks + w;
    }
};

__device__ __forceinline__ uint64_t warp_mag_max(uint64_t mx) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) mx = mag_max(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    return mx;
}
// exponent of a line as stored: 0 for an all-zero line (its digits are zero for any exponent)
__device__ __forceinline__ int stored_exponent(uint64_t mx) {
    const int e = line_exponent_bits(mx);
    return e == INT_MIN ? 0 : e;
}

__device__ __forceinline__ uint64_t ld_cluster_u64(uint32_t addr) {
    uint64_t v;
    asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(addr) : "memory");
    return v;
}

// four values w .. w+3 of a w-contiguous real line, zero from nw on
__device__ __forceinline__ void load4(const double* line, int64_t w, int64_t nw, bool vec, double (&x)[4]) {
    if (vec && w + 4 <= nw) {
        const double2 a = __ldcs(reinterpret_cast<const double2*>(line + w));
        const double2 b = __ldcs(reinterpret_cast<const double2*>(line + w + 2));
        x[0] = a.x; x[1] = a.y; x[2] = b.x; x[3] = b.y;
    } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) x[c] = (w + c < nw) ? __ldcs(line + w + c) : 0.0;
    }
}

// exponent of the line from the halfwise maxima of the 32 WL threads that share it (a CTA of eight
// warps holds 8 / WL lines; `red` has eight entries)
__device__ __forceinline__ uint64_t line_mag_max(uint64_t mx, int WL, uint64_t* red) {
    mx = warp_mag_max(mx);
    if (WL > 1) {
        if (lane_id() == 0) red[warp_id()] = mx;
        __syncthreads();
        const int w0 = int(warp_id()) / WL * WL;
        for (int i = 0; i < WL; ++i) mx = mag_max(mx, red[w0 + i]);
    }
    return mx;
}

template <int BITS, int S, bool BLOCKED>
__device__ __forceinline__ void split_w_real(const SplitJob& j, int64_t block, int bits, int s) {
    __shared__ uint64_t red[8];
    const int WL = j.warps, G = 32 * WL, t = int(threadIdx.x) & (G - 1);
    const int64_t v = block * (8 / WL) + warp_id() / WL;
    const bool live = v < j.nv;                             // the same in every warp of a line
    if (WL == 1 && !live) return;
    const double* line = j.M + (live ? v : 0) * j.ld;
    const int64_t step = 4 * G;
    const bool vec = j.vec_in != 0;
    double x[SPLIT_HELD][4];
    uint64_t mx = 0;
#pragma unroll
    for (int c = 0; c < SPLIT_HELD; ++c)
        if (c * step < j.nw) load4(line, c * step + 4 * t, j.nw, vec, x[c]);
#pragma unroll
    for (int c = 0; c < SPLIT_HELD; ++c)
        if (c * step < j.nw) {
#pragma unroll
            for (int i = 0; i < 4; ++i) mx = mag_max(mx, mag_bits(x[c][i]));
        }
    mx = line_mag_max(mx, WL, red);
    if (!live) return;
    const int e = stored_exponent(mx);
    if (t == 0) j.expo[v] = e;
    const SliceRow<BLOCKED> out(j, v);
#pragma unroll
    for (int c = 0; c < SPLIT_HELD; ++c) {
        const int64_t w = c * step + 4 * t;
        if (c * step >= j.nw) {
#pragma unroll
            for (int i = 0; i < 4; ++i) x[c][i] = 0.0;
        }
        if (w < j.ldq) slice_store4_any<BITS, S>(x[c], e, bits, s, out.at(w), j.plane, j.vec_out != 0);
    }
}

// Exponents of w-contiguous lines, 1 to 8 warps each (complex: 8), or all warps of the CTAs of a cluster
template <bool CPLX>
__device__ __forceinline__ void scan_w(const SplitJob& j, int64_t block) {
    __shared__ uint64_t red[8], cmax;
    const int rank = int(cluster_ctarank()), CS = int(cluster_nctarank());
    const int WL = CPLX ? 8 : j.warps, t = int(threadIdx.x) & (32 * WL - 1);
    const int64_t v = block / CS * (8 / WL) + warp_id() / WL;
    const bool live = v < j.nv;
    const double* line = j.M + (CPLX ? 2 : 1) * (live ? v : 0) * j.ld;
    const int64_t part = ((j.nw + CS - 1) / CS + 3) / 4 * 4, w0 = rank * part, w1 = live ? min(j.nw, w0 + part) : 0;
    uint64_t mx = 0;
    if constexpr (CPLX) {
        for (int64_t w = w0 + t; w < w1; w += 256 * 8) {
            double2 x[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                x[u] = w + 256 * u < w1 ? reinterpret_cast<const double2*>(line)[w + 256 * u] : make_double2(0.0, 0.0);
#pragma unroll
            for (int u = 0; u < 8; ++u) mx = mag_max(mx, mag_max(mag_bits(x[u].x), mag_bits(x[u].y)));
        }
    } else {
        const int64_t step = 128 * WL;
        for (int64_t w = w0 + 4 * t; w < w1; w += 4 * step) {
            double x[4][4];
#pragma unroll
            for (int u = 0; u < 4; ++u) load4(line, w + u * step, w1, j.vec_in != 0, x[u]);
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int i = 0; i < 4; ++i) mx = mag_max(mx, mag_bits(x[u][i]));
        }
    }
    mx = line_mag_max(mx, WL, red);
    if (CS == 1) {
        if (t == 0 && live) j.expo[v] = stored_exponent(mx);
        return;
    }
    if (threadIdx.x == 0) cmax = mx;        // WL = 8: the CTA's part of one line
    __syncwarp();
    cluster_sync_all();
    if (rank == 0 && threadIdx.x == 0) {
        for (int r = 1; r < CS; ++r) mx = mag_max(mx, ld_cluster_u64(mapa_shared(smem_u32(&cmax), uint32_t(r))));
        j.expo[v] = stored_exponent(mx);
    }
    __syncwarp();
    cluster_sync_all();                     // no CTA leaves while rank 0 may still read its maximum
}

// digits of four entries a thread, j.group threads to a line (of up to 1024 entries of it)
template <int BITS, int S, bool BLOCKED>
__device__ __forceinline__ void slice_w(const SplitJob& j, unsigned block, int bits, int s) {
    const int t = int(threadIdx.x) & (j.group - 1), lines = 256 / j.group;
    const unsigned row = block / j.pieces, piece = block - row * j.pieces;
    const int64_t v = int64_t(row) * lines + int(threadIdx.x) / j.group, w = (int64_t(piece) * j.group + t) * 4;
    if (v >= j.nv || w >= j.ldq) return;
    double x[4];
    load4(j.M + v * j.ld, w, j.nw, j.vec_in != 0, x);
    slice_store4_any<BITS, S>(x, j.expo[v], bits, s, SliceRow<BLOCKED>(j, v).at(w), j.plane, j.vec_out != 0);
}

// which part (0 real, 1 imaginary) of which entry stands at position p < 2 nw of row kind `second`
// (B'' rows nv + v), and whether negated
__device__ __forceinline__ int zpart_at(const SplitJob& j, int64_t p, bool second, int64_t& w, bool& flip) {
    const bool right = p >= j.nw;
    w = right ? p - j.nw : p;
    flip = right && j.role_b && !second;                    // -Im
    return int(right) ^ int(second);
}

// place of entry w in a cached line: four consecutive entries per lane without bank conflicts
__host__ __device__ __forceinline__ int cache_at(int w) { return w + (w >> 4); }

template <int BITS, int S, bool BLOCKED>
__device__ __forceinline__ void split_w_complex(const SplitJob& j, int64_t v, int bits, int s, double* cache) {
    __shared__ uint64_t red[8];
    const int t = int(threadIdx.x);
    const double2* line = reinterpret_cast<const double2*>(j.M) + v * j.ld;
    const int half = cache_at(int(j.nw)) + 1;                     // imaginary parts from here on
    uint64_t mx = 0;
    for (int64_t w0 = t; w0 < j.nw; w0 += 256 * 8) {
        double2 a[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) a[u] = w0 + 256 * u < j.nw ? line[w0 + 256 * u] : make_double2(0.0, 0.0);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int64_t w = w0 + 256 * u;
            mx = mag_max(mx, mag_max(mag_bits(a[u].x), mag_bits(a[u].y)));
            if (w < j.nw) {
                cache[cache_at(int(w))] = a[u].x;
                cache[half + cache_at(int(w))] = j.conj ? -a[u].y : a[u].y;
            }
        }
    }
    const int e = stored_exponent(line_mag_max(mx, 8, red));
    if (t == 0) j.expo[v] = e;
    const int64_t nw = j.nw;
    for (int second = 0; second <= (j.role_b ? 1 : 0); ++second) {
        const SliceRow<BLOCKED> out(j, second ? j.nv + v : v);
        for (int64_t p = 4 * t; p < j.ldq; p += 1024) {
            double x[4];
            const bool left = p + 4 <= nw, right = p >= nw && p + 4 <= 2 * nw;
            if (left || right) {                            // all four from one half of the row
                const int part = int(right) ^ second, w = int(right ? p - nw : p);
                const bool flip = right && j.role_b && second == 0;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const double y = cache[part * half + cache_at(w + c)];
                    x[c] = flip ? -y : y;
                }
            } else {
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    x[c] = 0.0;
                    if (p + c < 2 * nw) {
                        int64_t w;
                        bool flip;
                        const int part = zpart_at(j, p + c, second != 0, w, flip);
                        const double y = cache[part * half + cache_at(int(w))];
                        x[c] = flip ? -y : y;
                    }
                }
            }
            slice_store4_as<BITS, S>(x, e, bits, s, out.at(p), j.plane, true, 4);    // a workspace's slices are aligned
        }
    }
}

// digits of up to 1024 entries of a complex line, in the two places (A') or four (B'') they occupy
template <int BITS, int S, bool BLOCKED>
__device__ __forceinline__ void slice_w_complex(const SplitJob& j, unsigned block, int bits, int s) {
    __shared__ double part[2][1024 + 64];
    const unsigned row = block / j.pieces;
    const int64_t v = row, w0 = int64_t(block - row * j.pieces) * 1024;
    const int n = int(min(int64_t(1024), j.nw - w0)), t = int(threadIdx.x);
    const double2* line = reinterpret_cast<const double2*>(j.M) + v * j.ld + w0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int w = t + 256 * u;
        const double2 a = w < n ? __ldcs(line + w) : make_double2(0.0, 0.0);
        part[0][cache_at(w)] = a.x;
        part[1][cache_at(w)] = j.conj ? -a.y : a.y;
    }
    __syncthreads();
    const int e = j.expo[v];
    const SliceRow<BLOCKED> row1(j, v), row2(j, j.role_b ? j.nv + v : v);
    // part q to positions pos .. of a row, four at a time from the first multiple of four on
    const auto emit = [&](int q, const SliceRow<BLOCKED>& out, int64_t pos, bool flip) {
        const int lead = j.vec_out ? min(n, int(-pos & 3)) : 0;
        const auto group = [&](int first, int valid) {
            double x[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const double y = c < valid ? part[q][cache_at(first + c)] : 0.0;
                x[c] = flip ? -y : y;
            }
            slice_store4_as<BITS, S>(x, e, bits, s, out.at(pos + first), j.plane, j.vec_out && valid == 4, valid);
        };
        const int first = lead + 4 * t;
        if (first < n) group(first, min(4, n - first));
        if (lead > 0 && t == 255) group(0, lead);
    };
    emit(0, row1, w0, false);
    emit(1, row1, j.nw + w0, j.role_b != 0);
    if (j.role_b) {
        emit(1, row2, w0, false);
        emit(0, row2, j.nw + w0, false);
    }
    if (w0 == 0)                   // zeros from 2 nw to ldq
        for (int64_t p = 2 * j.nw + t; p < j.ldq; p += 256)
            for (int q = 0; q < s; ++q) {
                row1.at(p)[int64_t(q) * j.plane] = 0;
                if (j.role_b) row2.at(p)[int64_t(q) * j.plane] = 0;
            }
}

// entries [w0, w0 + n) of line vl of a tile (n <= 64, column v of row w at (v + w / 4) % 32) to
// positions base + w0 .. of its row, four at a time from the first position that is a multiple
// of four; thread wq of 16.  The entries before it and the last partial group go one by one.
template <int BITS, int S, bool BLOCKED>
__device__ __forceinline__ void emit_tile_row(const SplitJob& j, const double (*tile)[32], int vl, int wq, int n,
                                              int64_t pos, const SliceRow<BLOCKED>& row, int e, bool flip, int bits, int s) {
    const int lead = j.vec_out ? min(n, int(-pos & 3)) : 0;
    auto group = [&](int first, int valid) {
        double x[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int r = first + c;
            const double y = c < valid ? tile[r & 63][(vl + ((r & 63) >> 2)) & 31] : 0.0;
            x[c] = flip ? -y : y;
        }
        slice_store4_as<BITS, S>(x, e, bits, s, row.at(pos + first), j.plane, j.vec_out && valid == 4, valid);
    };
    const int first = lead + 4 * wq;
    if (first < n) group(first, min(4, n - first));
    if (lead > 0 && wq == 15) group(0, lead);
}

// Exponents of 2 LX v-contiguous lines: a cluster shares them, each CTA scans its part of w, LX
// lanes with two lines each by 256 / LX entries at a time.  Loads come in batches, the last one
// predicated (a remainder loop would take them one by one).  Six real loads a batch let four CTAs share
// an SM; with eight (78 registers, three CTAs) the 512 CTAs of 8192 lines took two waves, 96 -> 79 us.
template <int LX, bool CPLX>
__device__ __forceinline__ void scan_v(const SplitJob& j, int64_t block) {
    constexpr int R = 256 / LX, U = CPLX ? 4 : 6;
    __shared__ uint64_t red[R][2 * LX], cmax[2 * LX];
    const int rank = int(cluster_ctarank()), CS = int(cluster_nctarank());
    const int tx = int(threadIdx.x) % LX, ty = int(threadIdx.x) / LX;
    const int64_t v0 = block / CS * (2 * LX), v = v0 + 2 * tx;
    const int64_t part = (j.nw + CS - 1) / CS, w0 = rank * part, w1 = min(j.nw, w0 + part);
    const bool two = v + 1 < j.nv, vec = two && j.vec_in;
    uint64_t ma = 0, mb = 0;
    const int64_t step = R * j.ld;
    if (v < j.nv) {
        const auto batch = [&](auto full, int64_t w) {
            constexpr bool FULL = decltype(full)::value;
            const double* p = j.M + (CPLX ? 2 : 1) * (v + w * j.ld);
            if constexpr (CPLX) {
                double2 x[U], y[U];
#pragma unroll
                for (int u = 0; u < U; ++u, p += 2 * step) {
                    const bool in = FULL || w + R * u < w1;
                    x[u] = in ? reinterpret_cast<const double2*>(p)[0] : make_double2(0.0, 0.0);
                    y[u] = in && two ? reinterpret_cast<const double2*>(p)[1] : make_double2(0.0, 0.0);
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    ma = mag_max(ma, mag_max(mag_bits(x[u].x), mag_bits(x[u].y)));
                    mb = mag_max(mb, mag_max(mag_bits(y[u].x), mag_bits(y[u].y)));
                }
            } else {
                double2 x[U];
#pragma unroll
                for (int u = 0; u < U; ++u, p += step) {
                    const bool in = FULL || w + R * u < w1;
                    if (in && vec) x[u] = *reinterpret_cast<const double2*>(p);
                    else x[u] = make_double2(in ? p[0] : 0.0, in && two ? p[1] : 0.0);
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    ma = mag_max(ma, mag_bits(x[u].x));
                    mb = mag_max(mb, mag_bits(x[u].y));
                }
            }
        };
        int64_t w = w0 + ty;
        for (; w + R * (U - 1) < w1; w += R * U) batch(std::true_type{}, w);
        if (w < w1) batch(std::false_type{}, w);
    }
    red[ty][2 * tx] = ma;
    red[ty][2 * tx + 1] = mb;
    __syncthreads();
    const int t = int(threadIdx.x);
    uint64_t mx = 0;
    if (t < 2 * LX) {
#pragma unroll
        for (int i = 0; i < R; ++i) mx = mag_max(mx, red[i][t]);
        cmax[t] = mx;
    }
    __syncwarp();
    cluster_sync_all();
    if (rank == 0 && t < 2 * LX) {
        for (int r = 1; r < CS; ++r) mx = mag_max(mx, ld_cluster_u64(mapa_shared(smem_u32(&cmax[t]), uint32_t(r))));
        if (v0 + t < j.nv) j.expo[v0 + t] = stored_exponent(mx);
    }
    __syncwarp();
    cluster_sync_all();            // no CTA leaves while rank 0 may still read its maxima
}

// one tile of 64 w x 32 v-contiguous lines, transposed through shared memory
template <int BITS, int S, bool CPLX, bool BLOCKED>
__device__ __forceinline__ void slice_v(const SplitJob& j, unsigned block, int bits, int s) {
    // column v of row w at (v + w / 4) % 32: conflict-free both along v and for the four
    // consecutive w a thread slices
    __shared__ double tile[CPLX ? 2 : 1][64][32];
    const int tx = int(threadIdx.x) & 31, ty = int(threadIdx.x) >> 5;   // 32 x 8
    const int64_t len = CPLX ? j.nw : j.ldq;        // a real row's padding belongs to its last entries
    const unsigned row = block / j.pieces;
    const int64_t w0 = int64_t(block - row * j.pieces) * 64, v0 = int64_t(row) * 32, v = v0 + tx;
    const int n = int(min(int64_t(64), len - w0));
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int wl = ty + 8 * i;
        const int64_t w = w0 + wl;
        const bool in = v < j.nv && w < j.nw;
        const int col = (tx + (wl >> 2)) & 31;
        if constexpr (CPLX) {
            const double2 a = in ? __ldcs(reinterpret_cast<const double2*>(j.M) + v + w * j.ld) : make_double2(0.0, 0.0);
            tile[0][wl][col] = a.x;
            tile[CPLX ? 1 : 0][wl][col] = j.conj ? -a.y : a.y;
        } else {
            tile[0][wl][col] = in ? __ldcs(j.M + v + w * j.ld) : 0.0;
        }
    }
    __syncthreads();
    const int wq = int(threadIdx.x) & 15, vh = int(threadIdx.x) >> 4;   // 16 x 16
#pragma unroll 1
    for (int r = 0; r < 2; ++r) {
        const int vl = vh + 16 * r;
        if (v0 + vl >= j.nv) continue;
        const int e = j.expo[v0 + vl];
        const SliceRow<BLOCKED> row(j, v0 + vl);
        if constexpr (CPLX) {
            constexpr int IM = CPLX ? 1 : 0;
            emit_tile_row<BITS, S, BLOCKED>(j, tile[0], vl, wq, n, w0, row, e, false, bits, s);
            emit_tile_row<BITS, S, BLOCKED>(j, tile[IM], vl, wq, n, j.nw + w0, row, e, j.role_b != 0, bits, s);
            if (j.role_b) {
                const SliceRow<BLOCKED> row2(j, j.nv + v0 + vl);
                emit_tile_row<BITS, S, BLOCKED>(j, tile[IM], vl, wq, n, w0, row2, e, false, bits, s);
                emit_tile_row<BITS, S, BLOCKED>(j, tile[0], vl, wq, n, j.nw + w0, row2, e, false, bits, s);
            }
        } else if (4 * wq < n) {
            double x[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) x[c] = tile[0][4 * wq + c][(vl + wq) & 31];
            slice_store4_any<BITS, S>(x, e, bits, s, row.at(w0 + 4 * wq), j.plane, j.vec_out != 0);
        }
    }
    if constexpr (CPLX) {          // zeros from 2 nw to ldq
        if (w0 == 0 && v < j.nv)
            for (int64_t p = 2 * j.nw + ty; p < j.ldq; p += 8)
                for (int t = 0; t < s; ++t)
                    for (int second = 0; second <= (j.role_b ? 1 : 0); ++second)
                        SliceRow<BLOCKED>(j, (second ? j.nv : 0) + v).at(p)[int64_t(t) * j.plane] = 0;
    }
}

// Blocks 0 .. j0.blocks - 1 split the first operand, the rest the second.
template <int BITS, int S, bool CPLX, bool BLOCKED>
__global__ void __launch_bounds__(256, CPLX ? 4 : 2) ozaki_split_w_kernel(SplitJob j0, SplitJob j1, int bits, int s) {
    extern __shared__ double cache[];
    pdl_wait();
    pdl_trigger();
    const bool first = blockIdx.x < j0.blocks;
    const SplitJob& j = first ? j0 : j1;
    const int64_t block = first ? blockIdx.x : blockIdx.x - j0.blocks;
    if constexpr (CPLX) split_w_complex<BITS, S, BLOCKED>(j, block, bits, s, cache);
    else split_w_real<BITS, S, BLOCKED>(j, block, bits, s);
}
template <bool CPLX>
__global__ void __launch_bounds__(256) ozaki_scan_w_kernel(SplitJob j0, SplitJob j1) {
    pdl_wait();
    const bool first = blockIdx.x < j0.blocks;
    scan_w<CPLX>(first ? j0 : j1, first ? blockIdx.x : blockIdx.x - j0.blocks);
}
template <int BITS, int S, bool CPLX, bool BLOCKED>
__global__ void __launch_bounds__(256) ozaki_slice_w_kernel(SplitJob j0, SplitJob j1, int bits, int s) {
    pdl_trigger();
    const bool first = blockIdx.x < j0.blocks;
    const SplitJob& j = first ? j0 : j1;
    const unsigned block = first ? blockIdx.x : blockIdx.x - j0.blocks;
    if constexpr (CPLX) slice_w_complex<BITS, S, BLOCKED>(j, block, bits, s);
    else slice_w<BITS, S, BLOCKED>(j, block, bits, s);
}
template <int LX, bool CPLX>
__global__ void __launch_bounds__(256) ozaki_scan_v_kernel(SplitJob j0, SplitJob j1) {
    pdl_wait();
    const bool first = blockIdx.x < j0.blocks;
    scan_v<LX, CPLX>(first ? j0 : j1, first ? blockIdx.x : blockIdx.x - j0.blocks);
}
template <int BITS, int S, bool CPLX, bool BLOCKED>
__global__ void __launch_bounds__(256, CPLX ? 5 : BITS > 0 ? 8 : 5) ozaki_slice_v_kernel(SplitJob j0, SplitJob j1, int bits, int s) {
    pdl_trigger();
    const bool first = blockIdx.x < j0.blocks;
    slice_v<BITS, S, CPLX, BLOCKED>(first ? j0 : j1, first ? blockIdx.x : blockIdx.x - j0.blocks, bits, s);
}

}  // namespace

namespace {

// G 2^P as a double for an integer |G| < 2^53 (so double(G) is exact), built from
// integer operations: the exponent field takes P directly, no FP64 arithmetic.
// Results outside the normal range go through ldexp (exact or correctly rounded).
__device__ __forceinline__ double scaled_int(int64_t G, int P) {
    if (G == 0) return 0.0;
    const uint64_t neg = G < 0 ? 1u : 0u;
    const uint64_t mag = uint64_t(G < 0 ? -G : G);
    const int top = 63 - __clzll(int64_t(mag));                       // 0..52
    const int ef = top + P + 1023;
    if (ef < 1 || ef > 2046) return ldexp(double(G), P);
    const uint64_t mant = (mag << (52 - top)) & ((uint64_t(1) << 52) - 1);
    return __longlong_as_double(int64_t((neg << 63) | (uint64_t(ef) << 52) | mant));
}

// C_ij = alpha 2^(e_i + f_j) sum_{d=2}^{s+1} 2^(-bits d) S_d(i,j) + beta C_ij.
// Consecutive anti-diagonals are first combined exactly in INT64,
//   G = sum_{d=dl}^{dh} S_d 2^(bits (dh - d)),  |G| < 2^(31 + bits (g-1) + 1) <= 2^53,
// so G 2^(e_i + f_j - bits dh) is an exact double and each group costs one FP64
// addition (smallest group first).
// Complex: Re and Im of op(A) op(B) are columns j and n + j of the real form's S_d; C = alpha
// (Re + i Im) + beta C, alpha and beta complex.
//
// V rows per thread: 4 with 16-byte loads of every S_d plane (m, the plane pitch and ldc suitably
// aligned; checked by the host), else 1.  F77: s = 7 slices of 7 bits (groups d = 5..8 and d =
// 2..4), all planes loaded before any arithmetic, the same operations in the same order as the
// general loop; a loop over the planes keeps one load in flight per thread.  Bound by DRAM (4 s
// bytes in and 8 out per real element).
template <int V>
__device__ __forceinline__ void load_sums(const int32_t* p, int (&v)[V]) {
    if constexpr (V == 4) {
        const int4 x = __ldcs(reinterpret_cast<const int4*>(p));
        v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
    } else {
        v[0] = __ldcs(p);
    }
}

// the sums of V rows of one column, scaled by 2^E0[c]
template <int V, bool F77>
__device__ __forceinline__ void combine(const int32_t* p, int64_t plane, int s, int bits, int gsize, const int (&E0)[V],
                                        double (&acc)[V]) {
    if constexpr (F77) {
        int v[7][V];
#pragma unroll
        for (int d = 2; d <= 8; ++d) load_sums<V>(p + int64_t(d - 2) * plane, v[d - 2]);
#pragma unroll
        for (int c = 0; c < V; ++c) {
            int64_t G1 = 0, G2 = 0;
#pragma unroll
            for (int d = 5; d <= 8; ++d) G1 = G1 * 128 + int64_t(v[d - 2][c]);
#pragma unroll
            for (int d = 2; d <= 4; ++d) G2 = G2 * 128 + int64_t(v[d - 2][c]);
            acc[c] = scaled_int(G1, E0[c] - 7 * 8) + scaled_int(G2, E0[c] - 7 * 4);
        }
    } else {
        for (int dh = s + 1; dh >= 2; dh -= gsize) {
            const int dl = dh - gsize + 1 > 2 ? dh - gsize + 1 : 2;
            int64_t G[V];
#pragma unroll
            for (int c = 0; c < V; ++c) G[c] = 0;
            for (int d = dl; d <= dh; ++d) {
                int v[V];
                load_sums<V>(p + int64_t(d - 2) * plane, v);
#pragma unroll
                for (int c = 0; c < V; ++c) G[c] = G[c] * (int64_t(1) << bits) + int64_t(v[c]);
            }
#pragma unroll
            for (int c = 0; c < V; ++c) {
                const double gv = scaled_int(G[c], E0[c] - bits * dh);
                acc[c] = (dh == s + 1) ? gv : acc[c] + gv;      // the first group needs no FP64 addition
            }
        }
    }
}

struct RecombineArgs {
    int64_t m, n;
    int s, bits, gsize;
    const int32_t* sd;
    int64_t plane;
    const int32_t *ea, *eb;
    double2 alpha, beta;        // real: the first component
    double* C;                  // complex: pairs
    int64_t ldc;
};

template <int V, bool F77, bool CPLX>
__global__ void __launch_bounds__(256) ozaki_recombine_kernel(RecombineArgs g) {
    pdl_wait();
    pdl_trigger();
    const int64_t i = (int64_t(blockIdx.x) * 256 + threadIdx.x) * V;
    if (i >= g.m) return;
    int ei[V];
    if constexpr (V == 4) {
        const int4 e = *reinterpret_cast<const int4*>(g.ea + i);
        ei[0] = e.x; ei[1] = e.y; ei[2] = e.z; ei[3] = e.w;
    } else {
        ei[0] = g.ea[i];
    }
    for (int64_t j = blockIdx.y; j < g.n; j += gridDim.y) {
        const int fj = g.eb[j];
        int E0[V];
#pragma unroll
        for (int c = 0; c < V; ++c) E0[c] = ei[c] + fj;
        double re[V];
        combine<V, F77>(g.sd + i + j * g.m, g.plane, g.s, g.bits, g.gsize, E0, re);
        if constexpr (CPLX) {
            double im[V];
            combine<V, F77>(g.sd + i + (g.n + j) * g.m, g.plane, g.s, g.bits, g.gsize, E0, im);
            double2* cp = reinterpret_cast<double2*>(g.C) + i + j * g.ldc;
#pragma unroll
            for (int c = 0; c < V; ++c) {
                double vr = g.alpha.x * re[c] - g.alpha.y * im[c];
                double vi = g.alpha.x * im[c] + g.alpha.y * re[c];
                if (g.beta.x != 0.0 || g.beta.y != 0.0) {
                    const double2 c0 = cp[c];
                    vr = fma(g.beta.x, c0.x, fma(-g.beta.y, c0.y, vr));
                    vi = fma(g.beta.x, c0.y, fma(g.beta.y, c0.x, vi));
                }
                cp[c] = make_double2(vr, vi);
            }
        } else {
            double* cp = g.C + i + j * g.ldc;
#pragma unroll
            for (int c = 0; c < V; ++c) re[c] = (g.alpha.x == 1.0) ? re[c] : g.alpha.x * re[c];
            if constexpr (V == 4) {
                double2* c2 = reinterpret_cast<double2*>(cp);
                if (g.beta.x != 0.0) {
                    const double2 a = c2[0], b = c2[1];
                    re[0] = fma(g.beta.x, a.x, re[0]); re[1] = fma(g.beta.x, a.y, re[1]);
                    re[2] = fma(g.beta.x, b.x, re[2]); re[3] = fma(g.beta.x, b.y, re[3]);
                }
                c2[0] = make_double2(re[0], re[1]);
                c2[1] = make_double2(re[2], re[3]);
            } else {
                if (g.beta.x != 0.0) re[0] = fma(g.beta.x, cp[0], re[0]);
                cp[0] = re[0];
            }
        }
    }
}

template <bool CPLX>
hsmm_status_t launch_recombine(const RecombineArgs& g, cudaStream_t st) {
    // complex C is 16-byte aligned by its type; a real one needs an even ldc for 16-byte stores
    const bool vec4 = g.m % 4 == 0 && g.plane % 4 == 0 && aligned_to(g.sd, 16) && aligned_to(g.ea, 16) &&
                      aligned_to(g.C, 16) && (CPLX || g.ldc % 2 == 0);
    const bool f77 = g.s == 7 && g.bits == 7;
    const dim3 grid(unsigned(((vec4 ? g.m / 4 : g.m) + 255) / 256), unsigned(g.n < 65535 ? g.n : 65535));
    auto kern = vec4 && f77 ? ozaki_recombine_kernel<4, true, CPLX>
                : vec4      ? ozaki_recombine_kernel<4, false, CPLX>
                : f77       ? ozaki_recombine_kernel<1, true, CPLX>
                            : ozaki_recombine_kernel<1, false, CPLX>;
    const cudaError_t e = pdl_launch(kern, grid, 256, 0, 1, st, g);
    count_launches(1);
    if (e != cudaSuccess) return record_cuda(e);
    return check_launch();
}

}  // namespace

hsmm_status_t ozaki_recombine(int64_t m, int64_t n, int slices, int bits, const int32_t* sd, int64_t sd_plane,
                              const int32_t* ea, const int32_t* eb, double alpha, double beta, double* C, int64_t ldc,
                              cudaStream_t st) {
    return launch_recombine<false>(RecombineArgs{m, n, slices, bits, 1 + 21 / bits, sd, sd_plane, ea, eb,
                                                 make_double2(alpha, 0.0), make_double2(beta, 0.0), C, ldc}, st);
}

namespace {

constexpr size_t SPLIT_CACHE = 72 * 1024;      // shared memory for a complex line: three CTAs an SM
size_t split_cache_bytes(int64_t nw) { return size_t(16) * (size_t(nw) + size_t(nw) / 16 + 1); }

hsmm_status_t make_split_job(const SplitOperand& o, bool cplx, bool fixed, SplitJob* j) {
    if (o.nv > SPLIT_MAX_LINES) return fail(HSMM_STATUS_NOT_SUPPORTED, "ozaki: an operand of more than %lld lines",
                                            static_cast<long long>(SPLIT_MAX_LINES));
    j->M = static_cast<const double*>(o.M);
    j->ld = o.ld; j->nv = o.nv; j->nw = o.nw;
    j->expo = o.expo;
    const Slices& q = o.q;
    j->ldq = q.ldq; j->plane = q.plane;
    j->q = static_cast<uint16_t*>(q.q);
    j->wt = 0; j->block = 0; j->tail = 0; j->tail_at = 0;
    j->blocked = q.block_rows > 0;
    if (!j->blocked) {
        j->q += q.row0 * q.ldq;
    } else {
        j->wt = q.ldq / 64 * 64;
        j->block = q.block_rows * 64;
        j->tail = q.ldq - j->wt;
        j->tail_at = j->wt * q.block_rows + q.row0 * (j->tail - 64);   // from q, which starts 64 row0 later
        j->q += q.row0 * 64;
    }
    j->v_contig = o.v_contig; j->conj = o.conj; j->role_b = o.role_b;
    j->vec_in = o.ld % 2 == 0 && aligned_to(o.M, 16);
    j->vec_out = q.ldq % 4 == 0 && q.plane % 4 == 0 && aligned_to(q.q, 8);
    j->warps = 1;                  // as many warps per line as hold it in their registers
    while (j->warps < 8 && q.ldq > int64_t(SPLIT_HELD) * 128 * j->warps) j->warps *= 2;
    j->two_pass = !o.v_contig && (cplx ? split_cache_bytes(o.nw) > SPLIT_CACHE : !fixed || q.ldq > int64_t(SPLIT_HELD) * 1024);
    if (cplx) j->warps = 8;
    else if (j->two_pass)          // more where there are few lines
        while (j->warps < 8 && o.nv * j->warps < int64_t(num_sms()) * 16 && q.ldq > int64_t(128) * j->warps) j->warps *= 2;
    j->group = 32;
    while (j->group < 256 && q.ldq > int64_t(4) * j->group) j->group *= 2;
    const int lines = cplx ? 1 : 8 / j->warps;     // lines of a CTA (w contiguous)
    j->blocks = unsigned((o.nv + lines - 1) / lines);
    return HSMM_STATUS_SUCCESS;
}

template <int BITS, int S, bool CPLX, bool BLOCKED>
hsmm_status_t launch_split(SplitJob a, SplitJob b, int bits, int slices, cudaStream_t st) {
    cudaError_t e = cudaSuccess;
    if (a.v_contig) {
        // 128 lines per scanning CTA (1 KiB of a row of w), 32 where that leaves SMs idle; clusters
        // so that a CTA has a batch of loads and more
        const int64_t nv = std::max(a.nv, b.nv), nw = std::max(a.nw, b.nw);
        const int lines = (nv + 127) / 128 * SPLIT_CLUSTER >= 2 * num_sms() * 4 / 5 ? 128 : 32;
        unsigned cs = 1;
        while (cs < unsigned(SPLIT_CLUSTER) && nw > int64_t(128) * cs) cs *= 2;
        const auto scan_blocks = [cs, lines](const SplitJob& j) { return unsigned((j.nv + lines - 1) / lines * cs); };
        a.pieces = unsigned(((CPLX ? a.nw : a.ldq) + 63) / 64);
        b.pieces = unsigned(((CPLX ? b.nw : b.ldq) + 63) / 64);
        const auto slice_blocks = [](const SplitJob& j) { return (j.nv + 31) / 32 * int64_t(j.pieces); };
        if (slice_blocks(a) + slice_blocks(b) > INT32_MAX) return HSMM_STATUS_NOT_SUPPORTED;
        a.blocks = scan_blocks(a);
        b.blocks = scan_blocks(b);
        e = pdl_launch(lines == 128 ? ozaki_scan_v_kernel<64, CPLX> : ozaki_scan_v_kernel<16, CPLX>,
                       dim3(a.blocks + b.blocks), 256, 0, cs, st, a, b);
        count_launches(1);
        if (e != cudaSuccess) return record_cuda(e);
        a.blocks = unsigned(slice_blocks(a));
        b.blocks = unsigned(slice_blocks(b));
        ozaki_slice_v_kernel<BITS, S, CPLX, BLOCKED><<<a.blocks + b.blocks, 256, 0, st>>>(a, b, bits, slices);
    } else if (a.two_pass) {
        // a CTA to a line (or to some), or up to eight while there are under two CTAs an SM
        unsigned cs = 1;
        while (a.warps == 8 && (b.nv == 0 || b.warps == 8) && cs < unsigned(SPLIT_CLUSTER) &&
               (a.nv + b.nv) * cs < num_sms() * 2 && a.nw > int64_t(4096) * cs)
            cs *= 2;
        const auto slice_blocks = [](SplitJob& j) {
            if (j.nv == 0) return int64_t(0);
            const int64_t lines = CPLX ? 1 : 256 / j.group;
            j.pieces = unsigned(CPLX ? (j.nw + 1023) / 1024 : (j.ldq + 4 * j.group - 1) / (4 * j.group));
            return (j.nv + lines - 1) / lines * int64_t(j.pieces);
        };
        const int64_t na = slice_blocks(a), nb = slice_blocks(b);
        if (na + nb > INT32_MAX) return HSMM_STATUS_NOT_SUPPORTED;
        a.blocks *= cs;
        b.blocks *= cs;
        e = pdl_launch(ozaki_scan_w_kernel<CPLX>, dim3(a.blocks + b.blocks), 256, 0, cs, st, a, b);
        count_launches(1);
        if (e != cudaSuccess) return record_cuda(e);
        a.blocks = unsigned(na);
        b.blocks = unsigned(nb);
        ozaki_slice_w_kernel<BITS, S, CPLX, BLOCKED><<<a.blocks + b.blocks, 256, 0, st>>>(a, b, bits, slices);
    } else if constexpr (BITS > 0 || CPLX) {
        auto kern = ozaki_split_w_kernel<BITS, S, CPLX, BLOCKED>;
        size_t smem = 0;
        if (CPLX) {
            static std::atomic<uint64_t> attrs{0};
            const hsmm_status_t as = attrs_once_per_device(attrs, [kern] {
                return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(SPLIT_CACHE));
            });
            if (as != HSMM_STATUS_SUCCESS) return as;
            smem = std::max(split_cache_bytes(a.nw), split_cache_bytes(b.nw));
        }
        e = pdl_launch(kern, dim3(a.blocks + b.blocks), 256, smem, 1, st, a, b, bits, slices);
    }
    count_launches(1);
    if (e != cudaSuccess) return record_cuda(e);
    return check_launch();
}

hsmm_status_t launch_split(bool cplx, const SplitJob& a, const SplitJob& b, int bits, int slices, cudaStream_t st) {
    const bool fixed77 = bits == 7 && slices == 7;
    using Fn = hsmm_status_t (*)(SplitJob, SplitJob, int, int, cudaStream_t);
    static constexpr Fn fn[8] = {launch_split<0, 0, false, false>, launch_split<0, 0, false, true>,
                                 launch_split<0, 0, true, false>,  launch_split<0, 0, true, true>,
                                 launch_split<7, 7, false, false>, launch_split<7, 7, false, true>,
                                 launch_split<7, 7, true, false>,  launch_split<7, 7, true, true>};
    return fn[fixed77 * 4 + cplx * 2 + a.blocked](a, b, bits, slices, st);
}

}  // namespace

hsmm_status_t ozaki_split(bool cplx, const SplitOperand* ops, int count, int bits, int slices, cudaStream_t st) {
    SplitJob j[2] = {};
    for (int i = 0; i < count; ++i) {
        const hsmm_status_t r = make_split_job(ops[i], cplx, bits == 7 && slices == 7, &j[i]);
        if (r != HSMM_STATUS_SUCCESS) return r;
    }
    if (count == 1 || (j[0].v_contig == j[1].v_contig && j[0].blocked == j[1].blocked && j[0].two_pass == j[1].two_pass))
        return launch_split(cplx, j[0], j[1], bits, slices, st);
    const hsmm_status_t r = launch_split(cplx, j[0], SplitJob{}, bits, slices, st);
    return r != HSMM_STATUS_SUCCESS ? r : launch_split(cplx, j[1], SplitJob{}, bits, slices, st);
}

hsmm_status_t ozaki_zrecombine(int64_t m, int64_t n, int slices, int bits, const int32_t* sd, int64_t sd_plane,
                               const int32_t* ea, const int32_t* eb, const double* alpha, const double* beta, void* C,
                               int64_t ldc, cudaStream_t st) {
    return launch_recombine<true>(RecombineArgs{m, n, slices, bits, 1 + 21 / bits, sd, sd_plane, ea, eb,
                                                make_double2(alpha[0], alpha[1]), make_double2(beta[0], beta[1]),
                                                static_cast<double*>(C), ldc}, st);
}

}  // namespace hsmm
