// gemm_ozaki_tc.cu -- the slice products of the FP64-accurate form on the tcgen05 tensor cores.
//
// For split operands (BF16 slices of integer digits, see ozaki.cu) this computes the
// exact anti-diagonal sums S_d = sum_{t+u=d} Q^A_t (Q^B_u)^T, d = 2..s+1, as INT32 planes
// in the caller's workspace.  The main loop is that of the plain products (gemm_tc.cu):
// TMA -> shared memory -> tcgen05.mma -> TMEM, here with a k-schedule over the slice
// pairs and an epilogue that drains exact FP32 chunks into INT32 sums held in registers.
#include <algorithm>
#include <atomic>
#include <cstdint>
#include <cstdlib>
#include <cstring>

#include <cuda.h>
#include <cuda_runtime.h>

#include "common.cuh"
#include "tc_tile.cuh"
#include "internal.h"

namespace hsmm {

static __device__ uint32_t g_status_ozaki_tc;

uint32_t status_take_ozaki_tc() {
    uint32_t v = 0, z = 0;
    cudaMemcpyFromSymbol(&v, g_status_ozaki_tc, sizeof(v));
    cudaMemcpyToSymbol(g_status_ozaki_tc, &z, sizeof(z));
    return v;
}

namespace {

using namespace tc;

// ---------------------------------------------------------------------------
// Slice products of the FP64-accurate form
// ---------------------------------------------------------------------------
// Per 128 x 256 output tile the k-schedule runs over the anti-diagonals
// d = s+1 down to 2 of the slice pairs (t, u), t + u = d, and over k inside each
// pair.  Slice entries are integers with |q| <= 2^bits - 1, so an FP32 sum of
// kc products, kc (2^bits - 1)^2 <= 2^24, is exact; the MMA warp hands the
// accumulator over every kc_blocks k-blocks (and at the end of each d), the
// epilogue converts it to INT32 and adds it to S_d held in registers (exact:
// |S_d| <= s k (2^bits-1)^2 < 2^31 is checked on the host), and at the end of
// the anti-diagonal stores S_d.  No FP64 arithmetic runs in this kernel: the
// recombination (ozaki_recombine in ozaki.cu) reads the s INT32 planes once.
// Twelve warps: warpgroup 0 holds the TMA producer (warp 0) and the MMA issuer
// (warp 1) and lowers its register budget (setmaxnreg.dec to 152); warpgroups 1
// and 2 are eight epilogue warps that raise theirs (setmaxnreg.inc to 176).  The
// launch holds 384 x 168 = 64512 registers = 128 x 152 + 256 x 176; neither side
// spills (a tighter producer/MMA budget spilled inside the MMA issue loop and
// halved the tensor-pipe rate).  Epilogue warp w owns TMEM lanes 32*(w%4).. and
// the column half (w-4)/4 of the 256-column accumulator: 128 INT32 partial sums
// per thread, kept in registers.
struct OzakiArgs {
    int M, N, K;
    int slices, kc_blocks;
    int32_t* sd;        // S_d, d = 2..s+1, as [d-2][N][M] INT32 (column-major per anti-diagonal)
    int64_t sd_plane;   // elements between consecutive anti-diagonal planes
    uint64_t timeout_ns;
    int blocked;            // the slices are in blocks of 64 columns
};

constexpr int OZ_BN = 256;
constexpr int OZ_HALF = OZ_BN / 2;
constexpr int OZ_EPI_WARPS = 8;
constexpr int OZ_THREADS = 128 + 32 * OZ_EPI_WARPS;     // 384
constexpr uint32_t OZ_REGS_LAUNCH = 168, OZ_REGS_LOW = 152, OZ_REGS_HIGH = 176;
static_assert(OZ_THREADS * OZ_REGS_LAUNCH == 128 * OZ_REGS_LOW + 256 * OZ_REGS_HIGH, "register split must balance");

__host__ __device__ __forceinline__ int oz_tlo(int d, int s) { return d - s > 1 ? d - s : 1; }
__host__ __device__ __forceinline__ int oz_thi(int d, int s) { return d - 1 < s ? d - 1 : s; }

__host__ __device__ __forceinline__ int oz_weight(int d, int s) { return oz_thi(d, s) - oz_tlo(d, s) + 1; }

// Work of the CTA pairs of the slice-product kernel.  The tiles of the full waves are whole items
// (all anti-diagonals d = s+1 .. 2, tile t = pair + i npairs).  The tiles of the last, partial
// wave are dealt out in units of one anti-diagonal, or of part of its slice pairs: the host
// assigns them, largest first, to the least loaded pair and passes the table as a kernel
// parameter.  A unit that holds only part of an anti-diagonal adds its INT32 sums to S_d with
// reduction atomics (exact in any order) in a plane zeroed before.
// Units of one anti-diagonal, not groups of them with equal slice-pair counts: 20 tiles were 80
// groups on 76 pairs, two rounds of 7 slice pairs each, and are 8 at most now (7.4 the mean).
// Before -> now, same bits: 1000 x 1200 x 900 146.6 -> 109.9 us, complex 1500 x 1100 x 2301 706
// -> 676, 4096^3 from host memory (blocks of 64 tiles) 3279 -> 2952; 8192^3 (17.8 ms) within its spread.
struct OzWork {
    int t;         // tile
    int nd;        // anti-diagonals: s (whole tile, d = s+1 .. 2) or 1
    int d;         // of a unit: the anti-diagonal (0: whole tile), its first slice of A and slice pairs
    int ta, nt;
    bool add;      // S_d += (several units share the anti-diagonal)
};
constexpr int OZ_MAX_PAIRS = 100, OZ_MAX_UNITS = 1600;   // at most 16 units for each of 99 tail tiles

// The slices of one operand.  Row-major: `blocks` is all of them, boxes at (column, row, 0, slice).  In
// blocks of 64 columns (see Slices): `blocks` the whole ones, boxes at (0, row, block, slice), and
// `rest` the columns after them, zero-filled.
// Blocks of whole lines are what the tensor cores can be fed from: rows of a pitch of 8 to 56 columns
// more than a multiple of 64 cross a line with every 64 columns, and an odd multiple of 8 a sector,
// and the products then waited for loads (690 cycles a k-block instead of 523).  2048 x 2048 x 4100:
// 814 -> 592 us, 2048 x 2048 x 2056 406 -> 328, 1000 x 1200 x 900 78 -> 69 (whole product).
struct SliceMaps {
    CUtensorMap blocks, rest;
};

struct OzTable {
    uint16_t first[OZ_MAX_PAIRS + 1];    // units of a pair: first[pair] .. first[pair + 1] - 1
    uint32_t unit[OZ_MAX_UNITS];         // tail tile | d << 8 | first slice of A << 16 | pairs << 22 | add << 28
};
__device__ __forceinline__ int oz_items(const OzTable& tab, int ntiles, int npairs, int pair) {
    return ntiles / npairs + int(tab.first[pair + 1]) - int(tab.first[pair]);
}
__device__ __forceinline__ OzWork oz_item(const OzTable& tab, int i, int ntiles, int npairs, int pair, int s) {
    const int full = ntiles / npairs;
    if (i < full) return OzWork{pair + i * npairs, s, 0, 0, 0, false};
    const uint32_t u = tab.unit[int(tab.first[pair]) + i - full];
    return OzWork{full * npairs + int(u & 0xFFu), 1, int((u >> 8) & 0xFFu), int((u >> 16) & 0x3Fu),
                  int((u >> 22) & 0x3Fu), ((u >> 28) & 1u) != 0};
}
// the di-th anti-diagonal of an item: d, its first slice of A and its slice pairs
__device__ __forceinline__ void oz_item_d(const OzWork& it, int di, int s, int& d, int& ta, int& nt) {
    d = it.d != 0 ? it.d : s + 1 - di;
    ta = it.d != 0 ? it.ta : oz_tlo(d, s);
    nt = it.d != 0 ? it.nt : oz_weight(d, s);
}

__global__ void __launch_bounds__(OZ_THREADS, 1)
    gemm_ozaki_kernel(const __grid_constant__ SliceMaps mA, const __grid_constant__ SliceMaps mB, OzakiArgs g) {
    using C_ = Cfg<OZ_BN, false>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    Bars* bars = reinterpret_cast<Bars*>(smem + C_::STAGES * C_::STAGE_BYTES);
    const int warp = int(warp_id()), lane = int(lane_id());
    uint32_t* status = &g_status_ozaki_tc;

    if (threadIdx.x == 0) {
        for (int s = 0; s < C_::STAGES; ++s) {
            mbar_init(&bars->full[s], 1);
            mbar_init(&bars->empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&bars->acc_full[b], 1);
            mbar_init(&bars->acc_empty[b], OZ_EPI_WARPS);
        }
        mbar_init(&bars->mma_done, 1);
        bars->abort = 0;
        fence_mbar_init();
        tma_prefetch_desc(&mA.blocks);
        tma_prefetch_desc(&mB.blocks);
        tma_prefetch_desc(&mA.rest);
        tma_prefetch_desc(&mB.rest);
    }
    if (warp == 1) {
        tmem_alloc(&bars->tmem_base, C_::TMEM_COLS);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = bars->tmem_base;
    volatile int* abort = &bars->abort;

    const int tiles_m = (g.M + BM - 1) / BM;
    const int tiles_n = (g.N + OZ_BN - 1) / OZ_BN;
    const int ntiles = tiles_m * tiles_n;
    const int nkb = (g.K + C_::BK - 1) / C_::BK, nfull = g.K / C_::BK;
    const int s = g.slices;
    const int kcb = g.kc_blocks;

    if (warp < 4) regs_dec<OZ_REGS_LOW>();
    if (warp == 0) {
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0;
            int last_parity[8];
            for (int i = 0; i < 8; ++i) last_parity[i] = -1;
            bool ok = true;
            for (int t = blockIdx.x; t < ntiles && ok && !*abort; t += gridDim.x) {
                int tm, tn;
                tile_coords(t, tiles_m, tiles_n, tm, tn);
                for (int d = s + 1; d >= 2 && ok; --d)
                    for (int ta = oz_tlo(d, s); ta <= oz_thi(d, s) && ok; ++ta) {
                        const int ub = d - ta;
                        for (int kb = 0; kb < nkb; ++kb) {
                            if (!mbar_wait(&bars->empty[stage], phase ^ 1u, g.timeout_ns, status, abort)) { ok = false; break; }
                            uint8_t* a_dst = smem + stage * C_::STAGE_BYTES;
                            uint8_t* b_dst = a_dst + C_::A_BYTES;
                            mbar_arrive_expect_tx(&bars->full[stage], C_::STAGE_BYTES);
                            const bool rest = kb >= nfull;
                            const int col = g.blocked ? 0 : kb * C_::BK, block = g.blocked && !rest ? kb : 0;
                            tma_load_4d(a_dst, rest ? &mA.rest : &mA.blocks, &bars->full[stage], col, tm * BM, block, ta - 1);
                            tma_load_4d(b_dst, rest ? &mB.rest : &mB.blocks, &bars->full[stage], col, tn * OZ_BN, block,
                                        ub - 1);
                            last_parity[stage] = int(phase);
                            if (++stage == C_::STAGES) { stage = 0; phase ^= 1u; }
                        }
                    }
            }
            for (int i = 0; i < C_::STAGES; ++i)
                if (last_parity[i] >= 0) mbar_wait(&bars->full[i], uint32_t(last_parity[i]), g.timeout_ns, status, abort);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t idesc = make_idesc(1u, false, false, BM, OZ_BN);
            const uint64_t a0 = operand_desc<C_>(smem_u32(smem), 0, false);
            const uint64_t b0 = operand_desc<C_>(smem_u32(smem) + C_::A_BYTES, 0, false);
            const uint64_t kstep = ks_step<C_>(false);
            const uint64_t sstep = uint64_t(C_::STAGE_BYTES / 16);
            uint64_t acur = a0, bcur = b0;
            int stage = 0;
            uint32_t phase = 0;
            int abuf = 0;
            uint32_t aphase = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < ntiles && ok && !*abort; t += gridDim.x) {
                for (int d = s + 1; d >= 2 && ok; --d) {
                    int left_d = (oz_thi(d, s) - oz_tlo(d, s) + 1) * nkb;   // k-blocks left in this anti-diagonal
                    int left_c = 0;                                         // k-blocks left in this FP32 chunk
                    uint32_t d_tmem = tmem;
                    uint32_t acc_flag = 0;
                    while (left_d > 0) {
                        if (left_c == 0) {
                            if (!mbar_wait(&bars->acc_empty[abuf], aphase ^ 1u, g.timeout_ns, status, abort)) { ok = false; break; }
                            tc_fence_after();
                            left_c = kcb;
                            d_tmem = tmem + uint32_t(abuf * OZ_BN);
                            acc_flag = 0;
                        }
                        if (!mbar_wait(&bars->full[stage], phase, g.timeout_ns, status, abort)) { ok = false; break; }
                        tc_fence_after();
                        umma_f16(d_tmem, acur, bcur, idesc, acc_flag);
#pragma unroll
                        for (int ks = 1; ks < C_::KSTEPS; ++ks)
                            umma_f16(d_tmem, acur + ks * kstep, bcur + ks * kstep, idesc, 1u);
                        acc_flag = 1u;
                        umma_commit(&bars->empty[stage]);
                        if (++stage == C_::STAGES) { stage = 0; phase ^= 1u; acur = a0; bcur = b0; }
                        else { acur += sstep; bcur += sstep; }
                        --left_d;
                        if (--left_c == 0 || left_d == 0) {
                            umma_commit(&bars->acc_full[abuf]);
                            abuf ^= 1;
                            if (abuf == 0) aphase ^= 1u;
                            left_c = 0;
                        }
                    }
                }
            }
            umma_commit(&bars->mma_done);
            mbar_wait(&bars->mma_done, 0, g.timeout_ns, status, abort);
        }
    } else if (warp >= 4) {
        regs_inc<OZ_REGS_HIGH>();
        const int q = warp & 3;
        const int half = (warp - 4) >> 2;
        int abuf = 0;
        uint32_t aphase = 0;
        bool ok = true;
        for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
            int tm, tn;
            tile_coords(t, tiles_m, tiles_n, tm, tn);
            const int64_t row = int64_t(tm) * BM + q * 32 + lane;
            const int64_t col0 = int64_t(tn) * OZ_BN + half * OZ_HALF;
            const bool row_ok = row < g.M;
            for (int d = s + 1; d >= 2 && ok; --d) {
                int S[OZ_HALF];
#pragma unroll
                for (int j = 0; j < OZ_HALF; ++j) S[j] = 0;
                const int total = (oz_thi(d, s) - oz_tlo(d, s) + 1) * nkb;
                const int nch = (total + kcb - 1) / kcb;
                for (int c = 0; c < nch; ++c) {
                    int okw = 0;
                    if (lane == 0) okw = mbar_wait(&bars->acc_full[abuf], aphase, g.timeout_ns, status, abort) ? 1 : 0;
                    okw = __shfl_sync(0xffffffffu, okw, 0);
                    if (!okw) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t t_base = tmem + (uint32_t(q * 32) << 16) + uint32_t(abuf * OZ_BN + half * OZ_HALF);
#pragma unroll
                    for (int cc = 0; cc < OZ_HALF / 16; ++cc) {
                        uint32_t r[16];
                        tmem_ld16(t_base + uint32_t(cc * 16), r);
                        tmem_ld_wait();
#pragma unroll
                        for (int j = 0; j < 16; ++j) S[cc * 16 + j] += __float2int_rn(__uint_as_float(r[j]));
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&bars->acc_empty[abuf]);
                    abuf ^= 1;
                    if (abuf == 0) aphase ^= 1u;
                }
                if (!ok) break;
                // store S_d (INT32) for this row segment: lanes are consecutive rows, so
                // each column is one 128-byte coalesced store per warp
                if (!row_ok) continue;
                const int64_t rem = int64_t(g.N) - col0;
                const int jmax = rem < OZ_HALF ? int(rem) : OZ_HALF;
                int32_t* Sp = g.sd + int64_t(d - 2) * g.sd_plane + row + col0 * int64_t(g.M);
#pragma unroll
                for (int j = 0; j < OZ_HALF; ++j)
                    if (j < jmax) Sp[int64_t(j) * g.M] = S[j];
            }
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 1) tmem_dealloc(tmem, C_::TMEM_COLS);
}

// ---------------------------------------------------------------------------
// Slice products on a CTA pair (cta_group::2): one 256 x 256 tile per pair
// ---------------------------------------------------------------------------
// The same k-schedule, chunking and epilogue as gemm_ozaki_kernel, with the MMA
// spread over two SMs: the even CTA holds A rows 0-127 and B rows 0-127 of the
// tile, the odd CTA rows 128-255 of each; one tcgen05.mma.cta_group::2 (M = 256,
// N = 256) issued by the even CTA reads both CTAs' shared memory and writes the
// 128 x 256 accumulator of each CTA into that CTA's TMEM.  Each CTA stages only
// 32 KiB per k-block (7 stages instead of 4), half the L2 traffic per tile row.
// Both CTAs' TMA copies complete on the even CTA's `full` barrier; the MMA
// commits are multicast to both CTAs (stage release, accumulator ready); both
// CTAs' epilogue warps release an accumulator on the even CTA's `acc_empty`.
// The producer and MMA roles are run by whole warps (see gemm_tc.cu): 1000 x 1200 x 900 149.9 ->
// 146.6 us, 4096^3 from host memory 3318 -> 3279, complex 1500 x 1100 x 2301 714 -> 706; 8192^3
// is bound by the power cap (18.5 ms either way).

__global__ void __launch_bounds__(OZ_THREADS, 1)
    gemm_ozaki_pair_kernel(const __grid_constant__ SliceMaps mA, const __grid_constant__ SliceMaps mB,
                           OzakiArgs g, const __grid_constant__ OzTable tab) {
    using C_ = Cfg<OZ_BN, false>;                  // BK, KSTEPS, descriptors (K-major, 128-byte rows)
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    Bars* bars = reinterpret_cast<Bars*>(smem + PAIR_STAGES * PAIR_STAGE_BYTES);
    const int warp = warp_id_uniform(), lane = int(lane_id());
    uint32_t* status = &g_status_ozaki_tc;
    const uint32_t rank = cluster_ctarank() & 1u;  // role in the pair
    const bool leader = (rank == 0);

    if (threadIdx.x == 0) {
        for (int s = 0; s < PAIR_STAGES; ++s) {
            mbar_init(&bars->full[s], 1);
            mbar_init(&bars->empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&bars->acc_full[b], 1);
            mbar_init(&bars->acc_empty[b], 2 * OZ_EPI_WARPS);
        }
        mbar_init(&bars->mma_done, 1);
        bars->abort = 0;
        fence_mbar_init();
        tma_prefetch_desc(&mA.blocks);
        tma_prefetch_desc(&mB.blocks);
        tma_prefetch_desc(&mA.rest);
        tma_prefetch_desc(&mB.rest);
    }
    if (warp == 1) {
        tmem_alloc_pair(&bars->tmem_base, 512);
        tmem_relinquish_pair();
    }
    tc_fence_before();
    cluster_sync_all();            // barriers of every CTA initialised before anyone signals them
    tc_fence_after();
    const uint32_t tmem = bars->tmem_base;
    volatile int* abort = &bars->abort;
    pdl_wait();                    // the setup above overlaps the end of the split (or of the zeroing)

    const int tiles_m = (g.M + 2 * BM - 1) / (2 * BM);
    const int tiles_n = (g.N + PAIR_BN - 1) / PAIR_BN;
    const int ntiles = tiles_m * tiles_n;
    const int pair = int(blockIdx.x >> 1), npairs = int(gridDim.x >> 1);
    const int nkb = (g.K + C_::BK - 1) / C_::BK, nfull = g.K / C_::BK;
    const int s = g.slices;
    const int kcb = g.kc_blocks;
    const int nitems = oz_items(tab, ntiles, npairs, pair);

    if (warp < 4) regs_dec<OZ_REGS_LOW>();
    if (warp == 0) {
        // both roles are run by their whole warps, one elected lane issues (see elect_one)
        const bool issue = elect_one();
        int stage = 0, filled = 0;
        uint32_t phase = 0;
        bool ok = true;
        const uint32_t full0 = mapa_shared(smem_u32(&bars->full[0]), 0);
        for (int i = 0; i < nitems && ok && !*abort; ++i) {
            const OzWork it = oz_item(tab, i, ntiles, npairs, pair, s);
            int tm, tn;
            tile_coords(it.t, tiles_m, tiles_n, tm, tn);
            const int arow = tm * 2 * BM + int(rank) * BM;
            const int brow = tn * PAIR_BN + int(rank) * BM;
            for (int di = 0; di < it.nd && ok; ++di) {
                int d, ta0, nt;
                oz_item_d(it, di, s, d, ta0, nt);
                for (int ta = ta0; ta < ta0 + nt && ok; ++ta) {
                    const int ub = d - ta;
                    for (int kb = 0; kb < nkb; ++kb) {
                        // the first round of stages starts empty
                        if (filled >= PAIR_STAGES &&
                            !mbar_wait_warp(&bars->empty[stage], phase ^ 1u, g.timeout_ns, status, abort)) { ok = false; break; }
                        uint8_t* a_dst = smem + stage * PAIR_STAGE_BYTES;
                        const uint32_t full_leader = full0 + uint32_t(stage) * 8u;
                        mbar_arrive_expect_tx_if(issue && leader, &bars->full[stage], 2 * PAIR_STAGE_BYTES);
                        const bool rest = kb >= nfull;
                        const int col = g.blocked ? 0 : kb * C_::BK, block = g.blocked && !rest ? kb : 0;
                        tma_load_4d_pair_if(issue, a_dst, rest ? &mA.rest : &mA.blocks, full_leader, col, arow, block,
                                            ta - 1);
                        tma_load_4d_pair_if(issue, a_dst + BM * 128, rest ? &mB.rest : &mB.blocks, full_leader, col, brow,
                                            block, ub - 1);
                        ++filled;
                        if (++stage == PAIR_STAGES) { stage = 0; phase ^= 1u; }
                    }
                }
            }
        }
        // every issued stage is released (empty) only after its copies landed and were consumed
        for (int f = max(0, filled - PAIR_STAGES); f < filled; ++f)
            mbar_wait_warp(&bars->empty[f % PAIR_STAGES], uint32_t(f / PAIR_STAGES) & 1u, g.timeout_ns, status, abort);
    } else if (warp == 1) {
        if (leader) {
            const bool issue = elect_one();
            const uint32_t idesc = make_idesc(1u, false, false, 2 * BM, PAIR_BN);
            const uint64_t a0 = operand_desc<C_>(smem_u32(smem), 0, false);
            const uint64_t b0 = operand_desc<C_>(smem_u32(smem) + BM * 128, 0, false);
            const uint64_t kstep = ks_step<C_>(false);
            const uint64_t sstep = uint64_t(PAIR_STAGE_BYTES / 16);
            int stage = 0;
            uint32_t phase = 0;
            int abuf = 0;
            uint32_t aphase = 0;
            bool ok = true;
            // One warp issues every MMA of the pair, so its own instruction time per k-block
            // (one wait, four MMAs, one commit) has to stay below the 512 tensor-pipe cycles
            // the k-block takes.  The loop is kept lean for that: one counter per FP32 chunk,
            // descriptors formed from the stage index (no state carried between k-blocks
            // but the stage and its phase), and four k-blocks per unrolled iteration.
            for (int i = 0; i < nitems && ok && !*abort; ++i) {
                const OzWork it = oz_item(tab, i, ntiles, npairs, pair, s);
                for (int di = 0; di < it.nd && ok; ++di) {
                    int d, ta0, nt;
                    oz_item_d(it, di, s, d, ta0, nt);
                    int left_d = nt * nkb;
                    while (left_d > 0 && ok) {
                        if (!mbar_wait_warp(&bars->acc_empty[abuf], aphase ^ 1u, g.timeout_ns, status, abort)) { ok = false; break; }
                        tc_fence_after();
                        const uint32_t d_tmem = tmem + uint32_t(abuf * PAIR_BN);
                        const int nk = min(kcb, left_d);     // k-blocks of this exact FP32 chunk
#pragma unroll 4
                        for (int j = 0; j < nk; ++j) {
                            if (!mbar_wait_warp(&bars->full[stage], phase, g.timeout_ns, status, abort)) { ok = false; break; }
                            tc_fence_after();
                            const uint64_t ad = a0 + uint64_t(stage) * sstep, bd = b0 + uint64_t(stage) * sstep;
#pragma unroll
                            for (int ks = 0; ks < C_::KSTEPS; ++ks)   // j == 0, ks == 0 starts the chunk
                                umma_pair_if<false>(issue, d_tmem, ad + ks * kstep, bd + ks * kstep, idesc,
                                                    ks == 0 ? uint32_t(j) : 1u);
                            umma_commit_pair_if(issue, &bars->empty[stage], 0x3);
                            stage = (stage + 1 == PAIR_STAGES) ? 0 : stage + 1;
                            phase ^= (stage == 0) ? 1u : 0u;
                        }
                        if (!ok) break;
                        umma_commit_pair_if(issue, &bars->acc_full[abuf], 0x3);
                        abuf ^= 1;
                        if (abuf == 0) aphase ^= 1u;
                        left_d -= nk;
                    }
                }
            }
            umma_commit_pair_if(issue, &bars->mma_done, 0x1);
            mbar_wait_warp(&bars->mma_done, 0, g.timeout_ns, status, abort);
        }
    } else if (warp >= 4) {
        regs_inc<OZ_REGS_HIGH>();
        const int q = warp & 3;
        const int half = (warp - 4) >> 2;
        const uint32_t acc_empty_leader0 = mapa_shared(smem_u32(&bars->acc_empty[0]), 0);
        const uint32_t acc_empty_leader1 = mapa_shared(smem_u32(&bars->acc_empty[1]), 0);
        int abuf = 0;
        uint32_t aphase = 0;
        bool ok = true;
        for (int i = 0; i < nitems && ok; ++i) {
            const OzWork it = oz_item(tab, i, ntiles, npairs, pair, s);
            int tm, tn;
            tile_coords(it.t, tiles_m, tiles_n, tm, tn);
            const int64_t row = int64_t(tm) * 2 * BM + int64_t(rank) * BM + q * 32 + lane;
            const int64_t col0 = int64_t(tn) * PAIR_BN + half * OZ_HALF;
            const bool row_ok = row < g.M;
            for (int di = 0; di < it.nd && ok; ++di) {
                int d, ta0, nt;
                oz_item_d(it, di, s, d, ta0, nt);
                int S[OZ_HALF];
#pragma unroll
                for (int j = 0; j < OZ_HALF; ++j) S[j] = 0;
                const int total = nt * nkb;
                const int nch = (total + kcb - 1) / kcb;
                for (int c = 0; c < nch; ++c) {
                    int okw = 0;
                    if (lane == 0) okw = mbar_wait(&bars->acc_full[abuf], aphase, g.timeout_ns, status, abort) ? 1 : 0;
                    okw = __shfl_sync(0xffffffffu, okw, 0);
                    if (!okw) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t t_base = tmem + (uint32_t(q * 32) << 16) + uint32_t(abuf * PAIR_BN + half * OZ_HALF);
#pragma unroll
                    for (int cc = 0; cc < OZ_HALF / 16; ++cc) {
                        uint32_t r[16];
                        tmem_ld16(t_base + uint32_t(cc * 16), r);
                        tmem_ld_wait();
#pragma unroll
                        for (int j = 0; j < 16; ++j) S[cc * 16 + j] += __float2int_rn(__uint_as_float(r[j]));
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) {
                        if (leader) mbar_arrive(&bars->acc_empty[abuf]);
                        else mbar_arrive_remote(abuf ? acc_empty_leader1 : acc_empty_leader0);
                    }
                    abuf ^= 1;
                    if (abuf == 0) aphase ^= 1u;
                }
                if (!ok) break;
                if (!row_ok) continue;
                const int64_t rem = int64_t(g.N) - col0;
                const int jmax = rem < OZ_HALF ? int(rem) : OZ_HALF;
                int32_t* Sp = g.sd + int64_t(d - 2) * g.sd_plane + row + col0 * int64_t(g.M);
                if (it.add) {
#pragma unroll
                    for (int j = 0; j < OZ_HALF; ++j)
                        if (j < jmax) atomicAdd(Sp + int64_t(j) * g.M, S[j]);
                } else {
#pragma unroll
                    for (int j = 0; j < OZ_HALF; ++j)
                        if (j < jmax) Sp[int64_t(j) * g.M] = S[j];
                }
            }
        }
    }
    __syncwarp();
    tc_fence_before();
    cluster_sync_all();            // the peers' MMAs and remote arrivals are done before TMEM goes
    tc_fence_after();
    if (warp == 1) tmem_dealloc_pair(tmem, 512);
}

// Zeros in the planes d_lo .. s+1 of S_d under the tiles of the last, partial wave
__global__ void __launch_bounds__(256) ozaki_zero_kernel(OzakiArgs g, int first_tile, int d_lo) {
    const int tiles_m = (g.M + 2 * BM - 1) / (2 * BM), tiles_n = (g.N + PAIR_BN - 1) / PAIR_BN;
    int tm, tn;
    tile_coords(first_tile + int(blockIdx.x), tiles_m, tiles_n, tm, tn);
    const int64_t row = int64_t(tm) * 2 * BM + threadIdx.x;
    pdl_wait();
    pdl_trigger();
    if (row >= g.M) return;
    int32_t* p = g.sd + int64_t(d_lo - 2 + int(blockIdx.y)) * g.sd_plane + row;
    const int64_t c1 = min(int64_t(g.N), int64_t(tn + 1) * PAIR_BN);
    for (int64_t c = int64_t(tn) * PAIR_BN + blockIdx.z; c < c1; c += gridDim.z) p[c * g.M] = 0;
}

// Deal the anti-diagonals of `tiles` tiles to npairs pairs, each cut into pieces of at most `piece`
// slice pairs: largest piece first, to the least loaded pair.  Returns the largest load.
int deal_units(int tiles, int npairs, int s, int piece, OzTable* tab) {
    struct Unit {
        uint32_t code;
        uint8_t pair;
    };
    static thread_local Unit units[OZ_MAX_UNITS];
    int n = 0;
    int load[OZ_MAX_PAIRS] = {0}, count[OZ_MAX_PAIRS] = {0};
    // pairs by load: a ring of stacks, one per load value (loads stay within `s` of the least)
    int next[OZ_MAX_PAIRS], head[32];
    for (int i = 0; i < 32; ++i) head[i] = -1;
    for (int p = npairs - 1; p >= 0; --p) { next[p] = head[0]; head[0] = p; }
    int least = 0, most = 0;
    for (int w = std::min(s, piece); w >= 1; --w)
        for (int d = s + 1; d >= 2; --d) {
            const int total = oz_weight(d, s), parts = (total + piece - 1) / piece;
            for (int q = 0; q < parts; ++q) {
                const int lo = total * q / parts, hi = total * (q + 1) / parts;
                if (hi - lo != w) continue;
                for (int t = 0; t < tiles; ++t) {
                    while (head[least & 31] < 0) ++least;
                    const int p = head[least & 31];
                    head[least & 31] = next[p];
                    load[p] += w;
                    next[p] = head[load[p] & 31];
                    head[load[p] & 31] = p;
                    most = std::max(most, load[p]);
                    if (n == OZ_MAX_UNITS) return 1 << 30;
                    ++count[p];
                    units[n++] = Unit{uint32_t(t) | uint32_t(d) << 8 | uint32_t(oz_tlo(d, s) + lo) << 16 |
                                          uint32_t(w) << 22 | (parts > 1 ? 1u : 0u) << 28,
                                      uint8_t(p)};
                }
            }
        }
    int at = 0, pos[OZ_MAX_PAIRS];
    for (int p = 0; p < npairs; ++p) {
        tab->first[p] = uint16_t(at);
        pos[p] = at;
        at += count[p];
    }
    tab->first[npairs] = uint16_t(at);
    for (int i = 0; i < n; ++i) tab->unit[pos[units[i].pair]++] = units[i].code;
    return most;
}

// The table of a launch and the anti-diagonals (d >= zero_from) whose planes have to be zeroed
// under the tail tiles; the last ones of this host thread are kept (they depend on the counts only).
struct OzSchedule {
    int ntiles, npairs, s, nkb, zero_from;
    OzTable tab;
};
const OzSchedule& oz_schedule(int ntiles, int npairs, int s, int nkb) {
    static thread_local OzSchedule cache[4];
    static thread_local int turn = 0;
    for (const OzSchedule& c : cache)
        if (c.npairs == npairs && c.ntiles == ntiles && c.s == s && c.nkb == nkb) return c;
    OzSchedule& c = cache[turn];
    turn = (turn + 1) % 4;
    c.ntiles = ntiles; c.npairs = npairs; c.s = s; c.nkb = nkb; c.zero_from = 0;
    const int tail = ntiles % npairs;
    const int whole = deal_units(tail, npairs, s, s, &c.tab);
    const int total = tail * s * (s + 1) / 2, piece = std::max(1, (total + npairs - 1) / npairs);
    if (tail > 0 && piece < s) {
        // cutting anti-diagonals pays when the busiest pair saves more than the zeroing (a launch
        // and the planes' bytes) and the atomics cost
        OzTable cut;
        const int most = deal_units(tail, npairs, s, piece, &cut);
        const double saved_us = double(whole - most) * nkb * 0.26;
        const double cost_us = 5.0 + double(tail) * (s - piece) * 0.26 / 5.0;
        if (saved_us > cost_us) {
            c.tab = cut;
            c.zero_from = piece + 2;     // oz_weight(d) = d - 1 > piece
        }
    }
    return c;
}

}  // namespace

// The slice products run on CTA pairs; HSMM_OZAKI_KERNEL = single selects the one-CTA kernel
// (kept for comparison; both produce the same exact S_d).
static bool ozaki_pairs_enabled() {
    const char* v = std::getenv("HSMM_OZAKI_KERNEL");
    return !(v && std::strcmp(v, "single") == 0);
}

static hsmm_status_t launch_ozaki_pairs(const SliceMaps& mA, const SliceMaps& mB, const OzakiArgs& g, int slices,
                                        cudaStream_t st) {
    static std::atomic<uint64_t> attrs{0};
    hsmm_status_t as = attrs_once_per_device(attrs, [] {
        return cudaFuncSetAttribute(gemm_ozaki_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, PAIR_SMEM);
    });
    if (as != HSMM_STATUS_SUCCESS) return as;
    const int max_pairs = std::min(num_sms() / 2, OZ_MAX_PAIRS);
    const int tiles = ((g.M + 2 * BM - 1) / (2 * BM)) * ((g.N + PAIR_BN - 1) / PAIR_BN);
    // whole tiles while they fill every pair; the tiles of a partial wave go out in smaller units
    const int pairs = std::max(1, tiles >= max_pairs ? max_pairs : std::min(max_pairs, tiles * slices * (slices + 1) / 2));
    const OzSchedule& sc = oz_schedule(tiles, pairs, slices, (g.K + 63) / 64);
    if (sc.zero_from > 0) {
        const int tail = tiles % pairs;
        const cudaError_t ez = pdl_launch(ozaki_zero_kernel, dim3(unsigned(tail), unsigned(slices + 2 - sc.zero_from), 8),
                                          256, 0, 1, st, g, tiles - tail, sc.zero_from);
        count_launches(1);
        if (ez != cudaSuccess) return record_cuda(ez);
    }
    // A programmatic dependent is placed as SMs come free, not in order, and tiles that share operands
    // then sit on different halves of the chip: 8192^3 in a row, power-capped, 19.35 -> 19.95 ms.  The 2 us
    // it saves are worth that only while the products are short (1000 k-blocks a pair, 270 us; 2048^3,
    // 754, 307.6 -> 303.8 us a call).
    const bool is_short = double(tiles) * slices * (slices + 1) / 2 * ((g.K + 63) / 64) < 1000.0 * pairs;
    const cudaError_t e = cluster_launch(is_short, gemm_ozaki_pair_kernel, dim3(unsigned(2 * pairs)), OZ_THREADS, PAIR_SMEM, 2,
                                         st, mA, mB, g, sc.tab);
    count_launches(1);
    if (e != cudaSuccess) return record_cuda(e);
    return check_launch();
}

// Maps of the slices of `rows` rows and k columns, boxes of box_rows x 64.  Row-major slices are one
// tensor with all of k inside, so that an L2 fetch may take two neighbouring lines of a row.
static bool slice_maps(const Slices& q, int64_t rows, int64_t k, int slices, uint32_t box_rows, SliceMaps* m) {
    const uint16_t* base = static_cast<const uint16_t*>(q.q);
    auto encode = [&](CUtensorMap* map, int64_t from, int64_t cols, int64_t ld, int64_t blocks, int64_t step) {
        return encode_map(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base + from, uint64_t(cols), uint64_t(rows),
                          uint64_t(ld), 64, box_rows, uint64_t(slices), uint64_t(q.plane), CU_TENSOR_MAP_SWIZZLE_128B, 1,
                          uint64_t(blocks), uint64_t(step));
    };
    if (q.block_rows == 0) {
        if (!encode(&m->blocks, q.row0 * q.ldq, k, q.ldq, 1, 64)) return false;
        m->rest = m->blocks;
        return true;
    }
    const int64_t full = k / 64, rem = k % 64;    // ldq / 64 == full: ldq is k rounded up to 8, and not to 64
    const int64_t step = q.block_rows * 64, rest_pitch = q.ldq % 64;
    if (full > 0 && !encode(&m->blocks, q.row0 * 64, 64, 64, full, step)) return false;
    if (rem > 0 && !encode(&m->rest, full * step + q.row0 * rest_pitch, rem, rest_pitch, 1, 64)) return false;
    if (full == 0) m->blocks = m->rest;
    if (rem == 0) m->rest = m->blocks;
    return true;
}

hsmm_status_t gemm_ozaki_slices(int64_t m, int64_t n, int64_t k, int slices, int bits, const Slices& qa,
                                const Slices& qb, int32_t* sd, int64_t sd_plane, cudaStream_t st) {
    using C_ = Cfg<OZ_BN, false>;
    // exactness of the FP32 chunks and of the INT32 anti-diagonal sums
    const double qmax = double((1 << bits) - 1);
    const int64_t kc = int64_t(16777216.0 / (qmax * qmax));
    const int kc_blocks = int(kc / C_::BK);
    if (kc_blocks < 1) return fail(HSMM_STATUS_NOT_SUPPORTED, "ozaki: slice width leaves no exact FP32 chunk");
    if (double(slices) * double(k) * qmax * qmax >= 2147483648.0)
        return fail(HSMM_STATUS_NOT_SUPPORTED, "ozaki: s k (2^bits-1)^2 >= 2^31, the INT32 sums would not be exact");
    OzakiArgs g{};
    g.M = int(m); g.N = int(n); g.K = int(k);
    g.slices = slices; g.kc_blocks = kc_blocks;
    g.sd = sd;
    g.blocked = qa.block_rows > 0;      // A and B alike: it follows from ldq
    g.sd_plane = sd_plane;
    g.timeout_ns = wait_timeout_ns();
    if (ozaki_pairs_enabled()) {
        // pair kernel: boxes of 128 rows (each CTA stages its half of the 256 x 256 tile's A and B)
        SliceMaps mA2, mB2;
        if (!slice_maps(qa, m, k, slices, BM, &mA2) || !slice_maps(qb, n, k, slices, BM, &mB2))
            return HSMM_STATUS_NOT_SUPPORTED;
        return launch_ozaki_pairs(mA2, mB2, g, slices, st);
    }
    SliceMaps mA, mB;
    if (!slice_maps(qa, m, k, slices, BM, &mA) || !slice_maps(qb, n, k, slices, OZ_BN, &mB))
        return HSMM_STATUS_NOT_SUPPORTED;
    static std::atomic<uint64_t> attrs{0};
    hsmm_status_t as = attrs_once_per_device(attrs, [] {
        return cudaFuncSetAttribute(gemm_ozaki_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, C_::SMEM_BYTES);
    });
    if (as != HSMM_STATUS_SUCCESS) return as;
    const int tiles = ((g.M + BM - 1) / BM) * ((g.N + OZ_BN - 1) / OZ_BN);
    const int grid = std::min(tiles, num_sms());
    gemm_ozaki_kernel<<<grid, OZ_THREADS, C_::SMEM_BYTES, st>>>(mA, mB, g);
    count_launches(1);
    return check_launch();
}

}  // namespace hsmm
