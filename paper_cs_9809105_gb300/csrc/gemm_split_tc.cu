// gemm_split_tc.cu -- plain BF16/TF32 products with few output tiles: narrow tiles whose
// contraction is split over the CTAs of a thread-block cluster.
//
// The persistent kernels of gemm_tc.cu put one 256 x 256 (or 128 x 256) tile on a CTA pair (a
// CTA) and walk all of k there.  A product with few columns, or small on both sides, then has
// fewer tiles than the GPU has pairs, and its time is one pair's serial walk along k.  Here a
// tile is 128 x BN (BN a multiple of 16 up to 128) and a cluster of S = 1..8 CTAs shares it: CTA r runs the
// main loop of the plain kernel (TMA -> shared memory ring -> tcgen05.mma -> TMEM) over its
// S-th of the k-blocks and stores its FP32 partial sums of column c into the shared memory of
// rank c % S (distributed shared memory); after one cluster barrier every rank adds up its
// columns in rank order: deterministic, without workspace or atomics.
//
//   warps 0 and 2      TMA producers of A and of B over this rank's k-blocks
//   warp 1             MMA issuer, one TMEM accumulator of BN columns
//   warps 0..7         epilogue: 32 TMEM lanes and every other 16 columns each, then the sum and
//                      the stores of C
//
// What bounds it: with the tiles spread over all SMs, the 0.15 us (300 cycles) the producers need
// to issue a k-block's loads, or the ~150 GB/s an SM takes from L2 (DRAM for long thin products);
// hence roles run by whole warps (see elect_one: a k-block took 0.24 us with single-lane
// branches), one producer per operand, and as many stages as fit.  Partial sums are pushed to
// their owner (a pull through distributed shared memory, behind a second barrier, cost 0.4 us
// more).  Microseconds in a row in a CUDA graph, whole tiles -> here: 6144 x 16 x 4096 (T, N)
// 21.0 -> 10.9 (50 MB of A: 4.6 TB/s), 1280 x 520 x 1024 9.9 -> 5.5, 1280 x 1024 x 520 (N, T)
// 8.2 -> 5.3, 256 x 256 x 8192 39.4 -> 6.7, 1024^3 10.0 -> 5.8, 64 x 4392 x 5520 39.1 -> 13.9;
// 2048^3 15.5 on whole tiles and 16.6 here (whole tiles stay).
//
// The tile and the split follow from the sizes, the number of SMs and how many clusters fit the GPU (see
// split_plan): the order of the FP32 sums, and so their last bits, is the same in every call on one GPU
// but not on every GPU.  The error does not grow: the FP32 result of 16 x 4096 x 6144 is 2.1e-6 off its
// 64-bit value (norm) in eight parts, 4.4e-6 in one; over 51 shapes it was nowhere larger.
//
// When every CTA has an SM to itself it takes the whole shared memory for stages; else two share
// an SM, and one's prologue and epilogue overlap the other's main loop.
#include <algorithm>
#include <atomic>
#include <cstdint>
#include <mutex>

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "common.cuh"
#include "tc_tile.cuh"
#include "internal.h"

namespace hsmm {

static __device__ uint32_t g_status_split;

uint32_t status_take_split() {
    uint32_t v = 0, z = 0;
    cudaMemcpyFromSymbol(&v, g_status_split, sizeof(v));
    cudaMemcpyToSymbol(g_status_split, &z, sizeof(z));
    return v;
}

namespace {

using namespace tc;

constexpr int SP_THREADS = 256;                 // eight warps: two per TMEM lane quarter in the epilogue
constexpr int SP_WARPS = SP_THREADS / 32;
constexpr int SP_MAX_SPLIT = 8;                 // portable cluster size
constexpr int SP_MAX_BN = 128;
constexpr int SP_A_BYTES = BM * 128;
constexpr int SP_SPLIT_BN = 64;                 // widest tile that is split along k
constexpr int SP_SMEM2 = 111 * 1024, SP_SMEM1 = 208 * 1024;   // stages of one CTA: two or one per SM
constexpr int SP_SMEM_EXTRA = 1024 + 256;                     // alignment, barriers
static_assert(2 * (SP_SMEM2 + SP_SMEM_EXTRA + 1024) <= 228 * 1024 && SP_SMEM1 + SP_SMEM_EXTRA <= 227 * 1024,
              "split kernel shared memory");
static_assert(SP_SMEM2 / (SP_A_BYTES + SP_MAX_BN * 128) * (SP_A_BYTES + SP_MAX_BN * 128) >= BM * SP_MAX_BN * 4,
              "the partial tile reuses the stages");

// bytes of the incoming partial sums [rank][column of this rank][row] of a split tile
__host__ __device__ constexpr int split_part_bytes(int bn) { return (bn + SP_MAX_SPLIT) * BM * 4; }
static_assert((SP_SMEM2 - split_part_bytes(SP_SPLIT_BN)) / (SP_A_BYTES + SP_SPLIT_BN * 128) >= 3, "stages of a split tile");

// store into the shared memory of a CTA of the cluster (address from mapa_shared)
__device__ __forceinline__ void st_cluster_f32(uint32_t addr, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}

// four rows of one column of C: alpha s (+ beta C), `rows` of them inside the matrix
template <bool OUT_BF16>
__device__ __forceinline__ void store_c4(const SplitArgs& g, void* cp, const float4& s, int rows) {
    const float v[4] = {g.alpha * s.x, g.alpha * s.y, g.alpha * s.z, g.alpha * s.w};
    if (g.c_vec && rows >= 4) {
        if (OUT_BF16) {
            const __nv_bfloat162 lo = __floats2bfloat162_rn(v[0], v[1]), hi = __floats2bfloat162_rn(v[2], v[3]);
            uint2 pk;
            pk.x = *reinterpret_cast<const uint32_t*>(&lo);
            pk.y = *reinterpret_cast<const uint32_t*>(&hi);
            *static_cast<uint2*>(cp) = pk;
        } else {
            *static_cast<float4*>(cp) = make_float4(v[0], v[1], v[2], v[3]);
        }
        return;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (i >= rows) break;
        if (OUT_BF16) {
            __nv_bfloat16* c = static_cast<__nv_bfloat16*>(cp) + i;
            *c = __float2bfloat16_rn(g.beta != 0.f ? fmaf(g.beta, __bfloat162float(*c), v[i]) : v[i]);
        } else {
            float* c = static_cast<float*>(cp) + i;
            *c = g.beta != 0.f ? fmaf(g.beta, *c, v[i]) : v[i];
        }
    }
}

// Columns col, col + step, ... of C (n of them, every eighth from this warp), four rows per lane,
// from `part` [column][row], summed over S planes of `plane` floats in order
template <bool OUT_BF16>
__device__ __forceinline__ void sum_store(const SplitArgs& g, const float* part, int S, int plane, int warp, int lane,
                                          int64_t row0, int64_t col, int step, int n) {
    const int64_t row = row0 + 4 * lane;
    const int rows = row < g.M ? int(min(int64_t(4), g.M - row)) : 0;
    if (rows == 0) return;
    constexpr int ES = OUT_BF16 ? 2 : 4;
    uint8_t* cp = static_cast<uint8_t*>(g.C) + (row + (col + int64_t(warp) * step) * g.ldc) * ES;
    const int64_t cstep = int64_t(SP_WARPS) * step * g.ldc * ES;
    const float* p = part + warp * BM + 4 * lane;
#pragma unroll 4
    for (int c = warp; c < n; c += SP_WARPS) {
        float4 s = *reinterpret_cast<const float4*>(p);
        for (int q = 1; q < S; ++q) {
            const float4 v = *reinterpret_cast<const float4*>(p + q * plane);
            s.x += v.x;
            s.y += v.y;
            s.z += v.z;
            s.w += v.w;
        }
        store_c4<OUT_BF16>(g, cp, s, rows);
        cp += cstep;
        p += SP_WARPS * BM;
    }
}

template <bool TF32, bool OUT_BF16>
__global__ void __launch_bounds__(SP_THREADS, 2)
    gemm_tc_split_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                         SplitArgs g) {
    using C_ = Cfg<SP_MAX_BN, TF32>;               // BK, KSTEPS, descriptors; the tile width is g.bn
    const int stages = g.stages, BN = g.bn;
    const uint32_t stage_bytes = uint32_t(SP_A_BYTES + BN * 128);
    const uint32_t tmem_cols = BN <= 32 ? 32u : BN <= 64 ? 64u : 128u;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    Bars* bars = reinterpret_cast<Bars*>(smem + stages * stage_bytes);
    const int warp = warp_id_uniform(), lane = int(lane_id());
    uint32_t* status = &g_status_split;
    const int rank = int(cluster_ctarank()), S = int(cluster_nctarank());

    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) {
            mbar_init(&bars->full[s], 2);    // the two producers' expected bytes
            mbar_init(&bars->empty[s], 1);
        }
        mbar_init(&bars->acc_full[0], 1);
        mbar_init(&bars->mma_done, 1);
        bars->abort = 0;
        fence_mbar_init();
        tma_prefetch_desc(&tmA);
        tma_prefetch_desc(&tmB);
    }
    if (warp == 1) {
        tmem_alloc(&bars->tmem_base, tmem_cols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = bars->tmem_base;
    volatile int* abort = &bars->abort;
    if (S > 1) cluster_arrive();   // this CTA runs; the wait is before the first store to a peer
    // launched as a programmatic dependent (see gemm_tc.cu): the setup above overlapped the
    // previous kernel; the producer and the stores of C wait for it
    pdl_trigger();

    const int tiles_m = (g.M + BM - 1) / BM;
    const int t = int(blockIdx.x) / S;
    const int tm = t % tiles_m, tn = t / tiles_m;     // tiles of one column block run together
    const int nkb = (g.K + C_::BK - 1) / C_::BK;
    const int kb0 = int(int64_t(nkb) * rank / S), kb1 = int(int64_t(nkb) * (rank + 1) / S);

    if (warp == 0 || warp == 2) {
        // producers: warp 0 loads A, warp 2 loads B.  The issue of one warp, about 470 cycles per
        // k-block with both operands, was what bounded the main loop.
        const bool is_a = warp == 0;
        const void* map = is_a ? &tmA : &tmB;
        const bool mn = is_a ? g.a_mn : g.b_mn, mn3 = is_a ? g.a_mn3 : g.b_mn3;
        const int r0 = is_a ? tm * BM : tn * BN, rows = is_a ? BM : BN;
        const uint32_t bytes = uint32_t(rows) * 128u;
        uint8_t* dst0 = smem + (is_a ? 0 : SP_A_BYTES);
        const bool issue = elect_one();
        pdl_wait();   // A and B may be written by the previous kernel
        int stage = 0, filled = 0;
        uint32_t phase = 0;
        for (int kb = kb0; kb < kb1; ++kb) {
            // the first round of stages starts empty
            if (filled >= stages &&
                !mbar_wait_warp(&bars->empty[stage], phase ^ 1u, g.timeout_ns, status, abort)) break;
            uint8_t* dst = dst0 + stage * stage_bytes;
            mbar_arrive_expect_tx_if(issue, &bars->full[stage], bytes);
            if (!mn) {
                tma_load_2d_if(issue, dst, map, &bars->full[stage], kb * C_::BK, r0);
            } else if (mn3) {
                tma_load_3d_if(issue, dst, map, &bars->full[stage], 0, kb * C_::BK, r0 / C_::MN_CHUNK);
            } else {
                for (int c = 0; c < rows / C_::MN_CHUNK; ++c)
                    tma_load_2d_if(issue, dst + c * C_::BK * 128, map, &bars->full[stage], r0 + c * C_::MN_CHUNK,
                                   kb * C_::BK);
            }
            ++filled;
            if (++stage == stages) { stage = 0; phase ^= 1u; }
        }
        // no bulk copy may still land when the stages are reused below: the last fill of each stage
        for (int f = max(0, filled - stages); f < filled; ++f)
            mbar_wait_warp(&bars->full[f % stages], uint32_t(f / stages) & 1u, g.timeout_ns, status, abort);
    } else if (warp == 1) {
        // the whole warp runs the loop; the elected lane issues (see elect_one)
        const uint32_t idesc = make_idesc(TF32 ? 2u : 1u, g.a_mn != 0, g.b_mn != 0, BM, uint32_t(BN));
        const uint64_t a0 = operand_desc<C_>(smem_u32(smem), 0, g.a_mn != 0);
        const uint64_t b0 = operand_desc<C_>(smem_u32(smem) + SP_A_BYTES, 0, g.b_mn != 0);
        const uint64_t aks = ks_step<C_>(g.a_mn != 0), bks = ks_step<C_>(g.b_mn != 0);
        const uint64_t sstep = uint64_t(stage_bytes / 16);
        const bool issue = elect_one();
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true;
#pragma unroll 2
        for (int kb = kb0; kb < kb1; ++kb) {
            if (!mbar_wait_warp(&bars->full[stage], phase, g.timeout_ns, status, abort)) { ok = false; break; }
            tc_fence_after();
            const uint64_t ad = a0 + uint64_t(stage) * sstep, bd = b0 + uint64_t(stage) * sstep;
#pragma unroll
            for (int ks = 0; ks < C_::KSTEPS; ++ks)
                umma_if<TF32>(issue, tmem, ad + ks * aks, bd + ks * bks, idesc, ks == 0 ? uint32_t(kb - kb0) : 1u);
            umma_commit_if(issue, &bars->empty[stage]);
            stage = (stage + 1 == stages) ? 0 : stage + 1;
            phase ^= (stage == 0) ? 1u : 0u;
        }
        if (issue) {
            if (ok) umma_commit(&bars->acc_full[0]);
            // all issued MMAs complete before TMEM is released
            umma_commit(&bars->mma_done);
            mbar_wait(&bars->mma_done, 0, g.timeout_ns, status, abort);
        }
    }
    __syncwarp();

    // epilogue: warp w holds rows 32 w + lane of the tile in its TMEM lanes
    int done = 0;
    if (lane == 0) done = mbar_wait(&bars->acc_full[0], 0, g.timeout_ns, status, abort) ? 1 : 0;
    done = __shfl_sync(0xffffffffu, done, 0);
    tc_fence_after();
    const int64_t row0 = int64_t(tm) * BM, col0 = int64_t(tn) * BN;
    const int cols = min(BN, g.N - tn * BN);
    const int q = warp & 3;
    const uint32_t t_base = tmem + (uint32_t(q * 32) << 16);
    if (S == 1) {
        // the tile [column][row] into the stages: every MMA has read them, every copy has landed
        float* part = reinterpret_cast<float*>(smem);
        if (done) {
            float* mine = part + q * 32 + lane;
#pragma unroll 2
            for (int c0 = (warp >> 2) * 16; c0 < cols; c0 += 32) {
                uint32_t r[16];
                tmem_ld16(t_base + uint32_t(c0), r);
                tmem_ld_wait();
#pragma unroll
                for (int j = 0; j < 16; ++j) mine[(c0 + j) * BM] = __uint_as_float(r[j]);
            }
        }
        pdl_wait();   // C may be read or written by the previous kernel
        __syncthreads();
        sum_store<OUT_BF16>(g, part, 1, 0, warp, lane, row0, col0, 1, cols);
    } else {
        // column c of the tile belongs to rank c % S; every rank stores its partial column there,
        // plane `rank` of that rank's buffer (which nothing else uses, so one barrier is enough)
        float* part = reinterpret_cast<float*>(smem + stages * stage_bytes + sizeof(Bars));
        const int per_rank = (cols + S - 1) / S, plane = per_rank * BM;
        cluster_wait();
        if (done) {
            const uint32_t mine = smem_u32(part) + uint32_t(rank * plane + q * 32 + lane) * 4u;
#pragma unroll 1
            for (int c0 = (warp >> 2) * 16; c0 < cols; c0 += 32) {
                uint32_t r[16];
                tmem_ld16(t_base + uint32_t(c0), r);
                int owner = c0 % S;
                uint32_t addr = mine + uint32_t(c0 / S * BM) * 4u;
                tmem_ld_wait();
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    if (c0 + j < cols) st_cluster_f32(mapa_shared(addr, uint32_t(owner)), __uint_as_float(r[j]));
                    if (++owner == S) { owner = 0; addr += BM * 4; }
                }
            }
        }
        pdl_wait();
        __syncwarp();
        cluster_sync_all();
        sum_store<OUT_BF16>(g, part, S, plane, warp, lane, row0, col0 + rank, S, (cols - rank + S - 1) / S);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 1) tmem_dealloc(tmem, tmem_cols);
}

template <bool TF32, bool OUT_BF16>
hsmm_status_t split_attrs() {
    auto kern = gemm_tc_split_kernel<TF32, OUT_BF16>;
    static std::atomic<uint64_t> attrs{0};
    return attrs_once_per_device(attrs, [kern] {
        return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SP_SMEM1 + SP_SMEM_EXTRA);
    });
}

// Clusters of S CTAs that are resident together, with the shared memory of one CTA per SM
// (alone) or of two, looked up once per device: 76 pairs on 152 SMs, but fewer than 152 / S of
// the larger ones, whose CTAs have to lie in one GPC.  0 where the query fails.
struct Resident {
    int alone[SP_MAX_SPLIT + 1], shared[SP_MAX_SPLIT + 1];
};
Resident query_resident() {
    Resident r{};
    if (split_attrs<false, false>() != HSMM_STATUS_SUCCESS) return r;
    for (int s = 2; s <= SP_MAX_SPLIT; ++s)
        for (int k = 0; k < 2; ++k) {
            cudaLaunchConfig_t lc = {};
            lc.gridDim = dim3(unsigned(s), 1, 1);
            lc.blockDim = dim3(SP_THREADS, 1, 1);
            lc.dynamicSmemBytes = (k == 0 ? SP_SMEM1 : SP_SMEM2) + SP_SMEM_EXTRA;
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = unsigned(s);
            at[0].val.clusterDim.y = 1;
            at[0].val.clusterDim.z = 1;
            lc.attrs = at;
            lc.numAttrs = 1;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, gemm_tc_split_kernel<false, false>, &lc) != cudaSuccess) {
                cudaGetLastError();
                n = 0;
            }
            (k == 0 ? r.alone : r.shared)[s] = n;
        }
    return r;
}
const Resident& resident() {
    static std::once_flag once[64];
    static Resident table[64];
    static const Resident none{};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return none;
    std::call_once(once[dev], [dev] { table[dev] = query_resident(); });
    return table[dev];
}

// Stages of one CTA: deep when every CTA has an SM to itself, else what lets two share one
bool split_alone(const Resident& r, int sms, int64_t tiles, int split) {
    return split == 1 ? tiles <= sms : tiles <= r.alone[split];
}
int split_stages(bool alone, int bn, int split) {
    const int part = split == 1 ? 0 : split_part_bytes(bn);
    return std::min(8, ((alone ? SP_SMEM1 : SP_SMEM2) - part) / (SP_A_BYTES + bn * 128));
}

template <bool TF32, bool OUT_BF16>
hsmm_status_t launch_split(const CUtensorMap& ta, const CUtensorMap& tb, SplitArgs g, int split, cudaStream_t st) {
    auto kern = gemm_tc_split_kernel<TF32, OUT_BF16>;
    const hsmm_status_t as = split_attrs<TF32, OUT_BF16>();
    if (as != HSMM_STATUS_SUCCESS) return as;
    const int tiles = ((g.M + BM - 1) / BM) * ((g.N + g.bn - 1) / g.bn);
    g.stages = split_stages(split_alone(resident(), num_sms(), tiles, split), g.bn, split);
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(unsigned(tiles * split), 1, 1);
    lc.blockDim = dim3(SP_THREADS, 1, 1);
    lc.dynamicSmemBytes = size_t(g.stages) * (SP_A_BYTES + g.bn * 128) +
                          (split == 1 ? 0 : split_part_bytes(g.bn)) + SP_SMEM_EXTRA;
    lc.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = unsigned(split);
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // see pdl_wait in the kernel
    at[1].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = at;
    lc.numAttrs = 2;
    const cudaError_t e = cudaLaunchKernelEx(&lc, kern, ta, tb, g);
    count_launches(1);
    if (e != cudaSuccess) return record_cuda(e);
    return check_launch();
}

}  // namespace

// Tile width and split with the least estimated time (microseconds, fitted to launches in a row
// inside CUDA graphs): a launch and the epilogue of a tile cost 2.7 + bn / 100, a cluster another
// 1.0 (2.0 where its CTAs share SMs), and a k-block of a CTA the longest of the issue of its loads
// (0.15), the 150 GB/s an SM gets from L2, and the latency of a load (1.0) over the stages in
// flight.
SplitPlan split_plan(int64_t m, int64_t n, int64_t k, bool tf32, bool b_mn) {
    const int bk = tf32 ? 32 : 64, chunk = tf32 ? 32 : 64;
    const int sms = num_sms();
    const Resident& res = resident();
    const int64_t nkb = (k + bk - 1) / bk;
    const int64_t tiles_m = (m + BM - 1) / BM;
    SplitPlan best{0, 0, 0.0};
    for (int bn = 16; bn <= SP_MAX_BN; bn += 16) {
        if (b_mn && bn % chunk != 0) continue;     // an MN-major B comes in whole chunks
        const int64_t tiles = tiles_m * ((n + bn - 1) / bn);
        if (tiles > 2 * sms) continue;             // more than one wave
        for (int s = 1; s <= (bn <= SP_SPLIT_BN ? SP_MAX_SPLIT : 1) && s <= nkb && tiles * s <= 2 * sms; ++s) {
            const bool alone = split_alone(res, sms, tiles, s);
            if (s > 1 && !alone && tiles > res.shared[s]) continue;   // more than one wave
            const double per_sm = alone ? 1.0 : double((tiles * s + sms - 1) / sms);
            const double t_kb = std::max(std::max(0.15, per_sm * (16.0 + bn / 8.0) * 0.0066), 1.0 / split_stages(alone, bn, s));
            const double cost = 2.7 + 0.01 * bn + (s == 1 ? 0.0 : alone ? 1.0 : 2.0) + double((nkb + s - 1) / s) * t_kb;
            if (best.bn == 0 || cost < best.cost) best = SplitPlan{bn, s, cost};
        }
    }
    return best;
}

hsmm_status_t gemm_tc_split(bool tf32, bool out_bf16, const CUtensorMap& ta, const CUtensorMap& tb, const SplitArgs& g,
                            const SplitPlan& plan, cudaStream_t st) {
    if (tf32) return launch_split<true, false>(ta, tb, g, plan.split, st);
    return out_bf16 ? launch_split<false, true>(ta, tb, g, plan.split, st)
                    : launch_split<false, false>(ta, tb, g, plan.split, st);
}

}  // namespace hsmm
