// nbody.cu -- the two-array n^2 problem of Section 4, F_i = sum_j f(x_i, z_j), with the
// gravitational interaction Section 2 cites as the prototype hyper-systolic application:
//   f(x, z) = m_z (r_z - r_x) / (|r_z - r_x|^2 + eps2)^(3/2)   (0 for coincident bodies).
// Bodies are float4 (px, py, pz, m), results float4 (ax, ay, az, 0); FP32 arithmetic with the
// hardware reciprocal square root.  From eps2 = 2^-66 on the kernels work on pairs of x bodies with
// the packed FP32 instructions of this GPU (sub/mul/fma .f32x2: two interactions per
// instruction, the reciprocal square root per half).
//
// Two schedules:
//  * tiled: each lane owns x bodies; the z array streams through shared memory in tiles
//    that every CTA reads from L2 (the GPU's own way to share one array among all cells), split
//    over the warps of a CTA and the CTAs of a cluster;
//  * hyper-systolic (Section 4.1 with the regular bases of Definition REGULARBASE2): a
//    cluster of p CTAs is the ring of p cells, each owning a block of x; the K replicas of
//    x (A = (0, 1, ..., 1)) are the blocks of the K-1 right-hand neighbours, read once
//    through distributed shared memory; z passes through the cluster in rounds of p blocks,
//    each block moving K~-1 times by K cells (B = (0, K, ..., K)), and every cell adds the
//    interactions of its K replicas with the z block it holds into K intermediate results;
//    the collector then moves K-1 times by one cell against the replica shifts, adding the
//    intermediate results (back-shift phase).  Every (x block, z block) pair meets once per
//    round because the distances s K - t, 0 <= t < K, 0 <= s < K~, cover 0..p-1.
#include <cstdint>
#include <cuda_runtime.h>

#include "common.cuh"
#include "internal.h"

namespace hsmm {
namespace {

// tiled kernel: warps per CTA (each takes its share of a z tile of NB_THREADS bodies), x bodies
// per lane and per CTA, z bodies per unrolled step, CTAs of a cluster (the split of z)
constexpr int NB_WARPS = 8, NB_THREADS = 32 * NB_WARPS;
constexpr int NB_ILP = 4, NB_XB = 32 * NB_ILP, NB_UNROLL = 8;
constexpr int NB_ZS = 8, NB_ZS_WIDE = 4;   // see nbody_forces
constexpr int NB_RING = 128;    // bodies per cell and threads per CTA (hyper-systolic)

// a += f(x, z): m_z d / (|d|^2 + eps2)^(3/2), d = r_z - r_x
__device__ __forceinline__ void interact(const float4& x, const float4& z, float eps2, float3& a) {
    const float dx = z.x - x.x, dy = z.y - x.y, dz = z.z - x.z;
    const float r2 = fmaf(dx, dx, fmaf(dy, dy, fmaf(dz, dz, eps2)));
    const float inv = rsqrtf(r2);
    const float s = r2 > 0.f ? z.w * (inv * inv * inv) : 0.f;
    a.x = fmaf(s, dx, a.x);
    a.y = fmaf(s, dy, a.y);
    a.z = fmaf(s, dz, a.z);
}

// The forms of the interaction.  The cube of 1/r overflows below r^2 = 2^-85 and one body's pair with
// itself is then infinity times zero; so the packed form is taken for eps2 from 2^-66 on (1/r^3 <= 2^99,
// masses to 2^28), and smaller positive ones multiply in another order, one body at a time.
enum class Form { Zero, Small, Packed };
constexpr float PACKED_EPS2 = 1.3552527e-20f;      // 2^-66
__host__ __device__ __forceinline__ Form form_of(float eps2) {
    return eps2 >= PACKED_EPS2 ? Form::Packed : eps2 > 0.f ? Form::Small : Form::Zero;
}

// a += f(x, z) for any eps2 > 0: m / r and d / r, which stay finite (and 0 for d = 0), before the last 1/r
__device__ __forceinline__ void interact_small(const float4& x, const float4& z, float eps2, float3& a) {
    const float dx = z.x - x.x, dy = z.y - x.y, dz = z.z - x.z;
    const float inv = rsqrtf(fmaf(dx, dx, fmaf(dy, dy, fmaf(dz, dz, eps2))));
    const float m = z.w * inv;
    a.x = fmaf(m * (dx * inv), inv, a.x);
    a.y = fmaf(m * (dy * inv), inv, a.y);
    a.z = fmaf(m * (dz * inv), inv, a.z);
}
template <Form F>
__device__ __forceinline__ void interact_one(const float4& x, const float4& z, float eps2, float3& a) {
    if constexpr (F == Form::Small) interact_small(x, z, eps2, a);
    else interact(x, z, eps2, a);
}

// ---- packed FP32 pairs (f32x2): two x bodies against one z body per instruction ----
__device__ __forceinline__ uint64_t pk2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void upk2(uint64_t v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ float rsqrt_approx(float v) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

// two x bodies (packed coordinates X, Y, Z) against z (coordinates and mass broadcast to both
// halves); Form::Packed: r^2 >= eps2, no pair needs the r = 0 case
struct XPair {
    uint64_t X, Y, Z, ax, ay, az;
};
__device__ __forceinline__ void interact2(XPair& p, uint64_t zx, uint64_t zy, uint64_t zz, uint64_t zm,
                                          uint64_t eps2x2) {
    const uint64_t dx = sub2(zx, p.X), dy = sub2(zy, p.Y), dz = sub2(zz, p.Z);
    const uint64_t r2 = fma2(dx, dx, fma2(dy, dy, fma2(dz, dz, eps2x2)));
    float lo, hi;
    upk2(r2, lo, hi);
    const uint64_t inv = pk2(rsqrt_approx(lo), rsqrt_approx(hi));
    const uint64_t s = mul2(zm, mul2(mul2(inv, inv), inv));
    p.ax = fma2(s, dx, p.ax);
    p.ay = fma2(s, dy, p.ay);
    p.az = fma2(s, dz, p.az);
}

__device__ __forceinline__ XPair make_pair(const float4& a, const float4& b) {
    return XPair{pk2(a.x, b.x), pk2(a.y, b.y), pk2(a.z, b.z), pk2(0.f, 0.f), pk2(0.f, 0.f), pk2(0.f, 0.f)};
}

// 16-byte load from the shared memory of another CTA of the cluster
__device__ __forceinline__ float4 ld_peer_f4(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(addr)
                 : "memory");
    return v;
}

// Tiled schedule.  A CTA owns NB_XB = 128 x bodies, four per lane, and each of its eight warps
// works on its own eighth of every z tile; a cluster of eight CTAs, or four, shares the same x bodies
// and splits z.  Partial sums are added in the fixed order of warps, then cluster ranks, through
// shared and distributed shared memory (deterministic, no workspace).
//   Form::Packed: the four bodies as two packed pairs; else one body at a time.
// Bound by the FP32 pipe: 12 packed instructions per two interactions, so what counts is that
// every scheduler has warps to hide their latency behind.  The 64-way split of z (eight warps x
// eight CTAs) gives an x array of 20000 bodies 1256 CTAs, four resident per SM; with 1024 x bodies
// per CTA it had 140 CTAs on 152 SMs, two warps per scheduler.  z is kept duplicated, (x, x, y, y)
// and (z, z, m, m), so that both halves of a packed operand come from one 16-byte load without
// register moves, and the next tile is fetched into registers while one is used.
// G interactions/s before -> now: 1061 -> 2169 at 20000 bodies, 2236 -> 2490 at 131072; 6.3 us at
// 1000 bodies.  Also measured: four CTAs per cluster (1991 at 20000, 2461 at 131072), 16 (not
// portable, equal at 5000), 64 lanes x 4 warps (2011, 2494), unrolled by 4 (2146, 2468) or 16
// (1989, 2328), two bodies a lane (2011, 2265), six (1776, 2208).
// Launched as a programmatic dependent: resident while the kernel before still writes x or z, which are
// not const __restrict__ for that reason.
template <Form F>
__global__ void __launch_bounds__(NB_THREADS) nbody_tiled(int64_t nx, int64_t nz, const float4* x,
                                                          const float4* z, float eps2,
                                                          float4* out) {
    // two z tiles of NB_THREADS bodies (two float4 each), later the partial sums [warp][body]
    __shared__ float4 sm[2 * 2 * NB_THREADS];
    static_assert(2 * 2 * NB_THREADS >= NB_WARPS * NB_XB, "the partial sums reuse the z tiles");
    constexpr bool PACKED = F == Form::Packed;
    pdl_wait();
    const int lane = int(lane_id()), warp = int(warp_id());
    const int zs = int(cluster_ctarank()), ZS = int(cluster_nctarank());
    const int64_t xblock = int64_t(blockIdx.x / ZS) * NB_XB;
    // this CTA's share of z, in multiples of eight bodies per warp
    constexpr int ZU = NB_UNROLL * NB_WARPS;
    const int64_t zchunk = ((nz + ZS - 1) / ZS + ZU - 1) / ZU * ZU;
    const int64_t zbeg = int64_t(zs) * zchunk;
    const int64_t zend = min(nz, zbeg + zchunk);
    float4 xi[NB_ILP];
#pragma unroll
    for (int k = 0; k < NB_ILP; ++k) {
        const int64_t i = xblock + k * 32 + lane;
        xi[k] = i < nx ? load(x + i) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    float3 a[PACKED ? 1 : NB_ILP];
    XPair pr[PACKED ? NB_ILP / 2 : 1];
    if constexpr (PACKED) {
#pragma unroll
        for (int k = 0; k < NB_ILP / 2; ++k) pr[k] = make_pair(xi[2 * k], xi[2 * k + 1]);
    } else {
#pragma unroll
        for (int k = 0; k < NB_ILP; ++k) a[k] = make_float3(0.f, 0.f, 0.f);
    }
    const uint64_t e2 = pk2(eps2, eps2);
    // padding: zero mass, far from any body (at the origin a body there and a tiny eps2 would
    // give 0 x infinity)
    const float4 pad = make_float4(1e18f, 1e18f, 1e18f, 0.f);
    auto put = [&](int buf, const float4& v) {
        float4* t = sm + buf * 2 * NB_THREADS + 2 * threadIdx.x;
        t[0] = make_float4(v.x, v.x, v.y, v.y);
        t[1] = make_float4(v.z, v.z, v.w, v.w);
    };
    put(0, zbeg + threadIdx.x < zend ? load(z + zbeg + threadIdx.x) : pad);
    __syncthreads();
    int buf = 0;
    for (int64_t j0 = zbeg; j0 < zend; j0 += NB_THREADS) {
        const bool more = j0 + NB_THREADS < zend;
        const int64_t jn = j0 + NB_THREADS + threadIdx.x;
        float4 next = pad;
        if (more && jn < zend) next = load(z + jn);
        // bodies of this tile per warp: 32, fewer (a multiple of eight) in the last one
        const int64_t rem = zend - j0;
        const int cnt = rem >= NB_THREADS ? 32 : int((rem + ZU - 1) / ZU) * NB_UNROLL;
        const float4* t = sm + buf * 2 * NB_THREADS + warp * cnt * 2;
#pragma unroll 8
        for (int q = 0; q < cnt; ++q) {
            if constexpr (PACKED) {
                const ulonglong2 u = *reinterpret_cast<const ulonglong2*>(t + 2 * q);
                const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(t + 2 * q + 1);
#pragma unroll
                for (int k = 0; k < NB_ILP / 2; ++k) interact2(pr[k], u.x, u.y, w.x, w.y, e2);
            } else {
                const float4 u = t[2 * q], w = t[2 * q + 1];
#pragma unroll
                for (int k = 0; k < NB_ILP; ++k) interact_one<F>(xi[k], make_float4(u.x, u.z, w.x, w.z), eps2, a[k]);
            }
        }
        if (more) put(buf ^ 1, next);
        __syncthreads();
        buf ^= 1;
    }
#pragma unroll
    for (int k = 0; k < NB_ILP; ++k) {
        float3 r;
        if constexpr (PACKED) {
            float l0, h0, l1, h1, l2, h2;
            upk2(pr[k / 2].ax, l0, h0);
            upk2(pr[k / 2].ay, l1, h1);
            upk2(pr[k / 2].az, l2, h2);
            r = (k & 1) ? make_float3(h0, h1, h2) : make_float3(l0, l1, l2);
        } else {
            r = a[k];
        }
        sm[warp * NB_XB + k * 32 + lane] = make_float4(r.x, r.y, r.z, 0.f);
    }
    __syncthreads();
    if (threadIdx.x < NB_XB) {
        float4 sum = sm[threadIdx.x];
#pragma unroll
        for (int w = 1; w < NB_WARPS; ++w) {
            const float4 v = sm[w * NB_XB + threadIdx.x];
            sum.x += v.x;
            sum.y += v.y;
            sum.z += v.z;
        }
        sm[threadIdx.x] = sum;
    }
    __syncwarp();
    cluster_sync_all();
    // every rank adds up its 16 bodies of the x block (with eight ranks)
    const int share = (NB_XB + ZS - 1) / ZS;
    for (int b = zs * share + int(threadIdx.x); b < min(NB_XB, (zs + 1) * share); b += NB_THREADS) {
        float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int q = 0; q < ZS; ++q) {
            const float4 v = ld_peer_f4(mapa_shared(smem_u32(&sm[b]), uint32_t(q)));
            sum.x += v.x;
            sum.y += v.y;
            sum.z += v.z;
        }
        if (xblock + b < nx) out[xblock + b] = make_float4(sum.x, sum.y, sum.z, 0.f);
    }
    __syncwarp();
    cluster_sync_all();   // the other ranks keep their partial sums until they have been read
}

template <int K, Form F>
__global__ void __launch_bounds__(NB_RING) nbody_hsys(int64_t nx, int64_t nz, const float4* __restrict__ x,
                                                      const float4* __restrict__ z, float eps2,
                                                      float4* __restrict__ out, int P) {
    constexpr bool PACKED = F == Form::Packed;
    static_assert(!PACKED || K % 2 == 0, "packed replicas come in pairs");
    __shared__ float4 xs[NB_RING];          // this cell's block of x
    __shared__ float4 zb[2][NB_RING];       // the z block held in step s (buffer s % 2) and the next
    __shared__ float4 recv[2][NB_RING];     // back-shift: the collector arriving from the left
    const int c = int(cluster_ctarank());
    const int t = int(threadIdx.x);
    const int Kt = P / K;
    const int64_t cx = int64_t(blockIdx.x) / P;                  // cluster: x blocks cx*P .. cx*P + P-1
    const int64_t xi = (cx * P + c) * NB_RING + t;
    xs[t] = xi < nx ? x[xi] : make_float4(0.f, 0.f, 0.f, 0.f);
    cluster_sync_all();
    // replicas: x^_r at cell c is the block of cell c + r (r shifts of stride 1)
    float4 xr[K];
    float3 acc[K];
#pragma unroll
    for (int r = 0; r < K; ++r) {
        xr[r] = ld_peer_f4(mapa_shared(smem_u32(&xs[t]), uint32_t((c + r) % P)));
        acc[r] = make_float3(0.f, 0.f, 0.f);
    }
    XPair pr[PACKED ? K / 2 : 1];
    if constexpr (PACKED) {
#pragma unroll
        for (int r = 0; r < K / 2; ++r) pr[r] = make_pair(xr[2 * r], xr[2 * r + 1]);
    }
    const uint64_t e2 = pk2(eps2, eps2);
    const int64_t rounds = (nz + int64_t(P) * NB_RING - 1) / (int64_t(P) * NB_RING);
    for (int64_t rd = 0; rd < rounds; ++rd) {
        __syncthreads();                                          // done with buffer 0 of the last round
        const int64_t zj = (rd * P + c) * NB_RING + t;
        zb[0][t] = zj < nz ? z[zj] : make_float4(0.f, 0.f, 0.f, 0.f);   // padding: zero mass
        cluster_sync_all();                                       // every cell holds its own z block
        for (int s = 0; s < Kt; ++s) {
            const float4* zc = zb[s & 1];
#pragma unroll 4
            for (int q = 0; q < NB_RING; ++q) {
                const float4 zq = zc[q];
                if constexpr (PACKED) {
                    const uint64_t zx = pk2(zq.x, zq.x), zy = pk2(zq.y, zq.y), zz = pk2(zq.z, zq.z),
                                   zm = pk2(zq.w, zq.w);
#pragma unroll
                    for (int r = 0; r < K / 2; ++r) interact2(pr[r], zx, zy, zz, zm, e2);
                } else {
#pragma unroll
                    for (int r = 0; r < K; ++r) interact_one<F>(xr[r], zq, eps2, acc[r]);
                }
            }
            if (s + 1 < Kt) {
                // z <- cshift^K(z): this cell takes the block of cell c + K into its other buffer
                zb[(s + 1) & 1][t] = ld_peer_f4(mapa_shared(smem_u32(&zb[s & 1][t]), uint32_t((c + K) % P)));
                cluster_sync_all();
            }
        }
    }
    if constexpr (PACKED) {
#pragma unroll
        for (int r = 0; r < K / 2; ++r) {
            float l0, h0, l1, h1, l2, h2;
            upk2(pr[r].ax, l0, h0);
            upk2(pr[r].ay, l1, h1);
            upk2(pr[r].az, l2, h2);
            acc[2 * r] = make_float3(l0, l1, l2);
            acc[2 * r + 1] = make_float3(h0, h1, h2);
        }
    }
    // back-shift: the collector starts as acc[K-1] and moves one cell to the right K-1 times,
    // adding acc[r] (r = K-2 .. 0) at each arrival; it ends on the cell that owns its block
    float3 y = acc[K - 1];
    const uint32_t right = uint32_t((c + 1) % P);
#pragma unroll
    for (int u = 0; u < K - 1; ++u) {
        const uint32_t dst = mapa_shared(smem_u32(&recv[u & 1][t]), right);
        asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "f"(y.x), "f"(y.y), "f"(y.z),
                     "f"(0.f)
                     : "memory");
        cluster_sync_all();
        const float4 in = recv[u & 1][t];
        const int r = K - 2 - u;
        y = make_float3(in.x + acc[r].x, in.y + acc[r].y, in.z + acc[r].z);
    }
    if (xi < nx) out[xi] = make_float4(y.x, y.y, y.z, 0.f);
    __syncwarp();
    cluster_sync_all();                                           // no cell leaves while peers read it
}

}  // namespace

hsmm_status_t nbody_forces(int64_t nx, int64_t nz, const float* x, const float* z, float eps2, float* out,
                           int ring_p, int ring_k, cudaStream_t st) {
    const float4* x4 = reinterpret_cast<const float4*>(x);
    const float4* z4 = reinterpret_cast<const float4*>(z);
    float4* o4 = reinterpret_cast<float4*>(out);
    const Form form = form_of(eps2);
    if (ring_p == 0) {
        const int64_t xblocks = (nx + NB_XB - 1) / NB_XB;
        if (xblocks > INT32_MAX / NB_ZS) return HSMM_STATUS_NOT_SUPPORTED;
        // Eight CTAs share an x block, four where those alone fill the SMs one and a half times over (four
        // CTAs an SM) and z is at most a tile for each, or the bodies go one by one: a CTA then has
        // twice the z bodies to set up and add up for.  Us, four / eight: 70000 x 900 34.4 / 41.3, 30000 x
        // 1000 17.5 / 19.5, but 50000^2 1038 / 1034 and 20000^2 196 / 178; eps2 = 0: 70000 x 900 53.7 / 69.1,
        // 40000 x 10000 282 / 295, 131072^2 10665 / 11484.
        const bool few = nz <= NB_ZS_WIDE * NB_THREADS || form != Form::Packed;
        const int zs = few && xblocks * NB_ZS_WIDE >= int64_t(num_sms()) * 6 ? NB_ZS_WIDE : NB_ZS;
        const cudaError_t te = pdl_launch(form == Form::Packed  ? nbody_tiled<Form::Packed>
                                          : form == Form::Small ? nbody_tiled<Form::Small>
                                                                : nbody_tiled<Form::Zero>,
                                          dim3(unsigned(xblocks * zs)), NB_THREADS, 0, unsigned(zs), st, nx, nz, x4, z4, eps2, o4);
        count_launches(1);
        if (te != cudaSuccess) return record_cuda(te);
        return check_launch();
    }
    const int P = ring_p, K = ring_k;
    const int64_t clusters = (nx + int64_t(P) * NB_RING - 1) / (int64_t(P) * NB_RING);
    if (clusters * P > INT32_MAX) return HSMM_STATUS_NOT_SUPPORTED;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned(clusters * P), 1, 1);
    cfg.blockDim = dim3(NB_RING, 1, 1);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = unsigned(P);
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    // by K = 1, 2, 4 and form; one replica has no packed pair
    using Kern = void (*)(int64_t, int64_t, const float4*, const float4*, float, float4*, int);
    static constexpr Kern kerns[3][3] = {
        {nbody_hsys<1, Form::Zero>, nbody_hsys<1, Form::Small>, nbody_hsys<1, Form::Zero>},
        {nbody_hsys<2, Form::Zero>, nbody_hsys<2, Form::Small>, nbody_hsys<2, Form::Packed>},
        {nbody_hsys<4, Form::Zero>, nbody_hsys<4, Form::Small>, nbody_hsys<4, Form::Packed>}};
    static std::atomic<uint64_t> attrs{0};
    const hsmm_status_t as = attrs_once_per_device(attrs, [] {
        cudaError_t r = cudaSuccess;
        for (const auto& row : kerns)
            for (const Kern kern : row)
                if (r == cudaSuccess) r = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        return r;
    });
    if (as != HSMM_STATUS_SUCCESS) return as;
    if (K != 1 && K != 2 && K != 4) return HSMM_STATUS_INVALID_VALUE;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kerns[K / 2][int(form)], nx, nz, x4, z4, eps2, o4, P);
    count_launches(1);
    if (e != cudaSuccess) return record_cuda(e);
    return check_launch();
}

}  // namespace hsmm
