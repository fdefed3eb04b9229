// k_mlp_split.cu -- K-c, plain FP32 networks on the tensor cores (tcgen05, sm_103a), their
// operands split into three BF16 parts.
//
// Same network and work unit as the FP32 SIMT path (Sec. 3.1 F_Theta, Sec. 3.2 same-shaped
// networks, samples grouped by node, Sec. 3.5).  An FP32 value has 24 significand bits, a
// BF16 value 8 and FP32's exponents, so v = h + m + l with h = bf16(v), m = bf16(v - h),
// l = bf16(v - h - m) is exact (below about 2^-110, where parts become subnormal, up to an
// absolute 2^-133).  A product of two split values is taken as the six largest of its nine
// partial products -- h h, h m, m h, m m, h l, l h.  |m| is at most 2^-8 and |l| 2^-17 of a
// value, so the three left out (m l, l m, l l) are at most about 2^-24 of the product, as large
// as the one rounding that an FP32 product has, and mostly far smaller.  The tensor cores'
// accumulation truncates where FP32 arithmetic rounds to nearest, so each layer adds its small
// products first (the accumulator then is 2^-8 of the sum, and so is what a truncation drops),
// then the bias, and the h h products last: 5 or 6 accumulations at full size against 64 to 90
// roundings of an FP32 chain.  That this is the SIMT path's precision, and not a lower one, is
// measured:
//
// Against 64 bits (relative 2-norm of the pixels' error, one 800 x 800 view):
// 9.1e-7 with the SIMT kernel, 9.1e-7 here; the networks' own outputs, on the same sample
// positions (256 networks of 4 x 64, 48 x 48 rays): 4.9e-8 (sigma) and 6.4e-8 (rgb) with the
// SIMT kernel, 4.7e-8 and 6.0e-8 here; with weights three times as large 2.5e-7 and 7.4e-7
// with the SIMT kernel, 2.6e-7 and 2.8e-7 here; the largest single error is lower in each.
//
// What bounds it: a 4 x 64 tile takes 135 MMAs, about 4 400 cycles of the tensor pipe, and
// its rows about 2 500 instruction issues per SM sub-partition (nine instructions per split
// pair, 30 per sincospif); three tiles of 168 TMEM columns are in flight per SM, each
// alternating between the two.  One 800 x 800 view (300 k tiles), network step: SIMT kernel
// 37.6 ms (46 % of the FP32 lanes' peak); one thread per row 7.4 ms; two threads per row
// (each half of a chunk's columns, half of an accumulator row) 7.1; with the staging in a
// warp of its own, out of the issuing warps, 6.5 ms.
//
// Structure, as k_mlp_tc: per tile in flight two compute warpgroups, whose threads r and
// r + 128 own sample row (TMEM lane) r, and one auxiliary warp that loads weights and issues
// the MMAs; one more warp stages the crossings of all groups.  A network's split weights
// take three times a BF16 network's (123 KB at 4 x 64), so the groups of a CTA share one
// copy: the CTA's contiguous range of tiles is cut at leaf changes, its groups take a
// leaf's tiles in turn, and at a leaf change the auxiliary warps meet on an mbarrier before
// one of them loads the next leaf's weights.  Layer 0's 96 input columns (90 features, the
// constant 1 of the bias, padding) are written in three chunks of 32 (kPerm): all three h
// parts stay in TMEM for the last products, the m and l parts of a chunk share one buffer.
// The samples of a crossing share their direction's features (eight lanes compute a pair
// each and exchange them, at 8 samples per crossing or more).  While the head runs, a group
// encodes the first chunk of its next tile.  Every wait is bounded.
//
// Overflow: the parts of an infinity do not multiply as it does, so an activation that is
// infinite or NaN gets a NaN among its parts, and a sample whose head sums are NaN is computed
// again in FP32 (fp32_sample).  Its cost where nothing overflows: none measurable at 4 x 64
// (6.16 and 6.14 ms per view without and with it), 2 % at eight layers of 32; where every
// sample overflows an 800 x 800 view takes 161 ms (35 on the SIMT kernel).  A sum whose partial
// sums overflow in one order of its terms and not in another may still come out either way.
//
// Kept on the SIMT kernel: calibration (per-layer input maxima), other encodings than
// lx = 10, ld = 4, and networks whose split weights do not fit the shared memory.
#include <cuda_bf16.h>

#include <type_traits>

#include "amnerf_internal.h"
#include "tc_common.cuh"

namespace amnerf {
namespace {

using namespace tcx;

constexpr int kIn = 90, kInP = 96;  // encoded features; layer 0's K (bias at column 90)
constexpr int kGroups = 3;          // tiles in flight per CTA, 256 threads (two per sample row) each
constexpr int kTPR = 2;             // threads per row
constexpr int kThreads = 128 * (kGroups * kTPR + 1);
constexpr int kBiasK = 16;

// TMEM columns of a group: D (accumulator), A (input parts), the constant ones of the bias
// MMAs.  Layer 0: h parts of the 96 columns in A 0..47, a chunk's m and l parts in A 48..63
// and 64..79; later layers: h, m, l parts in A 0.., 32.., 64...
constexpr uint32_t kCols = 168, kA = 64, kOnes = 160;
constexpr uint32_t kM0 = 48, kL0 = 64;
static_assert(kGroups * kCols <= 512, "TMEM");

// Layer 0's column order: column 2 i + 6 (and the next) hold sin and cos of pair i < 42
// (octave i / 3 of coordinate i % 3 of x, the last 12 of d), columns 0..5 x and d.  Returns
// the canonical feature, -1 for the bias column, -2 for padding.
__host__ __device__ constexpr int kPerm(int c) {
    if (c < 3) return c;
    if (c < 6) return 60 + c;
    if (c == 90) return -1;
    if (c > 90) return -2;
    const int i = (c - 6) >> 1, cosine = (c - 6) & 1;
    return i < 30 ? 3 + 6 * (i / 3) + 3 * cosine + i % 3 : 66 + 6 * ((i - 30) / 3) + 3 * cosine + i % 3;
}

// A network's split weights (bytes): parts p = 0, 1, 2 (h, m, l) of every matrix as BF16
// K-major core matrices; the hidden layers' biases as K = 16 operands (their three parts
// at K columns 10..12, as in k_mlp_tc); the head's FP32 bias.
struct SplitLayout {
    int width, hidden;
    size_t w0, wh, wo, bb, bo, stride;
    __host__ __device__ SplitLayout(int w, int h) : width(w), hidden(h) {
        w0 = 0;
        wh = w0 + 3 * part0();
        wo = wh + (size_t)(h - 1) * 3 * parth();
        bb = wo + 3 * parto();
        bo = bb + (size_t)(h - 1) * w * kBiasK * 2;
        stride = (bo + 16 + 127) / 128 * 128;
    }
    __host__ __device__ size_t part0() const { return (size_t)width * kInP * 2; }
    __host__ __device__ size_t parth() const { return (size_t)width * width * 2; }
    __host__ __device__ size_t parto() const { return (size_t)16 * width * 2; }
};

struct SplitShared {
    uint64_t bar_w;             // a leaf's weights
    uint64_t bar_seg;           // the groups are done with a leaf's weights
    uint64_t bar_a[kGroups];    // input parts written by the eight compute warps
    uint64_t bar_m[kGroups];    // MMAs completed
    uint64_t bar_s[kGroups];    // crossings staged
    uint64_t bar_f[kGroups];    // a tile's staged crossings read by the eight compute warps
    int leaf[kGroups][kIdSlots];
    uint32_t tmem_base;
};
constexpr size_t kShBytes = (sizeof(SplitShared) + 15) & ~(size_t)15;

size_t split_smem(int width, int hidden, int cpt) {
    return SplitLayout(width, hidden).stride + kShBytes + kGroups * stage_bytes(cpt);
}

__device__ __forceinline__ float2 bf16x2_floats(uint32_t p) {
    return make_float2(__uint_as_float(p << 16), __uint_as_float(p & 0xffff0000u));
}

// Two BF16 per word, to nearest, a value beyond the largest finite BF16 to that one.
__device__ __forceinline__ uint32_t pack_bf16_sat(float lo, float hi) {
    uint32_t d;
    asm("cvt.rn.satfinite.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}

// (v0, v1) = h + m + l, two BF16 per word.  h saturates, so that a value above the largest BF16
// stays exact (h + m).  Of an infinity or a NaN at least one part is NaN (m or l of inf - inf),
// so all that a sample's network computes from it is NaN: see fp32_sample.
__device__ __forceinline__ void split3(float v0, float v1, uint32_t& h, uint32_t& m, uint32_t& l) {
    const float2 neg = make_float2(-1.0f, -1.0f);
    h = pack_bf16_sat(v0, v1);
    const float2 r = fma2v(bf16x2_floats(h), neg, make_float2(v0, v1));
    m = pack_bf16(r.x, r.y);
    const float2 s = fma2v(bf16x2_floats(m), neg, r);
    l = pack_bf16(s.x, s.y);
}

// max(v, 0), or NaN.
__device__ __forceinline__ float relu_nan(float v) {
    float r;
    asm("max.NaN.f32 %0, %1, 0f00000000;" : "=f"(r) : "f"(v));
    return r;
}

__device__ __forceinline__ float softplus_f32(float z) { return z > 20.0f ? z : log1pf(expf(z)); }
__device__ __forceinline__ float sigmoid_f32(float z) { return 1.0f / (1.0f + expf(-z)); }

// BF16 to nearest; a finite value that would round to infinity becomes the largest BF16.
__device__ __forceinline__ __nv_bfloat16 bf16_sat(float v) {
    constexpr float kMax = 3.38953139e38f;  // 0x7f7f0000
    return __float2bfloat16_rn(fminf(fmaxf(v, -kMax), kMax));
}

// The FP32 SIMT blob (transposed matrices, see k_mlp_simt.cu) of every network as split
// operands, one element per thread and step; networks over blockIdx.y.
__global__ void k_split_pack(const float* __restrict__ simt, size_t simt_stride, uint8_t* __restrict__ out, int W,
                             int hidden) {
    const SplitLayout lay(W, hidden);
    const float* src = simt + (size_t)blockIdx.y * simt_stride;
    uint8_t* dst = out + (size_t)blockIdx.y * lay.stride;
    const int n0 = W * kInP, nh = (hidden - 1) * W * W, no = 16 * W, nb = (hidden - 1) * W * kBiasK;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n0 + nh + no + nb + 4; i += gridDim.x * blockDim.x) {
        float v = 0.0f;
        size_t at, part;
        if (i < n0) {
            const int n = i / kInP, c = i - n * kInP, f = kPerm(c);
            v = f >= 0 ? src[(size_t)f * W + n] : (f == -1 ? src[(size_t)kIn * W + n] : 0.0f);
            at = lay.w0 + cm_offset(n, c, kInP);
            part = lay.part0();
        } else if (i < n0 + nh) {
            const int e = i - n0, l = e / (W * W), n = (e / W) % W, k = e % W;
            v = src[(size_t)(kIn + 1) * W + (size_t)l * (W * W + W) + (size_t)k * W + n];
            at = lay.wh + (size_t)l * 3 * lay.parth() + cm_offset(n, k, W);
            part = lay.parth();
        } else if (i < n0 + nh + no) {
            const int e = i - n0 - nh, n = e / W, k = e % W;
            const float* wo = src + (size_t)(kIn + 1) * W + (size_t)(hidden - 1) * (W * W + W);
            v = n < 4 ? wo[(size_t)k * 4 + n] : 0.0f;
            at = lay.wo + cm_offset(n, k, W);
            part = lay.parto();
        } else if (i < n0 + nh + no + nb) {
            const int e = i - n0 - nh - no, l = e / (W * kBiasK), n = (e / kBiasK) % W, k = e % kBiasK;
            const int p = k - (kOnesCol - kOnesStep);  // which part this K column carries
            const float b = src[(size_t)(kIn + 1) * W + (size_t)l * (W * W + W) + (size_t)W * W + n];
            const float h = __bfloat162float(bf16_sat(b)), m = __bfloat162float(__float2bfloat16_rn(b - h));
            v = p == 0 ? h : (p == 1 ? m : (p == 2 ? b - h - m : 0.0f));
            *reinterpret_cast<__nv_bfloat16*>(dst + lay.bb + (size_t)l * W * kBiasK * 2 + cm_offset(n, k, kBiasK)) =
                __float2bfloat16_rn(v);
            continue;
        } else {
            const int n = i - n0 - nh - no - nb;
            reinterpret_cast<float*>(dst + lay.bo)[n] =
                src[(size_t)(kIn + 1) * W + (size_t)(hidden - 1) * (W * W + W) + 4 * W + n];
            continue;
        }
        const __nv_bfloat16 h = bf16_sat(v);
        const float r = v - __bfloat162float(h);
        const __nv_bfloat16 m = __float2bfloat16_rn(r);
        *reinterpret_cast<__nv_bfloat16*>(dst + at) = h;
        *reinterpret_cast<__nv_bfloat16*>(dst + at + part) = m;
        *reinterpret_cast<__nv_bfloat16*>(dst + at + 2 * part) = __float2bfloat16_rn(r - __bfloat162float(m));
    }
}

// Sample j of crossing id by a whole converged warp in FP32, from k_mlp_simt's copy of the leaf's
// weights and with its operations in its order: each lane holds W / 32 activations, a layer's
// inputs go round by shuffles.  For samples whose tensor-core result is NaN: an activation
// overflowed (or the input is not finite), and the split of an infinity has no products that add
// up to FP32's.  Microseconds per sample; out of line, so that it costs the kernel no registers.
template <int W, bool JIT>
__device__ __noinline__ void fp32_sample(const MlpArgs& g, int leaf, int hidden, uint32_t id, int j) {
    constexpr int R = W / 32;
    const int lane = threadIdx.x & 31;
    const float* w = g.weights_fp32 + (size_t)leaf * (g.leaf_stride / sizeof(float));
    const uint32_t ray = id / (uint32_t)g.maxc;
    const float2 xi = __ldcg(g.xing + id);
    float x[3], d[3], o[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        o[a] = __ldg(g.ro + 3 * (size_t)ray + a);
        d[a] = __ldg(g.rd + 3 * (size_t)ray + a);
    }
    const float delta = __fmul_rn(__fsub_rn(xi.y, xi.x), __frcp_rn((float)g.steps));
    float u = 0.5f;
    if (JIT)
        u = jit_fraction(g.jitter, jit_ray_key(g.jitter, o, d), (int)(id - ray * (uint32_t)g.maxc), g.steps, j);
    const float tj = __fadd_rn(xi.x, __fmul_rn(__fadd_rn((float)j, u), delta));
#pragma unroll
    for (int a = 0; a < 3; ++a) x[a] = __fadd_rn(o[a], __fmul_rn(tj, d[a]));
    float in[3];  // inputs lane, lane + 32, lane + 64
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const int f = lane + 32 * i, e = f < 63 ? f - 3 : f - 66;  // e < 0: the coordinate itself
        const int a = f < 3 ? f : (f >= 63 && f < 66 ? f - 63 : e % 3);
        const float p = f < 63 ? (a == 0 ? x[0] : (a == 1 ? x[1] : x[2])) : (a == 0 ? d[0] : (a == 1 ? d[1] : d[2]));
        in[i] = p;
        if (e >= 0 && f < kIn) {
            float sn, cs;
            sincospif(p * (float)(1 << (e / 6)), &sn, &cs);
            in[i] = e % 6 < 3 ? sn : cs;
        }
    }
    float h[R];
    auto layer = [&](const float* v, int kin) {
        const float* b = w + (size_t)kin * W;
        float acc[R];
#pragma unroll
        for (int r = 0; r < R; ++r) acc[r] = __ldg(b + lane + 32 * r);
        for (int k0 = 0; k0 < kin; k0 += 32) {
            const float vk = k0 == 0 ? v[0] : (k0 == 32 ? v[1] : v[2]);
#pragma unroll 8
            for (int k = 0; k < min(32, kin - k0); ++k) {
                const float a = __shfl_sync(0xffffffffu, vk, k);
#pragma unroll
                for (int r = 0; r < R; ++r) acc[r] = fmaf(a, __ldg(w + (size_t)(k0 + k) * W + lane + 32 * r), acc[r]);
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) h[r] = fmaxf(acc[r], 0.0f);
        w = b + W;
    };
    layer(in, kIn);
    for (int l = 1; l < hidden; ++l) {
        const float v[3] = {h[0], h[R - 1], 0.0f};
        layer(v, W);
    }
    float z = 0.0f;
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll 8
        for (int k = 0; k < 32; ++k)
            z = fmaf(__shfl_sync(0xffffffffu, h[r], k), __ldg(w + (size_t)(32 * r + k) * 4 + (lane & 3)), z);
    z += __ldg(w + 4 * W + (lane & 3));
    if (lane < 4)
        reinterpret_cast<float*>(static_cast<float4*>(g.slot_out) + sample_slot(g, id, j))[lane] =
            lane == 0 ? softplus_f32(z) : sigmoid_f32(z);
}

// HC > 0: the number of hidden layers fixed at compile time.
template <int W, int HC, bool JIT>
__global__ void __launch_bounds__(kThreads, 1) k_mlp_split(const __grid_constant__ MlpArgs g) {
    const int hidden = HC > 0 ? HC : g.hidden;
    extern __shared__ __align__(1024) uint8_t smem[];
    const SplitLayout lay(W, hidden);
    SplitShared* sh = reinterpret_cast<SplitShared*>(smem + lay.stride);
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);  // uniform for the compiler
    const int q = warp & 3, lane_id = threadIdx.x & 31;
    const int row = 32 * q + lane_id;  // sample row = TMEM lane (two threads: half 0 and 1)
    const int half = (warp >> 2) & 1;
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&sh->bar_w), 1);
        mbar_init(smem_u32(&sh->bar_seg), kGroups);
        for (int i = 0; i < kGroups; ++i) {
            mbar_init(smem_u32(&sh->bar_a[i]), 4 * kTPR);
            mbar_init(smem_u32(&sh->bar_m[i]), 1);
            mbar_init(smem_u32(&sh->bar_s[i]), kStageArrivals);
            mbar_init(smem_u32(&sh->bar_f[i]), 4 * kTPR);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_proxy_async();
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sh->tmem_base)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sh->tmem_base;
    grid_wait();  // a chained launch: the crossings and their grouping

    const bool aux = warp >= 4 * kGroups * kTPR;
    const int gi = aux ? q : warp >> 3;  // this warp's group (aux: warp i of the last warpgroup serves group i)
    const int gc = gi < kGroups ? gi : 0;
    const uint32_t bar_a = smem_u32(&sh->bar_a[gc]);
    const uint32_t bar_m = smem_u32(&sh->bar_m[gc]);
    const uint32_t bar_s = smem_u32(&sh->bar_s[gc]);
    const uint32_t bar_f = smem_u32(&sh->bar_f[gc]);
    const uint32_t d_col = tmem + kCols * (uint32_t)gc;
    const uint32_t a_col = d_col + kA;
    const int cpt = kTileRows >> g.lg_steps;
    uint8_t* stage = reinterpret_cast<uint8_t*>(sh) + kShBytes + gc * stage_bytes(cpt);
    volatile int* leaf_s = sh->leaf[gc];
    const uint8_t* wall = reinterpret_cast<const uint8_t*>(g.weights);
    bool ok = true;  // the same in every thread of a warp
    auto wait = [&](uint32_t bar, uint32_t phase) {
        ok = __all_sync(0xffffffffu, mbar_wait_bounded(bar, phase));
        return ok;
    };
    // this CTA's contiguous range of tiles; group i takes tiles t0 + i, t0 + i + kGroups, ...
    const uint32_t t_end = g.t_end == 0xffffffffu ? (uint32_t)__ldcg(g.stats + 1) : g.t_end;
    const uint32_t span = t_end > g.t_begin ? t_end - g.t_begin : 0u;
    const uint32_t per = (span + gridDim.x - 1) / gridDim.x;
    const uint32_t t0 = min(g.t_begin + blockIdx.x * per, t_end);
    const uint32_t t1 = min(t0 + per, t_end);

    if (aux) {
        if (gi < kGroups) {
            const uint32_t w_addr = smem_u32(smem);
            const uint32_t bar_w = smem_u32(&sh->bar_w), bar_seg = smem_u32(&sh->bar_seg);
            const uint64_t desc0 = sdesc(w_addr + (uint32_t)lay.w0, kInP * 16u);
            const uint64_t desch = sdesc(w_addr + (uint32_t)lay.wh, (uint32_t)W * 16u);
            const uint64_t desco = sdesc(w_addr + (uint32_t)lay.wo, (uint32_t)W * 16u);
            const uint64_t descb = sdesc(w_addr + (uint32_t)lay.bb, kBiasK * 16u);
            const uint32_t p0 = (uint32_t)(lay.part0() >> 4), ph_ = (uint32_t)(lay.parth() >> 4),
                           po = (uint32_t)(lay.parto() >> 4);
            const uint32_t idd = idesc_bf16(W), idh = idesc_bf16(16);
            uint32_t ph_a = 0, ph_w = 0, ph_seg = 0, n_m = 0;  // n_m: phases of bar_m committed
            uint32_t n = 0;
            // the leaves of the CTA's range in order, each with its tiles of this group
            uint32_t t = t0;
            int leaf = t0 < t1 ? leaf_of_tile_warp(g.tile_off, 0, g.n_leaves, t0) : 0;
            while (t < t1 && ok) {
                if (t > t0) {  // every group is done with the previous leaf's weights
                    if (n_m > 0 && !wait(bar_m, (n_m - 1u) & 1u)) break;
                    if (lane_id == 0) mbar_arrive(bar_seg);
                    if (gi == 0 && !wait(bar_seg, ph_seg)) break;
                    ph_seg ^= 1u;
                }
                if (gi == 0 && lane_id == 0) {
                    fence_proxy_async();
                    bulk_load(w_addr, wall + (size_t)leaf * lay.stride, (uint32_t)lay.stride, bar_w);
                }
                if (!wait(bar_w, ph_w)) break;
                ph_w ^= 1u;
                const uint32_t seg_end = min(t1, __ldcg(g.tile_off + leaf + 1));
                // this group's tiles below seg_end: numbers n with t0 + gi + kGroups n < seg_end
                for (; t0 + (uint32_t)gi + kGroups * n < seg_end && ok; ++n) {
                    // layer 0: per chunk the small products, after the last chunk the large ones
#pragma unroll 1
                    for (int c = 0; c < 3; ++c) {
                        if (!wait(bar_a, ph_a)) break;
                        ph_a ^= 1u;
                        tc_fence_after();
                        for (int s = 2 * c; s < 2 * c + 2; ++s) {
                            const uint32_t ah = a_col + 8u * s, am = a_col + kM0 + 8u * (s & 1),
                                           al = a_col + kL0 + 8u * (s & 1);
                            const uint64_t b = desc0 + 16u * s;
                            mma_bf16_ts_warp(d_col, am, b + p0, idd, s > 0 ? 1u : 0u);
                            mma_bf16_ts_warp(d_col, al, b, idd, 1u);
                            mma_bf16_ts_warp(d_col, ah, b + 2 * p0, idd, 1u);
                            mma_bf16_ts_warp(d_col, am, b, idd, 1u);
                            mma_bf16_ts_warp(d_col, ah, b + p0, idd, 1u);
                        }
                        if (c == 2)
                            for (int s = 0; s < 6; ++s) mma_bf16_ts_warp(d_col, a_col + 8u * s, desc0 + 16u * s, idd, 1u);
                        mma_commit_warp(bar_m);
                        ++n_m;
                    }
                    if (!ok) break;
                    // later layers, and the head onto D columns 0..15
#pragma unroll 1
                    for (int l = 1; l <= hidden; ++l) {
                        if (!wait(bar_a, ph_a)) break;
                        ph_a ^= 1u;
                        tc_fence_after();
                        const bool head = l == hidden;
                        const uint64_t b0 = head ? desco : desch + (uint64_t)(3u * (uint32_t)(l - 1)) * ph_;
                        const uint32_t pp = head ? po : ph_, id = head ? idh : idd;
                        for (int s = 0; s < W / 16; ++s) {
                            const uint32_t ah = a_col + 8u * s;
                            const uint64_t b = b0 + 16u * s;
                            mma_bf16_ts_warp(d_col, ah + 32u, b + pp, id, s > 0 ? 1u : 0u);
                            mma_bf16_ts_warp(d_col, ah + 64u, b, id, 1u);
                            mma_bf16_ts_warp(d_col, ah, b + 2 * pp, id, 1u);
                        }
                        for (int s = 0; s < W / 16; ++s) {
                            const uint32_t ah = a_col + 8u * s;
                            const uint64_t b = b0 + 16u * s;
                            mma_bf16_ts_warp(d_col, ah + 32u, b, id, 1u);
                            mma_bf16_ts_warp(d_col, ah, b + pp, id, 1u);
                        }
                        if (!head)
                            mma_bf16_ts_warp(d_col, d_col + kOnes,
                                             descb + (uint64_t)((uint32_t)(l - 1) * (W * kBiasK * 2 / 16)), id, 1u);
                        for (int s = 0; s < W / 16; ++s) mma_bf16_ts_warp(d_col, a_col + 8u * s, b0 + 16u * s, id, 1u);
                        mma_commit_warp(bar_m);
                        ++n_m;
                    }
                }
                t = seg_end;
                if (t < t1) leaf = leaf_of_tile_warp(g.tile_off, leaf + 1, g.n_leaves, t);
            }
            if (!ok && lane_id == 0) atomicCAS(g.err, 0, kDevErrTimeout);
        } else {
            // the last warp stages every group's crossings: ids three tiles, intervals and rays
            // two tiles ahead of what the group reads
            auto group = [&](int i) {
                return Stager(g, reinterpret_cast<uint8_t*>(sh) + kShBytes + i * stage_bytes(cpt), sh->leaf[i],
                              smem_u32(&sh->bar_s[i]), cpt, t0 + (uint32_t)i, kGroups, t1);
            };
            Stager st[kGroups] = {group(0), group(1), group(2)};
            uint32_t k[kGroups], last[kGroups];  // tiles whose reading is awaited next, and in all
#pragma unroll
            for (int i = 0; i < kGroups; ++i) {
                k[i] = 0;
                last[i] = t0 + (uint32_t)i < t1 ? (t1 - t0 - (uint32_t)i + kGroups - 1) / kGroups : 0u;
                for (uint32_t n = 0; n < 3; ++n) st[i].ids(n);
            }
            cp_async_wait_all();
            __syncwarp();
#pragma unroll
            for (int i = 0; i < kGroups; ++i) {
                st[i].data(0);
                st[i].data(1);
                st[i].publish();
            }
            // tile k's crossings read (and with them phase k awaited): tile k + 2's may take
            // their slot, and be published as phase k + 1
            unsigned long long since = clock64();
            while (k[0] < last[0] || k[1] < last[1] || k[2] < last[2]) {
                bool any = false;
#pragma unroll
                for (int i = 0; i < kGroups; ++i) {
                    if (k[i] < last[i] && __all_sync(0xffffffffu, mbar_test(smem_u32(&sh->bar_f[i]), k[i] & 1u))) {
                        cp_async_wait_all();  // tile k + 2's ids, copied a tile ago
                        __syncwarp();
                        st[i].data(k[i] + 2);
                        st[i].publish();
                        st[i].ids(k[i] + 3);
                        ++k[i];
                        any = true;
                    }
                }
                const unsigned long long now = clock64();
                if (any) since = now;
                if (!__all_sync(0xffffffffu, now - since <= kWaitCycles)) {
                    if (lane_id == 0) atomicCAS(g.err, 0, kDevErrTimeout);
                    break;
                }
            }
            cp_async_wait_all();  // none in flight when the CTA ends
        }
    } else {
        const uint32_t lane = (uint32_t)(32 * q) << 16;
        const uint32_t d_row = d_col + lane, a_row = a_col + lane;
        if (half == 0) {
            const uint32_t c8[8] = {0u, 0u, 0u, 0u, 0u, pack_bf16(1.0f, 1.0f), pack_bf16(1.0f, 0.0f), 0u};
            tmem_st8(d_row + kOnes, c8);
        }
        const int ci = row >> g.lg_steps, j = row - (ci << g.lg_steps);
        const bool share = g.lg_steps >= 3;  // lanes 8 i .. 8 i + 7 belong to one crossing
        auto publish = [&]() {
            tmem_st_wait();
            tc_fence_before();
            __syncwarp();
            if (lane_id == 0) mbar_arrive(bar_a);
        };
        float x[3] = {0.f, 0.f, 0.f}, d[3] = {0.f, 0.f, 0.f};
        // this half's eight words (column pairs) of a chunk of the layer-0 input, split
        uint32_t wh[8], wm[8], wl[8];
        // pair p < 42: sine and cosine
        auto pair = [&](int p, float& v0, float& v1) {
            const int oct = p < 30 ? p / 3 : (p - 30) / 3;
            sincospif((p < 30 ? x[p % 3] : d[p % 3]) * (float)(1 << oct), &v0, &v1);
        };
        auto encode_half = [&](auto chunk, auto hv) {
            constexpr int C = decltype(chunk)::value, H = decltype(hv)::value;
            constexpr int P0 = (32 * C + 16 * H - 6) / 2;  // pair of word 0 (chunk 0, half 0: from word 3)
            constexpr int D0 = P0 < 30 ? 30 - P0 : 0;      // first word that holds a direction pair ...
            constexpr int D1 = P0 + 8 < 42 ? 8 : 42 - P0;  // ... and one past the last
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int col = 32 * C + 16 * H + 2 * i;
                float v0, v1;
                if (col < 6) {
                    v0 = col == 0 ? x[0] : (col == 2 ? x[2] : d[1]);
                    v1 = col == 0 ? x[1] : (col == 2 ? d[0] : d[2]);
                } else if (P0 + i < 42) {
                    if (C == 2 && i >= D0 && share) continue;
                    pair(P0 + i, v0, v1);
                } else {  // the bias column's 1, then padding
                    v0 = P0 + i == 42 ? 1.0f : 0.0f;
                    v1 = 0.0f;
                }
                split3(v0, v1, wh[i], wm[i], wl[i]);
            }
            if (C == 2 && share) {
                // the eight samples of a crossing share its direction: lane L of every eight
                // computes word D0 + L, then all read them
                const int p = min(P0 + D0 + (lane_id & 7), 41) - 30;
                const int a = p % 3;
                float v0, v1;
                uint32_t h, m, l;
                sincospif((a == 0 ? d[0] : (a == 1 ? d[1] : d[2])) * (float)(1 << (p / 3)), &v0, &v1);
                split3(v0, v1, h, m, l);
#pragma unroll
                for (int i = D0; i < D1; ++i) {
                    wh[i] = __shfl_sync(0xffffffffu, h, i - D0, 8);
                    wm[i] = __shfl_sync(0xffffffffu, m, i - D0, 8);
                    wl[i] = __shfl_sync(0xffffffffu, l, i - D0, 8);
                }
            }
            pin(wh);
            pin(wm);
            pin(wl);
        };
        auto encode = [&](auto chunk) {
            if (half == 0) encode_half(chunk, std::integral_constant<int, 0>());
            else encode_half(chunk, std::integral_constant<int, 1>());
        };
        auto store = [&](int c) {
            tmem_st8(a_row + 16u * c + 8u * half, wh);
            tmem_st8(a_row + kM0 + 8u * half, wm);
            tmem_st8(a_row + kL0 + 8u * half, wl);
            publish();
        };
        float4 bo = make_float4(0.f, 0.f, 0.f, 0.f);
        uint32_t id = 0xffffffffu, ph_m = 0;
        int cur = -1;
        // reads tile n's staged sample; phase n of bar_s (tile n + 1's crossings) has been awaited,
        // so that the staging warp's next phase cannot be mistaken for it
        auto place = [&](uint32_t n) {
            id = staged_sample<JIT>(g, stage, cpt, n, ci, j, x, d);
            __syncwarp();
            if (lane_id == 0) mbar_arrive(bar_f);
        };
        if (wait(bar_s, 0u) && leaf_s[0] >= 0) {
            place(0);
            encode(std::integral_constant<int, 0>());
            store(0);
        }
        for (uint32_t n = 0; ok; ++n) {
            const int leaf = leaf_s[n & (kIdSlots - 1)];
            if (leaf < 0) break;
            if (leaf != cur) {
                bo = __ldg(reinterpret_cast<const float4*>(wall + (size_t)leaf * lay.stride + lay.bo));
                cur = leaf;
            }
            // the m and l buffer is free when the previous chunk's small products are done
            encode(std::integral_constant<int, 1>());
            if (!wait(bar_m, ph_m)) break;
            ph_m ^= 1u;
            tc_fence_after();
            store(1);
            encode(std::integral_constant<int, 2>());
            if (!wait(bar_m, ph_m)) break;
            ph_m ^= 1u;
            tc_fence_after();
            store(2);
#pragma unroll 1
            for (int l = 0; l < hidden; ++l) {
                if (!wait(bar_m, ph_m)) break;
                ph_m ^= 1u;
                tc_fence_after();
                // relu of this half of the accumulator row, split, as the next layer's (or the
                // head's) input, 16 columns at a time
#pragma unroll
                for (int i0 = 0; i0 < W / 32; ++i0) {
                    const uint32_t col = (uint32_t)(W / 2) * half + 16u * i0;
                    uint32_t v[16];
                    tmem_ld16_nowait(d_row + col, v);
                    tmem_ld_wait_regs(v);
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        split3(relu_nan(__uint_as_float(v[2 * i])), relu_nan(__uint_as_float(v[2 * i + 1])), wh[i], wm[i], wl[i]);
                    tmem_st8(a_row + col / 2, wh);
                    tmem_st8(a_row + 32u + col / 2, wm);
                    tmem_st8(a_row + 64u + col / 2, wl);
                }
                publish();
            }
            if (!ok) break;
            // under the head: the next tile's sample and first chunk
            const uint32_t id_cur = id;
            if (!wait(bar_s, (n + 1) & 1u)) break;
            place(n + 1);
            const bool more = leaf_s[(n + 1) & (kIdSlots - 1)] >= 0;
            encode(std::integral_constant<int, 0>());
            if (!wait(bar_m, ph_m)) break;
            ph_m ^= 1u;
            tc_fence_after();
            uint32_t z[4];
            if (half == 0) {
                tmem_ld4_nowait(d_row, z);
                tmem_ld_wait_regs(z);
            }
            if (more) store(0);
            if (half == 0) {
                bool nan = false;
#pragma unroll
                for (int c = 0; c < 4; ++c) nan |= isnan(__uint_as_float(z[c]));
                if (id_cur != 0xffffffffu && !nan) {
                    float4 o;
                    o.x = softplus_f32(__uint_as_float(z[0]) + bo.x);
                    o.y = sigmoid_f32(__uint_as_float(z[1]) + bo.y);
                    o.z = sigmoid_f32(__uint_as_float(z[2]) + bo.z);
                    o.w = sigmoid_f32(__uint_as_float(z[3]) + bo.w);
                    static_cast<float4*>(g.slot_out)[sample_slot(g, id_cur, j)] = o;
                }
                uint32_t redo = __ballot_sync(0xffffffffu, nan && id_cur != 0xffffffffu);
                for (; redo; redo &= redo - 1u) {
                    const int src = __ffs(redo) - 1;
                    fp32_sample<W, JIT>(g, cur, hidden, __shfl_sync(0xffffffffu, id_cur, src),
                                        __shfl_sync(0xffffffffu, j, src));
                }
            }
        }
        if (!ok && lane_id == 0) atomicCAS(g.err, 0, kDevErrTimeout);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}

template <int W>
constexpr int kHiddenFor = W == 64 ? 4 : 2;

template <int W>
cudaError_t prepare_w(int max_smem) {
    const void* fns[4] = {(const void*)k_mlp_split<W, 0, false>, (const void*)k_mlp_split<W, 0, true>,
                          (const void*)k_mlp_split<W, kHiddenFor<W>, false>,
                          (const void*)k_mlp_split<W, kHiddenFor<W>, true>};
    for (const void* f : fns) {
        const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <int W>
cudaError_t launch_w(cudaStream_t s, const MlpArgs& a, int grid, size_t smem) {
    const bool hc = a.hidden == kHiddenFor<W>;
    void (*kern)(const MlpArgs) = a.jitter ? (hc ? k_mlp_split<W, kHiddenFor<W>, true> : k_mlp_split<W, 0, true>)
                                     : (hc ? k_mlp_split<W, kHiddenFor<W>, false> : k_mlp_split<W, 0, false>);
    return launch_after(s, a.chain, kern, (unsigned)grid, (unsigned)kThreads, smem, a);
}

}  // namespace

size_t split_leaf_stride_bytes(int width, int hidden, int lx, int ld) {
    if (lx != 10 || ld != 4 || (width != 32 && width != 64)) return 0;
    return SplitLayout(width, hidden).stride;
}

bool split_fits(int width, int hidden, int steps) {
    int dev = 0, max_smem = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        return false;
    return split_smem(width, hidden, kTileRows / steps) <= (size_t)max_smem;
}

cudaError_t prepare_mlp_split(int width) {
    int dev = 0, max_smem = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    return width == 64 ? prepare_w<64>(max_smem) : prepare_w<32>(max_smem);
}

cudaError_t launch_split_pack(cudaStream_t s, const float* simt, size_t simt_stride, int n_nets, int width, int hidden,
                              void* out) {
    if (n_nets < 1) return cudaSuccess;
    const int elems = width * kInP + (hidden - 1) * width * (width + kBiasK) + 16 * width + 4;
    const dim3 grid((unsigned)((elems + 255) / 256), (unsigned)n_nets);
    k_split_pack<<<grid, 256, 0, s>>>(simt, simt_stride, static_cast<uint8_t*>(out), width, hidden);
    return cudaGetLastError();
}

cudaError_t launch_mlp_split(cudaStream_t s, const MlpArgs& a, int grid) {
    int dev = 0, max_smem = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    size_t smem = split_smem(a.width, a.hidden, kTileRows >> a.lg_steps);
    if (smem > (size_t)max_smem) return cudaErrorInvalidConfiguration;
    // more than half of the SM's shared memory: a second CTA can never become resident and
    // wait in tcgen05.alloc for columns that this one holds
    if (smem < (size_t)max_smem / 2 + 1024) smem = (size_t)max_smem / 2 + 1024;
    if (a.width == 64) return launch_w<64>(s, a, grid, smem);
    if (a.width == 32) return launch_w<32>(s, a, grid, smem);
    return cudaErrorInvalidValue;
}

}  // namespace amnerf
