// Localized Gram matrices as one matrix product on the 5th-generation tensor cores (tcgen05).
//
// Every entry of A_p = sum_o G_po dy_o dy_o^T / sigma_o^2 and c_p = sum_o G_po dy_o d_o / sigma_o^2
// (Eqs. letkf_q, letkf_wa; R-localization of Sec. II-B) is the same weighted sum over the
// observation points: with z_o the upper triangle of sum_v dy_ov dy_ov^T / sigma_ov^2 followed by
// sum_v dy_ov d_ov / sigma_ov^2 (v the observed variables, which share the weight G_po),
//     [A_p | c_p] = sum_o G_po z_o        (points x observations) x (observations x pairs).
// The products dy dy^T are formed once per observation point (gram_z_kernel) instead of once per
// (grid point, observed scalar), and the operand built per grid point is one number per
// observation point instead of k per scalar.
//
// Precision: W = G and Z are split into three BF16 parts each (8 + 8 + 8 = 24 significant bits,
// the exponent range of FP32, so no scaling and no overflow), and the six products hh, hm, mh,
// mm, hl, lh are formed; what is dropped is below 2^-24 relative.  Z is formed with compensated
// FP32 arithmetic, so its split carries the exact products to 24 bits.  The tensor cores'
// FP32 accumulation truncates, which over a whole patch biased the sums by -2.8e-6 relative
// (228 accumulations at r = 12, every fourth point observed), so an accumulator only holds one
// step of 32 observation slots, small products first (two accumulations at full size), and the
// steps are added in registers with round-to-nearest.
//
// Tiling: D[128 pairs x 256 grid points] (M = pairs, so that a warp's lanes store neighbouring
// entries of a Gram slot; N = a 16 x 16 tile of grid points), two such accumulators in turn (all
// 512 tensor-memory columns).  Work items run pair-tile-major, so that the CTAs of the chip read
// the same columns of Z at a time and those stay in L2.
//
// Warp roles of one persistent CTA per SM, linked by mbarrier rings:
//   warp 0       meta: walks the tile's patch (per bin row of the observation bins the x range
//                within the cutoff, a contiguous run of Z's rows) and publishes steps of 32
//                observation slots in four groups of 8 consecutive rows
//   warp 1       TMA: the groups' rows of Z (three parts) into a ring of stages
//   warp 2       MMA issue: 2 K-steps x 6 products per step
//   warps 4..7   weights: each thread two grid points, G for the step's 32 slots, three parts
//   warps 8..15  sums: tensor memory added into registers per step, then stored to the Gram
//                slots and c in global memory
// Measured (Gram phase, z included): 1024^2, k = 64, r = 12, every fourth point observed 93.7 ms ->
// 15.05 ms (CUDA cores in FP32; the split-FP16 tensor form 48.4 ms); 256^2, k = 32, r = 8, every
// eighth point 0.393 -> 0.110 ms; 250 x 187, k = 40, three variables, Gaspari-Cohn 2.16 -> 0.33 ms.
// Relative error of A against 64 bits (256^2, k = 64, spread 5e-3): 4.2e-7 -> 1.8e-7.  The tensor
// pipe needs about 8 ms of the 15.05 (18 pair tiles x 20 steps x 12 MMAs of 128 cycles per tile);
// the weights' FP32 work (about 1,000 issue slots per scheduler and step) bounds it next.
// Every wait is bounded in time: on expiry the status word gets ST_TIMEOUT, all roles leave, the
// copies and MMAs in flight are awaited (bounded) and the tensor memory is freed.
//
// A non-finite product would reach every point of a tile through 0 x inf: gram_z_kernel puts zeros
// in its place and marks the row, and gram_fix() adds the marked rows' non-finite products to the
// points within their cutoff, after the sums are stored and only in tiles whose patch holds such a
// row.  Gram phase at 256^2, k = 64, r = 12: finite 0.97 ms, one NaN observation 1.16, a whole member
// NaN 2.5 (every point's own observations summed per entry in such a case: 372 ms).
#include <cuda.h>
#include <cuda_bf16.h>

#include <mutex>

#include "common.cuh"
#include "kernels.h"
#include "tcgen05.cuh"

namespace lk {
namespace {

using namespace tc;

constexpr int kTW = kGemmTile, kTH = kGemmTile, kPts = kTW * kTH;  // grid points per tile (N)
constexpr int kMT = 128;                       // pairs per accumulator (M)
constexpr int kKC = 32, kGroups = kKC / 8;     // observation slots per step, groups of 8 rows
constexpr int kBoxB = 3 * 8 * 128;             // one TMA box: 3 parts x 8 rows x 64 pairs
constexpr int kZStage = 2 * kGroups * kBoxB;   // 24576: two 64-pair halves
constexpr int kWPart = kPts * kKC * 2;         // 16384: one part of the weights
constexpr int kWStage = 3 * kWPart;
constexpr int kNZ = 4, kNW = 2, kNM = 6;       // ring lengths
constexpr int kWSbo = (kKC / 8) * 128;         // bytes between 8-point core blocks
constexpr int kThreads = 512;
constexpr int kWarpMeta = 0, kWarpTma = 1, kWarpMma = 2, kWarpProd = 4, kWarpSum = 8;
constexpr int kProdWarps = 4, kSumWarps = 8;
// registers per thread of the three roles (setmaxnreg): the sums hold 128 accumulators and read
// 16 columns at a time (32 would take 184 and leave the weights' warps 88: 15.5 ms against 15.05);
// the block is launched with 512 x 128
constexpr int kRegMisc = 56, kRegProd = 120, kRegSum = 168;
static_assert(kRegMisc + kRegProd + 2 * kRegSum <= 4 * 128, "the launch's registers");
constexpr uint32_t kCols = 512;

struct Step {                                  // one published step of 32 slots
    float2 xy[kKC];                            // coordinates from the tile's origin, the image
                                               // nearest its centre; NaN: none (weight 0)
    int start[kGroups];                        // first row of Z of each group
    int last;                                  // last step of the work item
    int pad[3];
};

constexpr int kOffZ = 0;
constexpr int kOffW = kOffZ + kNZ * kZStage;
constexpr int kOffM = kOffW + kNW * kWStage;
constexpr int kSmem = kOffM + kNM * (int)sizeof(Step);
static_assert(kSmem + 1024 <= 227 * 1024 - 512, "shared memory");

// tcgen05 descriptor of the pair operand: MN-major, 128-byte swizzle; LBO: next 64 pairs,
// SBO: next 8 observation rows
__device__ __forceinline__ uint64_t zdesc(uint32_t addr) {
    return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)((kGroups * kBoxB) >> 4) << 16) |
           ((uint64_t)(kBoxB >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
// instruction descriptor: FP32 accumulator, BF16 A (MN-major) and B (K-major)
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) |
                            ((uint32_t)(kPts >> 3) << 17) | ((uint32_t)(kMT >> 4) << 24);

__device__ __forceinline__ float2 bf2f(__nv_bfloat162 v) { return __bfloat1622float2(v); }
__device__ __forceinline__ uint32_t bits(__nv_bfloat162 v) {
    return *reinterpret_cast<uint32_t *>(&v);
}

// Localization weight of squared distance d2 (<= the cutoff).
template <int KIND>
__device__ __forceinline__ float weight_d2(const ObsNet &net, float d2) {
    if (KIND == 0) return 1.0f;
    if (KIND == 2) return gaspari_cohn(sqrtf(d2) * net.inv_c);
    return expf(-d2 * net.inv2r2);
}

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// gaspari_cohn() of two squared scaled distances z^2, in packed arithmetic: 1 / z by the hardware
// approximation and one Newton step serves both z = z^2 / z and the outer piece's division.
__device__ __forceinline__ float2 gaspari_cohn_pair(float2 z2) {
    auto dup = [](float v) { return make_float2(v, v); };
    float2 y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y.x) : "f"(fmaxf(z2.x, 1e-30f)));
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y.y) : "f"(fmaxf(z2.y, 1e-30f)));
    const float2 h = __fmul2_rn(__fmul2_rn(z2, dup(-0.5f)), y);
    y = __fmul2_rn(y, __ffma2_rn(h, y, dup(1.5f)));
    float2 z = __fmul2_rn(z2, y);
    float2 in = __ffma2_rn(dup(-0.25f), z, dup(0.5f));
    in = __ffma2_rn(in, z, dup(0.625f));
    in = __ffma2_rn(in, z, dup(-5.0f / 3.0f));
    in = __ffma2_rn(in, z2, dup(1.0f));
    const float2 zo = make_float2(fminf(z.x, 1.99999988f), fminf(z.y, 1.99999988f));
    const float2 t = __ffma2_rn(zo, dup(-1.0f), dup(2.0f));
    const float2 t2 = __fmul2_rn(t, t);
    float2 out = __ffma2_rn(dup(2.0f / 24.0f), zo, dup(4.0f / 24.0f));
    out = __ffma2_rn(out, zo, dup(-1.0f / 24.0f));
    out = __fmul2_rn(__fmul2_rn(__fmul2_rn(t2, t2), out), y);
    return make_float2(z.x <= 1.0f ? in.x : out.x, z.y <= 1.0f ? in.y : out.y);
}

// The weights of two squared distances.  The Gaussian is 2^t with t = -d2 log2(e) / (2 r^2)
// rounded to FP32 and its rounding error (from FMA, and the low word clo of the factor) applied
// to first order, in packed arithmetic.
template <int KIND>
__device__ __forceinline__ float2 weight_pair(const ObsNet &net, float2 d2, float2 c, float2 clo) {
    if (KIND == 0) return make_float2(1.0f, 1.0f);
    if (KIND == 2) return gaspari_cohn_pair(__fmul2_rn(d2, make_float2(net.inv_c * net.inv_c,
                                                                       net.inv_c * net.inv_c)));
    const float2 t = __fmul2_rn(d2, c);
    const float2 nt = make_float2(-t.x, -t.y);
    const float2 e = __fmul2_rn(__ffma2_rn(d2, clo, __ffma2_rn(d2, c, nt)),
                                make_float2(0.693147181f, 0.693147181f));
    const float2 w = make_float2(ex2(t.x), ex2(t.y));
    return __ffma2_rn(w, e, w);
}

// One x range of a bin row of a tile's patch: the bins within the cutoff at the row's distance
// from the tile; xr = 0 or 1 (the second range of a row that wraps).  Returns the row count.
__device__ inline int patch_run(const ObsNet &net, int nx, int ny, int tx0, int ty0, int by,
                                int xr, int *j0) {
    BinRanges rr;
    if (net.loc_none) {
        rr.n = 1;
        rr.lo[0] = 0;
        rr.hi[0] = net.ncx - 1;
    } else {
        const int gy = axis_gap(by * net.cs, min((by + 1) * net.cs, ny) - 1, ty0, ty0 + kTH - 1, ny);
        const long long rem = (long long)net.d2max - (long long)gy * gy;
        if (rem < 0) return 0;
        int w = (int)sqrtf((float)rem);
        while ((long long)(w + 1) * (w + 1) <= rem) ++w;
        while ((long long)w * w > rem) --w;
        rr = bin_ranges(tx0 - w, tx0 + kTW - 1 + w, nx, net.cs);
    }
    if (xr >= rr.n) return 0;
    const int blo = xr ? rr.lo[1] : rr.lo[0], bhi = xr ? rr.hi[1] : rr.hi[0];
    const int c0 = by * net.ncx + blo;
    *j0 = __ldg(net.cell_start + c0);
    return __ldg(net.cell_start + c0 + (bhi - blo) + 1) - *j0;
}

__device__ __forceinline__ BinRanges patch_rows(const ObsNet &net, int ny, int ty0) {
    BinRanges ry;
    if (net.loc_none) {
        ry.n = 1;
        ry.lo[0] = 0;
        ry.hi[0] = net.ncy - 1;
    } else {
        ry = bin_ranges(ty0 - net.cr, ty0 + kTH - 1 + net.cr, ny, net.cs);
    }
    return ry;
}

// One entry of z in two FP32 words (compensated): the sum over the observed variables of
// dy_i dy_j / sigma^2, from f(v) = (dy_vi, dy_vj, 1 / sigma_v^2).
template <class F>
__device__ __forceinline__ void z_entry(int V, F f, float &hi, float &lo) {
    float acc = 0.0f, err = 0.0f;
    for (int v = 0; v < V; ++v) {
        const float3 d = f(v);
        const float t = d.x * d.y;
        const float e = fmaf(d.x, d.y, -t);
        const float t2 = t * d.z;
        const float e2 = fmaf(e, d.z, fmaf(t, d.z, -t2));
        const float s = acc + t2, b = s - acc;
        err += ((acc - (s - b)) + (t2 - b)) + e2;
        acc = s;
    }
    hi = acc + err;
    lo = err - (hi - acc);
    if (!isfinite(hi)) {   // the plain sum keeps an overflowed error term out
        hi = acc;
        lo = 0.0f;
    }
}

// Whether the products take v as it is (its first BF16 part is finite).
__device__ __forceinline__ bool z_finite(float v) {
    return isfinite(__bfloat162float(__float2bfloat16_rn(v)));
}

// dy_i of observation o's variable v (i < k), or its innovation (i = k).
__device__ __forceinline__ float z_factor(const GemmArgs &a, int o, int v, int i) {
    const int s = o * a.net.V + v;
    return i < a.k ? a.yb[(size_t)s * a.kp + i] : (a.yo[s] - a.yref[v]) - a.ybar[s];
}

// Adds the products that gram_z_kernel left out (not finite) to the entries of a warp's 32 pairs and
// 8 rows of a tile, which its lanes have stored: the rows of the patch, 32 at a time, from the
// middle of the patch and of each run (near every point), until every entry is a NaN.  A NaN is
// stored without a look at the sum, so that nothing waits for a load.
template <int KIND>
__device__ __noinline__ void gram_fix(const GemmArgs &a, int tx0, int ty0, int mt, int warp,
                                      int lane) {
    const ObsNet net = a.net;   // (copies: a is in memory here, and the stores might alias it)
    const int nx = a.nx, ny = a.ny, y_begin = a.y_begin, y_end = a.y_end, k = a.k;
    const int *const zbad = a.zbad;
    const float2 *const oxy = a.oxy;
    const int m = mt * kMT + 32 * (warp & 3) + lane, off = a.offs[m], pr = a.pairs[m];
    const int yb = ty0 + ((warp - kWarpSum) >> 2) * (kTH / 2);
    const size_t stride = off >= kGemmC ? (size_t)k : (size_t)k * k;
    float *const base = off >= kGemmC ? a.cvec + (off - kGemmC) : a.gram + off;
    uint32_t todo[kTH / 4];   // a bit per point (two rows per word), cleared once it is a NaN
#pragma unroll
    for (int wd = 0; wd < kTH / 4; ++wd) {
        const int y = yb + 2 * wd;
        const uint32_t row = off < 0 || tx0 >= nx ? 0u : 0xffffu >> max(0, tx0 + kTW - nx);
        todo[wd] = (y >= y_begin && y < y_end ? row : 0u) |
                   (y + 1 >= y_begin && y + 1 < y_end ? row << kTW : 0u);
    }
    const BinRanges ry = patch_rows(net, ny, ty0);
    const int ly0 = ry.hi[0] - ry.lo[0] + 1;
    const int nyb = ly0 + (ry.n > 1 ? ry.hi[1] - ry.lo[1] + 1 : 0);
    for (int rb = 0; rb < 2 * nyb; rb += 32) {     // 32 runs at a time, one per lane
        int r = rb + lane + nyb, run0 = 0, runn = 0;
        r -= r >= 2 * nyb ? 2 * nyb : 0;
        if (rb + lane < 2 * nyb) {
            const int yi = r >> 1, by = yi < ly0 ? ry.lo[0] + yi : ry.lo[1] + (yi - ly0);
            runn = patch_run(net, nx, ny, tx0, ty0, by, r & 1, &run0);
        }
        for (unsigned runs = __ballot_sync(0xffffffffu, runn > 0); runs; runs &= runs - 1) {
            const int j0 = __shfl_sync(0xffffffffu, run0, __ffs(runs) - 1);
            const int cnt = __shfl_sync(0xffffffffu, runn, __ffs(runs) - 1);
            for (int c = 0; c < cnt; c += 32) {
                int jl = j0 + cnt / 2 + c + lane;
                jl -= jl >= j0 + cnt ? cnt : 0;
                unsigned marked = __ballot_sync(0xffffffffu, c + lane < cnt && zbad[jl]);
                for (; marked; marked &= marked - 1) {
                    const int j = __shfl_sync(0xffffffffu, jl, __ffs(marked) - 1);
                    const int o = net.cell_obs[j];
                    float v = 0.0f, lo = 0.0f;
                    if (off >= 0)
                        z_entry(net.V, [&](int w) {
                            return make_float3(z_factor(a, o, w, pr & 0xffff),
                                               z_factor(a, o, w, pr >> 16), a.rinv[o * net.V + w]);
                        }, v, lo);
                    const bool add = !z_finite(v), nan = isnan(v);
                    if (!__any_sync(0xffffffffu, add)) continue;
                    const float2 at = oxy[j];
#pragma unroll
                    for (int wd = 0; wd < kTH / 4; ++wd)
#pragma unroll 1
                        for (int h = 0; h < 2; ++h) {
                            const int y = yb + 2 * wd + h, dy = min_image((int)at.y - y, ny);
                            if (KIND != 0 && dy * dy > net.d2max) continue;
                            float *const row = base + ((ptrdiff_t)(y - y_begin) * nx + tx0) *
                                                          (ptrdiff_t)stride;
#pragma unroll 1
                            for (int i = 0; i < kTW; ++i) {
                                const int dx = min_image((int)at.x - (tx0 + i), nx);
                                const int d2 = dx * dx + dy * dy;
                                const uint32_t bit = 1u << (h * kTW + i);
                                if ((KIND != 0 && d2 > net.d2max) || !add || !(todo[wd] & bit))
                                    continue;
                                float t = v;
                                if (!nan) t = fmaf(weight_d2<KIND>(net, (float)d2), v, row[i * stride]);
                                row[i * stride] = t;
                                if (isnan(t)) todo[wd] &= ~bit;
                            }
                        }
                    uint32_t left = 0;
#pragma unroll
                    for (int wd = 0; wd < kTH / 4; ++wd) left |= todo[wd];
                    if (!__any_sync(0xffffffffu, left != 0)) return;
                }
            }
        }
    }
}

template <int KIND, bool WRAP>
__global__ void __launch_bounds__(kThreads, 1)
    gram_gemm_kernel(const __grid_constant__ GemmArgs a, const __grid_constant__ TmaMap zmap,
                     int *status) {
    extern __shared__ unsigned char dyn_raw[];
    __shared__ __align__(8) uint64_t meta_full[kNM], meta_empty[kNM];
    __shared__ __align__(8) uint64_t z_full[kNZ], z_empty[kNZ], w_full[kNW], w_empty[kNW];
    __shared__ __align__(8) uint64_t tm_full[2], tm_empty[2], mma_done;
    __shared__ uint32_t tmem_base;
    __shared__ volatile int abort_flag;
    unsigned char *dyn = dyn_raw + ((1024u - (smem_u32(dyn_raw) & 1023u)) & 1023u);
    Step *steps = reinterpret_cast<Step *>(dyn + kOffM);

    const ObsNet &net = a.net;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // tiles lie on multiples of 16 in the grid, so a point's sums do not depend on the chunk
    const int ty_first = a.y_begin / kTH * kTH;
    const int ntx = (a.nx + kTW - 1) / kTW, nty = (a.y_end - ty_first + kTH - 1) / kTH;
    const int ntiles = ntx * nty, nmt = a.np / kMT;
    const int nitems = ntiles * nmt;
    // item -> origin of its tile; returns its pair tile
    auto item_at = [&](int it, int &tx0, int &ty0) -> int {
        const int mt = it / ntiles, tile = it - mt * ntiles;
        tx0 = (tile % ntx) * kTW;
        ty0 = ty_first + (tile / ntx) * kTH;
        return mt;
    };

    if (tid == 0) {
        for (int i = 0; i < kNM; ++i) {
            bar_init(&meta_full[i], 32);
            bar_init(&meta_empty[i], 2 + kProdWarps + kSumWarps);   // TMA, MMA, weights, sums
        }
        for (int i = 0; i < kNZ; ++i) {
            bar_init(&z_full[i], 1);
            bar_init(&z_empty[i], 1);
        }
        for (int i = 0; i < kNW; ++i) {
            bar_init(&w_full[i], kProdWarps);
            bar_init(&w_empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            bar_init(&tm_full[i], 1);
            bar_init(&tm_empty[i], kSumWarps);
        }
        bar_init(&mma_done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;");
        abort_flag = 0;
    }
    if (warp == kWarpMma) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&tmem_base)),
                     "r"(kCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = tmem_base;

    auto fail = [&]() {
        abort_flag = 1;
        if (lane == 0) atomicOr(status, ST_TIMEOUT);
    };

    if (warp < kWarpProd) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegMisc));
    if (warp == kWarpMeta) {
        // ===================== the patch, in steps of 32 slots =====================
        uint32_t g = 0;
        const float nan = __int_as_float(0x7fc00000);
        for (int it = blockIdx.x; it < nitems && !abort_flag; it += gridDim.x) {
            int tx0, ty0;
            item_at(it, tx0, ty0);
            const BinRanges ry = patch_rows(net, a.ny, ty0);
            const int ly0 = ry.hi[0] - ry.lo[0] + 1;
            const int nyb = ly0 + (ry.n > 1 ? ry.hi[1] - ry.lo[1] + 1 : 0);
            const int nr = 2 * nyb;
            bool ok = true, closed = false;
            // one step: this lane's slot holds row j (or none), the groups' first rows in start
            auto publish = [&](int j, bool in, int start, int last) {
                const int s = g % kNM;
                float2 o = make_float2(nan, nan);
                if (in) {
                    o = __ldg(a.oxy + j);
                    o.x -= (float)tx0;
                    o.y -= (float)ty0;
                    const float cx = 0.5f * (kTW - 1), cy = 0.5f * (kTH - 1);
                    o.x -= (float)a.nx * rintf((o.x - cx) / (float)a.nx);
                    o.y -= (float)a.ny * rintf((o.y - cy) / (float)a.ny);
                }
                if (!(ok = wait_bar(&meta_empty[s], ((g / kNM) & 1) ^ 1, &abort_flag))) return;
                steps[s].xy[lane] = o;
                if ((lane & 7) == 0) steps[s].start[lane >> 3] = start;
                if (lane == 0) steps[s].last = last;
                bar_arrive(&meta_full[s]);
                ++g;
            };
            for (int rb = 0; rb < nr && ok; rb += 32) {
                int j0 = 0, cnt = 0;
                if (rb + lane < nr) {
                    const int yi = (rb + lane) >> 1;
                    const int by = yi < ly0 ? ry.lo[0] + yi : ry.lo[1] + (yi - ly0);
                    cnt = patch_run(net, a.nx, a.ny, tx0, ty0, by, (rb + lane) & 1, &j0);
                }
                const int ng = (cnt + 7) >> 3;
                int incl = ng;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int t = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += t;
                }
                const int tot = __shfl_sync(0xffffffffu, incl, 31);
                for (int fb = 0; fb < tot && ok; fb += kGroups) {
                    const int f = fb + (lane >> 3);          // this lane's group
                    const int fc = min(f, tot - 1);
                    int lo = 0;   // first run whose inclusive end exceeds fc
#pragma unroll
                    for (int step = 16; step > 0; step >>= 1) {
                        const int e = __shfl_sync(0xffffffffu, incl, lo + step - 1);
                        if (e <= fc) lo += step;
                    }
                    const int e_lo = __shfl_sync(0xffffffffu, incl, lo);
                    const int g_lo = __shfl_sync(0xffffffffu, ng, lo);
                    const int c_lo = __shfl_sync(0xffffffffu, cnt, lo);
                    const int b_lo = __shfl_sync(0xffffffffu, j0, lo);
                    const int r = 8 * (fc - (e_lo - g_lo)) + (lane & 7);   // row within the run
                    const int last = rb + 32 >= nr && fb + kGroups >= tot;
                    publish(b_lo + r, f < tot && r < c_lo, b_lo + r - (lane & 7), last);
                    closed = last;
                }
            }
            if (ok && !closed) publish(0, false, 0, 1);
            if (!ok) {
                fail();
                break;
            }
        }
    } else if (warp == kWarpTma) {
        // ===================== rows of Z =====================
        uint32_t g = 0;
        const uint32_t z0 = smem_u32(dyn + kOffZ);
        bool ok = true;
        for (int it = blockIdx.x; it < nitems && !abort_flag && ok; it += gridDim.x) {
            int tx0, ty0;
            const int mt = item_at(it, tx0, ty0);
            bool last = false;
            while (!last) {
                const int s = g % kNM, st = g % kNZ;
                if (!(ok = wait_bar(&meta_full[s], (g / kNM) & 1, &abort_flag))) break;
                last = steps[s].last != 0;
                int start[kGroups];
#pragma unroll
                for (int i = 0; i < kGroups; ++i) start[i] = steps[s].start[i];
                if (!(ok = wait_bar(&z_empty[st], ((g / kNZ) & 1) ^ 1, &abort_flag))) break;
                if (lane == 0) {
                    const uint32_t bar = smem_u32(&z_full[st]);
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                                 "r"((uint32_t)kZStage)
                                 : "memory");
#pragma unroll
                    for (int b = 0; b < 2 * kGroups; ++b) {
                        const uint32_t dst = z0 + st * kZStage + b * kBoxB;
                        asm volatile(
                            "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::"
                            "complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
                            "l"(reinterpret_cast<uint64_t>(&zmap)),
                            "r"(mt * kMT + (b / kGroups) * 64), "r"(start[b % kGroups]), "r"(0),
                            "r"(bar)
                            : "memory");
                    }
                    bar_arrive(&meta_empty[s]);
                }
                __syncwarp();
                ++g;
            }
        }
        if (!ok || abort_flag) {
            fail();
            // the copies in flight land before the CTA may exit (bounded)
            volatile int no_abort = 0;
            for (uint32_t i = g > kNZ ? g - kNZ : 0; i < g; ++i)
                wait_bar(&z_full[i % kNZ], (i / kNZ) & 1, &no_abort);
        }
    } else if (warp == kWarpMma) {
        // ===================== tensor-core issue =====================
        uint32_t g = 0;
        const uint32_t z0 = smem_u32(dyn + kOffZ), w0 = smem_u32(dyn + kOffW);
        bool ok = true;
        for (int it = blockIdx.x; it < nitems && !abort_flag && ok; it += gridDim.x) {
            bool last = false;
            while (!last) {
                const int s = g % kNM, ws = g % kNW, st = g % kNZ, tb = g & 1;
                if (!(ok = wait_bar(&meta_full[s], (g / kNM) & 1, &abort_flag))) break;
                last = steps[s].last != 0;
                __syncwarp();
                if (lane == 0) bar_arrive(&meta_empty[s]);
                if (!(ok = wait_bar(&tm_empty[tb], ((g >> 1) & 1) ^ 1, &abort_flag))) break;
                if (!(ok = wait_bar(&w_full[ws], (g / kNW) & 1, &abort_flag))) break;
                if (!(ok = wait_bar(&z_full[st], (g / kNZ) & 1, &abort_flag))) break;
                asm volatile("tcgen05.fence::after_thread_sync;");
                if (lane == 0) {
                    const uint32_t zb = z0 + st * kZStage, wb = w0 + ws * kWStage;
                    const uint32_t d = tmem + tb * kPts;
                    // parts (z, w) in ascending size; the leading products of both K-steps last
                    constexpr int pz[6] = {2, 0, 1, 1, 0, 0}, pw[6] = {0, 2, 1, 0, 1, 0};
#pragma unroll
                    for (int i = 0; i < 6; ++i)
#pragma unroll
                        for (int ks = 0; ks < kKC / 16; ++ks)
                            mma_f16(d, zdesc(zb + ks * 2 * kBoxB + pz[i] * 1024),
                                    sdesc(wb + pw[i] * kWPart + ks * 256, kWSbo), kIdesc,
                                    i == 0 && ks == 0 ? 0u : 1u);
                    mma_commit(&z_empty[st]);
                    mma_commit(&w_empty[ws]);
                    mma_commit(&tm_full[tb]);
                }
                __syncwarp();
                ++g;
            }
        }
        if (!ok) fail();
        // all MMAs issued by this CTA complete before its tensor memory is freed (bounded)
        if (lane == 0) mma_commit(&mma_done);
        __syncwarp();
        volatile int no_abort = 0;
        if (!wait_bar(&mma_done, 0, &no_abort)) fail();
    }
    } else if (warp < kWarpSum) {
        // ===================== weights =====================
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegProd));
        const int n = tid - 32 * kWarpProd;   // grid points n and n + 128 of the tile
        const float px = (float)(n % kTW);
        const float2 py = make_float2(-(float)(n / kTW), -(float)(n / kTW + kTH / 2));
        const float2 mper = make_float2(-(float)a.nx, -(float)a.ny);
        const float2 iper = make_float2(1.0f / (float)a.nx, 1.0f / (float)a.ny);
        const double ce = -1.4426950408889634 * (double)net.inv2r2;
        const float cf = (float)ce, cl = (float)(ce - (double)cf);
        const float2 c2 = make_float2(cf, cf), cl2 = make_float2(cl, cl);
        const float d2max = KIND == 0 ? __int_as_float(0x7f800000) : (float)net.d2max;
        uint32_t g = 0;
        bool ok = true;
        for (int it = blockIdx.x; it < nitems && !abort_flag && ok; it += gridDim.x) {
            bool last = false;
            while (!last) {
                const int s = g % kNM, ws = g % kNW;
                if (!(ok = wait_bar(&meta_full[s], (g / kNM) & 1, &abort_flag))) break;
                last = steps[s].last != 0;
                if (!(ok = wait_bar(&w_empty[ws], ((g / kNW) & 1) ^ 1, &abort_flag))) break;
                unsigned char *wb = dyn + kOffW + ws * kWStage + (n >> 3) * kWSbo + (n & 7) * 16;
#pragma unroll 1
                for (int kb = 0; kb < kKC / 8; ++kb) {
                    uint32_t part[2][3][4];   // [point][part][pair of slots]
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float4 o2 =
                            *reinterpret_cast<const float4 *>(&steps[s].xy[8 * kb + 2 * i]);
                        float2 w[2];          // [slot] (point n, point n + 128)
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            // squared distances, exact in FP32 (the launch's condition on
                            // d2max); far points stay beyond the cutoff
                            float dx = (h ? o2.z : o2.x) - px;
                            const float oy = h ? o2.w : o2.y;
                            float2 dy = __fadd2_rn(make_float2(oy, oy), py);
                            if (WRAP) {   // a grid narrower than the patch: nearest image
                                dx = fmaf(rintf(dx * iper.x), mper.x, dx);
                                dy.x = fmaf(rintf(dy.x * iper.y), mper.y, dy.x);
                                dy.y = fmaf(rintf(dy.y * iper.y), mper.y, dy.y);
                            }
                            const float dx2 = dx * dx;
                            const float2 d2 = __ffma2_rn(dy, dy, make_float2(dx2, dx2));
                            w[h] = weight_pair<KIND>(net, d2, c2, cl2);
                            w[h].x = d2.x <= d2max ? w[h].x : 0.0f;
                            w[h].y = d2.y <= d2max ? w[h].y : 0.0f;
                        }
#pragma unroll
                        for (int q = 0; q < 2; ++q) {
                            const float2 v = q ? make_float2(w[0].y, w[1].y)
                                               : make_float2(w[0].x, w[1].x);
                            const float2 m1 = make_float2(-1.0f, -1.0f);
                            const __nv_bfloat162 hb = __floats2bfloat162_rn(v.x, v.y);
                            const float2 r1 = __ffma2_rn(bf2f(hb), m1, v);
                            const __nv_bfloat162 mb = __floats2bfloat162_rn(r1.x, r1.y);
                            const float2 r2 = __ffma2_rn(bf2f(mb), m1, r1);
                            part[q][0][i] = bits(hb);
                            part[q][1][i] = bits(mb);
                            part[q][2][i] = bits(__floats2bfloat162_rn(r2.x, r2.y));
                        }
                    }
#pragma unroll
                    for (int q = 0; q < 2; ++q)
#pragma unroll
                        for (int p = 0; p < 3; ++p)
                            *reinterpret_cast<uint4 *>(wb + q * (kPts / 16) * kWSbo + p * kWPart +
                                                       kb * 128) =
                                make_uint4(part[q][p][0], part[q][p][1], part[q][p][2],
                                           part[q][p][3]);
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) {
                    bar_arrive(&w_full[ws]);
                    bar_arrive(&meta_empty[s]);
                }
                ++g;
            }
        }
        if (!ok) fail();
    } else {
        // ===================== sums, and their store =====================
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegSum));
        const int half = (warp - kWarpSum) >> 2;   // columns (grid points) 128 half ..
        const uint32_t src = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + half * (kPts / 2);
        uint32_t g = 0;
        bool ok = true;
        for (int it = blockIdx.x; it < nitems && !abort_flag && ok; it += gridDim.x) {
            int tx0, ty0;
            const int mt = item_at(it, tx0, ty0);
            const int off = __ldg(a.offs + mt * kMT + 32 * (warp & 3) + lane);
            float acc[kPts / 2];
#pragma unroll
            for (int i = 0; i < kPts / 2; ++i) acc[i] = 0.0f;
            bool last = false;
            while (!last) {
                const int s = g % kNM, tb = g & 1;
                if (!(ok = wait_bar(&meta_full[s], (g / kNM) & 1, &abort_flag))) break;
                last = steps[s].last != 0;
                __syncwarp();
                if (lane == 0) bar_arrive(&meta_empty[s]);
                if (!(ok = wait_bar(&tm_full[tb], (g >> 1) & 1, &abort_flag))) break;
                asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
                for (int c = 0; c < kPts / 2; c += 16) {
                    float v[16];
                    tmem_ld16(src + tb * kPts + c, v);
#pragma unroll
                    for (int i = 0; i < 16; i += 2) {
                        const float2 t = __fadd2_rn(make_float2(acc[c + i], acc[c + i + 1]),
                                                    make_float2(v[i], v[i + 1]));
                        acc[c + i] = t.x;
                        acc[c + i + 1] = t.y;
                    }
                }
                asm volatile("tcgen05.fence::before_thread_sync;");
                __syncwarp();
                if (lane == 0) bar_arrive(&tm_empty[tb]);
                ++g;
            }
            if (!ok) break;
            if (off >= 0) {
                const size_t stride = off >= kGemmC ? (size_t)a.k : (size_t)a.k * a.k;
                float *base = off >= kGemmC ? a.cvec + (off - kGemmC) : a.gram + off;
                const int yb = ty0 + half * (kTH / 2);
                base += ((ptrdiff_t)(yb - a.y_begin) * a.nx + tx0) * (ptrdiff_t)stride;
                const bool whole = tx0 + kTW <= a.nx;
#pragma unroll
                for (int r = 0; r < kTH / 2; ++r, base += (size_t)a.nx * stride) {
                    float *p = base;
                    if (yb + r < a.y_begin || yb + r >= a.y_end) continue;
#pragma unroll
                    for (int i = 0; i < kTW; ++i, p += stride)
                        if (whole || tx0 + i < a.nx) *p = acc[kTW * r + i];
                }
            }
        }
        if (!ok) fail();
        else if (*a.flag)   // written before this launch (read here: a register held through the
                            // sums, or a shared word, costs 2 % of the kernel)
            for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
                int tx0, ty0;
                const int mt = item_at(it, tx0, ty0);
                gram_fix<KIND>(a, tx0, ty0, mt, warp, lane);
            }
    }

    // ---- stop: every role has left its loop; free the tensor memory
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (warp == kWarpMma)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(kCols));
}

// z of every observation point in bin order, three BF16 parts: block per observation point, two
// neighbouring pairs per thread and round.  pairs[m] = i | j << 16 (j = k: the innovation), -1:
// padding.  An entry that is not finite becomes zero; its row is marked in zbad, and the flag raised
// (both cleared by the observation operator).
__global__ void __launch_bounds__(256) gram_z_kernel(const __grid_constant__ GemmArgs a) {
    __shared__ float dy[3][132];
    __shared__ float ri[3];
    const int j = blockIdx.x, o = a.net.cell_obs[j], V = a.net.V, k = a.k, np = a.np;
    for (int e = threadIdx.x; e < V * (k + 1); e += blockDim.x) {
        const int v = e / (k + 1), i = e - v * (k + 1);
        dy[v][i] = z_factor(a, o, v, i);
    }
    if (threadIdx.x < V) ri[threadIdx.x] = a.rinv[o * V + threadIdx.x];
    __syncthreads();
    bool bad = false;
    for (int m = 2 * threadIdx.x; m < np; m += 2 * blockDim.x) {
        const int2 pr = *reinterpret_cast<const int2 *>(a.pairs + m);
        float hi[2], lo[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int p = h ? pr.y : pr.x;
            hi[h] = lo[h] = 0.0f;
            if (p >= 0)
                z_entry(V, [&](int v) { return make_float3(dy[v][p & 0xffff], dy[v][p >> 16], ri[v]); },
                        hi[h], lo[h]);
        }
        __nv_bfloat162 hb = __floats2bfloat162_rn(hi[0], hi[1]);
        float2 hf = bf2f(hb);
        if (!isfinite(hf.x) || !isfinite(hf.y)) {   // (z_finite)
            bad = true;
            if (!isfinite(hf.x)) hi[0] = lo[0] = 0.0f;
            if (!isfinite(hf.y)) hi[1] = lo[1] = 0.0f;
            hb = __floats2bfloat162_rn(hi[0], hi[1]);
            hf = bf2f(hb);
        }
        const float a0 = (hi[0] - hf.x) + lo[0], a1 = (hi[1] - hf.y) + lo[1];
        const __nv_bfloat162 mb = __floats2bfloat162_rn(a0, a1);
        const float2 mf = bf2f(mb);
        const __nv_bfloat162 lb = __floats2bfloat162_rn(a0 - mf.x, a1 - mf.y);
        const size_t part = (size_t)a.net.L * np, at = (size_t)j * np + m;
        *reinterpret_cast<__nv_bfloat162 *>(a.z + at) = hb;
        *reinterpret_cast<__nv_bfloat162 *>(a.z + part + at) = mb;
        *reinterpret_cast<__nv_bfloat162 *>(a.z + 2 * part + at) = lb;
    }
    if (bad) {
        a.zbad[j] = 1;
        atomicOr(a.flag, 1);
    }
}

using EncodeTiled = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                 const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                 const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                 CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiled gemm_encoder() {
    static std::once_flag once;
    static EncodeTiled fn = nullptr;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000,
                                             cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiled>(p);
    });
    return fn;
}

}  // namespace

int gram_gemm_pairs(int k) {
    const int b = (k + 3) / 4;
    return ((8 * b * (b + 1) + k) + kMT - 1) / kMT * kMT;   // 4-wide runs of every row, and c
}

void gram_gemm_tables(int k, int *pairs, int *offs) {
    const int np = gram_gemm_pairs(k);
    int m = 0;
    auto put = [&](int i, int j, int off) {
        pairs[m] = off < 0 ? -1 : (i | (j << 16));
        offs[m++] = off;
    };
    for (int i = 0; i < (k + 3) / 4 * 4; ++i)
        for (int j = i / 4 * 4; j < (k + 3) / 4 * 4; ++j)
            put(i, j, i < k && j < k ? i * k + j : -1);
    for (int i = 0; i < k; ++i) put(i, k, kGemmC + i);
    while (m < np) put(0, 0, -1);
}

cudaError_t gram_gemm_prepare(const void *z, int L, int np, TmaMap *map, int *ok) {
    *ok = 0;
    const EncodeTiled enc = gemm_encoder();
    if (!enc) return cudaSuccess;
    const cuuint64_t dim[3] = {(cuuint64_t)np, (cuuint64_t)L, 3};
    const cuuint64_t str[2] = {(cuuint64_t)np * 2, (cuuint64_t)np * 2 * (cuuint64_t)L};
    const cuuint32_t box[3] = {64, 8, 3}, es[3] = {1, 1, 1};
    if (enc(reinterpret_cast<CUtensorMap *>(map), CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3,
            const_cast<void *>(z), dim, str, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    *ok = 1;
    for (auto f : {gram_gemm_kernel<0, false>, gram_gemm_kernel<1, false>,
                   gram_gemm_kernel<1, true>, gram_gemm_kernel<2, false>,
                   gram_gemm_kernel<2, true>}) {
        const cudaError_t e =
            cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem + 1024);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_gram_z(const GemmArgs &a, cudaStream_t s) {
    if (a.net.L <= 0) return cudaSuccess;
    gram_z_kernel<<<a.net.L, 256, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_gram_gemm(const GemmArgs &a, const TmaMap &map, int *status, int max_ctas,
                             cudaStream_t s) {
    if (a.y_end <= a.y_begin) return cudaSuccess;
    const long long tiles = (long long)((a.nx + kTW - 1) / kTW) *
                            ((a.y_end - a.y_begin / kTH * kTH + kTH - 1) / kTH);
    const long long items = tiles * (a.np / kMT);
    int lo = 0, hi = 0;
    cudaError_t e = cudaDeviceGetStreamPriorityRange(&lo, &hi);
    if (e != cudaSuccess) return e;
    // one CTA per SM (all of tensor memory), placed ahead of other streams' pending blocks
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributePriority;
    attr[0].val.priority = hi;
    cfg.gridDim = dim3((unsigned)(items < max_ctas ? items : max_ctas));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmem + 1024;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (a.net.loc_none) return cudaLaunchKernelEx(&cfg, gram_gemm_kernel<0, false>, a, map, status);
    // a grid at least as wide as a patch: the image of an observation nearest the tile's centre
    // is the nearest one to each of its points within the cutoff
    const bool wrap = a.nx < kTW + 2 * a.net.cr + 1 || a.ny < kTH + 2 * a.net.cr + 1;
    auto f = a.net.loc_gc ? (wrap ? gram_gemm_kernel<2, true> : gram_gemm_kernel<2, false>)
                          : (wrap ? gram_gemm_kernel<1, true> : gram_gemm_kernel<1, false>);
    return cudaLaunchKernelEx(&cfg, f, a, map, status);
}

}  // namespace lk
