// EVD-free transform by Chebyshev polynomials in Q (the LETKF_EIG_CHEBYSHEV schedule, FP32).
//
// The transform of a grid point needs two matrix functions of Q = d I + A, d = (k-1)/rho and A
// the localized Gram matrix (positive semidefinite), applied to the forecast (Sec. II-B, Eqs.
// letkf_wa, letkf_dwa, letkf_xa):
//     mean increment   dX Q^-1 c
//     perturbations    sqrt(k-1) dX Q^-1/2
// S = Q / d has its spectrum in [1, kappa] for every kappa >= 1 + lambda_max(A) / d, and on that
// interval t^-1/2 and t^-1 are approximated by Chebyshev expansions
//     t^-1/2 ~ sum_j a_j T_j(s),   t^-1 ~ sum_j b_j T_j(s),   s = (2 t - kappa - 1) / (kappa - 1),
// the interpolants at the Chebyshev points of the first kind (FP64 on the host, the degree
// chosen per kappa so that the relative error stays below 2e-8).  The ten rows R = [dX; c^T]
// (10 x k) are multiplied by these polynomials in S from the right with Clenshaw's recurrence,
// one product with Z = (2 S - (kappa + 1) I) / (kappa - 1) per degree.  Z = gamma A - I with
// gamma = 2 / (d (kappa - 1)): A enters directly, so nothing cancels when kappa is near 1.
// Rows 0..8 take the coefficients of t^-1/2, row 9 those of t^-1; then
//     dX Q^-1/2 = d^-1/2 dX S^-1/2,   Q^-1 c = d^-1 S^-1 c.
// No factorization, eigenvalue or eigenvector is formed.
//
// kappa comes from the cheapest upper bounds of lambda_max(A): the least of the Gershgorin
// bound, the Frobenius norm and the trace.  The degree grows like sqrt(kappa) (1 for kappa <=
// 1.0002, 2 for 1.005, 3 for 1.035, 4 for 1.1, 10 for 2, 36 for 16); a point beyond the last
// approximation goes to the rational schedule (tridiagonalization and Zolotarev's
// approximation) through a list.
//
// Layout, k <= 64 (eig_cheb_kernel): one warp per grid point.  A half warp holds half of the rows of
// A in registers, a lane four columns (two for k <= 32), loaded from the upper triangle of the Gram
// slot staged in shared memory.  A product R A reads the rows of R as 16-byte broadcasts to a half
// warp (five loads for 40 packed multiply-adds) and ends with a shuffle between the half warps.
// The rows of R are independent: five run through the whole recurrence, its values in
// registers, then the other five.  (Broadcasts to a whole warp took twice the shared-memory
// wavefronts, and two warps per point, halves of the rows, 1.5 times the instructions.)
// k <= 128 (eig_cheb_block_kernel): eight warps per point, quarters of the rows x halves of the
// columns, 32 rows of two columns per lane; the partial sums meet in shared memory.
#include <math.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "common.cuh"
#include "kernels.h"
#include "letkf.h"

namespace lk {

// ---- coefficients (host, FP64) ---------------------------------------------------------

namespace {

constexpr double kPiC = 3.14159265358979323846;

// Chebyshev series sum_j c_j T_j(s) at s (Clenshaw, FP64).
double cheb_eval(const double *c, int n, double s) {
    double b1 = 0.0, b2 = 0.0;
    for (int j = n; j >= 1; --j) {
        const double b0 = c[j] + 2.0 * s * b1 - b2;
        b2 = b1;
        b1 = b0;
    }
    return c[0] + s * b1 - b2;
}

// The degree-n interpolants of t^-1/2 (ca) and t^-1 (cb) on [1, kappa].
void cheb_interpolate(double kappa, int n, double *ca, double *cb) {
    const int m = n + 1;
    for (int j = 0; j <= n; ++j) {
        double sa = 0.0, sb = 0.0;
        for (int i = 0; i < m; ++i) {
            const double th = kPiC * (i + 0.5) / m;
            const double t = 1.0 + 0.5 * (cos(th) + 1.0) * (kappa - 1.0);
            const double cj = cos(j * th);
            sa += cj / sqrt(t);
            sb += cj / t;
        }
        ca[j] = (j == 0 ? 1.0 : 2.0) * sa / m;
        cb[j] = (j == 0 ? 1.0 : 2.0) * sb / m;
    }
}

}  // namespace

// Coefficients of the degree-n interpolants of t^-1/2 (ca) and t^-1 (cb) on [1, kappa] at the
// Chebyshev points of the first kind, in the variable s = (2 t - kappa - 1) / (kappa - 1);
// returns the larger of the two largest relative errors on a fine grid of the interval.
double chebyshev_coefficients(double kappa, int n, double *ca, double *cb) {
    cheb_interpolate(kappa, n, ca, cb);
    const int G = 20000;
    double err = 0.0;
    for (int g = 0; g <= G; ++g) {
        const double t = 1.0 + (kappa - 1.0) * g / G;
        const double s = (2.0 * t - kappa - 1.0) / (kappa - 1.0);
        err = fmax(err, fabs(cheb_eval(ca, n, s) * sqrt(t) - 1.0));
        err = fmax(err, fabs(cheb_eval(cb, n, s) * t - 1.0));
    }
    return err;
}

// The approximations the schedule chooses from: for each kappa_max the smallest degree whose
// error stays below 2e-8 in FP64, found once with chebyshev_coefficients.  The kernel reads the
// coefficients rounded to FP32; with them t^-1/2 and t^-1 are off by up to 6.9e-8 / 1.3e-7 at
// kappa_max = 16, 8.4e-8 / 6.9e-7 at 80 and 2.7e-7 / 4.5e-6 at 400 (relative, at the far end of the
// interval).  The sets beyond 16 serve k > kChebMaxK only and are built with it.  Against the split
// eigensolve that served those points before, on the same A and c (k = 65, 100, 128; observation
// errors falling across the grid, smooth and pointwise perturbations, innovations of noise and of a
// truth drawn with the ensemble): mean increment off by 4.3e-8 to 1.9e-6 against 7.3e-7 to 2.4e-5,
// the perturbations by 6.0e-8 to 9.5e-7 against 1.4e-6 to 1.1e-5; in every class of condition bounds
// at most 0.65 (increment) and 0.28 times as far from the FP64 transform as the split schedule.
// The sets 3.5, 5, 7, 12 and 14 save products where kappa is above 3: 250 x 187, k = 40 20.7 -> 19.0
// a point (eigensolve phase 1.67 -> 1.56 ms), 256 x 256, k = 64 28.4 -> 28.1 (3.82 -> 3.76 ms), 192 x
// 160, k = 128 13.4 -> 13.2.
namespace {
constexpr double kSetKappa[kChebBigSets] = {
    1.0002, 1.005, 1.035, 1.1,  1.2,  1.35, 1.5, 1.75, 2.0, 2.5, 3.0, 3.5, 4.0, 5.0,
    6.0,    7.0,   10.0,  12.0, 14.0, 16.0, 24,  36,   54,  80,  120, 180, 270, 400};
constexpr int kSetDegree[kChebBigSets] = {1,  2,  3,  4,  5,  7,  8,  9,  10, 12,  13,  15,  16,  19,
                                          21, 23, 28, 30, 33, 36, 44, 54, 67, 82, 100, 123, 151, 184};
constexpr int set_coefs(int sets) {
    int n = 0;
    for (int s = 0; s < sets; ++s) n += kSetDegree[s] + 1;
    return n;
}
static_assert(set_coefs(kChebBigSets) <= kChebCoefs, "the table holds every set's coefficients");

void cheb_set(ChebTable &t, int s, double kmax, int n) {
    // the interval the kernel maps onto [-1, 1] is the FP32 kappa_max: the coefficients and the
    // degree are those of that interval
    const float kf = (float)kmax;
    const double km = (double)kf;
    std::vector<double> ca(256), cb(256);
    cheb_interpolate(km, n, ca.data(), cb.data());
    t.kappa_max[s] = kf;
    t.n[s] = n;
    t.off[s] = s == 0 ? 0 : t.off[s - 1] + t.n[s - 1] + 1;
    for (int j = 0; j <= n; ++j) t.c[t.off[s] + j] = make_float2((float)ca[j], (float)cb[j]);
}
}  // namespace

const ChebTable &cheb_table(int k) {
    static ChebTable t, big;
    static std::once_flag once, once_big;
    std::call_once(once, [] {
        for (int s = 0; s < kChebSets; ++s) cheb_set(t, s, kSetKappa[s], kSetDegree[s]);
    });
    if (k <= kChebMaxK) return t;
    std::call_once(once_big, [] {
        big = t;
        for (int s = kChebSets; s < kChebBigSets; ++s) cheb_set(big, s, kSetKappa[s], kSetDegree[s]);
    });
    return big;
}

// The largest set the transform uses for ensemble size k.  k <= 64: degrees up to 9k/16 (at least
// 4): a product with A costs ~20 k^2 flops, the rational schedule's tridiagonalization and
// transform ~(4/3) k^3 + 40 k^2 at a lower issue efficiency, so the break-even degree scales with
// k.  The line was drawn where the two measured equal at k = 64 (degree 36) and stays, so that
// the same points take the same schedule, although products have become cheaper (break-even
// measured since at 7, 17, 24, 28, 31 and 55 for k = 8, 16, 20, 24, 32 and 40 to 64; a point beyond
// goes to the rational schedule).  k > 64: the alternative is the split eigensolve, ~2.5 us a
// point at k = 128 against ~10 ns a product: every set is used up to degree 7k/5 + 5, that is
// up to kappa 80 (degree 82) at k = 65, 180 (123) at k = 100 and 400 (184) at k = 128.  Where
// every point is beyond, the transform's look at the bounds costs 2 % of the phase at k = 72 (4.38
// -> 4.48 ms at 64 x 64), 0.4 % at k = 128.
int cheb_max_set(int k) {
    const ChebTable &t = cheb_table(k);
    const int nsets = k <= kChebMaxK ? kChebSets : kChebBigSets;
    const int nmax = k <= kChebMaxK ? std::max(4, 9 * k / 16) : 7 * k / 5 + 5;
    int s = 0;
    while (s + 1 < nsets && t.n[s + 1] <= nmax) ++s;
    return s;
}

// ---- the transform kernel ---------------------------------------------------------------

namespace {

constexpr unsigned kAllC = 0xffffffffu;
constexpr int kRowsC = 10;   // rows of R: the nine populations' perturbations, then c

// Eight warps per point (k <= 128).
struct ChebBlock {
    static constexpr int KM = 128, NW = 8;                       // warps per point
    static constexpr int CS = KM / 32;                           // 32-column slots of a row
    static constexpr int NC = 2;                                 // columns of a lane
    static constexpr int CG = CS / NC, RB = NW / CG;             // column groups, row blocks
    static constexpr int NE = kRowsC * CS / NW;                  // (row, slot) entries of a warp
    static constexpr int SP = KM + 4;                            // stride of the staged slot
    static constexpr int off_x = KM * SP;                        // [9][k] and c[k]
    static constexpr int off_b = off_x + kRowsC * KM;            // b_{j+1}, [10][KM]
    static constexpr int off_p = off_b + kRowsC * KM;            // partial sums
    static constexpr int off_r = off_p + RB * kRowsC * KM;       // reductions over the warps
    static constexpr int floats = off_r + 2 * NW + 2 * kRowsC * CS;
    static_assert(KM == 32 * RB && floats % 4 == 0, "32 rows per block, 16-byte aligned buffers");
};

// One warp per point, kWarpsC points per block.
constexpr int kWarpsC = 4;
template <int KM>
struct ChebShape {
    static constexpr int NC = KM / 16, HC = NC / 2;   // columns of a lane; kept after a product
    static constexpr int RH = KM / 2;                 // rows of a half warp
    static constexpr int SP = KM + 4;                 // stride of the staged slot
    static constexpr int off_x = KM * SP;             // [9][k] and c[k]
    static constexpr int off_r = off_x + kRowsC * KM; // rows 0..4, kept for the second pass
    static constexpr int off_b = off_r + 5 * KM;      // b_{j+1}, [5][KM]
    static constexpr int off_u = off_b + 5 * KM;      // Q^-1 c
    static constexpr int floats = off_u + KM;
    static_assert(floats % 4 == 0 && off_b % 4 == 0, "16-byte aligned buffers");
    // blocks per SM: 8 warps with 255 registers (128 of them A), 16 with 128
    static constexpr int MINB = KM == 32 ? 4 : 2;
};

constexpr unsigned long long kChebWaitNs = 2000000000ull;   // bound of a prefetch wait (2 s)

__device__ __forceinline__ bool cheb_bar_wait(uint32_t bar, uint32_t parity) {
    unsigned long long t0 = 0;
    for (bool first = true;; first = false) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
            " selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
        unsigned long long t;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (first) t0 = t;
        else if (t - t0 > kChebWaitNs) return false;
    }
}

__device__ __forceinline__ float warp_max_c(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(kAllC, v, o));
    return v;
}

// Four entries of a row of R.  At KM = 64 the load stays where it is written: moved ahead by the
// compiler, the loads pushed pointers and counters out of the 255 registers (256 x 256, 28 products
// 3.76 -> 3.63 ms, 1024 x 1024, three products 11.9 -> 11.2 ms); at KM = 32, with registers to
// spare, moving them is better (301 x 215, k = 24 0.428 ms pinned, 0.414 not).
template <int KM>
__device__ __forceinline__ float4 row4(const float4 *p) {
    if constexpr (KM == 32) return *p;
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"((uint32_t)__cvta_generic_to_shared(p))
                 : "memory");
    return v;
}

// Five rows of R (b, row stride KM, this half warp's first row of A) times NG groups of four rows of
// A per half warp; sums over both half warps, each lane keeping half of its columns.  (With a
// run-time bound on the groups every group waited for its own loads.)
template <int KM, int NG>
__device__ __forceinline__ void cheb_product_ng(
    const float *b, const float2 (&A)[ChebShape<KM>::NC][ChebShape<KM>::RH / 2], int half,
    float (&out)[5][ChebShape<KM>::HC]) {
    constexpr int NC = ChebShape<KM>::NC, HC = NC / 2;
    const float4 *B4 = reinterpret_cast<const float4 *>(b);
    float2 acc[5][NC];
#pragma unroll
    for (int g = 0; g < NG; ++g)
#pragma unroll
        for (int rr = 0; rr < 5; ++rr) {
            const float4 v = row4<KM>(B4 + rr * (KM / 4) + g);
#pragma unroll
            for (int q = 0; q < NC; ++q)
                acc[rr][q] = g ? __ffma2_rn(make_float2(v.x, v.y), A[q][2 * g], acc[rr][q])
                               : __fmul2_rn(make_float2(v.x, v.y), A[q][0]);
#pragma unroll
            for (int q = 0; q < NC; ++q)
                acc[rr][q] = __ffma2_rn(make_float2(v.z, v.w), A[q][2 * g + 1], acc[rr][q]);
        }
#pragma unroll
    for (int rr = 0; rr < 5; ++rr)
#pragma unroll
        for (int q = 0; q < HC; ++q) {
            const float lo = acc[rr][q].x + acc[rr][q].y;
            const float hi = acc[rr][HC + q].x + acc[rr][HC + q].y;
            out[rr][q] = (half ? hi : lo) + __shfl_xor_sync(kAllC, half ? lo : hi, 16);
        }
}

template <int KM>
__device__ __forceinline__ void cheb_product(
    const float *b, const float2 (&A)[ChebShape<KM>::NC][ChebShape<KM>::RH / 2], int ng, int half,
    float (&out)[5][ChebShape<KM>::HC]) {
    if constexpr (KM == 64) {   // k > 32: 5 to 8 groups
        if (ng > 7) cheb_product_ng<KM, 8>(b, A, half, out);
        else if (ng > 6) cheb_product_ng<KM, 7>(b, A, half, out);
        else if (ng > 5) cheb_product_ng<KM, 6>(b, A, half, out);
        else cheb_product_ng<KM, 5>(b, A, half, out);
    } else {
        if (ng > 3) cheb_product_ng<KM, 4>(b, A, half, out);
        else if (ng > 2) cheb_product_ng<KM, 3>(b, A, half, out);
        else cheb_product_ng<KM, 2>(b, A, half, out);
    }
}

// k <= 64.  What bounds it: 10 k^2 multiply-adds per product and point on the FP32 pipe, at two warps
// per scheduler (k <= 32: four), and before the products the assembly of A from the staged
// triangle (about two products' time at k = 64).  Eigensolve phase, two warps per point -> this form:
// 256 x 256, k = 64, 28.4 products a point 4.23 -> 3.83 ms; 1024 x 1024, k = 64, three products
// 13.7 -> 11.9 ms; 250 x 187, k = 40, 20.7 products 2.01 -> 1.67 ms; one warp per point with
// broadcasts to the whole warp -> this form: 256 x 256, k = 32, 5.8 products 0.378 -> 0.358 ms;
// 301 x 215, k = 24, 9.7 products 0.436 -> 0.414 ms.
template <int KM>
__global__ void __launch_bounds__(32 * kWarpsC, ChebShape<KM>::MINB)
    eig_cheb_kernel(EigArgs a, EigSplit sp, const __grid_constant__ ChebTable ct, int max_set) {
    using S = ChebShape<KM>;
    constexpr int NC = S::NC, HC = S::HC, SP = S::SP;
    extern __shared__ float4 smem_c4[];
    __shared__ __align__(8) uint64_t pbar[kWarpsC];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    float *G = reinterpret_cast<float *>(smem_c4) + (size_t)wib * S::floats;
    float *XS = G + S::off_x, *RS = G + S::off_r, *B = G + S::off_b, *U = G + S::off_u;
    const int k = a.k;
    const float d = a.diag, inv_d = 1.0f / a.diag;
    const float sc = sqrtf((float)(k - 1)) / sqrtf(a.diag);   // sqrt(k-1) d^-1/2
    const int half = lane >> 4, cj = 2 * (lane & 15);         // columns cj, cj + 1 (+ 32, + 33)
    const int col = KM == 64 ? 32 * half + cj : cj + half;    // of them this lane's own: col (, + 1)
    const int ng = (k + 7) / 8, row0 = 4 * ng * half;         // groups of four rows per half warp
    unsigned long long n_pts = 0, n_prod = 0, n_hand = 0;
    const long long nw = (long long)gridDim.x * kWarpsC;
    // Where the Gram slot's rows are 16-byte multiples (k a multiple of 4) the next point's upper
    // triangle (bulk copies of every row from its first multiple of 4), forecast block and c are
    // fetched into the stage while this point is worked on, counted in bytes on the warp's
    // mbarrier; otherwise the warp loads them when the point begins.
    const bool pf = (k & 3) == 0;
    const uint32_t bar = (uint32_t)__cvta_generic_to_shared(&pbar[wib]);
    uint32_t phase = 0;
    auto bulk = [&](float *dst, const float *src, int n) {
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, "
            "[%3];" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
            "l"(src), "r"((uint32_t)(n * 4)), "r"(bar)
            : "memory");
    };
    auto prefetch = [&](long long q) {
        const int g = k / 4;
        if (lane == 0)
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                         "r"((uint32_t)((8 * g * (g + 1) + kRowsC * k) * 4))
                         : "memory");
        __syncwarp();
        const float *src = a.gram + (size_t)q * k * k;
        for (int i = lane; i < k; i += 32)
            bulk(G + i * SP + (i & ~3), src + (size_t)i * k + (i & ~3), k - (i & ~3));
        if (lane == 0) bulk(XS, a.x + (size_t)(a.pt0 + q) * NV * k, NV * k);
        if (lane == 1) bulk(XS + NV * k, a.cvec + (size_t)q * k, k);
    };
    // the stage is zero beyond k rows and columns throughout
    for (int e = lane; e < S::floats; e += 32) G[e] = 0.0f;
    if (lane == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar));
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
    long long lp = (long long)blockIdx.x * kWarpsC + wib;
    if (pf && lp < a.npts) prefetch(lp);
    int nl = a.nloc && lp < a.npts ? __ldg(a.nloc + lp) : 1;

    for (; lp < a.npts; lp += nw) {
        float *X = a.x + (size_t)(a.pt0 + lp) * NV * k;
        const bool zero = nl == 0;
        const bool more = lp + nw < a.npts;
        if (a.nloc && more) nl = __ldg(a.nloc + lp + nw);
        if (pf) {
            // this point's data (bounded wait; a timeout is never expected: report it, give the
            // copies a second bounded wait, leave)
            if (!__all_sync(kAllC, cheb_bar_wait(bar, phase))) {
                if (lane == 0) atomicOr(a.status, ST_TIMEOUT);
                cheb_bar_wait(bar, phase);
                return;
            }
            phase ^= 1;
        } else if (!zero) {
            const float *src = a.gram + (size_t)lp * k * k;
            for (int i = 0; i < k; ++i)
                for (int c = (i & ~31) + lane; c < k; c += 32)
                    if (c >= i) G[i * SP + c] = __ldg(src + (size_t)i * k + c);
            for (int e = lane; e < NV * k; e += 32) XS[e] = __ldcg(X + e);
            for (int e = lane; e < k; e += 32) XS[NV * k + e] = __ldcg(a.cvec + (size_t)lp * k + e);
            __syncwarp();
        }
        if (zero) {
            if (pf && more) prefetch(lp + nw);
            // Q = (k-1)/rho I: wbar = 0 and dW = sqrt(rho) I (untouched for rho = 1)
            if (a.sqrt_infl != 1.0f)
                for (int r = 0; r < NV; ++r) {
                    float v[KM / 32], s = 0.0f;
#pragma unroll
                    for (int q = 0; q < KM / 32; ++q) {
                        const int c = lane + 32 * q;
                        v[q] = c < k ? __ldcg(X + r * k + c) : 0.0f;
                        s += v[q];
                    }
                    const float xb = warp_sum(s) / (float)k;
#pragma unroll
                    for (int q = 0; q < KM / 32; ++q) {
                        const int c = lane + 32 * q;
                        if (c < k) X[r * k + c] = fmaf(a.sqrt_infl, v[q] - xb, xb);
                    }
                }
            continue;
        }
        // ---- A, symmetric, from the staged upper triangle: column c takes A[i][c] for i <= c down
        // its column (two columns per load) and A[c][i] for i > c along its own row
        float2 A[NC][S::RH / 2];
        float f2 = 0.0f, gm = 0.0f;
#pragma unroll
        for (int q = 0; q < NC; q += 2) {
            const int c = cj + 16 * q;
            float s0 = 0.0f, s1 = 0.0f;
#pragma unroll
            for (int g = 0; g < S::RH / 4; ++g) {
                float v0[4] = {0.0f, 0.0f, 0.0f, 0.0f}, v1[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                if (g < ng) {
                    const int i0 = row0 + 4 * g;
                    float4 r0 = make_float4(0.0f, 0.0f, 0.0f, 0.0f), r1 = r0;
                    if (i0 + 3 > c) {
                        r0 = *reinterpret_cast<const float4 *>(G + c * SP + i0);
                        r1 = *reinterpret_cast<const float4 *>(G + (c + 1) * SP + i0);
                    }
                    const float t0[4] = {r0.x, r0.y, r0.z, r0.w}, t1[4] = {r1.x, r1.y, r1.z, r1.w};
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        float2 up = make_float2(0.0f, 0.0f);
                        if (i0 + u <= c + 1)
                            up = *reinterpret_cast<const float2 *>(G + (i0 + u) * SP + c);
                        v0[u] = i0 + u <= c ? up.x : t0[u];
                        v1[u] = i0 + u <= c + 1 ? up.y : t1[u];
                        s0 += fabsf(v0[u]);
                        s1 += fabsf(v1[u]);
                        f2 = fmaf(v0[u], v0[u], fmaf(v1[u], v1[u], f2));
                    }
                }
                A[q][2 * g] = make_float2(v0[0], v0[1]);
                A[q][2 * g + 1] = make_float2(v0[2], v0[3]);
                A[q + 1][2 * g] = make_float2(v1[0], v1[1]);
                A[q + 1][2 * g + 1] = make_float2(v1[2], v1[3]);
            }
            s0 += __shfl_xor_sync(kAllC, s0, 16);
            s1 += __shfl_xor_sync(kAllC, s1, 16);
            gm = fmaxf(gm, fmaxf(s0, s1));
        }
        float dg = 0.0f;
#pragma unroll
        for (int q = 0; q < KM / 32; ++q) dg += G[(lane + 32 * q) * (SP + 1)];
        // rows 5..9 of [x; c] in registers, rows 0..4 put aside: the stage is free again
        float R[5][HC];
#pragma unroll
        for (int r = 0; r < 5; ++r)
#pragma unroll
            for (int q = 0; q < HC; ++q) {
                R[r][q] = col + q < k ? XS[(5 + r) * k + col + q] : 0.0f;
                RS[r * KM + col + q] = col + q < k ? XS[r * k + col + q] : 0.0f;
            }
        if (pf) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (pf && more) prefetch(lp + nw);
        // ---- kappa >= 1 + lambda_max(A) / d from min(Gershgorin, Frobenius, trace)
        gm = warp_max_c(gm);
        f2 = warp_sum(f2);
        dg = warp_sum(dg);
        const float e = fmaxf(fminf(gm, fminf(sqrtf(f2), dg)), 0.0f);
        const float kap = fmaf(e * inv_d, 1.0001f, 1.000001f);   // rounding margin
        int set = 0;
        while (set <= max_set && !(kap <= ct.kappa_max[set])) ++set;
        if (set > max_set) {   // beyond the sets in use (or not finite): the rational schedule
            if (lane == 0) sp.pre_list[atomicAdd(sp.pre_count, 1)] = (int)lp;
            ++n_hand;
            continue;
        }
        const int n = ct.n[set], co = ct.off[set];
        const float gam = 2.0f / (d * (ct.kappa_max[set] - 1.0f));
        bool bad = false;
#pragma unroll 1
        for (int pass = 1; pass >= 0; --pass) {   // rows 5..9 (with c), then 0..4
            if (pass == 0)
#pragma unroll
                for (int r = 0; r < 5; ++r)
#pragma unroll
                    for (int q = 0; q < HC; ++q) R[r][q] = RS[r * KM + col + q];
            // ---- R = [dX; c^T]: the rows less their means
            float mean[5];
#pragma unroll
            for (int r = 0; r < 5; ++r) {
                float s = R[r][0];
#pragma unroll
                for (int q = 1; q < HC; ++q) s += R[r][q];
                mean[r] = warp_sum(s) / (float)k;
                if (r == 4 && pass) mean[r] = 0.0f;
#pragma unroll
                for (int q = 0; q < HC; ++q) R[r][q] = col + q < k ? R[r][q] - mean[r] : 0.0f;
            }
            // ---- Clenshaw: b_n = c_n R, b_j = c_j R + 2 b_{j+1} Z - b_{j+2}, result
            // c_0 R + b_1 Z - b_2, with b_{j+1} Z = gamma b_{j+1} A - b_{j+1}.  Bc holds b_{j+1}
            // (also in B for the products), Bp b_{j+2}.
            float Bc[5][HC], Bp[5][HC];
            auto publish = [&]() {
#pragma unroll
                for (int r = 0; r < 5; ++r) {
                    if constexpr (HC == 2)
                        *reinterpret_cast<float2 *>(B + r * KM + col) = make_float2(Bc[r][0], Bc[r][1]);
                    else
                        B[r * KM + col] = Bc[r][0];
                }
                __syncwarp();
            };
            {
                const float2 cn = ct.c[co + n];
#pragma unroll
                for (int r = 0; r < 5; ++r)
#pragma unroll
                    for (int q = 0; q < HC; ++q) {
                        Bc[r][q] = (r == 4 && pass ? cn.y : cn.x) * R[r][q];
                        Bp[r][q] = 0.0f;
                    }
            }
            __syncwarp();
            publish();
            for (int j = n - 1; j >= 0; --j) {
                const float2 cc = ct.c[co + j];
                float v[5][HC];
                cheb_product<KM>(B + row0, A, ng, half, v);
                const float two = j > 0 ? 2.0f : 1.0f;
#pragma unroll
                for (int r = 0; r < 5; ++r)
#pragma unroll
                    for (int q = 0; q < HC; ++q) {
                        const float cr = r == 4 && pass ? cc.y : cc.x;
                        const float z = fmaf(gam, v[r][q], -Bc[r][q]);
                        const float nb = fmaf(cr, R[r][q], fmaf(two, z, -Bp[r][q]));
                        Bp[r][q] = Bc[r][q];
                        Bc[r][q] = nb;
                    }
                __syncwarp();   // B is read
                if (j > 0) publish();
            }
            // ---- u = Q^-1 c = S^-1 c / d; X^a_r = xbar_r + dX_r . u + sqrt(k-1) d^-1/2 (dX S^-1/2)_r
            float u[HC];
#pragma unroll
            for (int q = 0; q < HC; ++q) {
                if (pass) U[col + q] = u[q] = Bc[4][q] * inv_d;
                else u[q] = U[col + q];
            }
#pragma unroll
            for (int r = 0; r < 5; ++r) {
                if (r == 4 && pass) break;
                float s = R[r][0] * u[0];
#pragma unroll
                for (int q = 1; q < HC; ++q) s = fmaf(R[r][q], u[q], s);
                const float base = mean[r] + warp_sum(s);
#pragma unroll
                for (int q = 0; q < HC; ++q)
                    if (col + q < k) {
                        const float x = fmaf(sc, Bc[r][q], base);
                        bad |= !isfinite(x);
                        X[(5 * pass + r) * k + col + q] = x;
                    }
            }
        }
        if (__any_sync(kAllC, bad) && lane == 0) atomicOr(a.status, ST_NONFINITE);
        ++n_pts;
        n_prod += (unsigned long long)n;
    }
    if (a.work && lane == 0 && (n_pts | n_hand)) {
        atomicAdd(a.work, n_pts);
        atomicAdd(a.work + 1, n_prod);
        atomicAdd(a.work + 2, n_hand);
    }
}

// Five rows of R times NG groups of four rows of A (the loads of later groups run ahead of the
// multiply-adds: a run-time bound on the groups kept every group waiting for its own loads).
template <int NG>
__device__ __forceinline__ void cheb_block_product_ng(const float *b,
                                                const float2 (&A)[ChebBlock::NC][16],
                                                float (&out)[5][ChebBlock::NC]) {
    constexpr int NC = ChebBlock::NC, KM = ChebBlock::KM;
    const float4 *B4 = reinterpret_cast<const float4 *>(b);
    float2 acc[5][NC];
#pragma unroll
    for (int rr = 0; rr < 5; ++rr)
#pragma unroll
        for (int q = 0; q < NC; ++q) acc[rr][q] = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int g = 0; g < NG; ++g)
#pragma unroll
        for (int rr = 0; rr < 5; ++rr) {
            const float4 v = B4[rr * (KM / 4) + g];
#pragma unroll
            for (int q = 0; q < NC; ++q) {
                acc[rr][q] = __ffma2_rn(make_float2(v.x, v.y), A[q][2 * g], acc[rr][q]);
                acc[rr][q] = __ffma2_rn(make_float2(v.z, v.w), A[q][2 * g + 1], acc[rr][q]);
            }
        }
#pragma unroll
    for (int rr = 0; rr < 5; ++rr)
#pragma unroll
        for (int q = 0; q < NC; ++q) out[rr][q] = acc[rr][q].x + acc[rr][q].y;
}

// ng groups of the warp's 8 (rows of A beyond them are zero)
__device__ __forceinline__ void cheb_block_product(const float *b,
                                             const float2 (&A)[ChebBlock::NC][16], int ng,
                                             float (&out)[5][ChebBlock::NC]) {
    if (ng > 6) cheb_block_product_ng<8>(b, A, out);
    else if (ng > 4) cheb_block_product_ng<6>(b, A, out);
    else cheb_block_product_ng<4>(b, A, out);
}

// k <= 128.  What bounds it: per product and point 10 k^2 multiply-adds on the FP32 pipe; between
// products the latency of two barriers and of the exchange, covered by the SM's other point.
// 192 x 160, k = 128, clustered network (13 products a point): 77.1 -> 3.4 ms against the split
// eigensolve that served k > 64 alone.
__global__ void __launch_bounds__(32 * ChebBlock::NW, 2)
    eig_cheb_block_kernel(EigArgs a, EigSplit sp, const __grid_constant__ ChebTable ct,
                          int max_set) {
    using S = ChebBlock;
    constexpr int KM = S::KM, NW = S::NW, CS = S::CS, NC = S::NC, NE = S::NE, SP = S::SP;
    extern __shared__ float4 smem_c4[];
    __shared__ __align__(8) uint64_t pbar;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    float *ws = reinterpret_cast<float *>(smem_c4);
    float *G = ws, *XS = ws + S::off_x, *B = ws + S::off_b, *P = ws + S::off_p, *RD = ws + S::off_r;
    const int k = a.k;
    const float d = a.diag, inv_d = 1.0f / a.diag;
    const float sc = sqrtf((float)(k - 1)) / sqrtf(a.diag);   // sqrt(k-1) d^-1/2
    const int cg = w % S::CG, rb = w / S::CG;
    const int rpb = ((k + S::RB - 1) / S::RB + 3) & ~3;       // rows of a block, in groups of 4
    const int row0 = rb * rpb, ng = max(0, min(k - row0, rpb) + 3) / 4;
    unsigned long long n_pts = 0, n_prod = 0, n_hand = 0;
    const long long stride = (long long)gridDim.x;
    // Where the Gram slot's rows are 16-byte multiples (k a multiple of 4) the next point's upper
    // triangle (bulk copies of every row from its first multiple of 4), forecast block and c are
    // fetched into the stage while this point is worked on, counted in bytes on an mbarrier;
    // otherwise the warps load them when the point begins.
    const bool pf = (k & 3) == 0;
    const uint32_t bar = (uint32_t)__cvta_generic_to_shared(&pbar);
    uint32_t phase = 0;
    auto bulk = [&](float *dst, const float *src, int n) {
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, "
            "[%3];" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
            "l"(src), "r"((uint32_t)(n * 4)), "r"(bar)
            : "memory");
    };
    auto prefetch = [&](long long q) {   // warp 0 of the point
        const int g = k / 4;
        if (lane == 0)
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                         "r"((uint32_t)((8 * g * (g + 1) + kRowsC * k) * 4))
                         : "memory");
        __syncwarp();
        const float *src = a.gram + (size_t)q * k * k;
        for (int i = lane; i < k; i += 32)
            bulk(G + i * SP + (i & ~3), src + (size_t)i * k + (i & ~3), k - (i & ~3));
        if (lane == 0) bulk(XS, a.x + (size_t)(a.pt0 + q) * NV * k, NV * k);
        if (lane == 1) bulk(XS + NV * k, a.cvec + (size_t)q * k, k);
    };
    // the stage is zero beyond k rows and columns throughout
    for (int e = lane + 32 * w; e < S::off_b; e += 32 * NW) ws[e] = 0.0f;
    if (lane == 0 && w == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar));
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    long long lp = blockIdx.x;
    if (pf && w == 0 && lp < a.npts) prefetch(lp);
    int nl = a.nloc && lp < a.npts ? __ldg(a.nloc + lp) : 1;

    for (; lp < a.npts; lp += stride) {
        float *X = a.x + (size_t)(a.pt0 + lp) * NV * k;
        const bool zero = nl == 0;
        const bool more = lp + stride < a.npts;
        if (a.nloc && more) nl = __ldg(a.nloc + lp + stride);
        if (pf) {
            // this point's data (bounded wait; a timeout is never expected: report it, give the
            // copies a second bounded wait, leave)
            if (!__syncthreads_and(cheb_bar_wait(bar, phase))) {
                if (lane == 0 && w == 0) atomicOr(a.status, ST_TIMEOUT);
                cheb_bar_wait(bar, phase);
                return;
            }
            phase ^= 1;
        } else if (!zero) {
            const float *src = a.gram + (size_t)lp * k * k;
            for (int i = w; i < k; i += NW)
                for (int c = (i & ~31) + lane; c < k; c += 32)
                    if (c >= i) G[i * SP + c] = __ldg(src + (size_t)i * k + c);
            for (int e = lane + 32 * w; e < NV * k; e += 32 * NW) XS[e] = __ldcg(X + e);
            for (int e = lane + 32 * w; e < k; e += 32 * NW)
                XS[NV * k + e] = __ldcg(a.cvec + (size_t)lp * k + e);
            __syncthreads();
        }
        if (zero) {
            if (pf && w == 0 && more) prefetch(lp + stride);
            // Q = (k-1)/rho I: wbar = 0 and dW = sqrt(rho) I (untouched for rho = 1)
            if (a.sqrt_infl != 1.0f)
                for (int r = w; r < NV; r += NW) {
                    float v[CS], s = 0.0f;
#pragma unroll
                    for (int q = 0; q < CS; ++q) {
                        const int c = lane + 32 * q;
                        v[q] = c < k ? __ldcg(X + r * k + c) : 0.0f;
                        s += v[q];
                    }
                    const float xb = warp_sum(s) / (float)k;
#pragma unroll
                    for (int q = 0; q < CS; ++q) {
                        const int c = lane + 32 * q;
                        if (c < k) X[r * k + c] = fmaf(a.sqrt_infl, v[q] - xb, xb);
                    }
                }
            continue;
        }
        // ---- A, symmetric, from the staged upper triangle: column c takes A[i][c] for i <= c down
        // its column and A[c][i] for i > c along its own row
        float2 A[NC][16];
        float csum[NC], f2 = 0.0f, dg = 0.0f;
#pragma unroll
        for (int q = 0; q < NC; ++q) {
            const int c = 32 * (NC * cg + q) + lane;
            csum[q] = 0.0f;
#pragma unroll
            for (int g = 0; g < 8; ++g) {
                float v[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                if (g < ng) {
                    const int i0 = row0 + 4 * g;
                    float4 r = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    if (i0 + 3 > c) r = *reinterpret_cast<const float4 *>(G + c * SP + i0);
                    v[0] = i0 <= c ? G[i0 * SP + c] : r.x;
                    v[1] = i0 + 1 <= c ? G[(i0 + 1) * SP + c] : r.y;
                    v[2] = i0 + 2 <= c ? G[(i0 + 2) * SP + c] : r.z;
                    v[3] = i0 + 3 <= c ? G[(i0 + 3) * SP + c] : r.w;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        csum[q] += fabsf(v[u]);
                        f2 = fmaf(v[u], v[u], f2);
                    }
                }
                A[q][2 * g] = make_float2(v[0], v[1]);
                A[q][2 * g + 1] = make_float2(v[2], v[3]);
            }
            if (rb == 0) dg += G[c * SP + c];
            P[rb * KM + c] = csum[q];
        }
        f2 = warp_sum(f2);
        dg = warp_sum(dg);
        if (lane == 0) {
            RD[2 * w] = f2;
            RD[2 * w + 1] = dg;
        }
        // ---- this warp's entries of [x; c]: (row, 32-column slot) NE w + t
        float R[NE], Bc[NE], Bp[NE];
        float *sums = RD + 2 * NW, *dots = sums + kRowsC * CS;
#pragma unroll
        for (int t = 0; t < NE; ++t) {
            const int s = NE * w + t, row = s / CS, col = 32 * (s % CS) + lane;
            R[t] = col < k ? XS[row * k + col] : 0.0f;
        }
#pragma unroll
        for (int t = 0; t < NE; ++t) {
            const float v = warp_sum(R[t]);
            if (lane == 0) sums[NE * w + t] = v;
        }
        if (pf) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();   // the stage is read: the next point's copies may land in it
        if (pf && w == 0 && more) prefetch(lp + stride);
        // ---- kappa >= 1 + lambda_max(A) / d from min(Gershgorin, Frobenius, trace)
        float gm = 0.0f;
#pragma unroll
        for (int q = 0; q < CS; ++q) {
            float g = 0.0f;
#pragma unroll
            for (int b = 0; b < S::RB; ++b) g += P[b * KM + 32 * q + lane];
            gm = fmaxf(gm, g);
        }
        gm = warp_max_c(gm);
        f2 = dg = 0.0f;
#pragma unroll
        for (int i = 0; i < NW; ++i) {
            f2 += RD[2 * i];
            dg += RD[2 * i + 1];
        }
        const float e = fmaxf(fminf(gm, fminf(sqrtf(f2), dg)), 0.0f);
        const float kap = fmaf(e * inv_d, 1.0001f, 1.000001f);   // rounding margin
        int set = 0;
        while (set <= max_set && !(kap <= ct.kappa_max[set])) ++set;
        if (set > max_set) {
            // beyond the sets in use (or not finite): the next schedule
            if (lane == 0 && w == 0) sp.pre_list[atomicAdd(sp.pre_count, 1)] = (int)lp;
            ++n_hand;
            __syncthreads();   // P and RD are read before the next point writes them
            continue;
        }
        // ---- R = [dX; c^T]: the nine rows less their means
        auto row_mean = [&](int row) {
            float v = 0.0f;
#pragma unroll
            for (int q = 0; q < CS; ++q) v += sums[row * CS + q];
            return row < NV ? v / (float)k : 0.0f;
        };
        float mean[NE];   // (another warp may be writing the next point's sums at the end)
#pragma unroll
        for (int t = 0; t < NE; ++t) {
            const int s = NE * w + t, row = s / CS, col = 32 * (s % CS) + lane;
            const float m = row_mean(row);
            mean[t] = m;
            R[t] = col < k ? R[t] - m : 0.0f;
        }
        // ---- Clenshaw: b_n = c_n R, b_j = c_j R + 2 b_{j+1} Z - b_{j+2}, result
        // c_0 R + b_1 Z - b_2, with b_{j+1} Z = gamma b_{j+1} A - b_{j+1}.  Bc holds b_{j+1}
        // (also in B for the products), Bp b_{j+2}.
        const int n = ct.n[set], co = ct.off[set];
        const float gam = 2.0f / (d * (ct.kappa_max[set] - 1.0f));
        const int last = kRowsC * CS - CS;   // entries of row 9 (c) start here
        {
            const float2 cn = ct.c[co + n];
#pragma unroll
            for (int t = 0; t < NE; ++t) {
                const int s = NE * w + t;
                Bc[t] = (s < last ? cn.x : cn.y) * R[t];
                Bp[t] = 0.0f;
                B[32 * s + lane] = Bc[t];
            }
        }
        __syncthreads();
        // rows r0 .. r0 + 4 of B times this warp's rows and columns of A
        auto product = [&](int r0, float (&out)[5][NC]) {
            cheb_block_product(B + r0 * KM + row0, A, ng, out);
        };
        for (int j = n - 1; j >= 0; --j) {
            const float2 cj = ct.c[co + j];
            float v[NE];
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                float o[5][NC];
                product(5 * p, o);
                float *pw = P + (rb * kRowsC + 5 * p) * KM + 32 * NC * cg + lane;
#pragma unroll
                for (int rr = 0; rr < 5; ++rr)
#pragma unroll
                    for (int q = 0; q < NC; ++q) pw[rr * KM + 32 * q] = o[rr][q];
            }
            __syncthreads();
#pragma unroll
            for (int t = 0; t < NE; ++t) {
                const float *pr = P + 32 * (NE * w + t) + lane;
                v[t] = (pr[0] + pr[kRowsC * KM]) + (pr[2 * kRowsC * KM] + pr[3 * kRowsC * KM]);
            }
#pragma unroll
            for (int t = 0; t < NE; ++t) {
                const int s = NE * w + t;
                const float cr = s < last ? cj.x : cj.y;
                const float z = fmaf(gam, v[t], -Bc[t]);
                const float nb = j > 0 ? fmaf(cr, R[t], fmaf(2.0f, z, -Bp[t]))
                                       : fmaf(cr, R[t], z - Bp[t]);
                Bp[t] = Bc[t];
                Bc[t] = nb;
                B[32 * s + lane] = nb;
            }
            __syncthreads();
        }
        // ---- u = Q^-1 c = S^-1 c / d; X^a_r = xbar_r + dX_r . u + sqrt(k-1) d^-1/2 (dX S^-1/2)_r
#pragma unroll
        for (int t = 0; t < NE; ++t) {
            const int s = NE * w + t;
            const float u = B[NV * KM + 32 * (s % CS) + lane] * inv_d;
            const float v = warp_sum(R[t] * u);
            if (lane == 0) dots[s] = v;
        }
        __syncthreads();
        bool bad = false;
#pragma unroll
        for (int t = 0; t < NE; ++t) {
            const int s = NE * w + t, row = s / CS, col = 32 * (s % CS) + lane;
            float v = 0.0f;
#pragma unroll
            for (int q = 0; q < CS; ++q) v += dots[row * CS + q];
            if (row < NV && col < k) {
                // mean and increment as two words: their rounded sum alone would be the same error
                // in every member, and so in the analysis mean
                const float s0 = mean[t] + v, b0 = s0 - mean[t];
                const float lo = (mean[t] - (s0 - b0)) + (v - b0);
                v = s0 + fmaf(sc, Bc[t], lo);
                bad |= !isfinite(v);
                X[row * k + col] = v;
            }
        }
        if (__any_sync(kAllC, bad) && lane == 0) atomicOr(a.status, ST_NONFINITE);
        ++n_pts;
        n_prod += (unsigned long long)n;
    }
    if (a.work && lane == 0 && w == 0 && (n_pts | n_hand)) {
        atomicAdd(a.work, n_pts);
        atomicAdd(a.work + 1, n_prod);
        atomicAdd(a.work + 2, n_hand);
    }
}

constexpr size_t kBlockSmem = (size_t)ChebBlock::floats * sizeof(float);
template <int KM>
constexpr size_t cheb_smem() {
    return (size_t)ChebShape<KM>::floats * kWarpsC * sizeof(float);
}

cudaError_t cheb_prepare(const void *kern, int threads, size_t smem, int k, int *grid) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0, per_sm = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
        return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    *grid = sms * per_sm;
    cheb_table(k);
    return cudaSuccess;
}

template <int KM>
cudaError_t cheb_launch_km(const EigArgs &a, const EigSplit &sp, int grid, cudaStream_t s) {
    const long long need = ((long long)a.npts + kWarpsC - 1) / kWarpsC;
    const unsigned blocks = (unsigned)(need < grid ? need : grid);
    eig_cheb_kernel<KM><<<blocks, 32 * kWarpsC, cheb_smem<KM>(), s>>>(
        a, sp, cheb_table(a.k), cheb_max_set(a.k));
    return cudaGetLastError();
}

}  // namespace

cudaError_t eigen_cheb_prepare(int k, int *grid) {
    if (k <= 32)
        return cheb_prepare((const void *)eig_cheb_kernel<32>, 32 * kWarpsC, cheb_smem<32>(), k, grid);
    if (k <= 64)
        return cheb_prepare((const void *)eig_cheb_kernel<64>, 32 * kWarpsC, cheb_smem<64>(), k, grid);
    if (k <= kChebSplitMaxK)
        return cheb_prepare((const void *)eig_cheb_block_kernel, 32 * ChebBlock::NW, kBlockSmem, k,
                            grid);
    return cudaErrorInvalidValue;
}

cudaError_t launch_eigen_cheb_transform(const EigArgs &a, const EigSplit &sp, int grid,
                                        cudaStream_t s) {
    if (a.npts <= 0) return cudaSuccess;
    if (!sp.pre_list || !sp.pre_count || grid < 1) return cudaErrorInvalidValue;
    if (a.k <= 32) return cheb_launch_km<32>(a, sp, grid, s);
    if (a.k <= 64) return cheb_launch_km<64>(a, sp, grid, s);
    if (a.k <= kChebSplitMaxK) {
        const unsigned blocks = (unsigned)(a.npts < grid ? a.npts : grid);
        eig_cheb_block_kernel<<<blocks, 32 * ChebBlock::NW, kBlockSmem, s>>>(
            a, sp, cheb_table(a.k), cheb_max_set(a.k));
        return cudaGetLastError();
    }
    return cudaErrorInvalidValue;
}

}  // namespace lk

extern "C" double letkf_chebyshev_coefficients(double kappa_max, int32_t n, double *c_rsqrt,
                                               double *c_inv) {
    if (!(kappa_max > 1.0) || !(kappa_max < 1e6) || n < 1 || n > 256 || !c_rsqrt || !c_inv)
        return -1.0;
    return lk::chebyshev_coefficients(kappa_max, n, c_rsqrt, c_inv);
}
