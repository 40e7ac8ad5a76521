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
// Layout: A in registers, 32 rows of two columns per lane (one column for k <= 32), loaded from
// the upper triangle of the Gram slot staged in shared memory; one warp per grid point for
// k <= 32, two (halves of the rows) for k <= 64, eight (quarters of the rows x halves of the
// columns) for k <= 128, so that 16 warps or more share an SM.  A product R A reads the rows of R
// as 16-byte broadcasts (five loads for 20 packed multiply-adds) and the warps' partial sums
// meet in shared memory; the recurrence's own values stay in registers.
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
// error stays below 2e-8 (under FP32 rounding of the result).  The sets beyond 16 serve
// k > kChebMaxK only and are built with it (degrees from the same criterion, found once).
namespace {
void cheb_set(ChebTable &t, int s, double kmax, int degree) {
    // the interval the kernel maps onto [-1, 1] is the FP32 kappa_max: the coefficients and the
    // degree are those of that interval
    const float kf = (float)kmax;
    const double km = (double)kf;
    std::vector<double> ca(256), cb(256);
    int n = degree;
    if (n == 0) {
        n = 1;
        while (n < kChebMaxDeg && chebyshev_coefficients(km, n, ca.data(), cb.data()) > 2e-8) ++n;
    }
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
        const double kmax[kChebSets] = {1.0002, 1.005, 1.035, 1.1, 1.2,  1.35, 1.5, 1.75,
                                        2.0,    2.5,   3.0,   4.0, 6.0, 10.0, 16.0};
        for (int s = 0; s < kChebSets; ++s) cheb_set(t, s, kmax[s], 0);
    });
    if (k <= kChebMaxK) return t;
    std::call_once(once_big, [] {
        big = t;
        const double kmax[kChebBigSets - kChebSets] = {24, 36, 54, 80, 120, 180, 270, 400};
        const int deg[kChebBigSets - kChebSets] = {44, 54, 67, 82, 100, 123, 151, 184};
        for (int i = 0; i < kChebBigSets - kChebSets; ++i)
            cheb_set(big, kChebSets + i, kmax[i], deg[i]);
    });
    return big;
}

// The largest set the transform uses for ensemble size k.  k <= 64: degrees up to 9k/16 (at least
// 4): a product with A costs ~20 k^2 flops, the rational schedule's tridiagonalization and
// transform ~(4/3) k^3 + 40 k^2 at a lower issue efficiency; at k = 64 the two measured equal
// near degree 36, and the break-even degree scales with k.  Points beyond go to the rational
// schedule, so the Chebyshev schedule never costs much more than the rational one.  k > 64: the
// alternative is the split eigensolve, ~2.5 us a point at k = 128 against ~10 ns a product:
// every set is used up to degree 1.4 k.
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

template <int KM>
struct ChebShape {
    static constexpr int NW = KM == 32 ? 1 : KM == 64 ? 2 : 8;   // warps per point
    static constexpr int PPB = NW == 1 ? 4 : 1;                  // points per block
    static constexpr int CS = KM / 32;                           // 32-column slots of a row
    static constexpr int NC = KM == 32 ? 1 : 2;                  // columns of a lane
    static constexpr int CG = CS / NC, RB = NW / CG;             // column groups, row blocks
    static constexpr int RR = KM / RB;                           // rows of a block
    static constexpr int NE = kRowsC * CS / NW;                  // (row, slot) entries of a warp
    static constexpr int SP = KM + 4;                            // stride of the staged slot
    static constexpr int off_x = KM * SP;                        // [9][k] and c[k]
    static constexpr int off_b = off_x + kRowsC * KM;            // b_{j+1}, [10][KM]
    static constexpr int off_p = off_b + kRowsC * KM;            // partial sums
    static constexpr int psize = RB == 1 ? KM : RB == 2 ? kRowsC * KM : RB * kRowsC * KM;
    static constexpr int off_r = off_p + psize;                  // reductions over the warps
    static constexpr int floats = off_r + 2 * NW + 2 * kRowsC * CS + (KM == 32 ? 6 : 0);
    static_assert(RR == 32 && psize >= RB * KM, "32 rows per block; the columns' sums fit");
    static_assert(floats % 4 == 0, "16-byte aligned point buffers");
    // blocks per SM: 12 warps with 168 registers (k <= 64; 16 warps of 128 spill and measured 8 %
    // slower at k = 64, 6 % at k = 32), 16 with 128 (k <= 128, by shared memory)
    static constexpr int MINB = KM == 32 ? 3 : KM == 64 ? 6 : 2;
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

template <int NW>
__device__ __forceinline__ void point_sync() {   // the warps of one point
    if constexpr (NW == 1) __syncwarp();
    else __syncthreads();
}

// Five rows of R times NG groups of four rows of A (the loads of later groups run ahead of the
// multiply-adds: a run-time bound on the groups kept every group waiting for its own loads).
template <int KM, int NG>
__device__ __forceinline__ void cheb_product_ng(const float *b,
                                                const float2 (&A)[ChebShape<KM>::NC][16],
                                                float (&out)[5][ChebShape<KM>::NC]) {
    constexpr int NC = ChebShape<KM>::NC;
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
template <int KM>
__device__ __forceinline__ void cheb_product(const float *b,
                                             const float2 (&A)[ChebShape<KM>::NC][16], int ng,
                                             float (&out)[5][ChebShape<KM>::NC]) {
    if (ng > 6) cheb_product_ng<KM, 8>(b, A, out);
    else if (ng > 4) cheb_product_ng<KM, 6>(b, A, out);
    else cheb_product_ng<KM, 4>(b, A, out);
}

// What bounds it: per product and point 10 k^2 multiply-adds on the FP32 pipe against 5 k^2 / 2
// 16-byte broadcasts per 20 k^2 / 4 packed instructions; between products the latency of two
// barriers and of the exchange, covered by the other points of the SM.  At k <= 64 the phase
// against A as rows of the block's lanes, re-read from shared memory: 256 x 256, k = 32, 5.8
// products a point 0.436 -> 0.378 ms; 250 x 187, k = 40, 20.7 products 2.46 -> 2.01 ms; 301 x 215,
// k = 24, 9.7 products 0.583 -> 0.436 ms; k = 64 the same (256 x 256, 28.4 products 4.28 -> 4.23
// ms).  192 x 160, k = 128, clustered network, 13.4 products: 77.1 -> 3.44 ms against the split
// eigensolve, which served k > 64 alone.
template <int KM>
__global__ void __launch_bounds__(32 * ChebShape<KM>::NW * ChebShape<KM>::PPB, ChebShape<KM>::MINB)
    eig_cheb_kernel(EigArgs a, EigSplit sp, const __grid_constant__ ChebTable ct, int max_set) {
    using S = ChebShape<KM>;
    constexpr int NW = S::NW, CS = S::CS, NC = S::NC, NE = S::NE, SP = S::SP;
    extern __shared__ float4 smem_c4[];
    __shared__ __align__(8) uint64_t pbar[S::PPB];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int pb = NW == 1 ? wib : 0, w = NW == 1 ? 0 : wib;   // point of the block, its warp
    float *ws = reinterpret_cast<float *>(smem_c4) + (size_t)pb * S::floats;
    float *G = ws, *XS = ws + S::off_x, *B = ws + S::off_b, *P = ws + S::off_p, *RD = ws + S::off_r;
    const int k = a.k;
    const float d = a.diag, inv_d = 1.0f / a.diag;
    const float sc = sqrtf((float)(k - 1)) / sqrtf(a.diag);   // sqrt(k-1) d^-1/2
    const int cg = w % S::CG, rb = w / S::CG;
    const int rpb = ((k + S::RB - 1) / S::RB + 3) & ~3;       // rows of a block, in groups of 4
    const int row0 = rb * rpb, ng = max(0, min(k - row0, rpb) + 3) / 4;
    unsigned long long n_pts = 0, n_prod = 0, n_hand = 0;
    const long long stride = (long long)gridDim.x * S::PPB;
    // Where the Gram slot's rows are 16-byte multiples (k a multiple of 4) the next point's upper
    // triangle (bulk copies of every row from its first multiple of 4), forecast block and c are
    // fetched into the stage while this point is worked on, counted in bytes on an mbarrier;
    // otherwise the warps load them when the point begins.
    const bool pf = (k & 3) == 0;
    const uint32_t bar = (uint32_t)__cvta_generic_to_shared(&pbar[pb]);
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
    point_sync<NW>();
    long long lp = (long long)blockIdx.x * S::PPB + pb;
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
            bool ok = cheb_bar_wait(bar, phase);
            if constexpr (NW == 1) ok = __all_sync(kAllC, ok);
            else ok = __syncthreads_and(ok);
            if (!ok) {
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
            point_sync<NW>();
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
        float2 A[NC][16];   // RR / 2
        float csum[NC], f2 = 0.0f, dg = 0.0f;
#pragma unroll
        for (int q = 0; q < NC; ++q) {
            const int c = 32 * (NC * cg + q) + lane;
            csum[q] = 0.0f;
#pragma unroll
            for (int g = 0; g < S::RR / 4; ++g) {
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
        point_sync<NW>();   // the stage is read: the next point's copies may land in it
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
            point_sync<NW>();   // P and RD are read before the next point writes them
            continue;
        }
        // ---- R = [dX; c^T]: the nine rows less their means
        auto row_mean = [&](int row) {
            float v = 0.0f;
#pragma unroll
            for (int q = 0; q < CS; ++q) v += sums[row * CS + q];
            return row < NV ? v / (float)k : 0.0f;
        };
        // (kept where another warp may already be writing the next point's sums at the end)
        constexpr bool kKeep = NW > 2;
        float mean[kKeep ? NE : 1];
#pragma unroll
        for (int t = 0; t < NE; ++t) {
            const int s = NE * w + t, row = s / CS, col = 32 * (s % CS) + lane;
            const float m = row_mean(row);
            if (kKeep) mean[t] = m;
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
        point_sync<NW>();
        // rows r0 .. r0 + 4 of B times this warp's rows and columns of A
        auto product = [&](int r0, float (&out)[5][NC]) {
            cheb_product<KM>(B + r0 * KM + row0, A, ng, out);
        };
        for (int j = n - 1; j >= 0; --j) {
            const float2 cj = ct.c[co + j];
            float v[NE];
            if constexpr (S::RB == 1) {          // one warp: both passes are its own
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    float o[5][NC];
                    product(5 * p, o);
#pragma unroll
                    for (int rr = 0; rr < 5; ++rr) v[5 * p + rr] = o[rr][0];
                }
                __syncwarp();
            } else if constexpr (S::RB == 2) {   // the other warp's rows first, then its own
                float o[5][NC];
                product(5 * (1 - w), o);
                float *pw = P + 5 * (1 - w) * KM + lane;
#pragma unroll
                for (int rr = 0; rr < 5; ++rr)
#pragma unroll
                    for (int q = 0; q < NC; ++q) pw[rr * KM + 32 * q] = o[rr][q];
                product(5 * w, o);
                point_sync<NW>();
                const float *pr = P + 5 * w * KM + lane;
#pragma unroll
                for (int rr = 0; rr < 5; ++rr)
#pragma unroll
                    for (int q = 0; q < NC; ++q)
                        v[2 * rr + q] = o[rr][q] + pr[rr * KM + 32 * q];
            } else {                             // every row block's sums through shared memory
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
                point_sync<NW>();
#pragma unroll
                for (int t = 0; t < NE; ++t) {
                    const float *pr = P + 32 * (NE * w + t) + lane;
                    v[t] = (pr[0] + pr[kRowsC * KM]) + (pr[2 * kRowsC * KM] + pr[3 * kRowsC * KM]);
                }
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
            point_sync<NW>();
        }
        // ---- u = Q^-1 c = S^-1 c / d; X^a_r = xbar_r + dX_r . u + sqrt(k-1) d^-1/2 (dX S^-1/2)_r
#pragma unroll
        for (int t = 0; t < NE; ++t) {
            const int s = NE * w + t;
            const float u = B[NV * KM + 32 * (s % CS) + lane] * inv_d;
            const float v = warp_sum(R[t] * u);
            if (lane == 0) dots[s] = v;
        }
        point_sync<NW>();
        bool bad = false;
#pragma unroll
        for (int t = 0; t < NE; ++t) {
            const int s = NE * w + t, row = s / CS, col = 32 * (s % CS) + lane;
            float v = kKeep ? mean[kKeep ? t : 0] : row_mean(row);
#pragma unroll
            for (int q = 0; q < CS; ++q) v += dots[row * CS + q];
            if (row < NV && col < k) {
                v = fmaf(sc, Bc[t], v);
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

template <int KM>
constexpr size_t cheb_smem() {
    return (size_t)ChebShape<KM>::floats * ChebShape<KM>::PPB * sizeof(float);
}

template <int KM>
cudaError_t cheb_prepare_km(int k, int *grid) {
    using S = ChebShape<KM>;
    const size_t smem = cheb_smem<KM>();
    cudaError_t e = cudaFuncSetAttribute(eig_cheb_kernel<KM>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0, per_sm = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
        return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, eig_cheb_kernel<KM>,
                                                      32 * S::NW * S::PPB, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    *grid = sms * per_sm;
    cheb_table(k);
    return cudaSuccess;
}

template <int KM>
cudaError_t cheb_launch_km(const EigArgs &a, const EigSplit &sp, int grid, cudaStream_t s) {
    using S = ChebShape<KM>;
    const long long need = ((long long)a.npts + S::PPB - 1) / S::PPB;
    const unsigned blocks = (unsigned)(need < grid ? need : grid);
    eig_cheb_kernel<KM><<<blocks, 32 * S::NW * S::PPB, cheb_smem<KM>(), s>>>(
        a, sp, cheb_table(a.k), cheb_max_set(a.k));
    return cudaGetLastError();
}

}  // namespace

cudaError_t eigen_cheb_prepare(int k, int *grid) {
    if (k <= 32) return cheb_prepare_km<32>(k, grid);
    if (k <= 64) return cheb_prepare_km<64>(k, grid);
    if (k <= kChebSplitMaxK) return cheb_prepare_km<128>(k, grid);
    return cudaErrorInvalidValue;
}

cudaError_t launch_eigen_cheb_transform(const EigArgs &a, const EigSplit &sp, int grid,
                                        cudaStream_t s) {
    if (a.npts <= 0) return cudaSuccess;
    if (!sp.pre_list || !sp.pre_count || grid < 1) return cudaErrorInvalidValue;
    if (a.k <= 32) return cheb_launch_km<32>(a, sp, grid, s);
    if (a.k <= 64) return cheb_launch_km<64>(a, sp, grid, s);
    if (a.k <= kChebSplitMaxK) return cheb_launch_km<128>(a, sp, grid, s);
    return cudaErrorInvalidValue;
}

}  // namespace lk

extern "C" double letkf_chebyshev_coefficients(double kappa_max, int32_t n, double *c_rsqrt,
                                               double *c_inv) {
    if (!(kappa_max > 1.0) || !(kappa_max < 1e6) || n < 1 || n > 256 || !c_rsqrt || !c_inv)
        return -1.0;
    return lk::chebyshev_coefficients(kappa_max, n, c_rsqrt, c_inv);
}
