// Batched ensemble D2Q9 lattice Boltzmann kernels (Sec. II-A).
//
// Time steps of Eq. 1 for every member at once: the nine populations of a node give the moments
// (Eqs. 2-3), the BGK relaxation towards the second-order D2Q9 equilibrium plus the body-force
// source F_q = 3 w_q c_q . F, and every post-collision population moves to the neighbour
// x + c_q (periodic).  The stored state is the post-streaming f.
//
// Layout: member-major structure of arrays g[m][q][y][x] (the paper's LBM layout
// X[m, N_v, N_x], Sec. IV-A), FP32, holding the deviation g_q = f_q - w_q from the
// rest state (exact weights).
//
// Up to four steps per launch (lbm_kernel<T>), in registers.  A warp owns a window of 64 columns of
// one member, two neighbouring ones per lane, and marches along y; the T steps run as a pipeline of
// T stages, stage s one row behind stage s - 1.  A collision's outputs stream to the stage after it:
// along x with one shuffle per direction and pair, along y by waiting in registers (those with
// c_y = -1 are used at once, c_y = 0 one row later, c_y = +1 two rows later).  The last stage's
// populations are streamed the same way and stored, coalesced.  A window loses one column per side
// and step, so neighbouring windows overlap by the halo, and so do the segments of rows a member
// is cut into.  Rows arrive by asynchronous copies three rows ahead in the warp's own ring in
// shared memory (nothing spills then, and a warp is never behind the memory's latency), the force
// in a longer one that every stage reads its row from.  A block is one warp, so that member,
// strip and row addresses are uniform, and there is no block barrier.  A form that kept four steps'
// rows in shared memory (36 accesses of 8 bytes per pair of nodes and step, four barriers per
// eight rows) was bound by them, at 1.26 to 1.45 ms per four steps of 1024^2, k = 64.
//
// Measured, four steps with a force: two launches of two steps through shared memory, the
// collision written as g + omega (g_eq - g) per direction -> this pipeline with the next row in
// registers -> with the ring:
//   1024^2, k = 64: 1759 -> 1031 -> 852 us (84 % of the copy rate in its own 4.8 GB);
//   256^2, k = 32: 71.1 -> 42.2 -> 39.1 us; 509 x 380, k = 20: 185 -> 74.5 -> 74.9 us;
//   64^2, k = 20: 8.6 -> 8.2 -> 7.4 us; 250 x 187, k = 40 (no force): 36.4 -> 34.8 us.
// Rings of two rows 962 us, two warps a block 865 us.  The row loop unrolled by four gains 1 to 6 %
// more from 128 x 128 on (847 us at 1024^2) but makes a 32^2 cycle, where fetching the code counts,
// 6 % slower.  Bound: memory at 1024^2; the FP32 pipe
// and the latency of three warps per scheduler (what 168 registers allow) at smaller grids.
#include <math.h>

#include "common.cuh"
#include "kernels.h"

namespace lk {
namespace {

// The collision works on two nodes at once: every quantity is a float2 (node pair) and every
// operation a packed FP32 instruction, which rounds each lane exactly as the scalar operation
// would.
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {   // a - b, one rounding
    return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a);
}
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }

// 1 / x for x near 1 (the density): the hardware approximation refined by one Newton-Raphson
// step y + y (1 - x y), which squares its relative error.
__device__ __forceinline__ float2 rcp2(float2 x) {
    float2 y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y.x) : "f"(x.x));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y.y) : "f"(x.y));
    const float2 e = fma2(neg2(x), y, dup2(1.0f));
    return fma2(y, e, y);
}

// Relaxation times beyond 2: 1 - omega is no FP32 number for omega < 1/2, and rounding it would
// change omega by up to 3e-8 absolutely (1.3e-5 of it at tau = 1000) with the same sign at every
// node and step.  The collision then keeps g apart from what it adds to it: out = g + (omega
// (g_eq - g) + 3 w c.F), nine additions more.
inline bool slow_relaxation(float tau) { return 1.0f / tau < 0.5f; }

// The collision's constants, from omega = 1 / tau in FP32 (host, FP64).  They satisfy
// rest + 9 rho = 1 and rest + 12 mom = 1 (slow relaxation: rest + 9 rho = 0 and rest + 12 mom = 0;
// rho, mom as two FP32 words each) and quad = 3 quad6 exactly, so that a collision conserves mass
// and momentum up to the rounding of its sums: a constant off by one ulp would act on every node
// and step with the same sign (an error of 6e-6 after 100 steps, measured, against 5e-7).
struct LbmCoef {
    float rest;             // 1 - omega (exact for omega >= 1/2); slow relaxation: -omega
    float rho, rho_lo;      // omega / 9
    float mom, mom_lo;      // omega / 12
    float nquad6, quad, quad8, quad4;   // -omega / 6, omega / 2, omega / 8, omega / 4
};
LbmCoef lbm_coef(float tau) {
    LbmCoef c;
    const double omega = (double)(1.0f / tau);
    c.rest = (float)(slow_relaxation(tau) ? -omega : 1.0 - omega);
    const double t = omega;
    c.rho = (float)(t / 9.0);
    c.rho_lo = (float)(t / 9.0 - (double)c.rho);
    c.mom = (float)(t / 12.0);
    c.mom_lo = (float)(t / 12.0 - (double)c.mom);
    int e = 0;
    const double m = frexp(t / 6.0, &e);     // 22 significant bits: 3 quad6 is an FP32 number
    const double q6 = ldexp(rint(ldexp(m, 22)), e - 22);
    c.nquad6 = (float)-q6;
    c.quad = (float)(3.0 * q6);
    c.quad8 = 0.25f * c.quad;
    c.quad4 = 0.5f * c.quad;
    return c;
}

// BGK collision with the body-force source for two nodes: post-collision populations out[q]
// from the nodes' deviations g[q] (Eq. 1, Sec. II-A).
//
// out = (1 - omega) g + omega g_eq + 3 w c.F, with the directions paired (q, 8 - q): the
// equilibrium's even part is w (drho + 4.5 (c.j)(c.u) - 1.5 j.u) and its odd part 3 w c.j (j = rho u),
// so no density multiplies the momentum again.  With P = j_x u_x, Q = j_y u_y, R = j_x u_y,
//   even (times omega): rest 4 b, x axis b + omega P / 2, y axis b + omega Q / 2, diagonals
//     b / 4 + omega (P + Q) / 8 +- omega R / 4, b = omega (drho / 9 - (P + Q) / 6);
//   odd: 4 m_x, 4 m_y, m_x +- m_y, m = (omega j + F) / 12.
// 61 packed operations for two nodes (the form g + omega (g_eq - g) per direction took 95).  Error
// after 100 steps against 64 bits (tau = 0.52, u = 0.02, emulated): 2.1e-6 -> 5e-7.  kSlow (the
// slow relaxation above): -omega g in place of (1 - omega) g, and g added last; error at tau = 30 /
// 100 / 1000 with 1 - omega rounded 1.5e-6 / 6.1e-7 / 7.7e-7, so 2.5e-7.
template <bool kForce, bool kSlow>
__device__ __forceinline__ void collide2(const float2 (&g)[NV], float2 fx, float2 fy,
                                         const LbmCoef &c, float2 (&out)[NV]) {
    const float2 s0 = add2(g[0], g[8]), s1 = add2(g[1], g[7]), s2 = add2(g[2], g[6]),
                 s3 = add2(g[3], g[5]);
    const float2 d0 = sub2(g[8], g[0]), d1 = sub2(g[7], g[1]), d2 = sub2(g[6], g[2]),
                 d3 = sub2(g[5], g[3]);
    const float2 drho = add2(add2(add2(s0, s2), add2(s1, s3)), g[4]);
    const float2 jx = add2(sub2(d0, d2), d3), jy = add2(add2(d0, d2), d1);
    const float2 rinv = rcp2(add2(dup2(1.0f), drho));
    const float2 ux = mul2(jx, rinv), uy = mul2(jy, rinv);
    const float2 P = mul2(jx, ux), Q = mul2(jy, uy), R = mul2(jx, uy), PQ = add2(P, Q);
    const float2 b =
        fma2(dup2(c.rho), drho, fma2(dup2(c.nquad6), PQ, mul2(dup2(c.rho_lo), drho)));
    const float2 ax = fma2(dup2(c.quad), P, b), ay = fma2(dup2(c.quad), Q, b);
    const float2 e = fma2(dup2(0.25f), b, mul2(dup2(c.quad8), PQ)), h = mul2(dup2(c.quad4), R);
    const float2 ap = add2(e, h), am = sub2(e, h);
    float2 lx = mul2(dup2(c.mom_lo), jx), ly = mul2(dup2(c.mom_lo), jy);
    if (kForce) {
        lx = fma2(dup2(1.0f / 12.0f), fx, lx);
        ly = fma2(dup2(1.0f / 12.0f), fy, ly);
    }
    const float2 mx = fma2(dup2(c.mom), jx, lx), my = fma2(dup2(c.mom), jy, ly);
    const float2 mp = add2(mx, my), mm = sub2(mx, my);
    const float2 r = dup2(c.rest);
    out[4] = fma2(dup2(4.0f), b, mul2(r, g[4]));
    out[8] = add2(fma2(r, g[8], ap), mp);
    out[0] = sub2(fma2(r, g[0], ap), mp);
    out[2] = add2(fma2(r, g[2], am), mm);
    out[6] = sub2(fma2(r, g[6], am), mm);
    out[7] = fma2(dup2(4.0f), my, fma2(r, g[7], ay));
    out[1] = fma2(dup2(-4.0f), my, fma2(r, g[1], ay));
    out[5] = fma2(dup2(4.0f), mx, fma2(r, g[5], ax));
    out[3] = fma2(dup2(-4.0f), mx, fma2(r, g[3], ax));
    if (kSlow)
#pragma unroll
        for (int q = 0; q < NV; ++q) out[q] = add2(out[q], g[q]);
}

constexpr int kWin = 64;                      // columns of a warp's window
constexpr int kLbmBlocks = 12;                // CTAs, of one warp, per SM
// rows of the staging ring (one less in flight), and of the force's, which the stages read up to
// T - 1 rows back (launches of one or two steps keep more warps per SM: with four rows a launch of
// one step takes 1075 us at 1024^2, k = 64, with two 820)
constexpr int lbm_ahead(int T) { return T > 2 ? 4 : 2; }
constexpr int lbm_force_ring(int T) { return T > 2 ? 8 : T > 1 ? 4 : 2; }
// halo columns on either side of a strip: T, rounded up to whole pairs
constexpr int lbm_halo(int T) { return (T + 1) & ~1; }
constexpr int lbm_strip(int T) { return kWin - 2 * lbm_halo(T); }

// Periodic wrap of a coordinate at most one period outside [0, n).
__device__ __forceinline__ int wrap1(int a, int n) {
    const int r = a < 0 ? a + n : (a >= n ? a - n : a);
    return (unsigned)r < (unsigned)n ? r : posmod(a, n);   // grids narrower than the halo
}

// Streamed populations whose consumers' rows are still to come: c_y = 0 of the last row, c_y = +1
// of the last and of the one before.
struct Waiting {
    float2 zero[3], up1[3], up2[3];
};

// A collision's outputs displaced by c_x: lane c holds columns 2c, 2c + 1.
__device__ __forceinline__ void stream_x(const float2 (&o)[NV], float2 (&s)[NV]) {
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        if (cx(q) == 0) s[q] = o[q];
        else if (cx(q) > 0) s[q] = make_float2(__shfl_up_sync(0xffffffffu, o[q].y, 1), o[q].x);
        else s[q] = make_float2(o[q].y, __shfl_down_sync(0xffffffffu, o[q].x, 1));
    }
}

// The populations that reach the row above the one just streamed (s), and the wait of the rest.
__device__ __forceinline__ void stream_y(const float2 (&s)[NV], Waiting &w, float2 (&g)[NV]) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        g[k] = s[k];                // c_y = -1
        g[3 + k] = w.zero[k];
        g[6 + k] = w.up2[k];
        w.up2[k] = w.up1[k];
        w.up1[k] = s[6 + k];
        w.zero[k] = s[3 + k];
    }
}

// Asynchronous copies of a lane's own 4, 8 or 16 bytes into its slot of the staging ring.
__device__ __forceinline__ void async4(void *d, const void *s) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(d)), "l"(s) : "memory");
}
__device__ __forceinline__ void async8(void *d, const void *s) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(d)), "l"(s) : "memory");
}
__device__ __forceinline__ void async16(void *d, const void *s) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(d)), "l"(s) : "memory");
}

// T steps.  Unit u: strip (fastest), segment of H rows, member.  kEven: nx is even, so a window's
// pairs are 8-byte aligned and never split by the periodic wrap.
template <int T, bool kForce, bool kEven, bool kSlow>
__global__ void __launch_bounds__(32, kLbmBlocks)
    lbm_kernel(const float *__restrict__ gin, float *__restrict__ gout,
               const float2 *__restrict__ force, int nx, int ny, int H, int strips, int segs,
               LbmCoef coef) {
    constexpr int HX = lbm_halo(T), TX = lbm_strip(T);
    constexpr int kAhead = lbm_ahead(T), kForceRing = lbm_force_ring(T);
    static_assert(kForceRing >= kAhead + T - 1, "a stage's row of the force is still there");
    const unsigned u = blockIdx.x;
    const int c = threadIdx.x;
    const int strip = (int)(u % strips), seg = (int)(u / strips % segs);
    const size_t npts = (size_t)nx * ny;
    const size_t mbase = (size_t)(u / strips / segs) * NV * npts;
    const int x0 = strip * TX, ys = seg * H, ye = min(ys + H, ny);
    const int xa = wrap1(x0 - HX + 2 * c, nx), xb = wrap1(x0 - HX + 2 * c + 1, nx);
    const float *const src = gin + mbase;
    // row l of the segment is y = ys - T + l (periodic), l < rows
    const int rows = ye - ys + 2 * T;
    int y = posmod(ys - T, ny);              // of the row to be loaded next
    // a lane reads only what it copied itself: no exchange, no barrier
    __shared__ float2 ring[kAhead][NV][32];
    __shared__ float4 fring[kForce ? kForceRing : 1][32];
    auto load = [&](int l) {                 // row l into its slot; a group even when there is none
        if (l < rows) {
            const size_t p = (size_t)y * nx;
#pragma unroll
            for (int q = 0; q < NV; ++q) {
                const float *a = src + (size_t)q * npts + p;
                float2 *d = ring[l & (kAhead - 1)][q];
                if (kEven) {
                    async8(d + c, a + xa);
                } else {
                    async4(&d[c].x, a + xa);
                    async4(&d[c].y, a + xb);
                }
            }
            if (kForce) {
                float4 *f = fring[l & (kForceRing - 1)];
                if (kEven) {                 // the pair's force: one 16-byte copy
                    async16(f + c, force + p + xa);
                } else {
                    async8(&f[c].x, force + p + xa);
                    async8(&f[c].z, force + p + xb);
                }
            }
            y = y + 1 == ny ? 0 : y + 1;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // targets: columns x0 + t, x0 + t + 1 of the strip and grid (for an even nx both or neither)
    const int t = 2 * c - HX;
    const bool in0 = t >= 0 && t < TX && x0 + t < nx, in1 = in0 && x0 + t + 1 < nx;
    float *const dst = gout + mbase + (x0 + t);

    Waiting w[T > 1 ? T - 1 : 1];
#pragma unroll
    for (int i = 0; i < (T > 1 ? T - 1 : 1); ++i)
#pragma unroll
        for (int k = 0; k < 3; ++k) w[i].zero[k] = w[i].up1[k] = w[i].up2[k] = make_float2(0.0f, 0.0f);
    if (kForce)                              // the rows before the first: any finite force
#pragma unroll
        for (int r = 0; r < kForceRing; ++r) fring[r][c] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
    for (int r = 0; r < kAhead - 1; ++r) load(r);
#pragma unroll 2
    for (int l = 0; l < rows; ++l) {
        float2 g[NV], o[NV], s[NV];
        asm volatile("cp.async.wait_group %0;" ::"n"(kAhead - 2) : "memory");
#pragma unroll
        for (int q = 0; q < NV; ++q) g[q] = ring[l & (kAhead - 1)][q][c];
        load(l + kAhead - 1);
#pragma unroll
        for (int i = 0; i < T; ++i) {        // stage i + 1, row l - i
            float2 fx = make_float2(0.0f, 0.0f), fy = fx;
            if (kForce) {
                const float4 f = fring[(l - i) & (kForceRing - 1)][c];
                fx = make_float2(f.x, f.z);
                fy = make_float2(f.y, f.w);
            }
            collide2<kForce, kSlow>(g, fx, fy, coef, o);
            stream_x(o, s);
            if (i + 1 < T) stream_y(s, w[i], g);
        }
        // the last stage's row l - T + 1, pushed along y
        const int yr = ys - T + l - (T - 1);
        if (l < 2 * T - 2 || !in0) continue;
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            if (yr + cy(q) < ys || yr + cy(q) >= ye) continue;
            float *d = dst + ((size_t)q * npts + (size_t)(yr + cy(q)) * nx);
            if (kEven) {
                __stcs(reinterpret_cast<float2 *>(d), s[q]);
            } else {
                __stcs(d, s[q].x);
                if (in1) __stcs(d + 1, s[q].y);
            }
        }
    }
}

// Rows per segment: the least estimated time.  A row of a segment (its 2 T halo rows and about two
// for the first load included) takes a scheduler with one, two or three warps 1.7, 2.4 or 3 units
// (a lone warp waits for its own chain of collisions); three warps fit.
template <int T>
int segment_rows(int nx, int ny, int nmem, int sms) {
    const long long lines = (long long)((nx + lbm_strip(T) - 1) / lbm_strip(T)) * nmem;
    constexpr int wmax = kLbmBlocks / 4;
    static_assert(wmax == 3, "the units of a row");
    const double unit[wmax] = {0.0, 1.7, 2.4};
    int best = ny;
    double least = 0.0;
    for (int n = 1; n <= ny; ++n) {          // segments
        const int H = (ny + n - 1) / n;
        const long long w = (lines * ((ny + H - 1) / H) + 4 * sms - 1) / (4 * sms);
        const double cost = ((double)(w / wmax * wmax) + unit[w % wmax]) * (H + 2 * T + 2);
        if (n == 1 || cost < least) {
            least = cost;
            best = H;
        }
        if (H < 2) break;
    }
    return best;
}

template <int T, bool kForce>
cudaError_t launch_steps(const float *gin, float *gout, const float2 *force, int nx, int ny,
                         int nmem, float tau, cudaStream_t s, int rows) {
    const int strips = (nx + lbm_strip(T) - 1) / lbm_strip(T), segs = (ny + rows - 1) / rows;
    const unsigned units = (unsigned)strips * segs * nmem;   // windows of 56 columns and more
    const LbmCoef coef = lbm_coef(tau);
    const bool slow = slow_relaxation(tau);
    auto *const f = nx % 2 == 0
        ? (slow ? lbm_kernel<T, kForce, true, true> : lbm_kernel<T, kForce, true, false>)
        : (slow ? lbm_kernel<T, kForce, false, true> : lbm_kernel<T, kForce, false, false>);
    f<<<units, 32, 0, s>>>(gin, gout, force, nx, ny, rows, strips, segs, coef);
    return cudaGetLastError();
}

// f -> g = (f - fl(w_q)) - dw_q and g -> f = fl(w_q) + (g + dw_q).
template <bool kToG>
__global__ void shift_kernel(const float *__restrict__ in, float *__restrict__ out, size_t npts) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= npts) return;
    const int q = blockIdx.y % NV;
    const size_t off = (size_t)blockIdx.y * npts + i;
    const int cls = q == 4 ? 4 : ((q & 1) ? 1 : 0);
    const float w = wq(cls), dw = dwq(cls);
    out[off] = kToG ? __fsub_rn(__fsub_rn(in[off], w), dw) : __fadd_rn(w, __fadd_rn(in[off], dw));
}

// g_q = f^eq_q(rho, u) - w_q = w_q ((rho - 1) + rho (3 c.u + 9/2 (c.u)^2 - 3/2 u.u)).
__global__ void macro_kernel(const float *__restrict__ rho, const float *__restrict__ ux,
                             const float *__restrict__ uy, float *__restrict__ g, size_t npts) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= npts) return;
    const size_t m = blockIdx.y;
    const float r = rho[m * npts + i], u = ux[m * npts + i], v = uy[m * npts + i];
    const float dr = r - 1.0f;
    const float usq = 1.5f * (u * u + v * v);
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        const float cu = (float)cx(q) * u + (float)cy(q) * v;
        g[(m * NV + q) * npts + i] = wq(q) * (dr + r * (3.0f * cu + 4.5f * cu * cu - usq));
    }
}

}  // namespace

void lbm_plan(int nx, int ny, int nmem, int sms, int rows[kLbmSteps]) {
    rows[0] = segment_rows<1>(nx, ny, nmem, sms);
    rows[1] = segment_rows<2>(nx, ny, nmem, sms);
    rows[2] = segment_rows<3>(nx, ny, nmem, sms);
    rows[3] = segment_rows<4>(nx, ny, nmem, sms);
}

cudaError_t launch_lbm(const float *gin, float *gout, const float2 *force, int nx, int ny, int nmem,
                       float tau, int steps, const int rows[kLbmSteps], cudaStream_t s) {
    if (nmem <= 0) return cudaSuccess;
#define LK_STEPS(T)                                                                             \
    case T:                                                                                     \
        return force ? launch_steps<T, true>(gin, gout, force, nx, ny, nmem, tau, s, rows[T - 1]) \
                     : launch_steps<T, false>(gin, gout, force, nx, ny, nmem, tau, s, rows[T - 1]);
    switch (steps) {
        LK_STEPS(1)
        LK_STEPS(2)
        LK_STEPS(3)
        LK_STEPS(4)
        default: return cudaErrorInvalidValue;
    }
#undef LK_STEPS
}

cudaError_t launch_f_to_g(const float *f, float *g, int nmem, size_t npts, cudaStream_t s) {
    if (nmem <= 0 || npts == 0) return cudaSuccess;
    dim3 grid((unsigned)((npts + 255) / 256), nmem * NV);
    shift_kernel<true><<<grid, 256, 0, s>>>(f, g, npts);
    return cudaGetLastError();
}

cudaError_t launch_g_to_f(const float *g, float *f, int nmem, size_t npts, cudaStream_t s) {
    if (nmem <= 0 || npts == 0) return cudaSuccess;
    dim3 grid((unsigned)((npts + 255) / 256), nmem * NV);
    shift_kernel<false><<<grid, 256, 0, s>>>(g, f, npts);
    return cudaGetLastError();
}

cudaError_t launch_macro_to_g(const float *rho, const float *ux, const float *uy, float *g,
                              int nmem, size_t npts, cudaStream_t s) {
    if (nmem <= 0 || npts == 0) return cudaSuccess;
    dim3 grid((unsigned)((npts + 255) / 256), nmem);
    macro_kernel<<<grid, 256, 0, s>>>(rho, ux, uy, g, npts);
    return cudaGetLastError();
}

}  // namespace lk
