// Dust temperature from the irradiation (Sect. 2.2, Eq. 16, in the frequency-
// dependent form of Sect. 2.3): with the stellar fluxes of every bin,
//     a T^4 = E_R + sum_i kappa_i |F_i| / (c kappa_P(T)),
// and over a cell sum_i kappa_i F_i = q_abs / rho = c a_rad, so
//     a T^4 = E_R + a_rad / kappa_P(T)
// per cell, from the tracer's radial acceleration (finite also where rho = 0).
// kappa_P(T) = sum_i kappa_i B_i(T) / sum_i B_i(T) is the Planck mean of the bin
// table, B_i(T) the Planck integral over bin i (the bins of Eq. 20 at T).
//
// The mean is tabulated once per table on 1024 points of ln T in [0, ln 1e5]
// (FP64 quadrature, stored as ln kappa_P) and read with cubic Hermite interpolation
// (Catmull-Rom tangents); outside the range it is held constant. Each cell solves
// 4 y + ln a = ln(E_R + a_rad e^{-L(y)}), y = ln T, L = ln kappa_P, in FP32: with a
// diffuse field by a Halley and a Newton step from a close start
// (diffuse_temperature), and by Newton's method from 300 K's opacity where those do
// not reach (the derivative 4 + w L'(y), 0 <= w <= 1, is positive wherever
// the mean grows slower than T^4). Where E_R = 0 the equation is
// 4 y + L(y) = ln a_rad - ln a: a cell reads T itself from the tabulated inverse of the
// left side (built once per table, each interval checked against the FP64 root) and
// takes Newton steps only in the intervals where that check failed.
#include <math.h>

#include <algorithm>
#include <string>
#include <vector>

#include "rt_internal.cuh"
#include "rt_planck.cuh"

namespace rt {

constexpr int kTempNodes = 1024;
// The inverse table of T (E_R = 0) sits on the grid v = lg2 a_rad with spacing 2^-e:
// node i at v = (v_org + i) 2^-e, v_org an integer, at most kTempInvNodes nodes.
constexpr int kTempInvNodes = 2048;
// the context's table buffer: lkp [kTempNodes]; 8 constants (X(y_lo), X(y_hi), 2^e,
// v_org, the node count of the inverse table, 1 / the step diffuse_temperature accepts); then (16-byte aligned) the cubic
// coefficients of lkp [kTempNodes - 1], of the inverse table [kTempInvNodes - 1] and of lkp in
// lg2 units [kTempNodes + 1], float4 each, and the inverse table's nodes while it is built
constexpr int kTempConsts = kTempNodes;
constexpr int kTempCoefLkp = kTempConsts + 8;
constexpr int kTempCoefInv = kTempCoefLkp + 4 * (kTempNodes - 1);
constexpr int kTempCoefLg2 = kTempCoefInv + 4 * (kTempInvNodes - 1);
constexpr float kTempLg2Top = kTempNodes + 0.999f;  // just inside the last entry of the lg2 table
constexpr int kTempInvYm = kTempCoefLg2 + 4 * (kTempNodes + 1);  // (y, dT/dt) of the inverse table's nodes, double2
constexpr int kTempTableFloats = kTempInvYm + 4 * kTempInvNodes;
constexpr double kTempLnLo = 0.0;                    // ln 1 K
constexpr double kTempLnHi = 11.512925464970229;     // ln 1e5 K

namespace {

// Planck mean of the table at temperature exp(y[n]); one warp per node, the bins'
// band integrals in FP64. kp_out[n] = kappa_P (double) and lkp[n] = ln kappa_P.
// Eight lanes per bin: 1024 nodes, 79 bins 2.3 -> 0.68 ms (the bands were one panel wide, one lane each).
__global__ void k_planck_mean(int n_nodes, const double *t_nodes, int n_nu, const double *nu_mid,
                              const double *kappa, int n_t, const double *t_grid, double *kp_out, float *lkp)
{
    const int lane = threadIdx.x & 31;
    const int node = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (node >= n_nodes) return;
    const double t = t_nodes[node];
    const double kt_h = kKB * t / kH;
    double num = 0.0, den = 0.0;
    for (int i0 = 0; i0 < n_nu; i0 += 4) {  // four bins at a time, 8 lanes each
        const int i = i0 + (lane >> 3);
        const bool on = i < n_nu;
        const double lo = (i == 0 || !on) ? 0.0 : 0.5 * (nu_mid[i - 1] + nu_mid[i]);
        const double hi = !on ? 0.0 : (i == n_nu - 1) ? INFINITY : 0.5 * (nu_mid[i] + nu_mid[i + 1]);
        const double b = planck_band_8(lo / kt_h, hi / kt_h, lane & 7);
        if (!on) continue;  // (the last round only)
        num += kappa_at(kappa + (size_t)i * n_t, n_t, t_grid, t) * b;
        den += b;
    }
    for (int o = 8; o < 32; o <<= 1) {
        den += __shfl_xor_sync(0xffffffffu, den, o);
        num += __shfl_xor_sync(0xffffffffu, num, o);
    }
    if (lane == 0) {
        const double kp = den > 0.0 ? num / den : 0.0;
        if (kp_out) kp_out[node] = kp;
        if (lkp) lkp[node] = (float)log(kp > 1e-300 ? kp : 1e-300);
    }
}

// ln kappa_P by the interpolation the cells use (cubic Hermite with Catmull-Rom
// tangents on the node table s, constant outside it), and its derivative, in FP64
__device__ double interp_d(const float *s, double y, double y0, double inv_dy, double *deriv = nullptr)
{
    double u = (y - y0) * inv_dy;
    if (!(u > 0.0) || u >= (double)(kTempNodes - 1)) {
        if (deriv) *deriv = 0.0;
        return !(u > 0.0) ? s[0] : s[kTempNodes - 1];
    }
    const int k = min((int)u, kTempNodes - 2);
    const double t = u - (double)k;
    const double p0 = s[k], p1 = s[k + 1];
    const double m0 = 0.5 * (p1 - s[k > 0 ? k - 1 : 0]) * (k > 0 ? 1.0 : 2.0);
    const double m1 = 0.5 * (s[k + 2 < kTempNodes ? k + 2 : kTempNodes - 1] - p0) * (k + 2 < kTempNodes ? 1.0 : 2.0);
    const double t2 = t * t, t3 = t2 * t;
    if (deriv)
        *deriv = ((6.0 * t2 - 6.0 * t) * p0 + (3.0 * t2 - 4.0 * t + 1.0) * m0 + (-6.0 * t2 + 6.0 * t) * p1 +
                  (3.0 * t2 - 2.0 * t) * m1) * inv_dy;
    return (2.0 * t3 - 3.0 * t2 + 1.0) * p0 + (t3 - 2.0 * t2 + t) * m0 + (-2.0 * t3 + 3.0 * t2) * p1 + (t3 - t2) * m1;
}

// the root y of 4 y + L(y) = x (bisection in [y0, y1], FP64); outside the table L is
// constant and the root is (x - L_end) / 4
__device__ double inverse_root(const float *s, double x, double y0, double y1, double inv_dy)
{
    const double x_lo = 4.0 * y0 + s[0], x_hi = 4.0 * y1 + s[kTempNodes - 1];
    if (x <= x_lo) return 0.25 * (x - s[0]);
    if (x >= x_hi) return 0.25 * (x - s[kTempNodes - 1]);
    double lo = y0, hi = y1;
    for (int it = 0; it < 64; ++it) {
        const double mid = 0.5 * (lo + hi);
        if (4.0 * mid + interp_d(s, mid, y0, inv_dy) < x) lo = mid;
        else hi = mid;
    }
    return 0.5 * (lo + hi);
}

// The inverse of X(y) = 4 y + L(y) (y = ln T): with E_R = 0, Eq. 16 reads
// X(y) = ln a_rad - ln a. The nodes are uniform in v = lg2 a_rad (spacing 2^-e, node i
// at v = (v_org + i) 2^-e, X = v ln 2 - ln a), so a cell finds its interval and its
// offset t in it from lg2 a_rad with exact arithmetic. Per interval the cubic Hermite
// of T = e^y in t in [0, 1] with the exact slopes dT/dX = T / (4 + L'(y)), as
// coefficients (c0, c1, c2, c3) like k_hermite_coeffs. Each interval is checked at 8
// points against the FP64 root, evaluated the way a cell does (FP32 FMAs); where the
// cubic is off by more than 4e-7 of T the lowest bit of c3 is set, and the cells
// there polish ln T with Newton steps. Two launches, one thread per node and 8 lanes per interval,
// over the chip: the FP64 pipe does two operations per SM and clock, and the 64-step bisections of
// one CTA took 8 ms (now 0.09 ms each).
__device__ __forceinline__ double inverse_node_x(double i, int v_org, int e, double ln_a)
{
    return (v_org + i) * ldexp(1.0, -e) * kLn2 - ln_a;
}

// the nodes: ym[i] = (y, dT/dt)
__global__ void __launch_bounds__(128) k_inverse_nodes(const float *lkp, float *consts, double2 *ym, double y0,
                                                       double y1, double ln_a, int e, int v_org, int n_inv,
                                                       float per_step)
{
    const double inv_dy = (kTempNodes - 1) / (y1 - y0);
    const double hx = ldexp(1.0, -e) * kLn2;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n_inv) {
        const double y = inverse_root(lkp, inverse_node_x(i, v_org, e, ln_a), y0, y1, inv_dy);
        double dl = 0.0;
        interp_d(lkp, y, y0, inv_dy, &dl);
        ym[i] = make_double2(y, hx * exp(y) / fmax(4.0 + dl, 0.5));
    }
    if (i == 0) {
        consts[0] = (float)(4.0 * y0 + lkp[0]);
        consts[1] = (float)(4.0 * y1 + lkp[kTempNodes - 1]);
        consts[2] = (float)ldexp(1.0, e);
        consts[3] = (float)v_org;
        consts[4] = (float)n_inv;
        consts[5] = per_step;
    }
}

// the intervals: coefficients, and the check at 8 points, one lane each
__global__ void __launch_bounds__(128) k_inverse_coeffs(const float *lkp, const double2 *ym, float4 *c, double y0,
                                                        double y1, double ln_a, int e, int v_org, int n_inv)
{
    const int k = (blockIdx.x * blockDim.x + threadIdx.x) >> 3, j = threadIdx.x & 7;
    const bool on = k < n_inv - 1;
    const double inv_dy = (kTempNodes - 1) / (y1 - y0);
    float c0 = 0.0f, c1 = 0.0f, c2 = 0.0f, c3 = 0.0f;
    bool bad = false;
    if (on) {
        const double2 a = ym[k], b = ym[k + 1];
        const double p0 = exp(a.x), p1 = exp(b.x), m0 = a.y, m1 = b.y;
        c0 = (float)p0;
        c1 = (float)m0;
        c2 = (float)(3.0 * (p1 - p0) - 2.0 * m0 - m1);
        c3 = __uint_as_float(__float_as_uint((float)(2.0 * (p0 - p1) + m0 + m1)) & ~1u);
        const float t = (j + 0.5f) * 0.125f;
        const float tc = fmaf(fmaf(fmaf(c3, t, c2), t, c1), t, c0);
        const double te = exp(inverse_root(lkp, inverse_node_x(k + (double)t, v_org, e, ln_a), y0, y1, inv_dy));
        bad = !(fabs((double)tc / te - 1.0) <= 4e-7);
    }
    const unsigned any = (__ballot_sync(0xffffffffu, bad) >> (threadIdx.x & 24)) & 255u;
    if (on && j == 0) c[k] = make_float4(c0, c1, c2, __uint_as_float(__float_as_uint(c3) | (any ? 1u : 0u)));
}

// Per-interval cubic coefficients of a node table (the cubic Hermite interpolation of
// interp_d, with the same tangents): on interval k, t in [0, 1],
//   f = c0 + t (c1 + t (c2 + t c3)),  c0 = p0, c1 = m0, c2 = 3 (p1 - p0) - 2 m0 - m1,
//   c3 = 2 (p0 - p1) + m0 + m1,
// so a cell evaluates one interval with one 16-byte load and three FMAs.
// c2: the same of lg2 kappa_P, interval k at entry k + 1, the end values held in the first entry
// and the last.
__global__ void k_hermite_coeffs(const float *s, float4 *c, float4 *c2)
{
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < kTempNodes - 1; k += gridDim.x * blockDim.x) {
        const double p0 = s[k], p1 = s[k + 1];
        const double m0 = 0.5 * (p1 - s[k > 0 ? k - 1 : 0]) * (k > 0 ? 1.0 : 2.0);
        const double m1 = 0.5 * (s[k + 2 < kTempNodes ? k + 2 : kTempNodes - 1] - p0) * (k + 2 < kTempNodes ? 1.0 : 2.0);
        const double q2 = 3.0 * (p1 - p0) - 2.0 * m0 - m1, q3 = 2.0 * (p0 - p1) + m0 + m1;
        c[k] = make_float4((float)p0, (float)m0, (float)q2, (float)q3);
        c2[k + 1] = make_float4((float)(p0 * kLog2e), (float)(m0 * kLog2e), (float)(q2 * kLog2e), (float)(q3 * kLog2e));
    }
    if (blockIdx.x == 0 && threadIdx.x < 2) {
        const double v = s[threadIdx.x ? kTempNodes - 1 : 0];
        c2[threadIdx.x ? kTempNodes : 0] = make_float4((float)(v * kLog2e), 0.0f, 0.0f, 0.0f);
    }
}

struct TempArgs {
    const float *a_rad;
    const float *e_rad;   // may be null (E_R = 0)
    float *t_out;
    const float *lkp;     // [kTempNodes] ln kappa_P on the uniform ln T grid
    const float *consts;  // X(y_lo), X(y_hi), 2^e, v_org, node count of the inverse table, per_step
    const float4 *c_lkp;  // [kTempNodes - 1] cubic coefficients of lkp per interval
    const float4 *c_inv;  // [n_inv - 1] cubic coefficients of T on the v = lg2 a_rad grid
    int vec;              // a_rad, e_rad (if any) and t_out are 16-byte aligned
    long long n;
    float y0, inv_dy;     // grid origin and 1 / spacing
    float ln_a;           // ln of the radiation constant a = 4 sigma / c
    float a, inv_a;       // a and 1 / a
    const float4 *c_lg2;  // [kTempNodes + 1] the coefficients of lkp in lg2 units, with a constant
                          // interval below and one above
    float s_hi, s_lo;     // nodes per unit of lg2 T, as a sum of two floats
    float l_scale, l_org; // lg2 T to [0, 1] over the entries of c_lg2
    float dl_dy;          // d ln kappa_P / dy per (lg2 units per node)
};

// ln kappa_P(e^y) and its derivative from the per-interval coefficients; lo, hi: the
// node values held outside the table.
__device__ __forceinline__ void interp_c(const float4 *c, float lo, float hi, float y, float y0, float inv_dy,
                                         float &L, float &dL)
{
    const float u = (y - y0) * inv_dy;
    if (!(u > 0.0f)) {  // below the table (or NaN): constant
        L = lo;
        dL = 0.0f;
        return;
    }
    if (u >= (float)(kTempNodes - 1)) {
        L = hi;
        dL = 0.0f;
        return;
    }
    const int k = min((int)u, kTempNodes - 2);
    const float t = u - (float)k;
    const float4 q = __ldg(c + k);
    L = fmaf(fmaf(fmaf(q.w, t, q.z), t, q.y), t, q.x);
    dL = fmaf(fmaf(3.0f * q.w, t, 2.0f * q.z), t, q.y) * inv_dy;
}

// e^y for |y| up to ~88 from the hardware 2^x: y log2(e) is formed as hi + lo with an
// FMA (Dekker's product, log2(e) split into two floats), so the rounding of the
// product does not grow with |y|; e^y = 2^hi (1 + lo ln 2) to about 2^-22.
__device__ __forceinline__ float exp_ex2(float y)
{
    constexpr float kL2eHi = 1.44269502162933349609375f;  // log2(e) rounded to float
    constexpr float kL2eLo = 1.92596298909109e-8f;        // log2(e) - kL2eHi
    const float hi = y * kL2eHi;
    const float lo = fmaf(y, kL2eHi, -hi) + y * kL2eLo;
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(hi));
    return fmaf(r, lo * 0.69314718055994530942f, r);
}

// the hardware log2 (absolute error ~2^-22)
__device__ __forceinline__ float lg2_approx(float x)
{
    float r;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// ln x for x > 0 from the hardware log2
__device__ __forceinline__ float log_lg2(float x) { return lg2_approx(x) * 0.69314718055994530942f; }

// The table ends and the inverse table's grid, read once per thread.
struct TempConsts {
    float l_lo, l_hi, v_scale, v_org, u_max;
    int k_max;
    float sat_scale, sat_org, u_top;  // lg2 a_rad to [0, 1] over the inverse table, and its last interval
    float per_step;                   // 1 / the last step of ln T that diffuse_temperature accepts
};

// rcp.approx (relative error below 2^-22)
__device__ __forceinline__ float rcp_fast(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ float2 splat(float v) { return make_float2(v, v); }

// T with a diffuse field (Eq. 16, E_R given) of N cells in l = lg2 T, N even; err[c] is below 1
// where t_out[c] holds.
// Start: a T^4 = E_R + a T_a^4 with T_a the E_R = 0 root from the inverse table, within a few per
// cent above the root (kappa_P grows with T, so the source at T is below its value at T_a). Then a
// Halley step on F(y) = 4 y + ln a - ln(E_R + a_rad / kappa_P), y = ln T, with F'' from L' alone
// (the error it leaves is cubic but for L''), and a Newton step. F is the log of a ratio near 1,
// so there is no cancellation, and the last step is applied to T itself: the rounding of ln T
// (5e-7) does not reach the result. A last step above what the table's curvature allows
// (accepted_step) is followed by further Newton steps of the thread's cells (diffuse_more: most
// cells of a table whose mean has kinks need one); where a value is beyond the tables or the
// hardware functions' range, or the steps do not settle, the cell takes the general solve.
// What bounds it: issue slots. So the intervals come from a saturating multiply and an FMA
// that rounds down to an integer (no conversions, no clamps; the lg2 kappa_P table has a constant
// interval at either end in place of range tests), and the arithmetic runs on pairs of cells.
// 8.4 M cells with E_R: 131 us for Newton steps from 300 K with accurate exp and log, 58 us for
// these steps cell by cell, 49 us four cells at once (175 instructions per cell), 41 us (116);
// further steps cost less than the general solve they spare (524 k cells, kappa(nu, T) linear
// between 24 temperatures: 19 us with the cells beyond 5e-4 sent there, 14 us now).
constexpr float kMagic = 12582912.0f;  // 1.5 2^23: adding it, rounding down, gives the floor
constexpr int kMagicBits = 0x4b400000;

template <bool HALLEY, int N>
__device__ __forceinline__ void diffuse_step(const TempArgs &p, const TempConsts &k, const float (&ar)[N],
                                             const float (&er)[N], float (&l)[N], float (&t_out)[N], float (&err)[N])
{
#pragma unroll
    for (int c = 0; c < N; c += 2) {
        // lg2 kappa_P and d ln kappa_P / dy: the interval, and the offset in it by FMA
        float L[2], dL[2], T[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const float x = l[c + i];
            const float m = __fmaf_rd(__saturatef(fmaf(x, p.l_scale, p.l_org)), kTempLg2Top, kMagic);
            // (node n of the table is entry n + 1)
            const float t = fmaf(x, p.s_lo, fmaf(x, p.s_hi, -(m - (kMagic + 1.0f))));
            const float4 q = __ldg(p.c_lg2 + (__float_as_int(m) - kMagicBits));
            L[i] = fmaf(fmaf(fmaf(q.w, t, q.z), t, q.y), t, q.x);
            dL[i] = fmaf(fmaf(3.0f * q.w, t, 2.0f * q.z), t, q.y);
            asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(T[i]) : "f"(x));
            asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(L[i]) : "f"(-L[i]));  // 1 / kappa_P
        }
        const float2 T2 = make_float2(T[0], T[1]), e2 = make_float2(er[c], er[c + 1]);
        const float2 d2 = __fmul2_rn(make_float2(dL[0], dL[1]), splat(p.dl_dy));
        const float2 src = __fmul2_rn(make_float2(ar[c], ar[c + 1]), make_float2(L[0], L[1]));
        const float2 rhs = __fadd2_rn(e2, src);
        const float2 tt = __fmul2_rn(T2, T2), t4 = __fmul2_rn(__fmul2_rn(splat(p.a), tt), tt);
        const float2 den = __ffma2_rn(src, d2, __fmul2_rn(rhs, splat(4.0f)));
        const float2 rt = make_float2(rcp_fast(t4.x), rcp_fast(t4.y));
        const float2 rd = make_float2(rcp_fast(den.x), rcp_fast(den.y));
        const float2 x = __ffma2_rn(rhs, rt, splat(-1.0f));  // rhs / (a T^4) - 1
        // ln(1 + x): to 1e-4 at x = 0.3 (the first step), to rounding where the last step is
        float2 f = splat(1.0f / 3.0f);
        if (HALLEY) f = __ffma2_rn(x, __ffma2_rn(x, splat(0.2f), splat(-0.25f)), f);
        f = __fmul2_rn(x, __ffma2_rn(x, __ffma2_rn(x, f, splat(-0.5f)), splat(1.0f)));
        float2 dy = __fmul2_rn(f, __fmul2_rn(rhs, rd));
        if (HALLEY) {
            // dy (1 + F F'' / (2 F'^2))
            const float2 sd = __fmul2_rn(__fmul2_rn(src, rd), d2);
            const float2 ed = __fmul2_rn(__fmul2_rn(e2, rd), d2);
            dy = __ffma2_rn(dy, __fmul2_rn(__fmul2_rn(f, splat(0.5f)), __fmul2_rn(sd, ed)), dy);
            l[c] = fmaf(dy.x, 1.44269504088896340736f, l[c]);
            l[c + 1] = fmaf(dy.y, 1.44269504088896340736f, l[c + 1]);
        } else {
            const float2 g = __ffma2_rn(__fmul2_rn(dy, splat(0.5f)), dy, dy);
            const float2 r = __ffma2_rn(T2, g, T2);
            t_out[c] = r.x;
            t_out[c + 1] = r.y;
            // (a NaN step gives err = NaN, which is not below 1)
            err[c] = fabsf(dy.x) * k.per_step;
            err[c + 1] = fabsf(dy.y) * k.per_step;
        }
    }
}

template <int N>
__device__ __forceinline__ void diffuse_temperature(const TempArgs &p, const TempConsts &k, const float (&ar)[N],
                                                    const float (&er)[N], float (&t_out)[N], float (&err)[N])
{
    float l[N];
#pragma unroll
    for (int c = 0; c < N; ++c) {
        const float lg = lg2_approx(ar[c]);
        // the interval: floor(u), u cut to [0, u_max)
        const float m = __fmaf_rd(__saturatef(fmaf(lg, k.sat_scale, -k.sat_org)), k.u_top, kMagic);
        const float t = fmaf(lg, k.v_scale, -(k.v_org + (m - kMagic)));
        const float4 q = __ldg(p.c_inv + (__float_as_int(m) - kMagicBits));
        const float tc = fmaf(fmaf(fmaf(q.w, t, q.z), t, q.y), t, q.x), t2 = tc * tc;
        // beyond the inverse table t leaves [0, 1]; a_rad = 0 (t = -Inf) has no source
        const bool in = fabsf(t - 0.5f) < 0.501f;
        const float l0 = 0.25f * lg2_approx(fmaf(er[c], p.inv_a, in ? t2 * t2 : 0.0f));
        // T in 1e-3 .. 6e7 K (a NaN start gives a NaN step)
        l[c] = (in || ar[c] == 0.0f) && fabsf(l0 - 8.0f) < 18.0f ? l0 : NAN;
    }
    diffuse_step<true, N>(p, k, ar, er, l, t_out, err);
    diffuse_step<false, N>(p, k, ar, er, l, t_out, err);
}

// Further Newton steps from t_out while a cell is short of its step but near (0.1 in ln T; three
// steps at most: quadratic from there), then the general solve of the rest.
__device__ float cell_temperature_general(const TempArgs &p, const TempConsts &k, float ar, float er);

template <int N>
__device__ __forceinline__ void diffuse_more(const TempArgs &p, const TempConsts &k, const float (&ar)[N],
                                             const float (&er)[N], float (&t_out)[N], float (&err)[N])
{
#pragma unroll 1
    for (int it = 0; it < 3; ++it) {
        bool more = false;
        float l[N];
#pragma unroll
        for (int c = 0; c < N; ++c) {
            more |= err[c] >= 1.0f && err[c] < 0.1f * k.per_step;
            l[c] = lg2_approx(t_out[c]);
        }
        if (!more) break;
        diffuse_step<false, N>(p, k, ar, er, l, t_out, err);
    }
#pragma unroll
    for (int c = 0; c < N; ++c)
        if (!(err[c] < 1.0f)) t_out[c] = cell_temperature_general(p, k, ar[c], er[c]);
}

// T of one cell (Eq. 16): a T^4 = E_R + a_rad / kappa_P(T); 0 where both sources vanish.
// ER: an E_R field is given (without one, E_R = 0 and every cell takes the table)
template <bool ER>
__device__ __forceinline__ float cell_temperature_body(const TempArgs &p, const TempConsts &k, float ar, float er)
{
    ar = fmaxf(ar, 0.0f);
    if constexpr (ER) er = fmaxf(er, 0.0f);
    if (!(ar > 0.0f) && (!ER || !(er > 0.0f))) return 0.0f;
    float L, dL, y;
    if (!ER || !(er > 0.0f)) {
        // X(y) = 4 y + L(y) = ln a_rad - ln a: T from the inverse table at v = lg2 a_rad.
        // The interval index from u = v 2^e - v_org, the offset in it from one FMA with
        // the exact integer v_org + k (so t keeps the full precision of v).
        const float lg = lg2_approx(ar);
        const float u = fmaf(lg, k.v_scale, -k.v_org);
        if (u > 0.0f && u < k.u_max) {
            const int kk = min((int)u, k.k_max);
            const float t = fmaf(lg, k.v_scale, -(k.v_org + (float)kk));
            const float4 q = __ldg(p.c_inv + kk);
            const float tc = fmaf(fmaf(fmaf(q.w, t, q.z), t, q.y), t, q.x);
            if (!(__float_as_uint(q.w) & 1u)) return tc;
            // an interval whose cubic failed its check: Newton steps on ln T from it,
            // until one is below 2e-6 (quadratic convergence: the root to FP32)
            const float x = fmaf(lg, 0.69314718055994530942f, -p.ln_a);
            y = log_lg2(tc);
            for (int it = 0; it < 24; ++it) {
                interp_c(p.c_lkp, k.l_lo, k.l_hi, y, p.y0, p.inv_dy, L, dL);
                float dy = -__fdividef(4.0f * y + L - x, fmaxf(4.0f + dL, 0.5f));  // the step, not the root
                dy = fminf(fmaxf(dy, -2.0f), 2.0f);
                y += dy;
                if (fabsf(dy) < 2e-6f) break;
            }
            return exp_ex2(y);
        }
        // beyond the table kappa_P is held constant: the root in closed form
        const float x = fmaf(lg, 0.69314718055994530942f, -p.ln_a);
        return exp_ex2(0.25f * (x - (u > 0.0f ? k.l_hi : k.l_lo)));
    }
    // the general solve (what diffuse_temperature leaves):
    // Newton on F(y) = 4 y + ln a - ln(E_R + a_rad e^{-L}) from 300 K's opacity; it
    // converges quadratically: once a step is below 1e-5 the next one reaches the FP32
    // resolution of ln T, so one more step ends the solve. F grows with y, so each
    // evaluation bounds the root from one side, and a step out of the bounds (a steep mean
    // sends Newton back and forth) halves them instead.
    interp_c(p.c_lkp, k.l_lo, k.l_hi, 5.7037825f, p.y0, p.inv_dy, L, dL);
    y = 0.25f * (logf(er + ar * expf(-L)) - p.ln_a);
    float y_lo = -100.0f, y_hi = 100.0f;  // (T of any float sources lies within e^(-20 .. 60))
    bool close = false;
    for (int it = 0; it < 48; ++it) {
        interp_c(p.c_lkp, k.l_lo, k.l_hi, y, p.y0, p.inv_dy, L, dL);
        const float src = ar * expf(-L);
        const float rhs = er + src;
        const float f = 4.0f * y + p.ln_a - logf(rhs);
        const float fp = 4.0f + dL * __fdividef(src, rhs);
        float dy = -__fdividef(f, fmaxf(fp, 0.5f));
        dy = fminf(fmaxf(dy, -2.0f), 2.0f);
        if (f < 0.0f) y_lo = y;
        if (f > 0.0f) y_hi = y;
        if (!close && fabsf(dy) >= 1e-5f && (y + dy <= y_lo || y + dy >= y_hi)) dy = 0.5f * (y_lo + y_hi) - y;
        y += dy;
        if (close) break;
        close = fabsf(dy) < 1e-5f;
    }
    return expf(y);
}

template <bool ER>
__device__ __forceinline__ float cell_temperature(const TempArgs &p, const TempConsts &k, float ar, float er)
{
    return cell_temperature_body<ER>(p, k, ar, er);
}
__device__ __noinline__ float cell_temperature_general(const TempArgs &p, const TempConsts &k, float ar, float er)
{
    return cell_temperature_body<true>(p, k, ar, er);
}

// Four cells per thread and iteration, moved as 16-byte vectors where the fields allow
// (p.vec): one load in flight per thread would leave HBM latency-bound. ER: p.e_rad is
// given (a separate instance, so the common E_R = 0 call carries none of its tests).
template <bool ER>
__global__ void __launch_bounds__(256) k_dust_temperature(const TempArgs p)
{
    TempConsts k;
    k.l_lo = __ldg(p.lkp);
    k.l_hi = __ldg(p.lkp + kTempNodes - 1);
    k.v_scale = __ldg(p.consts + 2);
    k.v_org = __ldg(p.consts + 3);
    k.k_max = (int)__ldg(p.consts + 4) - 2;
    k.u_max = (float)(k.k_max + 1);
    k.sat_scale = k.v_scale / k.u_max;
    k.sat_org = k.v_org / k.u_max;
    k.u_top = k.u_max - 0.001f;
    k.per_step = ER ? __ldg(p.consts + 5) : 0.0f;
    const long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long n4 = p.vec ? p.n / 4 : 0;
    // D quads in flight per thread: slot d holds the inputs of quad v + d stride, and is
    // refilled with quad v + (d + D) stride before quad v + d stride is solved (one with
    // an E_R field: the steps of its four cells need the registers)
    constexpr int D = ER ? 1 : 2;
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 an[D], en[D];
#pragma unroll
    for (int d = 0; d < D; ++d) {
        const long long v = tid + d * stride;
        an[d] = v < n4 ? __ldg(reinterpret_cast<const float4 *>(p.a_rad) + v) : zero4;
        en[d] = (ER && v < n4) ? __ldg(reinterpret_cast<const float4 *>(p.e_rad) + v) : zero4;
    }
    for (long long v0 = tid; v0 < n4; v0 += D * stride) {
#pragma unroll
        for (int d = 0; d < D; ++d) {
            const long long v = v0 + d * stride;
            if (v >= n4) break;
            const float4 a4 = an[d], e4 = en[d];
            const long long vn = v + D * stride;
            if (vn < n4) {
                an[d] = __ldg(reinterpret_cast<const float4 *>(p.a_rad) + vn);
                if constexpr (ER) en[d] = __ldg(reinterpret_cast<const float4 *>(p.e_rad) + vn);
            }
            float4 t4;
            if constexpr (ER) {
                const float ar[4] = {fmaxf(a4.x, 0.0f), fmaxf(a4.y, 0.0f), fmaxf(a4.z, 0.0f), fmaxf(a4.w, 0.0f)};
                const float er[4] = {fmaxf(e4.x, 0.0f), fmaxf(e4.y, 0.0f), fmaxf(e4.z, 0.0f), fmaxf(e4.w, 0.0f)};
                float t[4], err[4];
                diffuse_temperature<4>(p, k, ar, er, t, err);
                if (!(err[0] < 1.0f && err[1] < 1.0f && err[2] < 1.0f && err[3] < 1.0f))
                    diffuse_more<4>(p, k, ar, er, t, err);
                t4 = make_float4(t[0], t[1], t[2], t[3]);
            } else {
                t4.x = cell_temperature<ER>(p, k, a4.x, e4.x);
                t4.y = cell_temperature<ER>(p, k, a4.y, e4.y);
                t4.z = cell_temperature<ER>(p, k, a4.z, e4.z);
                t4.w = cell_temperature<ER>(p, k, a4.w, e4.w);
            }
            reinterpret_cast<float4 *>(p.t_out)[v] = t4;
        }
    }
    for (long long c = 4 * n4 + tid; c < p.n; c += stride) {
        if constexpr (ER) {
            const float a0 = fmaxf(p.a_rad[c], 0.0f), e0 = fmaxf(p.e_rad[c], 0.0f);
            const float ar[2] = {a0, a0}, er[2] = {e0, e0};
            float t[2], err[2];
            diffuse_temperature<2>(p, k, ar, er, t, err);
            if (!(err[0] < 1.0f)) diffuse_more<2>(p, k, ar, er, t, err);
            p.t_out[c] = t[0];
        } else {
            p.t_out[c] = cell_temperature<ER>(p, k, p.a_rad[c], 0.0f);
        }
    }
}

}  // namespace

// ---------------------------------------------------------------------------
// host: the table belongs to the context (built on first use, per table)
// ---------------------------------------------------------------------------
namespace {

int planck_means(const CtxInfo &in, const std::vector<double> &t_nodes, double *kp_host, float *lkp_dev,
                 cudaStream_t st, std::string &err)
{
    const int n = (int)t_nodes.size();
    // the table's opacities: one value per bin, or rows on a temperature grid
    const int n_t = in.n_t > 0 ? in.n_t : 1;
    const double *kap_h = in.n_t > 0 ? in.kappa_t_h : in.kappa_h;
    double *tn = nullptr, *nu = nullptr, *ka = nullptr, *kp = nullptr, *tg = nullptr;
    bool ok = cudaMalloc(&tn, sizeof(double) * n) == cudaSuccess &&
              cudaMalloc(&nu, sizeof(double) * in.n_nu) == cudaSuccess &&
              cudaMalloc(&ka, sizeof(double) * in.n_nu * n_t) == cudaSuccess &&
              cudaMalloc(&tg, sizeof(double) * n_t) == cudaSuccess &&
              cudaMalloc(&kp, sizeof(double) * n) == cudaSuccess;
    ok = ok && cudaMemcpyAsync(tn, t_nodes.data(), sizeof(double) * n, cudaMemcpyHostToDevice, st) == cudaSuccess &&
         cudaMemcpyAsync(nu, in.nu_h, sizeof(double) * in.n_nu, cudaMemcpyHostToDevice, st) == cudaSuccess &&
         cudaMemcpyAsync(ka, kap_h, sizeof(double) * in.n_nu * n_t, cudaMemcpyHostToDevice, st) == cudaSuccess;
    if (ok && in.n_t > 0)
        ok = cudaMemcpyAsync(tg, in.t_grid_h, sizeof(double) * n_t, cudaMemcpyHostToDevice, st) == cudaSuccess;
    if (ok) {
        k_planck_mean<<<(n + 7) / 8, 256, 0, st>>>(n, tn, in.n_nu, nu, ka, n_t, tg, kp, lkp_dev);
        ok = cudaGetLastError() == cudaSuccess;
    }
    if (ok && kp_host) ok = cudaMemcpyAsync(kp_host, kp, sizeof(double) * n, cudaMemcpyDeviceToHost, st) == cudaSuccess;
    ok = ok && cudaStreamSynchronize(st) == cudaSuccess;
    if (!ok) err = std::string("Planck-mean kernel: ") + cudaGetErrorString(cudaGetLastError());
    cudaFree(tn);
    cudaFree(nu);
    cudaFree(ka);
    cudaFree(tg);
    cudaFree(kp);
    return ok ? RT_OK : RT_ERR_CUDA;
}

// The last Newton step of ln T after which diffuse_temperature takes a cell. A step dy leaves
// F''/(2 F') dy^2, with F' = 4 + w L' and F'' = w L'' - w (1 - w) L'^2, 0 <= w <= 1 the source's
// share: the largest |L''| and |L'| of the table's cubics bound that by kLeft. 4e-4 to 5e-4 on
// means of kappa(nu) (L'' up to 5), 2e-5 to 1e-4 on tables whose kappa(T) is linear between 8 to 32
// temperatures (kinks in the mean: L'' 90 to 750; with 5e-4 there, up to one cell in a thousand was
// off by up to 2e-5).
double accepted_step(const std::vector<float> &h)
{
    constexpr double kLeft = 1.5e-7;
    const double per_y = (kTempNodes - 1) / (kTempLnHi - kTempLnLo);
    double curve = 0.0, slope = 0.0, fall = 0.0;
    for (int k = 0; k < kTempNodes - 1; ++k) {  // the cubics of k_hermite_coeffs
        const double p0 = h[k], p1 = h[k + 1];
        const double m0 = k > 0 ? 0.5 * (p1 - h[k - 1]) : p1 - p0;
        const double m1 = k + 2 < kTempNodes ? 0.5 * (h[k + 2] - p0) : p1 - p0;
        const double q2 = 3.0 * (p1 - p0) - 2.0 * m0 - m1, q3 = 2.0 * (p0 - p1) + m0 + m1;
        curve = std::max({curve, fabs(2.0 * q2), fabs(2.0 * q2 + 6.0 * q3)});
        for (double t : {0.0, 1.0, q3 != 0.0 ? -q2 / (3.0 * q3) : 0.0}) {
            if (!(t >= 0.0 && t <= 1.0)) continue;
            const double d = m0 + t * (2.0 * q2 + t * 3.0 * q3);
            slope = std::max(slope, fabs(d));
            fall = std::max(fall, -d);
        }
    }
    curve *= per_y * per_y;
    slope *= per_y;
    fall *= per_y;
    const double left = (curve + 0.25 * slope * slope) / (2.0 * std::max(4.0 - fall, 0.5));
    return std::min(5e-4, std::max(1e-6, sqrt(kLeft / left)));  // (a NaN or infinite curve: 1e-6 or less)
}

}  // namespace
}  // namespace rt

using namespace rt;

extern "C" {

int rt_planck_mean_opacity(rt_ctx *ctx, double t, double *kappa_p)
{
    if (!ctx || !kappa_p) return RT_ERR_INVALID_ARG;
    CtxInfo in;
    ctx_info(ctx, &in);
    if (!in.configured) return ctx_fail(ctx, RT_ERR_NOT_CONFIGURED, "call rt_set_star and rt_set_opacity_table first");
    if (!(t > 0.0) || !isfinite(t)) return ctx_fail(ctx, RT_ERR_INVALID_ARG, "t must be finite and > 0");
    if (cudaSetDevice(in.dev) != cudaSuccess) return ctx_fail(ctx, RT_ERR_CUDA, "cudaSetDevice");
    std::string err;
    const int rc = planck_means(in, std::vector<double>{t}, kappa_p, nullptr, in.stream, err);
    return rc == RT_OK ? RT_OK : ctx_fail(ctx, rc, err);
}

int rt_dust_temperature(rt_ctx *ctx, const float *a_rad, const float *e_rad, float *t_dust)
{
    if (!ctx) return RT_ERR_INVALID_ARG;
    CtxInfo in;
    ctx_info(ctx, &in);
    if (!in.configured) return ctx_fail(ctx, RT_ERR_NOT_CONFIGURED, "call rt_set_star and rt_set_opacity_table first");
    if (!a_rad || !t_dust) return ctx_fail(ctx, RT_ERR_INVALID_ARG, "a_rad and t_dust must be non-NULL");
    if (cudaSetDevice(in.dev) != cudaSuccess) return ctx_fail(ctx, RT_ERR_CUDA, "cudaSetDevice");
    const double sigma = 2.0 * pow(kPi, 5) * pow(kKB, 4) / (15.0 * kH * kH * kH * kC * kC);
    const double ln_a = log(4.0 * sigma / kC);
    float *&lkp = ctx_temp_table(ctx);
    unsigned long long &fp = ctx_temp_fingerprint(ctx);
    if (!lkp || fp != in.table_fingerprint) {
        if (!lkp && cudaMalloc(&lkp, sizeof(float) * kTempTableFloats) != cudaSuccess) {
            lkp = nullptr;
            cudaGetLastError();
            return ctx_fail(ctx, RT_ERR_NO_MEMORY, "Planck-mean table");
        }
        std::vector<double> tn(kTempNodes);
        for (int i = 0; i < kTempNodes; ++i)
            tn[i] = exp(kTempLnLo + (kTempLnHi - kTempLnLo) * i / (kTempNodes - 1));
        std::string err;
        const int rc = planck_means(in, tn, nullptr, lkp, in.stream, err);
        if (rc != RT_OK) return ctx_fail(ctx, rc, err);
        // the inverse table's grid in v = lg2 a_rad: the finest spacing 2^-e whose nodes
        // (whole steps from v_org) cover X(y_lo)..X(y_hi) within kTempInvNodes
        std::vector<float> h(kTempNodes);
        if (cudaMemcpyAsync(h.data(), lkp, sizeof(float) * kTempNodes, cudaMemcpyDeviceToHost, in.stream) != cudaSuccess ||
            cudaStreamSynchronize(in.stream) != cudaSuccess)
            return ctx_fail(ctx, RT_ERR_CUDA, "Planck-mean table");
        const double v_lo = (4.0 * kTempLnLo + h[0] + ln_a) / kLn2, v_hi = (4.0 * kTempLnHi + h[kTempNodes - 1] + ln_a) / kLn2;
        int e = 6, v_org = 0, n_inv = 0;
        for (; e >= 0; --e) {
            v_org = (int)floor(ldexp(v_lo, e));
            n_inv = (int)ceil(ldexp(v_hi, e)) - v_org + 1;
            if (n_inv <= kTempInvNodes) break;
        }
        if (e < 0 || n_inv < 2) return ctx_fail(ctx, RT_ERR_INVALID_ARG, "Planck mean outside the tabulated range");
        double2 *ym = reinterpret_cast<double2 *>(lkp + kTempInvYm);
        k_inverse_nodes<<<(n_inv + 127) / 128, 128, 0, in.stream>>>(lkp, lkp + kTempConsts, ym, kTempLnLo, kTempLnHi, ln_a,
                                                                    e, v_org, n_inv, (float)(1.0 / accepted_step(h)));
        k_inverse_coeffs<<<(8 * (n_inv - 1) + 127) / 128, 128, 0, in.stream>>>(
            lkp, ym, reinterpret_cast<float4 *>(lkp + kTempCoefInv), kTempLnLo, kTempLnHi, ln_a, e, v_org, n_inv);
        k_hermite_coeffs<<<4, 256, 0, in.stream>>>(lkp, reinterpret_cast<float4 *>(lkp + kTempCoefLkp),
                                                   reinterpret_cast<float4 *>(lkp + kTempCoefLg2));
        if (cudaGetLastError() != cudaSuccess) return ctx_fail(ctx, RT_ERR_CUDA, "inverse temperature table");
        fp = in.table_fingerprint;
    }
    TempArgs p;
    p.a_rad = a_rad;
    p.e_rad = e_rad;
    p.t_out = t_dust;
    p.lkp = lkp;
    p.consts = lkp + kTempConsts;
    p.c_lkp = reinterpret_cast<const float4 *>(lkp + kTempCoefLkp);
    p.c_inv = reinterpret_cast<const float4 *>(lkp + kTempCoefInv);
    p.vec = ((reinterpret_cast<size_t>(a_rad) | reinterpret_cast<size_t>(e_rad) | reinterpret_cast<size_t>(t_dust)) % 16) == 0;
    p.n = in.ncells;
    p.y0 = (float)kTempLnLo;
    p.inv_dy = (float)((kTempNodes - 1) / (kTempLnHi - kTempLnLo));
    p.ln_a = (float)ln_a;
    p.a = (float)exp(ln_a);
    p.inv_a = (float)exp(-ln_a);
    static_assert(kTempLnLo == 0.0, "the node index of lg2 T has no offset");
    const double per_lg2 = (kTempNodes - 1) / (kTempLnHi - kTempLnLo) * kLn2;
    p.s_hi = (float)per_lg2;
    p.s_lo = (float)(per_lg2 - (double)p.s_hi);
    p.c_lg2 = reinterpret_cast<const float4 *>(lkp + kTempCoefLg2);
    p.l_scale = (float)(per_lg2 / (kTempNodes + 1));
    p.l_org = (float)(1.0 / (kTempNodes + 1));
    p.dl_dy = (float)((kTempNodes - 1) / (kTempLnHi - kTempLnLo) * kLn2);
    int nsm = 0;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, in.dev);
    long long blocks = (in.ncells / 4 + 255) / 256;
    if (blocks > 8LL * nsm) blocks = 8LL * nsm;
    if (blocks < 1) blocks = 1;
    if (e_rad) k_dust_temperature<true><<<(unsigned)blocks, 256, 0, in.stream>>>(p);
    else k_dust_temperature<false><<<(unsigned)blocks, 256, 0, in.stream>>>(p);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return ctx_fail(ctx, RT_ERR_CUDA, std::string("temperature kernel: ") + cudaGetErrorString(e));
    return RT_OK;
}

}  // extern "C"
