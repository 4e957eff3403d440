// One implicit flux-limited-diffusion step of the radiation energy density E = E_R
// (Sect. 2.1, Eqs. 7-15) with the absorbed stellar power as source (Eq. 15):
//     (E' - E) / dt = f_c (div(D grad E') + q_abs),   f_c = 1 / (c_V rho / (4 a T^3) + 1),
//     D = lambda c / (kappa_R rho),  lambda = (2 + R) / (6 + 3 R + R^2),  R = |grad E| / (kappa_R rho E),
// coefficients frozen at the old state and written D = c (2 s + g) / (6 s^2 + 3 s g + g^2)
// with s = kappa_R rho, g = |grad E| / E (finite as s -> 0; D = 0 where s = g = 0).
//
// Finite volumes on the spherical grid: a face carries the harmonic mean of its two
// cells' D times area over centre distance; no flux through the inner radius or the
// theta ends; E = a T_bg^4 half a cell beyond the outer radius; periodic in phi
// (nphi > 1). Lengths are in units of the outer radius L (r^3 in cm overflows FP32)
// and the system is divided by c L^2, so with tau = c dt / L
//     (V'/(tau f_c)) (E'_c - E_c) + sum_faces F_f A'/d' (E'_c - E'_nb) = V' q_c L / c,
// F = (2 s' + g') / (6 s'^2 + 3 s' g' + g'^2), s' = kappa_R rho L, g' = L |grad E| / E.
//
// The matrix is symmetric positive definite. It is applied matrix-free and solved
// by multigrid-preconditioned conjugate gradients with residual replacement (FP32
// vectors, FP64 reductions, every scalar and the loop itself on the device), from
// E_old, until a group of steps changed no cell by more than tol relative.
#include <cuda_bf16.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <string>
#include <type_traits>
#include <vector>

#include "rt_internal.cuh"
#include "rt_planck.cuh"

namespace rt {

constexpr int kRossNodes = 1024;
constexpr double kRossLnLo = 0.0, kRossLnHi = 11.512925464970229;  // ln 1 K .. ln 1e5 K

struct FldState {
    long long cap = 0;
    float *buf = nullptr;  // F (then the second p), tc (then x), b0, w[3], s, 1/dg, b, d, r, p, q, z:
                           // 14 n floats, then BF16 copies of s, w[3], 1/dg (5 n halves) for the
                           // finest V-cycle
    float *mg_buf = nullptr;              // coarse levels: s, w[3], 1/dg, b, x each
    float *line_buf = nullptr;            // phi-line smoother: factors, separator inverses, x
    int line_j0 = 0, line_j1 = 0;         // rows j < line_j0 and j >= line_j1 are smoothed by phi lines
    bool lines_set = false;
    std::vector<int> mg_dims;             // (nr, ntheta, nphi) of every level, finest first
    double *part = nullptr, *scal = nullptr;
    unsigned *bad = nullptr, *count = nullptr;
    int part_cap = 0;
    float *geo = nullptr;  // axis tables
    float *lkr = nullptr;  // ln kappa_R on the ln T nodes
    unsigned long long lkr_fp = 0;
    bool lkr_valid = false;
    // the solve runs on a private stream, after the context's stream; its loop is a graph with
    // a conditional node that points at this workspace only (built once per context)
    cudaStream_t gs = nullptr;
    cudaEvent_t ev_in = nullptr;
    cudaGraphExec_t loop = nullptr;
    bool no_graph = false;  // the graph could not be built: the host drives the loop
    double *scal_h = nullptr;  // pinned: the scalars and the validity word of the last solve
};

namespace {

// Rosseland mean of the table at t_nodes[n] (FP64, one warp per node):
// 1/kappa_R = sum_i w_i / kappa_i / sum_i w_i with w_i the band integral of dB/dT.
// A bin with kappa = 0 and nonzero weight makes the mean 0. (1024 nodes, 79 bins: 2.26 -> 0.79 ms;
// the FP64 pipe and bands of unequal width.)
__global__ void k_rosseland(int n_nodes, const double *t_nodes, int n_nu, const double *nu_mid, const double *kappa,
                            int n_t, const double *t_grid, double *kr_out, float *lkr)
{
    const int lane = threadIdx.x & 31;
    const int node = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (node >= n_nodes) return;
    const double t = t_nodes[node];
    const double kt_h = kKB * t / kH;
    double num = 0.0, den = 0.0;
    bool gap = false;
    for (int i0 = 0; i0 < n_nu; i0 += 4) {  // four bins at a time, 8 lanes each
        const int i = i0 + (lane >> 3);
        const bool on = i < n_nu;
        const double lo = (i == 0 || !on) ? 0.0 : 0.5 * (nu_mid[i - 1] + nu_mid[i]);
        const double hi = !on ? 0.0 : (i == n_nu - 1) ? INFINITY : 0.5 * (nu_mid[i] + nu_mid[i + 1]);
        const double w = rosseland_band_8(lo / kt_h, hi / kt_h, lane & 7);
        if (!on) continue;  // (the last round only)
        const double k = kappa_at(kappa + (size_t)i * n_t, n_t, t_grid, t);
        den += w;
        if (k > 0.0) num += w / k;
        else if (w > 0.0) gap = true;
    }
    for (int o = 8; o < 32; o <<= 1) {
        den += __shfl_xor_sync(0xffffffffu, den, o);
        num += __shfl_xor_sync(0xffffffffu, num, o);
    }
    gap = __any_sync(0xffffffffu, gap);
    if (lane == 0) {
        const double kr = (gap || !(num > 0.0)) ? 0.0 : den / num;
        if (kr_out) kr_out[node] = kr;
        if (lkr) lkr[node] = (float)log(kr > 1e-300 ? kr : 1e-300);
    }
}

struct FldGeo {
    const float *rif;       // [nr+1] r / L
    const float *rc;        // [nr]   centre radii
    const float *drc;       // [nr]   rc[k+1] - rc[k] (last entry unused)
    const float *d3;        // [nr]   (r+^3 - r-^3) / 3
    const float *dr2;       // [nr]   (r+^2 - r-^2) / 2
    const float *sin_thif;  // [nth+1]
    const float *dthc;      // [nth]  thc[j+1] - thc[j] (last entry unused)
    const float *sin_thc;   // [nth]
    const float *dcos;      // [nth]  cos th- - cos th+
    const float *dth;       // [nth]  th+ - th-
    const float *dph;       // [nph]  phi+ - phi-
    const float *dphc;      // [nph]  phi centre l to centre l+1, wrapped
    int nr, nth, nph;
    FastDiv div_nr, div_nth;
};

// (k, j, l) of flat cell c of the [nphi][ntheta][nr] layout (c < 2^31)
__device__ __forceinline__ void cell_ijk(unsigned c, int nr, int nth, const FastDiv &dr, const FastDiv &dt, int &k,
                                         int &j, int &l)
{
    const unsigned rest = dr.div(c);
    k = (int)(c - rest * (unsigned)nr);
    l = (int)dt.div(rest);
    j = (int)(rest - (unsigned)l * (unsigned)nth);
}

__device__ __forceinline__ float lnk_interp(const float *s, float y, float y0, float inv_dy)
{
    const float u = (y - y0) * inv_dy;
    if (!(u > 0.0f)) return s[0];
    if (u >= (float)(kRossNodes - 1)) return s[kRossNodes - 1];
    const int k = min((int)u, kRossNodes - 2);
    const float t = u - (float)k;
    const float p0 = s[k], p1 = s[k + 1];
    const float m0 = k > 0 ? 0.5f * (p1 - s[k - 1]) : p1 - p0;
    const float m1 = k + 2 < kRossNodes ? 0.5f * (s[k + 2] - p0) : p1 - p0;
    const float t2 = t * t, t3 = t2 * t;
    return (2.0f * t3 - 3.0f * t2 + 1.0f) * p0 + (t3 - 2.0f * t2 + t) * m0 + (-2.0f * t3 + 3.0f * t2) * p1 +
           (t3 - t2) * m1;
}

struct FldCellArgs {
    FldGeo g;
    const float *rho, *t, *q, *e;
    const float *lkr;
    float y0, inv_dy;   // ln T nodes
    float L;            // outer radius, cm
    float c_v, four_a;  // specific heat, 4 a
    float inv_tau;      // L / (c dt)
    float q_scale;      // L / c
    float *F, *tc, *b0;
    unsigned *bad;
    long long n;
};

// per cell: the face factor F, the storage term V'/(tau f_c) and the old-state
// right-hand side; flags invalid input (rho < 0, T <= 0, E_old < 0, q < 0, NaN/Inf)
__global__ void __launch_bounds__(256) k_fld_cell(const FldCellArgs p)
{
    __shared__ float s_l[kRossNodes];
    for (int i = threadIdx.x; i < kRossNodes; i += blockDim.x) s_l[i] = p.lkr[i];
    __syncthreads();
    const FldGeo &g = p.g;
    const long long plane = (long long)g.nr * g.nth;
    bool bad = false;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < p.n;
         c += (long long)gridDim.x * blockDim.x) {
        int k, j, l;
        cell_ijk((unsigned)c, g.nr, g.nth, g.div_nr, g.div_nth, k, j, l);
        const float rho = p.rho[c], t = p.t[c], e = p.e[c], q = p.q[c];
        if (!(rho >= 0.0f && rho < INFINITY && t > 0.0f && t < INFINITY && e >= 0.0f && e < INFINITY &&
              q >= 0.0f && q < INFINITY)) {
            bad = true;
            p.F[c] = 0.0f;
            p.tc[c] = 1.0f;
            p.b0[c] = 0.0f;
            continue;
        }
        const float kr = expf(lnk_interp(s_l, logf(t), p.y0, p.inv_dy));
        const float s = (kr * rho) * p.L;
        // |grad E| / E in units of 1/L: central differences, one-sided at the r and
        // theta ends, periodic in phi (relative to this cell's E)
        const float inv_e = e > 0.0f ? 1.0f / e : 0.0f;
        float gr = 0.0f, gt = 0.0f, gp = 0.0f;
        if (g.nr > 1) {
            const int ka = k > 0 ? k - 1 : k, kb = k < g.nr - 1 ? k + 1 : k;
            float d = 0.0f;
            for (int i = ka; i < kb; ++i) d += g.drc[i];
            gr = (p.e[c + (kb - k)] - p.e[c + (ka - k)]) * inv_e / d;
        }
        if (g.nth > 1) {
            const int ja = j > 0 ? j - 1 : j, jb = j < g.nth - 1 ? j + 1 : j;
            float d = 0.0f;
            for (int i = ja; i < jb; ++i) d += g.dthc[i];
            gt = (p.e[c + (long long)(jb - j) * g.nr] - p.e[c + (long long)(ja - j) * g.nr]) * inv_e /
                 (g.rc[k] * d);
        }
        if (g.nph > 1) {
            const int la = (l + g.nph - 1) % g.nph, lb = (l + 1) % g.nph;
            const float dphi = g.nph == 2 ? 6.283185307179586f : g.dphc[la] + g.dphc[l];
            gp = (p.e[c + (long long)(lb - l) * plane] - p.e[c + (long long)(la - l) * plane]) * inv_e /
                 (g.rc[k] * g.sin_thc[j] * dphi);
        }
        const float gg = sqrtf(gr * gr + gt * gt + gp * gp);
        const float num = 2.0f * s + gg;
        p.F[c] = num > 0.0f ? num / (6.0f * s * s + 3.0f * s * gg + gg * gg) : 0.0f;
        const float t3 = t * t * t;
        const float fc = 1.0f / (p.c_v * rho / (p.four_a * t3) + 1.0f);
        const float vol = g.dcos[j] * g.dph[l] * g.d3[k];
        const float tc = vol * p.inv_tau / fc;
        p.tc[c] = tc;
        p.b0[c] = tc * e + vol * q * p.q_scale;
    }
    if (bad) atomicOr(p.bad, 1u);
}

struct FldFaceArgs {
    FldGeo g;
    const float *F, *tc, *b0;
    float e_bg;               // a T_bg^4
    const float *e;           // E_old, the solve's start value x
    float *w, *s, *idg, *b, *x;  // w [3][n]: to the k+1, j+1 and l+1 neighbours
    unsigned short *hs, *hw, *hidg;  // BF16 copies of s, w, 1/dg (the finest V-cycle's operator)
    long long n;
};

__device__ __forceinline__ float harm(float a, float b)
{
    return (a > 0.0f && b > 0.0f) ? 2.0f * a * b / (a + b) : 0.0f;
}

// face weights to the + neighbours; s = storage + outer-boundary weight; the
// inverse of the Jacobi diagonal s + all six face weights; the right-hand side
__global__ void __launch_bounds__(256) k_fld_faces(const FldFaceArgs p)
{
    const FldGeo &g = p.g;
    const long long plane = (long long)g.nr * g.nth, n = p.n;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n;
         c += (long long)gridDim.x * blockDim.x) {
        int k, j, l;
        cell_ijk((unsigned)c, g.nr, g.nth, g.div_nr, g.div_nth, k, j, l);
        const float Fc = p.F[c];
        const float dom = g.dcos[j] * g.dph[l];
        float sc = p.tc[c], rhs = p.b0[c], faces = 0.0f;
        float wr = 0.0f, wt = 0.0f, wp = 0.0f;
        if (k + 1 < g.nr) {
            wr = harm(Fc, p.F[c + 1]) * dom * (g.rif[k + 1] * g.rif[k + 1]) / g.drc[k];
            faces += wr;
        } else {  // outer boundary: E_bg half a cell beyond the last centre
            const float wo = Fc * dom * (g.rif[g.nr] * g.rif[g.nr]) / (g.rif[g.nr] - g.rc[k]);
            sc += wo;
            rhs += wo * p.e_bg;
        }
        if (k > 0) faces += harm(Fc, p.F[c - 1]) * dom * (g.rif[k] * g.rif[k]) / g.drc[k - 1];
        if (j + 1 < g.nth) {
            wt = harm(Fc, p.F[c + g.nr]) * g.dph[l] * g.sin_thif[j + 1] * g.dr2[k] / (g.rc[k] * g.dthc[j]);
            faces += wt;
        }
        if (j > 0)
            faces += harm(Fc, p.F[c - g.nr]) * g.dph[l] * g.sin_thif[j] * g.dr2[k] / (g.rc[k] * g.dthc[j - 1]);
        if (g.nph > 1) {
            const int lb = (l + 1) % g.nph, la = (l + g.nph - 1) % g.nph;
            const float area = g.dth[j] * g.dr2[k] / (g.rc[k] * g.sin_thc[j]);
            wp = harm(Fc, p.F[c + (long long)(lb - l) * plane]) * area / g.dphc[l];
            faces += wp;
            faces += harm(Fc, p.F[c + (long long)(la - l) * plane]) * area / g.dphc[la];
        }
        const float idg = 1.0f / (sc + faces);
        p.w[c] = wr;
        p.w[n + c] = wt;
        p.w[2 * n + c] = wp;
        p.s[c] = sc;
        p.idg[c] = idg;
        p.b[c] = rhs;
        p.x[c] = p.e[c];  // x may be tc's buffer: this cell's tc is read above, no other's
        p.hw[c] = __bfloat16_as_ushort(__float2bfloat16_rn(wr));
        p.hw[n + c] = __bfloat16_as_ushort(__float2bfloat16_rn(wt));
        p.hw[2 * n + c] = __bfloat16_as_ushort(__float2bfloat16_rn(wp));
        p.hs[c] = __bfloat16_as_ushort(__float2bfloat16_rn(sc));
        p.hidg[c] = __bfloat16_as_ushort(__float2bfloat16_rn(idg));
    }
}

// --- the solve -----------------------------------------------------------------
// A v = s v + sum_faces w (v_c - v_nb) is applied in this flux form: the storage
// and boundary term s is stored apart from the face weights, so nothing small is
// left as the difference of large rounded numbers (a diagonal holding s + sum w
// would bury s under the rounding of the face weights wherever diffusion dominates).
//
// Preconditioned conjugate gradients with group-wise residual replacement (Sleijpen and
// van der Vorst 1996): the steps of a group add up in d; once r.z fell by kGroupDrop^2, d
// goes into x, r is taken afresh as b - A x (FP32 recurrences lose the true residual after a
// few hundred steps) and the directions carry on. The groups end when max |d| / |x| < tol.
// Keeping the directions over a replacement took 37 steps against 41 with restarts (FP64
// emulation, 128x64x64), and a group costs one stencil pass in place of an update.
//
// One iteration is a fixed list of kernels whose scalars live on the device:
//   k_it_flush     (at a group's end only) x += d; max |d| / |x|; done?
//   k_it_residual  r -= alpha q, or r = b - A x after a flush; the phi lines' first solve
//   k_mg_down ... k_mg_tail ... k_mg_up: z = M^-1 r, r.z, beta (k_it_jacobi on small grids)
//   k_it_apply     d += alpha p; p = z + beta p; q = A p; alpha = r.z / p.q
// so p, q, d move once per iteration (the direction update and the step are folded into
// passes that read their arrays anyway). The loop is a graph with a conditional node, kUnroll
// iterations per body: no host round trip until the solve is done, no idle launches but the
// last body's.
constexpr double kGroupDrop = 0.1;
constexpr int kUnroll = 4;  // even: p alternates between two buffers

// device scalars of the solve
enum : int {
    kRz = 0,   // r.z
    kRz0,      // r.z at the start of the group
    kAlpha,
    kBeta,
    kPend,     // 1: the step alpha p is not yet in d
    kDLive,    // 1: d holds steps of this group (else it counts as 0)
    kFlush,    // 1: the group ends before the next residual; 2: first residual of the solve
    kLast,     // 1: max_iter reached, the next flush ends the solve
    kDone,     // 1: x is final (or the input was invalid); every later launch returns at once
    kIters,
    kPasses,   // groups
    kCorr,     // max |d| / |x| of the last group (infinite: x not finite)
    kTol,
    kMaxIter,
    kLoops,    // bodies of the loop run so far
    kNScal
};

struct CgArgs {
    int nr, nth, nph;
    FastDiv div_nr, div_nth;
    long long n;
    const float *w, *s, *idg, *b;
    float *x, *d, *r, *q, *z;
    double *part;     // [grid]
    double *scal;     // kNScal
    unsigned *count;  // blocks finished (last-block reductions)
};

__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ void st4(float *p, float4 v) { *reinterpret_cast<float4 *>(p) = v; }
// operator entries in FP32, or the finest V-cycle's BF16 copies
__device__ __forceinline__ float4 ldo4(const float *p) { return ld4(p); }
__device__ __forceinline__ float ldo1(const float *p) { return *p; }
__device__ __forceinline__ float4 ldo4(const unsigned short *p)
{
    const uint2 u = *reinterpret_cast<const uint2 *>(p);
    return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u), __uint_as_float(u.y << 16),
                       __uint_as_float(u.y & 0xffff0000u));
}
__device__ __forceinline__ float ldo1(const unsigned short *p) { return __uint_as_float((unsigned)*p << 16); }

// A v at cell c = (k, j, l); v(i, k', j', l') gives the neighbours' values
template <class T, class V>
__device__ __forceinline__ float flux_one(int nr, int nth, int nph, unsigned n, const T *s, const T *w, const V &v,
                                          unsigned c, int k, int j, int l, float vc)
{
    const unsigned plane = (unsigned)nr * (unsigned)nth;
    float acc = ldo1(s + c) * vc;
    if (k + 1 < nr) acc = fmaf(ldo1(w + c), vc - v(c + 1, k + 1, j, l), acc);
    if (k > 0) acc = fmaf(ldo1(w + c - 1), vc - v(c - 1, k - 1, j, l), acc);
    if (j + 1 < nth) acc = fmaf(ldo1(w + n + c), vc - v(c + nr, k, j + 1, l), acc);
    if (j > 0) acc = fmaf(ldo1(w + n + c - nr), vc - v(c - nr, k, j - 1, l), acc);
    if (nph > 1) {
        const int lb = l + 1 < nph ? l + 1 : 0, la = l > 0 ? l - 1 : nph - 1;
        const unsigned cb = c + (unsigned)(lb - l) * plane, ca = c + (unsigned)(la - l) * plane;
        acc = fmaf(ldo1(w + 2 * n + c), vc - v(cb, k, j, lb), acc);
        acc = fmaf(ldo1(w + 2 * n + ca), vc - v(ca, k, j, la), acc);
    }
    return acc;
}

// A v on the quad c .. c+3 of one ray (nr % 4 == 0: the four cells share (j, l) and every
// offset is a multiple of 16 bytes); vrow gives the quad at the same k of another row, v one cell
template <class T, class VR, class V>
__device__ __forceinline__ float4 flux_quad(int nr, int nth, int nph, unsigned n, const T *s_, const T *w_,
                                            const VR &vrow, const V &v, unsigned c, int k, int j, int l, float4 vc)
{
    const unsigned plane = (unsigned)nr * (unsigned)nth;
    const float4 s = ldo4(s_ + c), wr = ldo4(w_ + c);
    float4 acc = make_float4(s.x * vc.x, s.y * vc.y, s.z * vc.z, s.w * vc.w);
    acc.x = fmaf(wr.x, vc.x - vc.y, acc.x);
    acc.y = fmaf(wr.y, vc.y - vc.z, acc.y);
    acc.z = fmaf(wr.z, vc.z - vc.w, acc.z);
    acc.y = fmaf(wr.x, vc.y - vc.x, acc.y);
    acc.z = fmaf(wr.y, vc.z - vc.y, acc.z);
    acc.w = fmaf(wr.z, vc.w - vc.z, acc.w);
    if (k + 4 < nr) acc.w = fmaf(wr.w, vc.w - v(c + 4, k + 4, j, l), acc.w);
    if (k > 0) acc.x = fmaf(ldo1(w_ + c - 1), vc.x - v(c - 1, k - 1, j, l), acc.x);
    auto face4 = [&](float4 w, float4 u) {
        acc.x = fmaf(w.x, vc.x - u.x, acc.x);
        acc.y = fmaf(w.y, vc.y - u.y, acc.y);
        acc.z = fmaf(w.z, vc.z - u.z, acc.z);
        acc.w = fmaf(w.w, vc.w - u.w, acc.w);
    };
    if (j + 1 < nth) face4(ldo4(w_ + n + c), vrow(c + nr, k, j + 1, l));
    if (j > 0) face4(ldo4(w_ + n + c - nr), vrow(c - nr, k, j - 1, l));
    if (nph > 1) {
        const int lb = l + 1 < nph ? l + 1 : 0, la = l > 0 ? l - 1 : nph - 1;
        const unsigned cb = c + (unsigned)(lb - l) * plane, ca = c + (unsigned)(la - l) * plane;
        face4(ldo4(w_ + 2 * n + c), vrow(cb, k, j, lb));
        face4(ldo4(w_ + 2 * n + ca), vrow(ca, k, j, la));
    }
    return acc;
}

// a + b as their rounded sum and the rest, exactly (Knuth)
__device__ __forceinline__ float2 two_sum(float a, float b)
{
    const float t = a + b, bp = t - a;
    return make_float2(t, (a - (t - bp)) + (b - bp));
}

// Per-thread sums in compensated FP32 (TwoSum; GB300's FP64 rate is a small
// fraction of its FP32 rate).
struct KSum {
    float s = 0.0f, c = 0.0f;
    __device__ __forceinline__ void add(float v)
    {
        const float2 t = two_sum(s, v);
        c += t.y;
        s = t.x;
    }
};
// A block's sum of them: three floats (what a TwoSum leaves goes into the next one), which lose
// less than FP64 does; the block's partial is FP64. In FP64 the block sums took 1.5 us more per
// iteration (64x32x64: 1.72 against 1.67 ms per step), pairs of floats lost 2^-48 per addition.
struct BSum {
    float s = 0.0f, c = 0.0f, d = 0.0f;
    BSum() = default;
    __device__ __forceinline__ BSum(const KSum &k) : s(k.s), c(k.c) {}
    __device__ __forceinline__ void add(const BSum &o)
    {
        const float2 t = two_sum(s, o.s), u = two_sum(c, o.c), v = two_sum(u.x, t.y);
        s = t.x;
        c = v.x;
        d = (d + o.d) + (u.y + v.y);
    }
    __device__ __forceinline__ BSum shfl(int m) const
    {
        BSum r;
        r.s = __shfl_xor_sync(0xffffffffu, s, m);
        r.c = __shfl_xor_sync(0xffffffffu, c, m);
        r.d = __shfl_xor_sync(0xffffffffu, d, m);
        return r;
    }
    __device__ __forceinline__ double value() const { return ((double)d + (double)c) + (double)s; }
};
struct KMax {
    float s = 0.0f;
    __device__ __forceinline__ void add(const KMax &o) { s = fmaxf(s, o.s); }
    __device__ __forceinline__ KMax shfl(int m) const
    {
        KMax r;
        r.s = __shfl_xor_sync(0xffffffffu, s, m);
        return r;
    }
    __device__ __forceinline__ double value() const { return (double)s; }
};
struct DSum {  // the last block's sum of the FP64 partials
    double s = 0.0;
    __device__ __forceinline__ void add(const DSum &o) { s += o.s; }
    __device__ __forceinline__ DSum shfl(int m) const
    {
        DSum r;
        r.s = __shfl_xor_sync(0xffffffffu, s, m);
        return r;
    }
};

// block reduction into thread 0: two levels of shuffles
template <class S>
__device__ __forceinline__ S block_reduce(S v)
{
    __shared__ S s_w[32];
    for (int o = 16; o > 0; o >>= 1) v.add(v.shfl(o));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __syncthreads();
    if (lane == 0) s_w[warp] = v;
    __syncthreads();
    if (warp == 0) {
        v = lane < nw ? s_w[lane] : S();
        for (int o = 16; o > 0; o >>= 1) v.add(v.shfl(o));
    }
    return v;
}

// Writes this block's partial at part[at + blockIdx.x]; the block that finishes last reduces the
// first at + gridDim.x partials in a fixed order (deterministic) and returns true in its thread 0
// with the total. (at: the partials an earlier kernel left for this one.)
template <class S>
__device__ bool grid_reduce(const CgArgs &a, const S &v, double *out, int at = 0)
{
    __shared__ bool s_last;
    constexpr bool kMax = std::is_same<S, KMax>::value;
    const S t = block_reduce(v);
    if (threadIdx.x == 0) {
        a.part[at + blockIdx.x] = t.value();
        __threadfence();
        s_last = atomicAdd(a.count, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return false;
    DSum u;
    KMax m;
    for (int i = threadIdx.x; i < at + (int)gridDim.x; i += blockDim.x) {
        const double pi = __ldcg(a.part + i);
        if (kMax) m.s = fmaxf(m.s, (float)pi);
        else u.s += pi;
    }
    double tot;
    if constexpr (kMax) tot = block_reduce(m).value();
    else tot = block_reduce(u).s;
    if (threadIdx.x == 0) {
        *out = tot;
        *a.count = 0u;
    }
    return threadIdx.x == 0;
}

// the level-0 kernels' cells: quads of one ray (Q) or single cells, the blocks from b0 on
template <bool Q, class F>
__device__ __forceinline__ void for_cells(const CgArgs &a, unsigned b0, const F &f)
{
    constexpr unsigned W = Q ? 4u : 1u;
    for (unsigned c = W * ((blockIdx.x - b0) * blockDim.x + threadIdx.x); c < (unsigned)a.n;
         c += W * (gridDim.x - b0) * blockDim.x) {
        int k, j, l;
        cell_ijk(c, a.nr, a.nth, a.div_nr, a.div_nth, k, j, l);
        f(c, k, j, l);
    }
}

// Rows smoothed by whole phi lines on the finest level. Next to the poles the phi faces are
// close together and a row couples to itself in phi far more strongly (as 1 / sin^2 theta) than
// to its neighbours, which a point smoother and 2 x 2 x 2 aggregates cannot follow: the slowest
// modes of the point-smoothed V-cycle all sat there. So in the rows where the phi faces hold
// more than kLineShare of the diagonal (geometry only; a run of rows at each theta end) the
// Jacobi diagonal of the smoother is replaced by the row's periodic tridiagonal blocks T (one
// phi ring per (j, k)): x0 = omega T^-1 b before the restriction and x1 + omega T^-1 (b - A x1)
// after the prolongation, symmetric as before and omega lambda(T^-1 A) < 2 as for the points.
// FP64 PCG on the CPU to a 1e-8 residual: 79 -> 31 iterations on 128x64x64 with 12 % of the
// rows; lines in every row 29, radial lines 79. On the GPU 256 -> 56 iterations per step on
// 256x128x256 (dt = 1e4 s), and the error against 64 bits 4.3e-6 -> 2.9e-7 (2-norm).
struct LineOp {
    int j0, j1, nl;             // rows j < j0 and j >= j1: nl of them (j0 = 0, j1 = nth: none)
    int seg;                    // segments a ring is cut into (its last cells are the separators)
    int blocks;                 // CTAs of the line role: one per row and 32 k
    float *m, *vl, *vr, *inv;   // [nph][nl][nr]: pivots, responses to the left and right separator;
                                // [nl][seg][seg][nr]: inverse of the separators' Schur complement
    float *x, *res;             // [nph][nl][nr]: omega T^-1 b, and the residual of the second solve
    __device__ __forceinline__ bool has(int j) const { return j < j0 || j >= j1; }
    __device__ __forceinline__ unsigned at(int nr, int k, int j, int l) const
    {
        return ((unsigned)l * (unsigned)nl + (unsigned)(j < j0 ? j : j - j1 + j0)) * (unsigned)nr + (unsigned)k;
    }
};
constexpr int kLineMaxSeg = 16;
constexpr int kLineChunk = 8;        // cells whose loads a thread has in flight together
constexpr double kLineShare = 0.85;  // of the diagonal held by the phi faces
constexpr int kLineMinPhi = 16;
constexpr int kLineSmemPhi = 1024;   // rings up to this keep the sweep's values in shared memory

// The ring of one row j and 32 consecutive k per block: lane = k, warp = ring segment
// (coalesced along k; a ring's cells lie a plane apart). Each segment eliminates its interior
// with zero separators, the separators (its last cell) follow from the precomputed inverse of
// their cyclic Schur complement, and the interior takes the two separators' responses: the
// dependent chain is nph / seg cells instead of nph. The few rings are latency-bound, so the
// loads of a chunk of cells are issued before its arithmetic and its stores (256x128x256: 26 and
// 39 us per solve with loads and stores interleaved, 22 us, 512 threads at 64 registers).
// lb(c, i) and sb(c, b): load and keep the right-hand side of cell c; ld(c, i, e) loads what out
// needs; out(c, i, x, e) takes the solution (i: the cell's index in the line arrays).
// SM: the sweep's values in shared memory, else in gy (a line array that lb has read).
template <bool SM, class LB, class SB, class LD, class OUT>
__device__ __forceinline__ void line_solve(const LineOp &L, const CgArgs &a, float *gy, const LB &lb, const SB &sb,
                                           const LD &ld, const OUT &out)
{
    extern __shared__ float s_y[];  // [longest interior][threads]
    __shared__ float s_f[kLineMaxSeg][32], s_r[kLineMaxSeg][32], s_s[kLineMaxSeg][32];
    constexpr int U = kLineChunk;
    const int lane = threadIdx.x & 31, sg = threadIdx.x >> 5, S = L.seg, T = blockDim.x;
    const int kt = (a.nr + 31) / 32;
    const int jl = blockIdx.x / kt, k = (blockIdx.x - jl * kt) * 32 + lane;
    const int j = jl < L.j0 ? jl : jl - L.j0 + L.j1;
    const bool act = k < a.nr;
    const int l0 = sg * a.nph / S, le = (sg + 1) * a.nph / S - 1;  // interior [l0, le), separator le
    const unsigned plane = (unsigned)a.nr * (unsigned)a.nth, lp = (unsigned)L.nl * (unsigned)a.nr;
    const unsigned c0 = (unsigned)j * a.nr + k, i0 = (unsigned)jl * a.nr + k;
    const float *wp = a.w + 2 * a.n + c0;
    auto yv = [&](int l) -> float & {
        if constexpr (SM) return s_y[(l - l0) * T + threadIdx.x];
        else return gy[i0 + l * lp];
    };
    float y = 0.0f, w0 = 0.0f, bs = 0.0f, wsep = 0.0f;
    float mm[U], ww[U];
    if (act) {
        bs = lb(c0 + le * plane, i0 + le * lp);
        wsep = __ldg(wp + le * plane);
        for (int lc = l0; lc < le; lc += U) {
            float bb[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (lc + u < le) {
                    bb[u] = lb(c0 + (lc + u) * plane, i0 + (lc + u) * lp);
                    mm[u] = __ldg(L.m + i0 + (lc + u) * lp);
                    ww[u] = __ldg(wp + (lc + u) * plane);
                }
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (lc + u < le) {
                    y = fmaf(w0, y, bb[u]) * mm[u];
                    w0 = ww[u];
                    yv(lc + u) = y;
                    sb(c0 + (lc + u) * plane, bb[u]);
                }
        }
        sb(c0 + le * plane, bs);
        // backward: from the last chunk (its factors are in registers) to the first
        float x = 0.0f;
        for (int lc = l0 + (le - 1 - l0) / U * U; lc >= l0; lc -= U) {
            if (lc + U < le) {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    mm[u] = __ldg(L.m + i0 + (lc + u) * lp);
                    ww[u] = __ldg(wp + (lc + u) * plane);
                }
            }
#pragma unroll
            for (int u = U - 1; u >= 0; --u)
                if (lc + u < le) {  // (x starts at 0: the last interior cell keeps its y)
                    x = fmaf(ww[u] * mm[u], x, yv(lc + u));
                    yv(lc + u) = x;
                }
        }
        s_f[sg][lane] = x;
    }
    __syncthreads();
    if (act) s_r[sg][lane] = bs + w0 * y + wsep * s_f[sg + 1 < S ? sg + 1 : 0][lane];
    float iv[kLineMaxSeg];
    if (act) {
        const float *inv = L.inv + ((size_t)jl * S + sg) * S * a.nr + k;
#pragma unroll
        for (int t = 0; t < kLineMaxSeg; ++t) iv[t] = t < S ? __ldg(inv + (size_t)t * a.nr) : 0.0f;
    }
    __syncthreads();
    float sr = 0.0f;
    if (act) {
#pragma unroll
        for (int t = 0; t < kLineMaxSeg; ++t)
            if (t < S) sr = fmaf(iv[t], s_r[t][lane], sr);
        s_s[sg][lane] = sr;
    }
    __syncthreads();
    if (!act) return;
    const float sl = s_s[sg > 0 ? sg - 1 : S - 1][lane];
    float2 es;
    ld(c0 + le * plane, i0 + le * lp, es);
    for (int lc = l0; lc < le; lc += U) {
        float2 e[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (lc + u < le) {
                ld(c0 + (lc + u) * plane, i0 + (lc + u) * lp, e[u]);
                mm[u] = __ldg(L.vl + i0 + (lc + u) * lp);
                ww[u] = __ldg(L.vr + i0 + (lc + u) * lp);
            }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (lc + u < le)
                out(c0 + (lc + u) * plane, i0 + (lc + u) * lp,
                    fmaf(ww[u], sr, fmaf(mm[u], sl, yv(lc + u))), e[u]);
    }
    out(c0 + le * plane, i0 + le * lp, sr, es);
}

// the factors of every ring: pivots, separator responses and the inverse of the separators'
// cyclic tridiagonal Schur complement (FP64 recurrences; once per step)
__global__ void __launch_bounds__(512) k_line_setup(const LineOp L, const CgArgs a)
{
    __shared__ double s_d[kLineMaxSeg][32], s_e[kLineMaxSeg][32], s_v[kLineMaxSeg][32];
    const int lane = threadIdx.x & 31, sg = threadIdx.x >> 5, S = L.seg;
    const int kt = (a.nr + 31) / 32;
    const int jl = blockIdx.x / kt, k = (blockIdx.x - jl * kt) * 32 + lane;
    const int j = jl < L.j0 ? jl : jl - L.j0 + L.j1;
    const bool act = k < a.nr;
    const int l0 = sg * a.nph / S, l1 = (sg + 1) * a.nph / S;
    const unsigned n = (unsigned)a.n, plane = (unsigned)a.nr * (unsigned)a.nth;
    const unsigned lp = (unsigned)L.nl * (unsigned)a.nr, i0 = (unsigned)jl * a.nr + k;
    auto cell = [&](int l) { return (unsigned)l * plane + (unsigned)j * a.nr + k; };
    auto wph = [&](int l) { return (double)__ldg(a.w + 2 * n + cell(l)); };
    auto diag = [&](int l) {
        const unsigned c = cell(l);
        double d = (double)__ldg(a.s + c) + wph(l) + wph(l > 0 ? l - 1 : a.nph - 1);
        if (k + 1 < a.nr) d += (double)__ldg(a.w + c);
        if (k > 0) d += (double)__ldg(a.w + c - 1);
        if (j + 1 < a.nth) d += (double)__ldg(a.w + n + c);
        if (j > 0) d += (double)__ldg(a.w + n + c - a.nr);
        return d;
    };
    double m = 0.0, v = 0.0, w0 = 0.0, dsep = 0.0;
    if (act) {
        // interior pivots, and the forward part of the left separator's response
        const double wl = wph(l0 > 0 ? l0 - 1 : a.nph - 1);  // left separator to the first interior cell
#pragma unroll 4
        for (int l = l0; l < l1 - 1; ++l) {
            const double piv = diag(l) - w0 * w0 * m;
            m = piv > 0.0 ? 1.0 / piv : 0.0;
            v = (l == l0 ? wl : w0 * v) * m;
            w0 = wph(l);
            L.m[i0 + l * lp] = (float)m;
            L.vl[i0 + l * lp] = (float)v;
        }
        // backward; w0 couples the last interior cell and the separator
        double u = w0 * m;  // the right separator's response
        const double vlast = v, ulast = u;
        L.vr[i0 + (l1 - 2) * lp] = (float)u;
#pragma unroll 4
        for (int l = l1 - 3; l >= l0; --l) {
            const double g = wph(l) * (double)L.m[i0 + l * lp];
            u *= g;
            v = fma(g, v, (double)L.vl[i0 + l * lp]);
            L.vl[i0 + l * lp] = (float)v;
            L.vr[i0 + l * lp] = (float)u;
        }
        // Schur complement: own diagonal here, the left neighbour's share through s_v
        dsep = diag(l1 - 1) - w0 * ulast;
        s_v[sg][lane] = wl * v;      // first cell's response to the left separator, times its coupling
        s_e[sg][lane] = w0 * vlast;  // coupling of separators sg - 1 and sg
    }
    __syncthreads();
    if (act) s_d[sg][lane] = dsep - s_v[sg + 1 < S ? sg + 1 : 0][lane];
    __syncthreads();
    if (!act) return;
    // column sg of the inverse: cyclic tridiagonal solve (Thomas, with Sherman and Morrison's
    // rank-one correction for the wrap), couplings e[t] between separators t - 1 and t
    double cp[kLineMaxSeg], y[kLineMaxSeg], q[kLineMaxSeg];
    const double wrap = s_e[0][lane], gam = -s_d[0][lane];
    double den = 0.0;
    for (int t = 0; t < S; ++t) {
        double d = s_d[t][lane];
        if (t == 0) d -= gam;
        if (t == S - 1) d -= wrap * wrap / gam;
        const double e = t > 0 ? s_e[t][lane] : 0.0;
        den = 1.0 / (t > 0 ? d - e * cp[t - 1] : d);
        cp[t] = t + 1 < S ? s_e[t + 1][lane] * den : 0.0;
        y[t] = ((t == sg ? 1.0 : 0.0) + (t > 0 ? e * y[t - 1] : 0.0)) * den;
        q[t] = ((t == 0 ? gam : t == S - 1 ? -wrap : 0.0) + (t > 0 ? e * q[t - 1] : 0.0)) * den;
    }
    for (int t = S - 2; t >= 0; --t) {
        y[t] += cp[t] * y[t + 1];
        q[t] += cp[t] * q[t + 1];
    }
    const double f = (y[0] - wrap * y[S - 1] / gam) / (1.0 + q[0] - wrap * q[S - 1] / gam);
    for (int t = 0; t < S; ++t) L.inv[(((size_t)jl * S + t) * S + sg) * a.nr + k] = (float)(y[t] - f * q[t]);
}

// --- the iteration ----------------------------------------------------------------
// the scalars of a new solve (bad: the input was invalid, nothing runs)
__global__ void k_it_start(double *sc, const unsigned *bad, unsigned *count, double tol, double max_iter)
{
    *count = 0u;
    for (int i = 0; i < kNScal; ++i) sc[i] = 0.0;
    sc[kFlush] = 2.0;
    sc[kCorr] = INFINITY;
    sc[kTol] = tol;
    sc[kMaxIter] = max_iter;
    sc[kDone] = *bad ? 1.0 : 0.0;
}

// a group's end: x += d (and the step still to go into d); kCorr = max |d| / |x|, capped at
// 1e30 (infinite if an x is not finite). pc: the current direction
template <bool Q>
__global__ void __launch_bounds__(256) k_it_flush(const CgArgs a, const float *pc)
{
    double *sc = a.scal;
    if (sc[kDone] != 0.0 || sc[kFlush] != 1.0) return;
    const bool pend = sc[kPend] != 0.0, live = sc[kDLive] != 0.0;
    const float alpha = (float)sc[kAlpha];
    KMax m;
    auto one = [&](float x, float d) {
        if (!isfinite(x)) m.s = INFINITY;
        else if (d != 0.0f) m.s = fmaxf(m.s, fminf(fabsf(d) / fmaxf(fabsf(x), 1e-37f), 1e30f));
    };
    constexpr unsigned W = Q ? 4u : 1u;
    for (unsigned c = W * (blockIdx.x * blockDim.x + threadIdx.x); c < (unsigned)a.n; c += W * gridDim.x * blockDim.x) {
        if constexpr (Q) {
            float4 d = make_float4(0.0f, 0.0f, 0.0f, 0.0f), x = ld4(a.x + c);
            if (live) d = ld4(a.d + c);
            if (pend) {
                const float4 p = ld4(pc + c);
                d = make_float4(fmaf(alpha, p.x, d.x), fmaf(alpha, p.y, d.y), fmaf(alpha, p.z, d.z), fmaf(alpha, p.w, d.w));
            }
            x = make_float4(x.x + d.x, x.y + d.y, x.z + d.z, x.w + d.w);
            st4(a.x + c, x);
            one(x.x, d.x);
            one(x.y, d.y);
            one(x.z, d.z);
            one(x.w, d.w);
        } else {
            float d = live ? a.d[c] : 0.0f;
            if (pend) d = fmaf(alpha, pc[c], d);
            const float x = a.x[c] + d;
            a.x[c] = x;
            one(x, d);
        }
    }
    double tot;
    if (grid_reduce(a, m, &tot)) {
        sc[kCorr] = tot;
        sc[kPasses] += 1.0;
        sc[kPend] = 0.0;
        sc[kDLive] = 0.0;
        if (tot < sc[kTol] || isinf(tot) || sc[kLast] != 0.0) sc[kDone] = 1.0;
    }
}

constexpr float kMgOmega = 0.8f;

// r -= alpha q, or r = b - A x after a flush; in the line rows (the first blocks) also
// x0 = omega T^-1 r, the V-cycle's first smoothing step there
template <bool Q, bool SM>
__global__ void __launch_bounds__(512, 2) k_it_residual(const CgArgs a, const LineOp L)
{
    const double *sc = a.scal;
    if (sc[kDone] != 0.0) return;
    const bool fresh = sc[kFlush] != 0.0;
    const float alpha = (float)sc[kAlpha];
    const unsigned n = (unsigned)a.n;
    auto xv = [&](unsigned i, int, int, int) { return a.x[i]; };
    if ((int)blockIdx.x < L.blocks) {
        if (fresh) {  // the block's rings first, then solved from r
            const int kt = (a.nr + 31) / 32, jl = blockIdx.x / kt, k = (blockIdx.x - jl * kt) * 32 + (threadIdx.x & 31);
            const int j = jl < L.j0 ? jl : jl - L.j0 + L.j1;
            if (k < a.nr) {
#pragma unroll 1
                for (int l = threadIdx.x >> 5; l < a.nph; l += blockDim.x >> 5) {
                    const unsigned c = ((unsigned)l * a.nth + j) * a.nr + k;
                    a.r[c] = a.b[c] - flux_one(a.nr, a.nth, a.nph, n, a.s, a.w, xv, c, k, j, l, a.x[c]);
                }
            }
            __syncthreads();
        }
        line_solve<SM>(L, a, L.x, [&](unsigned c, unsigned) { return fresh ? a.r[c] : fmaf(-alpha, a.q[c], a.r[c]); },
                       [&](unsigned c, float r) { if (!fresh) a.r[c] = r; }, [](unsigned, unsigned, float2 &) {},
                       [&](unsigned, unsigned i, float x, float2) { L.x[i] = kMgOmega * x; });
        return;
    }
    if (Q && !fresh) {  // four quads in flight per thread: the line role's registers leave few warps
        const unsigned step = 4u * (gridDim.x - L.blocks) * blockDim.x;
        for (unsigned c0 = 4u * ((blockIdx.x - L.blocks) * blockDim.x + threadIdx.x); c0 < n; c0 += 4u * step) {
            float4 q[4], r[4];
            bool on[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const unsigned c = c0 + u * step;
                int k, j, l;
                cell_ijk(c, a.nr, a.nth, a.div_nr, a.div_nth, k, j, l);
                on[u] = c < n && !L.has(j);
                if (on[u]) {
                    q[u] = ld4(a.q + c);
                    r[u] = ld4(a.r + c);
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (on[u])
                    st4(a.r + c0 + u * step, make_float4(fmaf(-alpha, q[u].x, r[u].x), fmaf(-alpha, q[u].y, r[u].y),
                                                         fmaf(-alpha, q[u].z, r[u].z), fmaf(-alpha, q[u].w, r[u].w)));
        }
        return;
    }
    for_cells<Q>(a, L.blocks, [&](unsigned c, int k, int j, int l) {
        if (L.has(j)) return;
        if constexpr (Q) {
            auto xr = [&](unsigned i, int, int, int) { return ld4(a.x + i); };
            const float4 ax = flux_quad(a.nr, a.nth, a.nph, n, a.s, a.w, xr, xv, c, k, j, l, ld4(a.x + c));
            const float4 b = ld4(a.b + c);
            st4(a.r + c, make_float4(b.x - ax.x, b.y - ax.y, b.z - ax.z, b.w - ax.w));
        } else {
            a.r[c] = fresh ? a.b[c] - flux_one(a.nr, a.nth, a.nph, n, a.s, a.w, xv, c, k, j, l, a.x[c])
                           : fmaf(-alpha, a.q[c], a.r[c]);
        }
    });
}

// d += alpha p, p = z + beta p (pc -> pn), q = A p and alpha = r.z / p.q, the new p formed at the
// stencil's points from z and the old one
template <bool Q>
__global__ void __launch_bounds__(256, Q ? 4 : 6) k_it_apply(const CgArgs a, const float *pc, float *pn)
{
    double *sc = a.scal;
    if (sc[kDone] != 0.0) return;
    const float alpha = (float)sc[kAlpha], beta = (float)sc[kBeta];
    const bool pend = sc[kPend] != 0.0, live = sc[kDLive] != 0.0, carry = beta != 0.0f;
    const float *z = a.z;
    const unsigned n = (unsigned)a.n;
    KSum pq;
    auto p1 = [&](unsigned i, int, int, int) { return carry ? fmaf(beta, pc[i], z[i]) : z[i]; };
    for_cells<Q>(a, 0u, [&](unsigned c, int k, int j, int l) {
        if constexpr (Q) {
            auto pr = [&](unsigned i, int, int, int) {
                const float4 zz = ld4(z + i);
                if (!carry) return zz;
                const float4 p = ld4(pc + i);
                return make_float4(fmaf(beta, p.x, zz.x), fmaf(beta, p.y, zz.y), fmaf(beta, p.z, zz.z),
                                   fmaf(beta, p.w, zz.w));
            };
            const float4 p = pr(c, k, j, l);
            const float4 q = flux_quad(a.nr, a.nth, a.nph, n, a.s, a.w, pr, p1, c, k, j, l, p);
            if (pend) {
                const float4 o = ld4(pc + c);
                float4 d = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (live) d = ld4(a.d + c);
                st4(a.d + c, make_float4(fmaf(alpha, o.x, d.x), fmaf(alpha, o.y, d.y), fmaf(alpha, o.z, d.z),
                                         fmaf(alpha, o.w, d.w)));
            }
            st4(pn + c, p);
            st4(a.q + c, q);
            pq.add(p.x * q.x);
            pq.add(p.y * q.y);
            pq.add(p.z * q.z);
            pq.add(p.w * q.w);
        } else {
            const float p = p1(c, k, j, l);
            const float q = flux_one(a.nr, a.nth, a.nph, n, a.s, a.w, p1, c, k, j, l, p);
            if (pend) a.d[c] = fmaf(alpha, pc[c], live ? a.d[c] : 0.0f);
            pn[c] = p;
            a.q[c] = q;
            pq.add(p * q);
        }
    });
    double tot;
    if (grid_reduce(a, BSum(pq), &tot)) {
        if (pend) sc[kDLive] = 1.0;
        sc[kAlpha] = tot > 0.0 ? sc[kRz] / tot : 0.0;
        sc[kPend] = sc[kLast] != 0.0 ? 0.0 : 1.0;  // past max_iter the new step is not taken
        if (!(tot > 0.0)) sc[kFlush] = 1.0;
    }
}

// r.z closes a step: beta, the iteration count, and whether the group ends. A group's first
// r.z is of the true residual: where that exceeds the recurrence's the directions restart.
__device__ __forceinline__ void close_step(const CgArgs &a, double tot)
{
    double *sc = a.scal;
    const double flush = sc[kFlush], old = sc[kRz];
    if (flush == 2.0) {  // the first residual
        sc[kBeta] = 0.0;
        sc[kRz0] = tot;
        if (!(tot > 0.0)) {  // x solves the system as it is (or it is not finite)
            sc[kCorr] = tot == 0.0 ? 0.0 : INFINITY;
            sc[kPasses] = 1.0;
            sc[kDone] = 1.0;
        }
        sc[kFlush] = 0.0;
    } else {
        double beta = old > 0.0 ? tot / old : 0.0;
        if (flush == 1.0) {
            sc[kRz0] = tot;
            if (tot > old) beta = 0.0;
        }
        sc[kBeta] = beta;
        sc[kIters] += 1.0;
        const bool last = sc[kIters] >= sc[kMaxIter];
        sc[kLast] = last ? 1.0 : 0.0;
        sc[kFlush] = last || !(tot > kGroupDrop * kGroupDrop * sc[kRz0]) ? 1.0 : 0.0;
    }
    sc[kRz] = tot;
}

// z = r / dg: the preconditioner of grids too small for levels
__global__ void __launch_bounds__(256) k_it_jacobi(const CgArgs a)
{
    if (a.scal[kDone] != 0.0) return;
    KSum rz;
    for_cells<false>(a, 0u, [&](unsigned c, int, int, int) {
        const float r = a.r[c], z = r * a.idg[c];
        a.z[c] = z;
        rz.add(r * z);
    });
    double tot;
    if (grid_reduce(a, BSum(rz), &tot)) close_step(a, tot);
}

// the loop's condition, at the end of its body (with a limit of its own: whatever the scalars
// say, the loop ends)
__global__ void k_it_loop(double *sc, cudaGraphConditionalHandle h)
{
    sc[kLoops] += 1.0;
    cudaGraphSetConditional(h, sc[kDone] == 0.0 && sc[kLoops] * kUnroll < sc[kMaxIter] + 4.0 * kUnroll ? 1u : 0u);
}

// the step's result, unless the input was invalid
__global__ void __launch_bounds__(256) k_it_store(const float *x, float *out, long long n, const unsigned *bad)
{
    if (*bad) return;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x)
        out[c] = x[c];
}

// --- aggregation multigrid preconditioner ---------------------------------------
// Levels coarsen by 2 in every direction longer than one cell. The coarse operator
// is the Galerkin product with piecewise-constant prolongation: the storage terms
// of an aggregate add up, and a coarse face carries the sum of the fine faces that
// cross from one aggregate into the next (faces inside an aggregate drop out), so
// every level keeps the flux form. One V-cycle per CG iteration: a damped Jacobi
// step from zero, the restricted residual, the coarser levels, the prolonged
// correction and one more Jacobi step (symmetric, so CG keeps its guarantees);
// kMgCoarseSweeps Jacobi sweeps on the coarsest level (8 against 16: 25 / 33 iterations against
// 24 / 33 in the CPU emulation). The intermediates are formed on the fly at the stencil's
// points, never stored. The levels of at most kTailCells cells run in one CTA (k_mg_tail).
constexpr int kMgCoarseSweeps = 8;
constexpr unsigned kMgCoarsest = 512;  // coarsen while a level has more cells
constexpr unsigned kTailCells = 2048;
constexpr int kTailLevels = 8;

struct MgLevel {
    int nr, nth, nph;
    FastDiv dnr, dnth;
    unsigned n;
    float *s, *w, *idg;  // operator in flux form, w [3][n]
    float *b, *x;        // right-hand side and result of the level
};

// BF16 copies of the finest level's operator. The V-cycle is a preconditioner: it
// needs a symmetric positive definite approximation of A, not A itself (CG applies
// the FP32 operator), so the finest level's restriction and prolongation read these
// (BF16 keeps FP32's exponent range; s, w and 1/dg move 10 bytes per cell, not 20).
struct HalfOp {
    const unsigned short *s, *w, *idg;
};

struct MgPair {
    MgLevel f, c;    // fine and coarse level
    int sr, st, sp;  // log2 of the aggregation factors (0 or 1)
    CgArgs cg;       // scalars and reduction scratch
    HalfOp h;        // the finest level's BF16 operator (finest pair, four-cell kernels)
    LineOp ln;       // the finest level's phi lines (finest pair)
};

#define MG_LOOP(i, N) for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < (N); i += gridDim.x * blockDim.x)

// coarse storage terms and face weights of an aggregate
__global__ void __launch_bounds__(256) k_mg_coarsen(const MgPair P)
{
    const MgLevel &F = P.f, &C = P.c;
    MG_LOOP(cc, C.n)
    {
        int K, J, L;
        cell_ijk(cc, C.nr, C.nth, C.dnr, C.dnth, K, J, L);
        float sum = 0.0f, wr = 0.0f, wt = 0.0f, wp = 0.0f;
#pragma unroll
        for (int dl = 0; dl < 2; ++dl)
#pragma unroll
            for (int dj = 0; dj < 2; ++dj)
#pragma unroll
                for (int dk = 0; dk < 2; ++dk) {
                    const int l = (L << P.sp) + dl, j = (J << P.st) + dj, k = (K << P.sr) + dk;
                    if (!((dl <= P.sp && l < F.nph) && (dj <= P.st && j < F.nth) && (dk <= P.sr && k < F.nr)))
                        continue;
                    const unsigned c = ((unsigned)l * F.nth + j) * F.nr + k;
                    sum += F.s[c];
                    if (k + 1 < F.nr && ((k + 1) >> P.sr) != (k >> P.sr)) wr += F.w[c];
                    if (j + 1 < F.nth && ((j + 1) >> P.st) != (j >> P.st)) wt += F.w[F.n + c];
                    if (F.nph > 1 && (((l + 1) % F.nph) >> P.sp) != (l >> P.sp)) wp += F.w[2 * F.n + c];
                }
        C.s[cc] = sum;
        C.w[cc] = wr;
        C.w[C.n + cc] = wt;
        C.w[2 * C.n + cc] = wp;
    }
}

// inverse diagonal of a level
__global__ void __launch_bounds__(256) k_mg_diag(const MgLevel L)
{
    const unsigned n = L.n, plane = (unsigned)L.nr * (unsigned)L.nth;
    MG_LOOP(c, n)
    {
        int k, j, l;
        cell_ijk(c, L.nr, L.nth, L.dnr, L.dnth, k, j, l);
        float d = L.s[c];
        if (k + 1 < L.nr) d += L.w[c];
        if (k > 0) d += L.w[c - 1];
        if (j + 1 < L.nth) d += L.w[n + c];
        if (j > 0) d += L.w[n + c - L.nr];
        if (L.nph > 1) {
            const unsigned ca = l > 0 ? c - plane : c + (unsigned)(L.nph - 1) * plane;
            d += L.w[2 * n + c] + L.w[2 * n + ca];
        }
        L.idg[c] = d > 0.0f ? 1.0f / d : 0.0f;
    }
}

// coarse right-hand side: the aggregate's sum of the fine residuals after the
// first smoothing step x0 (omega b / dg; the stored line solution in line rows, LINES). Eight
// threads per coarse cell, one fine cell each, summed by shuffles: the coarse levels have few
// cells and a thread that walked all eight was a chain of loads (6.5 us on 2048 coarse cells and
// 12.6 us on 131072; 3.1 and 4.5 us now).
template <bool LINES>
__global__ void __launch_bounds__(256) k_mg_down(const MgPair P)
{
    if (P.cg.scal[kDone] != 0.0) return;
    const MgLevel &F = P.f, &C = P.c;
    const float *idg = F.idg, *b = F.b;
    auto x0 = [&](unsigned i, int k, int j, int l) {
        if constexpr (LINES) {
            if (P.ln.has(j)) return P.ln.x[P.ln.at(F.nr, k, j, l)];
        }
        return kMgOmega * idg[i] * b[i];
    };
    const int sub = threadIdx.x & 7, dk = sub & 1, dj = (sub >> 1) & 1, dl = sub >> 2;
    const unsigned step = (gridDim.x * blockDim.x) >> 3;
    // (every thread of a warp walks the same number of rounds: the shuffles need them all)
    for (unsigned c0 = (blockIdx.x * blockDim.x) >> 3; c0 < C.n; c0 += step) {
        const unsigned cc = c0 + (threadIdx.x >> 3);
        float res = 0.0f;
        if (cc < C.n) {
            int K, J, L;
            cell_ijk(cc, C.nr, C.nth, C.dnr, C.dnth, K, J, L);
            const int l = (L << P.sp) + dl, j = (J << P.st) + dj, k = (K << P.sr) + dk;
            if ((dl <= P.sp && l < F.nph) && (dj <= P.st && j < F.nth) && (dk <= P.sr && k < F.nr)) {
                const unsigned c = ((unsigned)l * F.nth + j) * F.nr + k;
                res = b[c] - flux_one(F.nr, F.nth, F.nph, F.n, F.s, F.w, x0, c, k, j, l, x0(c, k, j, l));
            }
        }
        for (int o = 1; o < 8; o <<= 1) res += __shfl_xor_sync(0xffffffffu, res, o);
        if (sub == 0 && cc < C.n) C.b[cc] = res;
    }
}

// prolonged correction and the second Jacobi step of a coarse level: x = x1 + omega (b - A x1)
// / dg, x1 = omega b / dg + x_coarse[aggregate]
__global__ void __launch_bounds__(256) k_mg_up(const MgPair P)
{
    if (P.cg.scal[kDone] != 0.0) return;
    const MgLevel &F = P.f, &C = P.c;
    const float *idg = F.idg, *b = F.b, *xc = C.x;
    auto x1 = [&](unsigned i, int k, int j, int l) {
        return fmaf(kMgOmega * idg[i], b[i], xc[((unsigned)(l >> P.sp) * C.nth + (j >> P.st)) * C.nr + (k >> P.sr)]);
    };
    MG_LOOP(c, F.n)
    {
        int k, j, l;
        cell_ijk(c, F.nr, F.nth, F.dnr, F.dnth, k, j, l);
        const float vc = x1(c, k, j, l);
        F.x[c] = fmaf(kMgOmega * idg[c], b[c] - flux_one(F.nr, F.nth, F.nph, F.n, F.s, F.w, x1, c, k, j, l, vc), vc);
    }
}

// The levels of at most kTailCells cells in one CTA, everything in shared memory: one launch in
// place of two per level and the coarsest solve, whose few cells are all launch latency.
struct MgTail {
    MgLevel lv[kTailLevels];
    int n_lv;
    const double *scal;
};

size_t tail_smem(const MgTail &t)
{
    size_t n = 0;
    for (int i = 0; i < t.n_lv; ++i) n += t.lv[i].n;
    return sizeof(float) * 8 * n;
}

__global__ void __launch_bounds__(1024) k_mg_tail(const __grid_constant__ MgTail T)
{
    if (T.scal[kDone] != 0.0) return;
    extern __shared__ float sm[];
    // per level: s, w[3], 1/dg, b, x as in memory (one run of 7 n floats over the levels), then
    // n floats y: residuals
    unsigned n7 = 0;
    for (int i = 0; i < T.n_lv; ++i) n7 += 7 * T.lv[i].n;
    const float *src = T.lv[0].s;
    for (unsigned c = threadIdx.x; c < n7; c += 8 * blockDim.x) {
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (c + u * blockDim.x < n7) v[u] = src[c + u * blockDim.x];
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (c + u * blockDim.x < n7) sm[c + u * blockDim.x] = v[u];
    }
    __syncthreads();
    float *o = sm, *y = sm + n7;
    for (int i = 0; i + 1 < T.n_lv; ++i) {  // down
        const MgLevel &F = T.lv[i], &C = T.lv[i + 1];
        const float *id = o + 4 * F.n, *b = o + 5 * F.n;
        auto x0 = [&](unsigned q, int, int, int) { return kMgOmega * id[q] * b[q]; };
        for (unsigned c = threadIdx.x; c < F.n; c += blockDim.x) {
            int k, j, l;
            cell_ijk(c, F.nr, F.nth, F.dnr, F.dnth, k, j, l);
            y[c] = b[c] - flux_one(F.nr, F.nth, F.nph, F.n, o, o + F.n, x0, c, k, j, l, x0(c, 0, 0, 0));
        }
        __syncthreads();
        o += 7 * F.n;
        const int sr = F.nr > 1, st = F.nth > 1, sp = F.nph > 1;
        for (unsigned cc = threadIdx.x; cc < C.n; cc += blockDim.x) {
            int K, J, L;
            cell_ijk(cc, C.nr, C.nth, C.dnr, C.dnth, K, J, L);
            float sum = 0.0f;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int dk = q & 1, dj = (q >> 1) & 1, dl = q >> 2;
                const int k = (K << sr) + dk, j = (J << st) + dj, l = (L << sp) + dl;
                if (dk <= sr && k < F.nr && dj <= st && j < F.nth && dl <= sp && l < F.nph)
                    sum += y[((unsigned)l * F.nth + j) * F.nr + k];
            }
            o[5 * C.n + cc] = sum;
        }
        __syncthreads();
    }
    {  // the coarsest level (at most kMgCoarsest cells, one per thread): damped Jacobi sweeps from
       // zero, the row of the operator in registers, x and y in turn
        const MgLevel &L = T.lv[T.n_lv - 1];
        const unsigned n = L.n, c = threadIdx.x;
        const unsigned warps = (n + 31) / 32;
        if (threadIdx.x < 32 * warps) {
            const bool in = c < n;
            float *x = o + 6 * n;
            const float *w = o + n;
            const unsigned plane = (unsigned)L.nr * (unsigned)L.nth;
            float wv[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f}, dia = 0.0f, g = 0.0f, bb = 0.0f, v = 0.0f;
            unsigned nb[6] = {c, c, c, c, c, c};
            if (in) {
                int k, j, l;
                cell_ijk(c, L.nr, L.nth, L.dnr, L.dnth, k, j, l);
                if (k + 1 < L.nr) { wv[0] = w[c]; nb[0] = c + 1; }
                if (k > 0) { wv[1] = w[c - 1]; nb[1] = c - 1; }
                if (j + 1 < L.nth) { wv[2] = w[n + c]; nb[2] = c + L.nr; }
                if (j > 0) { wv[3] = w[n + c - L.nr]; nb[3] = c - L.nr; }
                if (L.nph > 1) {
                    nb[4] = l + 1 < L.nph ? c + plane : c - (unsigned)l * plane;
                    nb[5] = l > 0 ? c - plane : c + (unsigned)(L.nph - 1) * plane;
                    wv[4] = w[2 * n + c];
                    wv[5] = w[2 * n + nb[5]];
                }
                dia = o[c];
                g = kMgOmega * o[4 * n + c];
                bb = o[5 * n + c];
                v = g * bb;
                x[c] = v;
            }
            float *cur = x, *nxt = y;
            for (int t = 1; t < kMgCoarseSweeps; ++t) {
                asm volatile("bar.sync 1, %0;" ::"r"(32 * warps) : "memory");
                if (in) {
                    float acc = dia * v;
#pragma unroll
                    for (int q = 0; q < 6; ++q) acc = fmaf(wv[q], v - cur[nb[q]], acc);
                    v = fmaf(g, bb - acc, v);
                    nxt[c] = v;
                }
                float *h = cur;
                cur = nxt;
                nxt = h;
            }
            asm volatile("bar.sync 1, %0;" ::"r"(32 * warps) : "memory");
            if (in) x[c] = v;
        }
        __syncthreads();
    }
    for (int i = T.n_lv - 2; i >= 0; --i) {  // up
        const MgLevel &F = T.lv[i], &C = T.lv[i + 1];
        const float *xc = o + 6 * C.n;
        o -= 7 * F.n;
        const float *id = o + 4 * F.n, *b = o + 5 * F.n;
        const int sr = F.nr > 1, st = F.nth > 1, sp = F.nph > 1;
        auto x1 = [&](unsigned q, int k, int j, int l) {
            return fmaf(kMgOmega * id[q], b[q], xc[((unsigned)(l >> sp) * C.nth + (j >> st)) * C.nr + (k >> sr)]);
        };
        float *xo = i == 0 ? T.lv[0].x : o + 6 * F.n;
        for (unsigned c = threadIdx.x; c < F.n; c += blockDim.x) {
            int k, j, l;
            cell_ijk(c, F.nr, F.nth, F.dnr, F.dnth, k, j, l);
            const float vc = x1(c, k, j, l);
            xo[c] = fmaf(kMgOmega * id[c], b[c] - flux_one(F.nr, F.nth, F.nph, F.n, o, o + F.n, x1, c, k, j, l, vc), vc);
        }
        __syncthreads();
    }
    if (T.n_lv == 1)
        for (unsigned c = threadIdx.x; c < T.lv[0].n; c += blockDim.x) T.lv[0].x[c] = sm[6 * T.lv[0].n + c];
}

// k_mg_down on the finest level with nr % 4 == 0: four threads per pair of coarse cells (K0,
// K0 + 1) of one coarse row, each a four-cell quad of one of the aggregate's fine rows, summed by
// shuffles; the BF16 operator in 64-bit loads. (One thread per pair walked the four rows one
// after the other: 8.9 us on 64x32x64, where 32 CTAs held the level; 4.5 us now, and 46 us on
// 256x128x256 either way.)
__global__ void __launch_bounds__(256) k_mg_down4(const MgPair P)
{
    if (P.cg.scal[kDone] != 0.0) return;
    const MgLevel &F = P.f, &C = P.c;
    const unsigned short *idg = P.h.idg;
    const float *b = F.b;
    const LineOp &ln = P.ln;
    auto vrow = [&](unsigned c0, int k, int j, int l) {
        if (ln.has(j)) return ld4(ln.x + ln.at(F.nr, k, j, l));
        const float4 d = ldo4(idg + c0), bb = ld4(b + c0);
        return make_float4(kMgOmega * d.x * bb.x, kMgOmega * d.y * bb.y, kMgOmega * d.z * bb.z, kMgOmega * d.w * bb.w);
    };
    auto vone = [&](unsigned i, int k, int j, int l) {
        return ln.has(j) ? ln.x[ln.at(F.nr, k, j, l)] : kMgOmega * ldo1(idg + i) * b[i];
    };
    const unsigned qr = (unsigned)(F.nr / 4), nq = qr * (unsigned)C.nth * (unsigned)C.nph;
    // a warp holds 8 consecutive quads of the four rows: 128 bytes per row
    const int dj = (threadIdx.x >> 3) & 1, dl = (threadIdx.x >> 4) & 1;
    const unsigned step = (gridDim.x * blockDim.x) >> 2;
    for (unsigned t0 = (blockIdx.x * blockDim.x + (threadIdx.x & ~31u)) >> 2; t0 < nq; t0 += step) {
        const unsigned t = t0 + (threadIdx.x & 7);
        float lo = 0.0f, hi = 0.0f;
        unsigned cc = 0u;
        if (t < nq) {
            const unsigned rest = t / qr;
            const int m = (int)(t - rest * qr);
            const int J = (int)(rest % (unsigned)C.nth), L = (int)(rest / (unsigned)C.nth);
            const int k = 4 * m, l = (L << P.sp) + dl, j = (J << P.st) + dj;
            cc = ((unsigned)L * C.nth + J) * C.nr + 2 * m;
            if (dl <= P.sp && l < F.nph && dj <= P.st && j < F.nth) {
                const unsigned c = ((unsigned)l * F.nth + j) * F.nr + k;
                const float4 vc = vrow(c, k, j, l), bb = ld4(b + c);
                const float4 ax = flux_quad(F.nr, F.nth, F.nph, F.n, P.h.s, P.h.w, vrow, vone, c, k, j, l, vc);
                lo = (bb.x - ax.x) + (bb.y - ax.y);
                hi = (bb.z - ax.z) + (bb.w - ax.w);
            }
        }
        for (int o = 8; o < 32; o <<= 1) {
            lo += __shfl_xor_sync(0xffffffffu, lo, o);
            hi += __shfl_xor_sync(0xffffffffu, hi, o);
        }
        if (t < nq && (threadIdx.x & 24) == 0) *reinterpret_cast<float2 *>(C.b + cc) = make_float2(lo, hi);
    }
}

// The finest level's prolongation and second smoothing step, z = M^-1 r, and r.z, which closes
// the CG step: as k_mg_up, four cells per thread and the BF16 operator where nr % 4 == 0 (Q). Of
// the line rows it leaves x1 in z and the residual b - A x1 to k_line_post. (Residual and line
// solve in blocks of their own beside the streaming ones: 140 us on 256x128x256 against 44 + 22.)
template <bool Q>
__global__ void __launch_bounds__(256, Q ? 5 : 6) k_mg_up0(const MgPair P)
{
    if (P.cg.scal[kDone] != 0.0) return;
    const MgLevel &F = P.f, &C = P.c;
    using T = typename std::conditional<Q, unsigned short, float>::type;
    const T *os, *ow, *idg;
    if constexpr (Q) {
        os = P.h.s;
        ow = P.h.w;
        idg = P.h.idg;
    } else {
        os = F.s;
        ow = F.w;
        idg = F.idg;
    }
    const float *b = F.b, *xc = C.x;
    const int sr = P.sr, st = P.st, sp = P.sp, cnr = C.nr, cnth = C.nth;
    const LineOp &ln = P.ln;
    auto crow = [=](int j, int l) { return ((unsigned)(l >> sp) * cnth + (j >> st)) * cnr; };
    auto vone = [&](unsigned i, int k, int j, int l) {
        const float cv = xc[crow(j, l) + (k >> sr)];
        return ln.has(j) ? ln.x[ln.at(F.nr, k, j, l)] + cv : fmaf(kMgOmega * ldo1(idg + i), b[i], cv);
    };
    KSum rz;
    for_cells<Q>(P.cg, 0u, [&](unsigned c, int k, int j, int l) {
        if constexpr (Q) {
            auto vrow = [&](unsigned c0, int k, int j, int l) {
                const float2 x2 = *reinterpret_cast<const float2 *>(xc + crow(j, l) + (k >> 1));
                if (ln.has(j)) {
                    const float4 x0 = ld4(ln.x + ln.at(F.nr, k, j, l));
                    return make_float4(x0.x + x2.x, x0.y + x2.x, x0.z + x2.y, x0.w + x2.y);
                }
                const float4 d = ldo4(idg + c0), bb = ld4(b + c0);
                return make_float4(fmaf(kMgOmega * d.x, bb.x, x2.x), fmaf(kMgOmega * d.y, bb.y, x2.x),
                                   fmaf(kMgOmega * d.z, bb.z, x2.y), fmaf(kMgOmega * d.w, bb.w, x2.y));
            };
            const float4 vc = vrow(c, k, j, l);
            const float4 ax = flux_quad(F.nr, F.nth, F.nph, F.n, os, ow, vrow, vone, c, k, j, l, vc);
            const float4 bb = ld4(b + c);
            const float4 res = make_float4(bb.x - ax.x, bb.y - ax.y, bb.z - ax.z, bb.w - ax.w);
            if (ln.has(j)) {
                st4(F.x + c, vc);
                st4(ln.res + ln.at(F.nr, k, j, l), res);
                return;
            }
            const float4 d = ldo4(idg + c);
            const float4 z = make_float4(fmaf(kMgOmega * d.x, res.x, vc.x), fmaf(kMgOmega * d.y, res.y, vc.y),
                                         fmaf(kMgOmega * d.z, res.z, vc.z), fmaf(kMgOmega * d.w, res.w, vc.w));
            st4(F.x + c, z);
            rz.add(bb.x * z.x);
            rz.add(bb.y * z.y);
            rz.add(bb.z * z.z);
            rz.add(bb.w * z.w);
        } else {
            const float vc = vone(c, k, j, l);
            const float res = b[c] - flux_one(F.nr, F.nth, F.nph, F.n, os, ow, vone, c, k, j, l, vc);
            if (ln.has(j)) {
                F.x[c] = vc;
                ln.res[ln.at(F.nr, k, j, l)] = res;
                return;
            }
            const float z = fmaf(kMgOmega * ldo1(idg + c), res, vc);
            F.x[c] = z;
            rz.add(b[c] * z);
        }
    });
    if (ln.nl > 0) {  // k_line_post sums these partials with its own
        const BSum t = block_reduce(BSum(rz));
        if (threadIdx.x == 0) P.cg.part[blockIdx.x] = t.value();
        return;
    }
    double tot;
    if (grid_reduce(P.cg, BSum(rz), &tot)) close_step(P.cg, tot);
}

// z = x1 + omega T^-1 (b - A x1) of the line rows, and their share of r.z (after the partials of
// k_mg_up0, rows_partials of them)
template <bool SM>
__global__ void __launch_bounds__(512, 2) k_line_post(const CgArgs a, const LineOp L, int rows_partials)
{
    if (a.scal[kDone] != 0.0) return;
    KSum rz;
    line_solve<SM>(L, a, L.res, [&](unsigned, unsigned i) { return L.res[i]; }, [](unsigned, float) {},
                   [&](unsigned c, unsigned, float2 &e) { e = make_float2(a.z[c], a.r[c]); },
                   [&](unsigned c, unsigned, float x, float2 e) {
                       const float z = fmaf(kMgOmega, x, e.x);
                       a.z[c] = z;
                       rz.add(e.y * z);
                   });
    double tot;
    if (grid_reduce(a, BSum(rz), &tot, rows_partials)) close_step(a, tot);
}

#undef MG_LOOP

int rosseland_nodes(const CtxInfo &in, const std::vector<double> &t_nodes, double *kr_host, float *lkr_dev,
                    cudaStream_t st, std::string &err)
{
    const int n = (int)t_nodes.size();
    const int n_t = in.n_t > 0 ? in.n_t : 1;
    const double *kap_h = in.n_t > 0 ? in.kappa_t_h : in.kappa_h;
    double *tn = nullptr, *nu = nullptr, *ka = nullptr, *tg = nullptr, *kr = nullptr;
    bool ok = cudaMalloc(&tn, sizeof(double) * n) == cudaSuccess &&
              cudaMalloc(&nu, sizeof(double) * in.n_nu) == cudaSuccess &&
              cudaMalloc(&ka, sizeof(double) * in.n_nu * n_t) == cudaSuccess &&
              cudaMalloc(&tg, sizeof(double) * n_t) == cudaSuccess && cudaMalloc(&kr, sizeof(double) * n) == cudaSuccess;
    ok = ok && cudaMemcpyAsync(tn, t_nodes.data(), sizeof(double) * n, cudaMemcpyHostToDevice, st) == cudaSuccess &&
         cudaMemcpyAsync(nu, in.nu_h, sizeof(double) * in.n_nu, cudaMemcpyHostToDevice, st) == cudaSuccess &&
         cudaMemcpyAsync(ka, kap_h, sizeof(double) * in.n_nu * n_t, cudaMemcpyHostToDevice, st) == cudaSuccess;
    if (ok && in.n_t > 0)
        ok = cudaMemcpyAsync(tg, in.t_grid_h, sizeof(double) * n_t, cudaMemcpyHostToDevice, st) == cudaSuccess;
    if (ok) {
        k_rosseland<<<(n + 7) / 8, 256, 0, st>>>(n, tn, in.n_nu, nu, ka, n_t, tg, kr, lkr_dev);
        ok = cudaGetLastError() == cudaSuccess;
    }
    if (ok && kr_host) ok = cudaMemcpyAsync(kr_host, kr, sizeof(double) * n, cudaMemcpyDeviceToHost, st) == cudaSuccess;
    ok = ok && cudaStreamSynchronize(st) == cudaSuccess;
    if (!ok) err = std::string("Rosseland-mean kernel: ") + cudaGetErrorString(cudaGetLastError());
    cudaFree(tn);
    cudaFree(nu);
    cudaFree(ka);
    cudaFree(tg);
    cudaFree(kr);
    return ok ? RT_OK : RT_ERR_CUDA;
}

// the axis tables of FldGeo, in units of the outer radius, computed in FP64
std::vector<float> geometry_tables(const CtxInfo &in)
{
    const int nr = in.nr, nth = in.ntheta, nph = in.nphi;
    const double *ri = in.r_if_h, *ti = in.theta_if_h, *pi = in.phi_if_h;
    const double L = ri[nr];
    std::vector<float> h;
    auto rc = [&](int k) { return 0.5 * (ri[k] + ri[k + 1]) / L; };
    auto thc = [&](int j) { return 0.5 * (ti[j] + ti[j + 1]); };
    auto phc = [&](int l) { return 0.5 * (pi[l] + pi[l + 1]); };
    for (int k = 0; k <= nr; ++k) h.push_back((float)(ri[k] / L));
    for (int k = 0; k < nr; ++k) h.push_back((float)rc(k));
    for (int k = 0; k < nr; ++k) h.push_back(k + 1 < nr ? (float)(rc(k + 1) - rc(k)) : 0.0f);
    for (int k = 0; k < nr; ++k) {
        const double a = ri[k] / L, b = ri[k + 1] / L;
        h.push_back((float)((b - a) * (a * a + a * b + b * b) / 3.0));
    }
    for (int k = 0; k < nr; ++k) {
        const double a = ri[k] / L, b = ri[k + 1] / L;
        h.push_back((float)(0.5 * (b - a) * (a + b)));
    }
    for (int j = 0; j <= nth; ++j) h.push_back((float)sin(ti[j]));
    for (int j = 0; j < nth; ++j) h.push_back(j + 1 < nth ? (float)(thc(j + 1) - thc(j)) : 0.0f);
    for (int j = 0; j < nth; ++j) h.push_back((float)sin(thc(j)));
    for (int j = 0; j < nth; ++j) h.push_back((float)(cos(ti[j]) - cos(ti[j + 1])));
    for (int j = 0; j < nth; ++j) h.push_back((float)(ti[j + 1] - ti[j]));
    for (int l = 0; l < nph; ++l) h.push_back((float)(pi[l + 1] - pi[l]));
    for (int l = 0; l < nph; ++l) {
        double d = fmod(phc((l + 1) % nph) - phc(l), 2.0 * kPi);
        if (d < 0.0) d += 2.0 * kPi;
        h.push_back((float)d);
    }
    return h;
}

FldGeo geo_view(const float *gp, int nr, int nth, int nph)
{
    FldGeo g;
    g.rif = gp; gp += nr + 1;
    g.rc = gp; gp += nr;
    g.drc = gp; gp += nr;
    g.d3 = gp; gp += nr;
    g.dr2 = gp; gp += nr;
    g.sin_thif = gp; gp += nth + 1;
    g.dthc = gp; gp += nth;
    g.sin_thc = gp; gp += nth;
    g.dcos = gp; gp += nth;
    g.dth = gp; gp += nth;
    g.dph = gp; gp += nph;
    g.dphc = gp;
    g.nr = nr;
    g.nth = nth;
    g.nph = nph;
    g.div_nr = FastDiv::make((unsigned)nr);
    g.div_nth = FastDiv::make((unsigned)nth);
    return g;
}

// largest dynamic shared memory of the step's kernels: the line kernels' 32 rings of
// kLineSmemPhi cells; a tail of 2048 + 1024 + 512 cells (one direction only) takes 112 KB
constexpr size_t kMaxFldSmem = sizeof(float) * 32 * kLineSmemPhi;

// segments a ring of nph cells is cut into (k_line_*: one warp each)
int line_segments(int nph) { return std::max(4, std::min(kLineMaxSeg, nph / 8)); }

// share of the diagonal the phi faces of row j hold where D is uniform, at the middle radius
std::vector<double> phi_shares(const CtxInfo &in)
{
    const int nth = in.ntheta, nph = in.nphi, k = in.nr / 2;
    const double *ri = in.r_if_h, *ti = in.theta_if_h;
    const double dph = (in.phi_if_h[nph] - in.phi_if_h[0]) / nph;
    const double rc = 0.5 * (ri[k] + ri[k + 1]), dr = ri[k + 1] - ri[k], dr2 = dr * rc;
    std::vector<double> share(nth);
    for (int j = 0; j < nth; ++j) {
        const double th = 0.5 * (ti[j] + ti[j + 1]), dth = ti[j + 1] - ti[j];
        const double p = 2.0 * dth * dr2 / (rc * fabs(sin(th)) * dph);
        const double t = dph * (sin(ti[j]) + sin(ti[j + 1])) * dr2 / (rc * dth);
        const double r = in.nr > 1 ? 2.0 * dph * (cos(ti[j]) - cos(ti[j + 1])) * rc * rc / dr : 0.0;
        share[j] = p / (p + t + r);
    }
    return share;
}

double radiation_constant()
{
    const double sigma = 2.0 * pow(kPi, 5) * pow(kKB, 4) / (15.0 * kH * kH * kH * kC * kC);
    return 4.0 * sigma / kC;
}

}  // namespace

void fld_free(FldState *s)
{
    if (!s) return;
    cudaFree(s->buf);
    cudaFree(s->mg_buf);
    cudaFree(s->line_buf);
    cudaFree(s->part);
    cudaFree(s->scal);
    cudaFree(s->bad);
    cudaFree(s->count);
    cudaFree(s->geo);
    cudaFree(s->lkr);
    if (s->loop) cudaGraphExecDestroy(s->loop);
    cudaFreeHost(s->scal_h);
    if (s->ev_in) cudaEventDestroy(s->ev_in);
    if (s->gs) cudaStreamDestroy(s->gs);
    delete s;
}

}  // namespace rt

using namespace rt;

extern "C" {

int rt_rosseland_mean_opacity(rt_ctx *ctx, double t, double *kappa_r)
{
    if (!ctx || !kappa_r) return RT_ERR_INVALID_ARG;
    CtxInfo in;
    ctx_info(ctx, &in);
    if (!in.configured) return ctx_fail(ctx, RT_ERR_NOT_CONFIGURED, "call rt_set_star and rt_set_opacity_table first");
    if (!(t > 0.0) || !isfinite(t)) return ctx_fail(ctx, RT_ERR_INVALID_ARG, "t must be finite and > 0");
    if (cudaSetDevice(in.dev) != cudaSuccess) return ctx_fail(ctx, RT_ERR_CUDA, "cudaSetDevice");
    std::string err;
    const int rc = rosseland_nodes(in, std::vector<double>{t}, kappa_r, nullptr, in.stream, err);
    return rc == RT_OK ? RT_OK : ctx_fail(ctx, rc, err);
}

int rt_fld_step(rt_ctx *ctx, const float *rho, const float *t_gas, const float *q_abs, const float *e_old,
                float *e_new, double dt, double c_v, double t_bg, double tol, int max_iter, rt_fld_stats *stats)
{
    if (!ctx) return RT_ERR_INVALID_ARG;
    CtxInfo in;
    ctx_info(ctx, &in);
    if (!in.configured) return ctx_fail(ctx, RT_ERR_NOT_CONFIGURED, "call rt_set_star and rt_set_opacity_table first");
    if (!rho || !t_gas || !q_abs || !e_old || !e_new) return ctx_fail(ctx, RT_ERR_INVALID_ARG, "NULL field pointer");
    if (!(dt > 0.0) || !(c_v >= 0.0) || !isfinite(c_v) || !(t_bg >= 0.0) || !isfinite(t_bg) || !(tol > 0.0) ||
        max_iter < 1)
        return ctx_fail(ctx, RT_ERR_INVALID_ARG, "need dt > 0, finite c_v >= 0 and t_bg >= 0, tol > 0, max_iter >= 1");
    if (e_new == e_old) return ctx_fail(ctx, RT_ERR_INVALID_ARG, "e_new must not alias e_old");
    if (in.ncells >= (1LL << 31) - 1) return ctx_fail(ctx, RT_ERR_INVALID_ARG, "FLD step needs fewer than 2^31 cells");
    if (cudaSetDevice(in.dev) != cudaSuccess) return ctx_fail(ctx, RT_ERR_CUDA, "cudaSetDevice");
    FldState *&fs = ctx_fld(ctx);
    if (!fs) fs = new FldState();
    if (!fs->gs) {
        if (cudaStreamCreateWithFlags(&fs->gs, cudaStreamNonBlocking) != cudaSuccess ||
            cudaEventCreateWithFlags(&fs->ev_in, cudaEventDisableTiming) != cudaSuccess) {
            cudaGetLastError();
            return ctx_fail(ctx, RT_ERR_CUDA, "FLD stream");
        }
    }
    // everything below runs on the private stream, after the context stream's work so far
    if (cudaEventRecord(fs->ev_in, in.stream) != cudaSuccess || cudaStreamWaitEvent(fs->gs, fs->ev_in, 0) != cudaSuccess)
        return ctx_fail(ctx, RT_ERR_CUDA, "FLD stream order");
    cudaStream_t st = fs->gs;
    const long long n = in.ncells;
    const int nr = in.nr, nth = in.ntheta, nph = in.nphi;
    int nsm = 0;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, in.dev);
    if (nsm < 1) nsm = 1;
    const int grid = (int)std::max(1LL, std::min<long long>((n + 255) / 256, 8LL * nsm));
    if (fs->cap < n) {
        cudaFree(fs->buf);
        fs->buf = nullptr;
        fs->cap = 0;
        if (cudaMalloc(&fs->buf, sizeof(float) * (14 * (size_t)n + (5 * (size_t)n + 1) / 2)) != cudaSuccess) {
            cudaGetLastError();
            return ctx_fail(ctx, RT_ERR_NO_MEMORY, "FLD workspace");
        }
        fs->cap = n;
    }
    // at most 16 resident CTAs per SM (128 threads and more), and one CTA per 32 rings before them
    const int grid_max = 16 * nsm + nth * ((nr + 31) / 32);
    if (fs->part_cap < grid_max) {
        cudaFree(fs->part);
        fs->part = nullptr;
        fs->part_cap = 0;
        if (cudaMalloc(&fs->part, sizeof(double) * grid_max) != cudaSuccess) {
            cudaGetLastError();
            return ctx_fail(ctx, RT_ERR_NO_MEMORY, "FLD partials");
        }
        fs->part_cap = grid_max;
    }
    if (!fs->scal) {
        if (cudaMalloc(&fs->scal, sizeof(double) * kNScal) != cudaSuccess ||
            cudaMalloc(&fs->bad, sizeof(unsigned)) != cudaSuccess ||
            cudaMalloc(&fs->count, sizeof(unsigned)) != cudaSuccess ||
            cudaMallocHost(&fs->scal_h, sizeof(double) * (kNScal + 1)) != cudaSuccess ||
            cudaMemset(fs->count, 0, sizeof(unsigned)) != cudaSuccess) {
            cudaGetLastError();
            cudaFree(fs->scal);
            cudaFree(fs->bad);
            cudaFree(fs->count);
            cudaFreeHost(fs->scal_h);
            fs->scal_h = nullptr;
            fs->scal = nullptr;
            fs->bad = fs->count = nullptr;
            return ctx_fail(ctx, RT_ERR_NO_MEMORY, "FLD scalars");
        }
    }
    if (!fs->geo) {
        const std::vector<float> h = geometry_tables(in);
        if (cudaMalloc(&fs->geo, sizeof(float) * h.size()) != cudaSuccess ||
            cudaMemcpy(fs->geo, h.data(), sizeof(float) * h.size(), cudaMemcpyHostToDevice) != cudaSuccess) {
            cudaGetLastError();
            cudaFree(fs->geo);
            fs->geo = nullptr;
            return ctx_fail(ctx, RT_ERR_CUDA, "FLD geometry tables");
        }
    }
    if (fs->mg_dims.empty()) {  // multigrid levels: halve every direction longer than one cell
        int a = nr, b2 = nth, c3 = nph;
        size_t coarse = 0;
        fs->mg_dims = {a, b2, c3};
        while ((unsigned long long)a * b2 * c3 > kMgCoarsest && (a > 1 || b2 > 1 || c3 > 1)) {
            a = a > 1 ? (a + 1) / 2 : 1;
            b2 = b2 > 1 ? (b2 + 1) / 2 : 1;
            c3 = c3 > 1 ? (c3 + 1) / 2 : 1;
            fs->mg_dims.insert(fs->mg_dims.end(), {a, b2, c3});
            coarse += (size_t)a * b2 * c3;
        }
        if (coarse > 0 && cudaMalloc(&fs->mg_buf, sizeof(float) * 7 * coarse) != cudaSuccess) {
            cudaGetLastError();
            fs->mg_dims.clear();
            return ctx_fail(ctx, RT_ERR_NO_MEMORY, "FLD multigrid levels");
        }
    }
    if (!fs->lines_set) {  // the rows smoothed by phi lines: a run at each theta end (LineOp)
        fs->line_j0 = 0;
        fs->line_j1 = nth;
        if (fs->mg_dims.size() > 3 && nph >= kLineMinPhi) {
            const std::vector<double> share = phi_shares(in);
            while (fs->line_j0 < nth && share[fs->line_j0] > kLineShare) ++fs->line_j0;
            while (fs->line_j1 > fs->line_j0 && share[fs->line_j1 - 1] > kLineShare) --fs->line_j1;
        }
        const size_t rows = (size_t)(fs->line_j0 + nth - fs->line_j1) * nr;
        const size_t S = line_segments(nph);
        if (rows > 0 && cudaMalloc(&fs->line_buf, sizeof(float) * rows * (5 * (size_t)nph + S * S)) != cudaSuccess) {
            cudaGetLastError();
            return ctx_fail(ctx, RT_ERR_NO_MEMORY, "FLD line smoother");
        }
        fs->lines_set = true;
    }
    if (!fs->lkr_valid || fs->lkr_fp != in.table_fingerprint) {
        if (!fs->lkr && cudaMalloc(&fs->lkr, sizeof(float) * kRossNodes) != cudaSuccess) {
            cudaGetLastError();
            return ctx_fail(ctx, RT_ERR_NO_MEMORY, "Rosseland table");
        }
        std::vector<double> tn(kRossNodes);
        for (int i = 0; i < kRossNodes; ++i) tn[i] = exp(kRossLnLo + (kRossLnHi - kRossLnLo) * i / (kRossNodes - 1));
        std::string err;
        const int rc = rosseland_nodes(in, tn, nullptr, fs->lkr, st, err);
        if (rc != RT_OK) return ctx_fail(ctx, rc, err);
        fs->lkr_fp = in.table_fingerprint;
        fs->lkr_valid = true;
    }
    const FldGeo g = geo_view(fs->geo, nr, nth, nph);
    const double L = in.r_if_h[nr];
    const double a_rad = radiation_constant();
    float *F = fs->buf, *tc = F + n, *b0 = tc + n, *w = b0 + n, *sv = w + 3 * n, *idg = sv + n, *b = idg + n;
    float *d = b + n, *r = d + n, *p = r + n, *q = p + n, *z = q + n;
    float *x = tc, *pbuf[2] = {p, F};  // tc and F are free once the face kernel has run
    unsigned short *hs = reinterpret_cast<unsigned short *>(z + n), *hw = hs + n, *hidg = hw + 3 * n;

    FldCellArgs ca;
    ca.g = g;
    ca.rho = rho;
    ca.t = t_gas;
    ca.q = q_abs;
    ca.e = e_old;
    ca.lkr = fs->lkr;
    ca.y0 = (float)kRossLnLo;
    ca.inv_dy = (float)((kRossNodes - 1) / (kRossLnHi - kRossLnLo));
    ca.L = (float)L;
    ca.c_v = (float)c_v;
    ca.four_a = (float)(4.0 * a_rad);
    ca.inv_tau = (float)(L / (kC * dt));
    ca.q_scale = (float)(L / kC);
    ca.F = F;
    ca.tc = tc;
    ca.b0 = b0;
    ca.bad = fs->bad;
    ca.n = n;
    FldFaceArgs fa;
    fa.g = g;
    fa.F = F;
    fa.tc = tc;
    fa.b0 = b0;
    fa.e_bg = (float)(a_rad * pow(t_bg, 4));
    fa.w = w;
    fa.s = sv;
    fa.idg = idg;
    fa.b = b;
    fa.hs = hs;
    fa.hw = hw;
    fa.hidg = hidg;
    fa.e = e_old;
    fa.x = x;
    fa.n = n;
    CgArgs cg;
    cg.nr = nr;
    cg.nth = nth;
    cg.nph = nph;
    cg.div_nr = g.div_nr;
    cg.div_nth = g.div_nth;
    cg.n = n;
    cg.w = w;
    cg.s = sv;
    cg.idg = idg;
    cg.b = b;
    cg.x = x;
    cg.d = d;
    cg.r = r;
    cg.q = q;
    cg.z = z;
    cg.part = fs->part;
    cg.scal = fs->scal;
    cg.count = fs->count;

    // multigrid levels and pairs (level 0: the fine operator, b = r, x = z)
    const int n_lv = (int)fs->mg_dims.size() / 3;
    const bool use_mg = n_lv > 1;
    std::vector<MgLevel> lv(n_lv);
    {
        float *cursor = fs->mg_buf;
        for (int i = 0; i < n_lv; ++i) {
            MgLevel &L = lv[i];
            L.nr = fs->mg_dims[3 * i];
            L.nth = fs->mg_dims[3 * i + 1];
            L.nph = fs->mg_dims[3 * i + 2];
            L.dnr = FastDiv::make((unsigned)L.nr);
            L.dnth = FastDiv::make((unsigned)L.nth);
            L.n = (unsigned)L.nr * (unsigned)L.nth * (unsigned)L.nph;
            if (i == 0) {
                L.s = sv;
                L.w = w;
                L.idg = idg;
                L.b = r;
                L.x = z;
            } else {
                L.s = cursor;
                L.w = L.s + L.n;
                L.idg = L.w + 3 * (size_t)L.n;
                L.b = L.idg + L.n;
                L.x = L.b + L.n;
                cursor = L.x + L.n;
            }
        }
    }
    std::vector<MgPair> pairs(n_lv > 0 ? n_lv - 1 : 0);
    for (int i = 0; i + 1 < n_lv; ++i) {
        pairs[i].f = lv[i];
        pairs[i].c = lv[i + 1];
        pairs[i].sr = lv[i].nr > 1 ? 1 : 0;
        pairs[i].st = lv[i].nth > 1 ? 1 : 0;
        pairs[i].sp = lv[i].nph > 1 ? 1 : 0;
        pairs[i].cg = cg;
        pairs[i].h = HalfOp{hs, hw, hidg};
    }
    // phi lines of the finest level
    LineOp ln{0, nth, 0, 0, 0, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
    const int nl = fs->line_j0 + nth - fs->line_j1;
    const bool lines = use_mg && nl > 0;
    if (lines) {
        const size_t rows = (size_t)nl * nr;
        ln.j0 = fs->line_j0;
        ln.j1 = fs->line_j1;
        ln.nl = nl;
        ln.seg = line_segments(nph);
        ln.blocks = nl * ((nr + 31) / 32);
        ln.m = fs->line_buf;
        ln.vl = ln.m + rows * nph;
        ln.vr = ln.vl + rows * nph;
        ln.x = ln.vr + rows * nph;
        ln.res = ln.x + rows * nph;
        ln.inv = ln.res + rows * nph;
    }
    if (use_mg) pairs[0].ln = ln;
    // the levels of the one-CTA tail
    MgTail tail{};
    int t0 = n_lv;
    if (use_mg) {
        for (t0 = 1; lv[t0].n > kTailCells || n_lv - t0 > kTailLevels;) ++t0;
        for (int i = t0; i < n_lv; ++i) tail.lv[tail.n_lv++] = lv[i];
        tail.scal = fs->scal;
    }

    // grids of one full wave: the CTAs resident per SM (from each kernel's registers) times the
    // SM count, capped by the work
    const bool quads = nr % 4 == 0;  // four cells per thread where a ray holds a multiple of four
    auto wave = [&](const void *kern, int threads, size_t smem, long long work) {
        int per_sm = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem) != cudaSuccess || per_sm < 1)
            per_sm = 1;
        return (int)std::max(1LL, std::min<long long>((work + threads - 1) / threads, (long long)per_sm * nsm));
    };
    const long long work = quads ? n / 4 : n;
    const int t_line = lines ? 32 * ln.seg : 256;
    const bool ring_sm = nph <= kLineSmemPhi;
    const size_t sm_line = lines && ring_sm ? sizeof(float) * t_line * (size_t)(nph / ln.seg) : 0;
    const size_t sm_tail = use_mg ? tail_smem(tail) : 0;
    using LevelFn = void (*)(const MgPair);
    const LevelFn up0 = quads ? k_mg_up0<true> : k_mg_up0<false>;
    const LevelFn down0 = quads ? k_mg_down4 : lines ? k_mg_down<true> : k_mg_down<false>;
    const auto residual = quads ? (ring_sm ? k_it_residual<true, true> : k_it_residual<true, false>)
                                : (ring_sm ? k_it_residual<false, true> : k_it_residual<false, false>);
    const auto line_post = ring_sm ? k_line_post<true> : k_line_post<false>;
    const auto apply = quads ? k_it_apply<true> : k_it_apply<false>;
    const auto flush = quads ? k_it_flush<true> : k_it_flush<false>;
    // (one limit for all contexts: another thread's smaller step must not lower it; the kernels'
    // static part, at most 6.8 KB, counts towards the 48 KB a launch has without asking)
    auto big_smem = [](const void *kern, size_t bytes) {
        return bytes <= 40 * 1024 ||
               (bytes <= kMaxFldSmem && cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                             (int)kMaxFldSmem) == cudaSuccess);
    };
    if (!big_smem((const void *)residual, sm_line) || !big_smem((const void *)line_post, sm_line) ||
        !big_smem((const void *)k_mg_tail, sm_tail))
        return ctx_fail(ctx, RT_ERR_CUDA, "FLD shared memory");
    const int g_res = ln.blocks + wave((const void *)residual, t_line, sm_line, work);
    const int g_up0 = wave((const void *)up0, 256, 0, work);
    const int g_app = wave((const void *)apply, 256, 0, work), g_flu = wave((const void *)flush, 256, 0, work);
    const int g_jac = wave((const void *)k_it_jacobi, 256, 0, n);
    std::vector<int> g_down(n_lv, 1), g_up(n_lv, 1);
    for (int i = 0; i + 1 < n_lv; ++i) {
        g_down[i] = wave(i == 0 ? (const void *)down0 : (const void *)k_mg_down<false>, 256, 0,
                         i == 0 && quads ? 2LL * lv[1].n : 8LL * lv[i + 1].n);
        g_up[i] = wave((const void *)k_mg_up, 256, 0, lv[i].n);
    }
    // one iteration; p goes from pbuf[i & 1] to the other buffer
    auto iteration = [&](int i) {
        const float *pc = pbuf[i & 1];
        flush<<<g_flu, 256, 0, st>>>(cg, pc);
        residual<<<g_res, t_line, sm_line, st>>>(cg, ln);
        if (use_mg) {
            down0<<<g_down[0], 256, 0, st>>>(pairs[0]);
            for (int v = 1; v < t0; ++v) k_mg_down<false><<<g_down[v], 256, 0, st>>>(pairs[v]);
            k_mg_tail<<<1, 1024, sm_tail, st>>>(tail);
            for (int v = t0 - 1; v >= 1; --v) k_mg_up<<<g_up[v], 256, 0, st>>>(pairs[v]);
            up0<<<g_up0, 256, 0, st>>>(pairs[0]);
            if (lines) line_post<<<ln.blocks, t_line, sm_line, st>>>(cg, ln, g_up0);
        } else {
            k_it_jacobi<<<g_jac, 256, 0, st>>>(cg);
        }
        apply<<<g_app, 256, 0, st>>>(cg, pc, pbuf[(i + 1) & 1]);
    };
    if (!fs->loop && !fs->no_graph) {  // the loop's graph
        // (none of its launches may be refused: the kernel would be missing from the body)
        bool fit = launch_fits((const void *)flush, 256, 0) && launch_fits((const void *)residual, t_line, sm_line) &&
                   launch_fits((const void *)apply, 256, 0) && launch_fits((const void *)k_it_loop, 1, 0);
        if (use_mg)
            fit = fit && launch_fits((const void *)down0, 256, 0) && launch_fits((const void *)k_mg_down<false>, 256, 0) &&
                  launch_fits((const void *)k_mg_tail, 1024, sm_tail) && launch_fits((const void *)k_mg_up, 256, 0) &&
                  launch_fits((const void *)up0, 256, 0) &&
                  (!lines || launch_fits((const void *)line_post, t_line, sm_line));
        else
            fit = fit && launch_fits((const void *)k_it_jacobi, 256, 0);
        if (!fit) return ctx_fail(ctx, RT_ERR_CUDA, "FLD step: a kernel of the loop does not fit its launch");
        cudaGetLastError();  // (an older call's error is none of these launches')
        cudaError_t refused = cudaSuccess;
        cudaGraph_t graph = nullptr, body = nullptr, end = nullptr;
        cudaGraphConditionalHandle h{};
        cudaGraphNode_t node = nullptr;
        cudaGraphNodeParams par = {};
        bool cap = cudaGraphCreate(&graph, 0) == cudaSuccess &&
                   cudaGraphConditionalHandleCreate(&h, graph, 1, cudaGraphCondAssignDefault) == cudaSuccess;
        if (cap) {
            par.type = cudaGraphNodeTypeConditional;
            par.conditional.handle = h;
            par.conditional.type = cudaGraphCondTypeWhile;
            par.conditional.size = 1;
            cap = cudaGraphAddNode(&node, graph, nullptr, nullptr, 0, &par) == cudaSuccess;
        }
        if (cap) {
            body = par.conditional.phGraph_out[0];
            cap = cudaStreamBeginCaptureToGraph(st, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal) ==
                  cudaSuccess;
        }
        if (cap) {
            for (int i = 0; i < kUnroll; ++i) iteration(i);
            k_it_loop<<<1, 1, 0, st>>>(fs->scal, h);
            refused = cudaGetLastError();
            cap = cudaStreamEndCapture(st, &end) == cudaSuccess && refused == cudaSuccess;
        }
        cap = cap && cudaGraphInstantiate(&fs->loop, graph, 0) == cudaSuccess;
        if (graph) cudaGraphDestroy(graph);
        if (!cap) {
            cudaGetLastError();
            fs->loop = nullptr;
            // (the host-driven loop would have the same launch refused)
            if (refused != cudaSuccess)
                return ctx_fail(ctx, RT_ERR_CUDA, std::string("FLD loop: ") + cudaGetErrorString(refused));
            fs->no_graph = true;
        }
    }

    auto sync_read = [&]() {
        return cudaGetLastError() == cudaSuccess &&
               cudaMemcpyAsync(fs->scal_h, fs->scal, sizeof(double) * kNScal, cudaMemcpyDeviceToHost, st) == cudaSuccess &&
               cudaMemcpyAsync(fs->scal_h + kNScal, fs->bad, sizeof(unsigned), cudaMemcpyDeviceToHost, st) ==
                   cudaSuccess &&
               cudaStreamSynchronize(st) == cudaSuccess;
    };
    bool ok = cudaMemsetAsync(fs->bad, 0, sizeof(unsigned), st) == cudaSuccess;
    k_fld_cell<<<grid, 256, 0, st>>>(ca);
    k_fld_faces<<<grid, 256, 0, st>>>(fa);
    for (int i = 0; i + 1 < n_lv; ++i) {  // coarse operators of this step
        k_mg_coarsen<<<wave((const void *)k_mg_coarsen, 256, 0, lv[i + 1].n), 256, 0, st>>>(pairs[i]);
        k_mg_diag<<<wave((const void *)k_mg_diag, 256, 0, lv[i + 1].n), 256, 0, st>>>(lv[i + 1]);
    }
    if (lines) k_line_setup<<<ln.blocks, t_line, 0, st>>>(ln, cg);
    k_it_start<<<1, 1, 0, st>>>(fs->scal, fs->bad, fs->count, tol, (double)max_iter);
    if (fs->loop) {
        ok = ok && cudaGraphLaunch(fs->loop, st) == cudaSuccess;
    } else {
        for (double left = max_iter + 4.0 * kUnroll; ok && left > 0.0; left -= kUnroll) {
            for (int i = 0; i < kUnroll; ++i) iteration(i);
            ok = sync_read();
            if (ok && fs->scal_h[kDone] != 0.0) break;
        }
    }
    k_it_store<<<grid, 256, 0, st>>>(x, e_new, n, fs->bad);
    ok = ok && sync_read();
    if (!ok) return ctx_fail(ctx, RT_ERR_CUDA, std::string("FLD step: ") + cudaGetErrorString(cudaGetLastError()));
    unsigned h_bad = 0;
    memcpy(&h_bad, fs->scal_h + kNScal, sizeof(unsigned));
    if (h_bad)
        return ctx_fail(ctx, RT_ERR_NONFINITE_INPUT,
                        "FLD input holds rho < 0, T <= 0, E_old < 0, q_abs < 0 or a NaN/Inf");
    const int iters = (int)fs->scal_h[kIters], passes = (int)fs->scal_h[kPasses];
    const double corr = fs->scal_h[kCorr];
    if (stats) {
        stats->levels = use_mg ? n_lv : 1;
        stats->iterations = iters;
        stats->passes = passes;
        stats->rel_change = corr;
    }
    if (isinf(corr)) return ctx_fail(ctx, RT_ERR_CUDA, "FLD solve broke down (non-finite E')");
    return corr < tol ? RT_OK
                      : ctx_fail(ctx, RT_ERR_TIMEOUT, "FLD solve did not reach tol within max_iter iterations");
}

}  // extern "C"
