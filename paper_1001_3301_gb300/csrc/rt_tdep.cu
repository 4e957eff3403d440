// Tracer with temperature-dependent opacity tables: kappa_i(T) per bin, linear in T
// between the points of a temperature grid (the ends beyond it), zero above the
// sublimation temperature. Each cell has its own kappa per bin, so the optical
// depth of every bin is its own scan along the ray (Eq. 19; no single column serves
// all bins as in rt_ray.cu):
//   tau_i,in(k) = sum_{k' < k} kappa_i(T_k') rho_k' dr_k',
// then the attenuated flux (Eq. 17) and the absorbed fraction of the cell
// (Eqs. 31-32, 36) per (cell, bin) as in the per-bin loop of rt_device.cuh.
//
// One warp per ray, lane l owns cells [l C, (l+1) C). The bins go in pairs (2p, 2p + 1),
// one f32x2 register per cell holding both: every cell's two kappa from the table (one
// 16-byte shared-memory read of both rows' bracketing points), the lane's two sums (C
// terms, plain FP32), one compensated warp scan of both (packed: half the scan
// instructions per bin), then a second pass over the lane's cells carrying the
// exclusive prefix (no per-cell prefix is stored).
// The bins are ordered by their largest tabulated kappa; the Taylor classes of the
// absorbed fraction (1, 2, 3, 5 terms) come from that largest kappa and the warp's
// largest column, the remaining bins take the per-cell select between the 5-term
// series and 1 - ex2 (kappa's smallest value need not follow the same order). A pair
// takes the class of its upper bin, which holds for the lower one too.
//
// Where the rays fill the chip the bins go across the lanes instead (k_ray_tdep_bins below; the
// line is in tdep_default).
#include "rt_device.cuh"

namespace rt {
namespace {

struct TdepTab {
    const float2 *kt2;  // [nnu_pad][n_t] (kappa_j, kappa_{j+1}) of every sorted bin (global)
    const float *tg;    // [n_t] temperature grid (K)
    int n_t;
};

// Bins [i0, i1) of one class: scan, attenuation, absorption for the lane's cells,
// two cells per f32x2 register pair (packed FMA/ADD/MUL on the column, the exponent,
// the absorbed fraction and the accumulators; the two cells' kappa come from
// different table rows, so the interpolation itself stays scalar).
template <int CLASS, int C>
__device__ __forceinline__ void tdep_range(int i0, int i1, const float *s_lf, const float2 *s_kt, int n_t,
                                           const int (&jt)[C], const float (&wt)[C], const float (&wb)[C],
                                           const float2 (&d2)[C / 2],
                                           float2 (&a2)[C / 2], float2 (&a02)[C / 2], bool any_zero, int lane,
                                           float &esc)
{
    const float2 nl2e = f2(-(float)kLog2e);
    for (int i = i0; i < i1; ++i) {
        const float lf = s_lf[i];
        const float2 *row = s_kt + i * n_t;
        auto kappa2 = [&](int m) {  // the two cells' kappa of this bin
            // kappa_j (T_{j+1} - T) / dT + kappa_{j+1} (T - T_j) / dT: two non-negative
            // terms, no cancellation where the row falls towards zero
            const float2 k0 = row[jt[2 * m]], k1 = row[jt[2 * m + 1]];
            return make_float2(fmaf(k0.y, wt[2 * m], k0.x * wb[2 * m]), fmaf(k1.y, wt[2 * m + 1], k1.x * wb[2 * m + 1]));
        };
        float2 dt2[C / 2];
        float2 ls2 = f2(0.0f);  // the lane's sum, at most C terms in two halves (plain FP32)
#pragma unroll
        for (int m = 0; m < C / 2; ++m) {
            dt2[m] = __fmul2_rn(kappa2(m), d2[m]);
            ls2 = __fadd2_rn(ls2, dt2[m]);
        }
        // compensated warp scan of the lane sums (the ray-long sum)
        KahanSum inc;
        inc.zero();
        inc.add(ls2.x + ls2.y);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const KahanSum v = inc.shfl_up(o);
            if (lane >= o) inc.add(v);
        }
        KahanSum pre = inc.shfl_up(1);
        if (lane == 0) pre.zero();
        if (lane == 31) esc += ex2_approx(fmaf(-(float)kLog2e, inc.value(), lf));
        // the lane's exclusive prefix: the warp offset (hi + lo) plus a plain partial sum
        const float2 bhi = f2(pre.hi), blo = f2(pre.lo), lf2 = f2(lf);
        float part = 0.0f;
#pragma unroll
        for (int m = 0; m < C / 2; ++m) {
            const float2 p2 = make_float2(part, part + dt2[m].x);
            const float2 tau = __fadd2_rn(bhi, __fadd2_rn(blo, p2));
            const float2 g = ex2_approx2(__ffma2_rn(nl2e, tau, lf2));
            const float2 y = __fmul2_rn(nl2e, dt2[m]);  // -dtau log2(e)
            float2 om;                                   // 1 - 2^y
            if constexpr (CLASS <= 5) {
                om = taylor_fraction<CLASS>(y);
            } else {
                const float2 big = __ffma2_rn(ex2_approx2(y), f2(-1.0f), f2(1.0f));
                const float2 small = taylor_fraction<5>(y);
                om = make_float2(y.x > -kYSplit ? small.x : big.x, y.y > -kYSplit ? small.y : big.y);
            }
            a2[m] = __ffma2_rn(g, om, a2[m]);
            if (any_zero) a02[m] = __ffma2_rn(g, kappa2(m), a02[m]);  // (rare: re-read, not kept)
            part = p2.y + dt2[m].y;
        }
    }
}

// Bin pairs [p0, p1) of one class: scan, attenuation, absorption for the lane's cells,
// one cell per f32x2 register pair holding the pair's two bins (packed FMA/ADD/MUL on the
// opacity, the column, the exponent, the absorbed fraction). s_kt4[p n_t + j] =
// (kappa_2p(T_j), kappa_2p+1(T_j), kappa_2p(T_j+1), kappa_2p+1(T_j+1)).
template <int CLASS, int C>
__device__ __forceinline__ void tdep_pairs(int p0, int p1, const float *s_lf, const float4 *s_kt4, int n_t,
                                           const int (&jt)[C], const float (&wt)[C], const float (&wb)[C],
                                           const Cells<float, C> &dc, Cells<float, C> &ac, Cells<float, C> &ac0,
                                           bool any_zero, int lane, float &esc)
{
    const float2 nl2e = f2(-(float)kLog2e);
    for (int pp = p0; pp < p1; ++pp) {
        const float2 lf2 = make_float2(s_lf[2 * pp], s_lf[2 * pp + 1]);
        const float4 *row = s_kt4 + pp * n_t;
        auto kappa2 = [&](int j) {  // the pair's kappa in cell j
            // kappa_j (T_{j+1} - T) / dT + kappa_{j+1} (T - T_j) / dT: two non-negative
            // terms, no cancellation where the row falls towards zero
            const float4 k = row[jt[j]];
            return __ffma2_rn(make_float2(k.z, k.w), f2(wt[j]), __fmul2_rn(make_float2(k.x, k.y), f2(wb[j])));
        };
        float2 dt2[C];
        float2 ls2 = f2(0.0f);  // the lane's two sums, C terms each (plain FP32)
#pragma unroll
        for (int j = 0; j < C; ++j) {
            dt2[j] = __fmul2_rn(kappa2(j), f2(dc.get(j)));
            ls2 = __fadd2_rn(ls2, dt2[j]);
        }
        // compensated warp scan of both bins' lane sums (the ray-long sums): a Kahan pair
        // per bin, the two bins side by side
        float2 ih = ls2, il = f2(0.0f);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const float2 vh = make_float2(__shfl_up_sync(0xffffffffu, ih.x, o), __shfl_up_sync(0xffffffffu, ih.y, o));
            const float2 vl = make_float2(__shfl_up_sync(0xffffffffu, il.x, o), __shfl_up_sync(0xffffffffu, il.y, o));
            if (lane >= o) {
                // two_sum(vh, ih) exactly, then the low parts
                const float2 sm = __fadd2_rn(vh, ih);
                const float2 bb = __fadd2_rn(sm, __fmul2_rn(vh, f2(-1.0f)));
                const float2 ea = __fadd2_rn(vh, __fmul2_rn(__fadd2_rn(sm, __fmul2_rn(bb, f2(-1.0f))), f2(-1.0f)));
                const float2 eb = __fadd2_rn(ih, __fmul2_rn(bb, f2(-1.0f)));
                il = __fadd2_rn(__fadd2_rn(il, vl), __fadd2_rn(ea, eb));
                ih = sm;
            }
        }
        // exclusive prefix: the inclusive one of the lane before
        float2 bhi = make_float2(__shfl_up_sync(0xffffffffu, ih.x, 1), __shfl_up_sync(0xffffffffu, ih.y, 1));
        float2 blo = make_float2(__shfl_up_sync(0xffffffffu, il.x, 1), __shfl_up_sync(0xffffffffu, il.y, 1));
        if (lane == 0) bhi = blo = f2(0.0f);
        if (lane == 31) {
            const float2 tot = __fadd2_rn(ih, il);
            const float2 ee = ex2_approx2(__ffma2_rn(nl2e, tot, lf2));
            esc += ee.x + ee.y;
        }
        // the lane's exclusive prefix: the warp offset (hi + lo) plus a plain partial sum
        float2 part = f2(0.0f);
#pragma unroll
        for (int j = 0; j < C; ++j) {
            const float2 tau = __fadd2_rn(bhi, __fadd2_rn(blo, part));
            const float2 g = ex2_approx2(__ffma2_rn(nl2e, tau, lf2));
            const float2 y = __fmul2_rn(nl2e, dt2[j]);  // -dtau log2(e)
            float2 om;                                  // 1 - 2^y
            if constexpr (CLASS <= 5) {
                om = taylor_fraction<CLASS>(y);
            } else {
                const float2 big = __ffma2_rn(ex2_approx2(y), f2(-1.0f), f2(1.0f));
                const float2 small = taylor_fraction<5>(y);
                om = make_float2(y.x > -kYSplit ? small.x : big.x, y.y > -kYSplit ? small.y : big.y);
            }
            ac.set(j, fmaf(g.y, om.y, fmaf(g.x, om.x, ac.get(j))));
            if (any_zero) {  // (rare: the kappa read again, not kept)
                const float2 k2 = kappa2(j);
                ac0.set(j, fmaf(g.y, k2.y, fmaf(g.x, k2.x, ac0.get(j))));
            }
            part = __fadd2_rn(part, dt2[j]);
        }
    }
}

// PAIRS: the bins in pairs (tdep_pairs; 2C more registers for both bins' column
// increments), else one at a time (tdep_range), for the shapes whose register cap the
// pair form overflows
template <int C, int W, int MINB, bool PAIRS>
__global__ void __launch_bounds__(W * 32, MINB) k_ray_tdep(const TraceArgs p, const TdepTab t)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nr = p.nr;
    const int c0 = lane * C;
    const int nv = nr - c0 < 0 ? 0 : (nr - c0 > C ? C : nr - c0);

    __shared__ float s_dr[C][32], s_gq[C][32], s_ga[C][32];
    __shared__ float s_tg[32], s_idt[32];  // grid, 1 / (T_{j+1} - T_j)
    __shared__ KahanSum s_red[W][2];
    extern __shared__ __align__(16) unsigned char smem[];
    float4 *s_nu = reinterpret_cast<float4 *>(smem);                 // [nnu_pad] (nk_max, ., lf, .)
    float *s_lf = reinterpret_cast<float *>(s_nu + p.nnu_pad);        // [nnu_pad]
    // [nnu_pad][n_t] rows of (kappa_j, kappa_j+1), or [nnu_pad / 2][n_t] bin-pair rows of
    // both bins' (kappa_j, kappa_j+1) (the same bytes); 16-byte aligned
    float4 *s_kt4 = reinterpret_cast<float4 *>((reinterpret_cast<size_t>(s_lf + p.nnu_pad) + 15) & ~size_t(15));
    float2 *s_kt = reinterpret_cast<float2 *>(s_kt4);

    for (int i = tid; i < p.nnu_pad; i += W * 32) {
        const NuEntry e = p.nu[i];
        s_nu[i] = make_float4(e.nk, e.nk, e.lf, e.lf);
        s_lf[i] = e.lf;
    }
    if constexpr (PAIRS) {
        for (int i = tid; i < (p.nnu_pad / 2) * t.n_t; i += W * 32) {
            const int pp = i / t.n_t, j = i - pp * t.n_t;
            const float2 a = t.kt2[2 * pp * t.n_t + j], b = t.kt2[(2 * pp + 1) * t.n_t + j];
            s_kt4[i] = make_float4(a.x, b.x, a.y, b.y);
        }
    } else {
        for (int i = tid; i < p.nnu_pad * t.n_t; i += W * 32) s_kt[i] = t.kt2[i];
    }
    for (int i = tid; i < t.n_t; i += W * 32) {
        s_tg[i] = t.tg[i];
        s_idt[i] = i + 1 < t.n_t ? 1.0f / (t.tg[i + 1] - t.tg[i]) : 0.0f;
    }
    for (int i = tid; i < 32 * C; i += W * 32) {
        const int l = i / C, j = i % C, k = l * C + j;
        const float4 g = (k < nr) ? __ldg(&p.rtab[k]) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        s_dr[j][l] = g.x;
        s_gq[j][l] = g.y;
        s_ga[j][l] = g.z;
    }
    __syncthreads();
    const int nt = t.n_t;

    KahanSum eabs, eesc;
    eabs.zero();
    eesc.zero();
    for (unsigned ray = blockIdx.x * W + warp; ray < p.nrays; ray += gridDim.x * W) {
        const size_t base = (size_t)ray * nr + c0;
        Cells<float, C> d, acc, acc0;
        float wt[C], wb[C];  // the weights of the upper and the lower point
        int jt[C];
        unsigned zero_m = 0;
        bool bad = false;
        float dmax = 0.0f;
#pragma unroll
        for (int j = 0; j < C; ++j) {
            float rho = 0.0f, td = 0.0f;
            if (j < nv) {
                rho = __ldg(p.rho + base + j);
                td = __ldg(p.tdust + base + j);
                bad |= !(rho >= 0.0f && rho <= FLT_MAX) || (td != td);
            }
            const bool dust = j < nv && td <= p.t_sub;
            const float dj = dust ? rho * s_dr[j][lane] : 0.0f;
            d.set(j, dj);
            if (dust && dj == 0.0f) zero_m |= 1u << j;
            dmax = fmaxf(dmax, dj);
            acc.set(j, 0.0f);
            acc0.set(j, 0.0f);
            // bracketing temperature points and the weight of the upper one
            int lo = 0;
            for (int s = 16; s > 0; s >>= 1)
                if (lo + s < nt - 1 && s_tg[lo + s] <= td) lo += s;
            jt[j] = lo;
            wt[j] = fminf(fmaxf((td - s_tg[lo]) * s_idt[lo], 0.0f), 1.0f);
            wb[j] = fminf(fmaxf((s_tg[lo + 1] - td) * s_idt[lo], 0.0f), 1.0f);
        }
        if (__any_sync(0xffffffffu, bad) && lane == 0) atomicMax(p.bad_input, p.seq);
        for (int o = 16; o > 0; o >>= 1) dmax = fmaxf(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
        const bool any_zero = __any_sync(0xffffffffu, zero_m != 0u);

        const int na = p.n_active;
        const BinClasses bc = classify_bins(s_nu, na, lane, dmax, 0.0f);
        float esc = 0.0f;
        if constexpr (PAIRS) {
            // pair p (bins 2p, 2p + 1) belongs to the class of its upper bin: the pairs
            // below a class boundary b are those with 2p + 1 < b; a last odd bin pairs with
            // a padding bin (kappa 0, no flux: it adds nothing)
            const int q1 = bc.b1 / 2, q2 = max(bc.b2 / 2, q1), q3 = max(bc.b3 / 2, q2), q5 = max(bc.b5 / 2, q3);
            const int qn = (na + 1) / 2;
            tdep_pairs<1, C>(0, q1, s_lf, s_kt4, nt, jt, wt, wb, d, acc, acc0, any_zero, lane, esc);
            tdep_pairs<2, C>(q1, q2, s_lf, s_kt4, nt, jt, wt, wb, d, acc, acc0, any_zero, lane, esc);
            tdep_pairs<3, C>(q2, q3, s_lf, s_kt4, nt, jt, wt, wb, d, acc, acc0, any_zero, lane, esc);
            tdep_pairs<5, C>(q3, q5, s_lf, s_kt4, nt, jt, wt, wb, d, acc, acc0, any_zero, lane, esc);
            tdep_pairs<6, C>(q5, qn, s_lf, s_kt4, nt, jt, wt, wb, d, acc, acc0, any_zero, lane, esc);
        } else {
            tdep_range<1, C>(0, bc.b1, s_lf, s_kt, nt, jt, wt, wb, d.v, acc.v, acc0.v, any_zero, lane, esc);
            tdep_range<2, C>(bc.b1, bc.b2, s_lf, s_kt, nt, jt, wt, wb, d.v, acc.v, acc0.v, any_zero, lane, esc);
            tdep_range<3, C>(bc.b2, bc.b3, s_lf, s_kt, nt, jt, wt, wb, d.v, acc.v, acc0.v, any_zero, lane, esc);
            tdep_range<5, C>(bc.b3, bc.b5, s_lf, s_kt, nt, jt, wt, wb, d.v, acc.v, acc0.v, any_zero, lane, esc);
            tdep_range<6, C>(bc.b5, na, s_lf, s_kt, nt, jt, wt, wb, d.v, acc.v, acc0.v, any_zero, lane, esc);
        }

        const float w = __ldg(p.domega32 + ray);
        if (lane == 31) eesc.add(esc * w);
        float lane_abs = 0.0f;
#pragma unroll
        for (int j = 0; j < C; ++j) {
            const bool zc = (zero_m >> j) & 1u;
            const float aj = acc.get(j), dj = d.get(j);
            const float qv = zc ? 0.0f : s_gq[j][lane] * aj;
            const float av = s_ga[j][lane] * (zc ? acc0.get(j) : (dj > 0.0f ? __fdividef(aj, dj) : 0.0f));
            lane_abs += (j < nv && !zc) ? aj : 0.0f;
            if (j < nv) {
                p.q[base + j] = qv;
                p.a[base + j] = av;
            }
        }
        eabs.add(lane_abs * w);
    }

    for (int o = 16; o > 0; o >>= 1) {
        eabs.add(eabs.shfl_xor(o));
        eesc.add(eesc.shfl_xor(o));
    }
    if (lane == 0) {
        s_red[warp][0] = eabs;
        s_red[warp][1] = eesc;
    }
    __syncthreads();
    if (tid == 0) {
        KahanSum sa = s_red[0][0], se = s_red[0][1];
        for (int w2 = 1; w2 < W; ++w2) {
            sa.add(s_red[w2][0]);
            se.add(s_red[w2][1]);
        }
        p.partials[blockIdx.x] = make_double2(to_double(sa), to_double(se));
    }
}

// ---------------------------------------------------------------------------
// the bins across the lanes
// ---------------------------------------------------------------------------
// Eight lanes per ray (four rays per warp): lane l of a ray owns the bin pairs l, 8 + l, 16 + l, ..
// and walks outwards in chunks of 8 cells: every bin's optical depth is a running sum in its own
// lane, so no bin needs a warp scan, and the table rows of a cell are read by the lanes of its ray
// as consecutive 16-byte words, whatever the temperatures (with the cells across the lanes, lanes
// in different temperature intervals collide in the banks). A slot (8 pairs with consecutive
// opacities) takes one class per chunk, from its largest opacity and the chunk's largest column.
// The running sums start at lf, so that hi + lo is the exponent itself (a Kahan pair, one
// compensated addition per chunk; inside the chunk a plain partial sum of at most 8 terms).
constexpr int kBinLanes = 8, kBinCells = 8;  // (the lanes of a ray also hold one cell of the chunk each)

// Slots [m0, m1) of one class over the chunk's cells: rows of (kappa_2p(T_j), kappa_2p+1(T_j),
// kappa_2p(T_j+1), kappa_2p+1(T_j+1)) at kt + row[c] + the slot's offset; wt, wb the interpolation
// weights times -rho dr log2 e, or times -log2 e for a zero-density dust cell (bit c of zm; ZERO:
// the chunk holds one), whose sum is of g y alone (y = -kappa log2 e) and whose step does not enter
// the column. The sums are of (1 - 2^y) / p0, p0 = -ln 2 the first Taylor coefficient: one term is y.
template <int CLASS, bool ZERO>
__device__ __forceinline__ void bins_chunk(int m0, int m1, const unsigned char *kt, unsigned char *state,
                                           const int (&row)[kBinCells], const float2 (&wt)[kBinCells],
                                           const float2 (&wb)[kBinCells], unsigned zm, float2 (&acc)[kBinCells])
{
    constexpr double p0 = taylor_coeff(0);
    for (int m = m0; m < m1; ++m) {
        float4 *sp = reinterpret_cast<float4 *>(state + m * (32 * (int)sizeof(float4)));
        const float4 st = *sp;
        const float2 hi = make_float2(st.x, st.y);
        float2 part = make_float2(st.z, st.w);
#pragma unroll
        for (int c = 0; c < kBinCells; ++c) {
            const float4 k = *reinterpret_cast<const float4 *>(kt + (row[c] + m * (kBinLanes * (int)sizeof(float4))));
            const float2 y = __ffma2_rn(make_float2(k.z, k.w), wt[c], __fmul2_rn(make_float2(k.x, k.y), wb[c]));
            const float2 g = ex2_approx2(__fadd2_rn(hi, part));
            float2 om = y;  // (1 - 2^y) / p0
            if constexpr (CLASS > 1) {
                constexpr int N = CLASS <= 5 ? CLASS : 5;
                float2 pl = f2((float)(taylor_coeff(N - 1) / p0));
#pragma unroll
                for (int k2 = N - 2; k2 >= 0; --k2) pl = __ffma2_rn(pl, y, f2((float)(taylor_coeff(k2) / p0)));
                om = __fmul2_rn(y, pl);
            }
            if constexpr (CLASS == 6) {
                const float2 big = __ffma2_rn(ex2_approx2(y), f2((float)(-1.0 / p0)), f2((float)(1.0 / p0)));
                if (!(y.x > -kYSplit)) om.x = big.x;
                if (!(y.y > -kYSplit)) om.y = big.y;
            }
            if constexpr (ZERO) {
                const bool z = (zm >> c) & 1u;
                if (z) om = y;
                part = __ffma2_rn(y, f2(z ? 0.0f : 1.0f), part);
            } else {
                part = __fadd2_rn(part, y);
            }
            acc[c] = __ffma2_rn(g, om, acc[c]);
        }
        const float2 t = __fadd2_rn(hi, part);
        const float2 rest = __ffma2_rn(__ffma2_rn(hi, f2(-1.0f), t), f2(-1.0f), part);
        *sp = make_float4(t.x, t.y, rest.x, rest.y);
    }
}

// every slot over the chunk, class by class (lane m holds the largest |nk| of slot m; live: the
// slots before the first one whose exponents have all gone under)
template <bool ZERO>
__device__ __forceinline__ void bins_slots(int live, float km, float dmax, const unsigned char *kt,
                                           unsigned char *state, const int (&row)[kBinCells],
                                           const float2 (&wt)[kBinCells], const float2 (&wb)[kBinCells], unsigned zm,
                                           float2 (&acc)[kBinCells])
{
    const float ym = km * dmax;
    const int b1 = min(live, __popc(__ballot_sync(0xffffffffu, ym < kYT1)));
    const int b2 = min(live, __popc(__ballot_sync(0xffffffffu, ym < kYT2)));
    const int b3 = min(live, __popc(__ballot_sync(0xffffffffu, ym < kYT3)));
    const int b5 = min(live, __popc(__ballot_sync(0xffffffffu, ym < kYSplit)));
    bins_chunk<1, ZERO>(0, b1, kt, state, row, wt, wb, zm, acc);
    bins_chunk<2, ZERO>(b1, b2, kt, state, row, wt, wb, zm, acc);
    bins_chunk<3, ZERO>(b2, b3, kt, state, row, wt, wb, zm, acc);
    bins_chunk<5, ZERO>(b3, b5, kt, state, row, wt, wb, zm, acc);
    bins_chunk<6, ZERO>(b5, live, kt, state, row, wt, wb, zm, acc);
}

// Bound by issue (110 M warp instructions for 4.2 M cells x 79 bins, 60 % of the issue slots with 16
// warps per SM) and by latency beside the slots: 256x128x128 cells, 79 bins, 24 temperatures 306 ->
// 186 us, the cells-across-lanes form above spending 17 instructions per (cell, bin) where this one
// spends 11, and 64x256x256 567 -> 164. Tried and slower: 16 or 32 lanes per ray (254, 397 us), the
// chunk's weights in shared memory with 20-28 warps per SM (231-295), sub-chunks of 4 cells (186-208).
template <int W, int MINB>
__global__ void __launch_bounds__(W * 32, MINB) k_ray_tdep_bins(const TraceArgs p, const TdepTab t, int nslot)
{
    constexpr int L = kBinLanes, R = 32 / L;  // rays per warp
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, l = lane % L;
    const int nr = p.nr, nt = t.n_t, np = nslot * L;  // bin pairs with padding
    __shared__ float s_tg[kMaxTdepPoints], s_idt[kMaxTdepPoints];
    __shared__ KahanSum s_red[W][2];
    extern __shared__ __align__(16) unsigned char smem[];
    float4 *s_kt = reinterpret_cast<float4 *>(smem);       // [n_t][np]
    float4 *s_st = s_kt + nt * np;                         // [W][nslot][32] running pairs (hi, hi, lo, lo)
    float2 *s_lf = reinterpret_cast<float2 *>(s_st + W * nslot * 32);  // [np]
    const int na = p.n_active;
    for (int i = tid; i < nt * np; i += W * 32) {
        const int j = i / np, q = i - j * np;
        const float2 a = 2 * q < na ? t.kt2[2 * q * nt + j] : make_float2(0.0f, 0.0f);
        const float2 b = 2 * q + 1 < na ? t.kt2[(2 * q + 1) * nt + j] : make_float2(0.0f, 0.0f);
        s_kt[i] = make_float4(a.x, b.x, a.y, b.y);
    }
    for (int q = tid; q < np; q += W * 32)  // (no flux: an exponent that gives 0 and stays finite)
        s_lf[q] = make_float2(2 * q < na ? fmaxf(p.nu[2 * q].lf, -1e4f) : -1e4f,
                              2 * q + 1 < na ? fmaxf(p.nu[2 * q + 1].lf, -1e4f) : -1e4f);
    for (int i = tid; i < nt; i += W * 32) {
        s_tg[i] = t.tg[i];
        s_idt[i] = i + 1 < nt ? 1.0f / (t.tg[i + 1] - t.tg[i]) : 0.0f;
    }
    __syncthreads();

    float4 *state = s_st + warp * nslot * 32 + lane;  // the lane's own, slot by slot
    // the largest |nk| of slot `lane` (at most 8 slots; lanes behind them: never in a class)
    const float km = lane < nslot ? -p.nu[min(2 * L * (lane + 1), na) - 1].nk : INFINITY;
    KahanSum eabs, eesc;
    eabs.zero();
    eesc.zero();
    for (unsigned w0 = (blockIdx.x * W + warp) * R; w0 < p.nrays; w0 += gridDim.x * W * R) {
        const unsigned ray = w0 + lane / L;
        const bool live = ray < p.nrays;
        const size_t base = (size_t)ray * nr;
        const float w = live ? __ldg(p.domega32 + ray) : 0.0f;
        for (int m = 0; m < nslot; ++m) {
            const float2 lf = s_lf[m * L + l];
            state[m * 32] = make_float4(lf.x, lf.y, 0.0f, 0.0f);
        }
        int nlive = nslot;
        bool bad = false;
        float rho_n = 0.0f, td_n = 0.0f;
        if (live && l < nr) {
            rho_n = __ldg(p.rho + base + l);
            td_n = __ldg(p.tdust + base + l);
        }
        for (int c0 = 0; c0 < nr; c0 += kBinCells) {
            const int k = c0 + l;
            const bool in = live && k < nr;
            const float rho = rho_n, td = td_n;
            float4 geo = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (in) {
                geo = __ldg(&p.rtab[k]);
                bad |= !(rho >= 0.0f && rho <= FLT_MAX) || (td != td);
            }
            if (live && k + kBinCells < nr) {  // the next chunk's
                rho_n = __ldg(p.rho + base + k + kBinCells);
                td_n = __ldg(p.tdust + base + k + kBinCells);
            }
            const bool dust = in && td <= p.t_sub;
            const float d = dust ? rho * geo.x : 0.0f;
            const bool zero = dust && d == 0.0f;
            const float dmax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(d, 0.0f))));
            const unsigned zall = __ballot_sync(0xffffffffu, zero);
            float sum = 0.0f;
            if (dmax > 0.0f || zall) {
                // bracketing temperature points; two non-negative terms, no cancellation
                // where a row falls towards zero
                int j = 0;
                for (int s = 16; s > 0; s >>= 1)
                    if (j + s < nt - 1 && s_tg[j + s] <= td) j += s;
                const float f = zero ? -(float)kLog2e : -(float)kLog2e * d;
                const float wu = f * fminf(fmaxf((td - s_tg[j]) * s_idt[j], 0.0f), 1.0f);
                const float wl = f * fminf(fmaxf((s_tg[j + 1] - td) * s_idt[j], 0.0f), 1.0f);
                const int rw = j * np * (int)sizeof(float4);  // (row of the cell's lower temperature)
                int row[kBinCells];
                float2 wt[kBinCells], wb[kBinCells], acc[kBinCells];
#pragma unroll
                for (int c = 0; c < kBinCells; ++c) {
                    row[c] = __shfl_sync(0xffffffffu, rw, c, 8) + l * (int)sizeof(float4);
                    wt[c] = f2(__shfl_sync(0xffffffffu, wu, c, 8));
                    wb[c] = f2(__shfl_sync(0xffffffffu, wl, c, 8));
                    acc[c] = f2(0.0f);
                }
                const unsigned zm = zall >> (lane & 24);
                unsigned char *sb = reinterpret_cast<unsigned char *>(state);
                if (zall) bins_slots<true>(nlive, km, dmax, smem, sb, row, wt, wb, zm, acc);
                else bins_slots<false>(nlive, km, dmax, smem, sb, row, wt, wb, zm, acc);
                // 2^-128 and below is flushed to zero and columns only grow: the last slots,
                // of the largest opacities, drop out first
                while (nlive > 0) {
                    const float4 st = state[(nlive - 1) * 32];
                    if (__any_sync(0xffffffffu, fmaxf(st.x, st.y) > -130.0f)) break;
                    --nlive;
                }
                // lane l of the ray gets cell l: halve the cells, double the lanes summed
                float v[kBinCells];
#pragma unroll
                for (int c = 0; c < kBinCells; ++c) v[c] = acc[c].x + acc[c].y;
#pragma unroll
                for (int h = 4; h > 0; h >>= 1) {
                    const bool upper = lane & h;
#pragma unroll
                    for (int c = 0; c < h; ++c) {
                        const float keep = upper ? v[c + h] : v[c], give = upper ? v[c] : v[c + h];
                        v[c] = keep + __shfl_xor_sync(0xffffffffu, give, h);
                    }
                }
                sum = v[0] * (float)taylor_coeff(0);
            }
            if (in) {
                p.q[base + k] = zero ? 0.0f : geo.y * sum;
                p.a[base + k] = geo.z * (zero ? sum : (d > 0.0f ? __fdividef(sum, d) : 0.0f));
                if (!zero) eabs.add(sum * w);
            }
        }
        if (__any_sync(0xffffffffu, bad) && lane == 0) atomicMax(p.bad_input, p.seq);
        // the flux leaving the ray (Eq. 33)
        float esc = 0.0f;
        for (int m = 0; m < nslot; ++m) {
            const float4 st = state[m * 32];
            esc += ex2_approx(st.x + st.z) + ex2_approx(st.y + st.w);
        }
#pragma unroll
        for (int o = 1; o < L; o <<= 1) esc += __shfl_xor_sync(0xffffffffu, esc, o);
        if (l == 0) eesc.add(esc * w);
    }

    for (int o = 16; o > 0; o >>= 1) {
        eabs.add(eabs.shfl_xor(o));
        eesc.add(eesc.shfl_xor(o));
    }
    if (lane == 0) {
        s_red[warp][0] = eabs;
        s_red[warp][1] = eesc;
    }
    __syncthreads();
    if (tid == 0) {
        KahanSum sa = s_red[0][0], se = s_red[0][1];
        for (int w2 = 1; w2 < W; ++w2) {
            sa.add(s_red[w2][0]);
            se.add(s_red[w2][1]);
        }
        p.partials[blockIdx.x] = make_double2(to_double(sa), to_double(se));
    }
}

// kt2[a][j] = (kappa[order[a]][j], kappa[order[a]][j + 1]) for the sorted active
// bins; padding bins get zero opacity
__global__ void k_build_tdep(int n_active, int nnu_pad, int n_t, const double *kappa_t, const int *order,
                             float2 *kt2)
{
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= nnu_pad * n_t) return;
    const int a = idx / n_t, j = idx % n_t;
    if (a >= n_active) {
        kt2[idx] = make_float2(0.0f, 0.0f);
        return;
    }
    const double *row = kappa_t + (size_t)order[a] * n_t;
    kt2[idx] = make_float2((float)row[j], (float)row[j + 1 < n_t ? j + 1 : j]);
}

// persistent blocks of W warps, `rays` rays per warp and turn
template <typename K, typename... Extra>
cudaError_t launch_rays(K kern, int W, int rays, size_t smem, const TraceArgs &a, cudaStream_t stream,
                        unsigned *grid_out, const Extra &...extra)
{
    int dev = 0, nsm = 0, per_sm = 0;
    cudaError_t e = cudaSuccess;
    if (smem > 40 * 1024) {  // the static part counts towards the 48 KB a launch has without asking
        int most = 0;
        e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        cudaFuncAttributes fa;
        if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, kern);
        if (e == cudaSuccess)  // one value for every caller: another thread's smaller call cannot lower it
            e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)fa.sharedSizeBytes);
        if (e != cudaSuccess) return e;
    }
    e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, W * 32, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    unsigned grid = (unsigned)nsm * (unsigned)per_sm;
    const unsigned need = (a.nrays + W * rays - 1) / (W * rays);
    if (grid > need) grid = need;
    if (grid < 1) grid = 1;
    kern<<<grid, W * 32, smem, stream>>>(a, extra...);
    *grid_out = grid;
    return cudaGetLastError();
}

template <int C, int W, int MINB, bool PAIRS>
cudaError_t launch_tdep_shape(const TraceArgs &a, const TdepTab &t, cudaStream_t stream, unsigned *grid_out)
{
    const size_t smem = (size_t)a.nnu_pad * (16 + 4) + 16 + (size_t)(a.nnu_pad / 2) * t.n_t * sizeof(float4);
    return launch_rays(k_ray_tdep<C, W, MINB, PAIRS>, W, 1, smem, a, stream, grid_out, t);
}

template <int W, int MINB>
cudaError_t launch_tdep_bins(const TraceArgs &a, const TdepTab &t, cudaStream_t stream, unsigned *grid_out)
{
    constexpr int L = kBinLanes;
    const int nslot = (a.n_active + 2 * L - 1) / (2 * L);
    const size_t np = (size_t)nslot * L;
    const size_t smem = np * t.n_t * sizeof(float4) + (size_t)W * nslot * 32 * sizeof(float4) + np * sizeof(float2);
    return launch_rays(k_ray_tdep_bins<W, MINB>, W, 32 / L, smem, a, stream, grid_out, t, nslot);
}

struct TdepEntry {
    int c, w, minb;
    cudaError_t (*fn)(const TraceArgs &, const TdepTab &, cudaStream_t, unsigned *);
};
// the bin-pair form where its registers fit the cap without more than a few bytes of spill
// the kernel with the bins across the lanes takes every ray length: it stands in every class of nr,
// as (C, 4, 1)
#define RT_TB(C) {C, 4, 1, &launch_tdep_bins<4, 4>}
#define RT_TD(C, W, MB, PR) {C, W, MB, &launch_tdep_shape<C, W, MB, PR>}
const TdepEntry kTdepShapes[] = {RT_TD(2, 4, 8, true),  RT_TD(4, 4, 8, false),  RT_TD(4, 4, 6, true),
                                 RT_TD(8, 4, 6, false), RT_TD(8, 4, 4, true),   RT_TD(16, 4, 3, false),
                                 RT_TD(32, 4, 2, false),
                                 RT_TB(2), RT_TB(4), RT_TB(8), RT_TB(16), RT_TB(32)};
#undef RT_TD
#undef RT_TB

}  // namespace

// The shapes whose rays fill the warp: the fewest cells per lane that hold nr
// (with each of its register caps); a wider one would leave lanes idle.
int tdep_shapes(int nr, Shape *out, int max_out)
{
    int c_fit = 0;
    for (const TdepEntry &s : kTdepShapes)
        if (32 * s.c >= nr && (c_fit == 0 || s.c < c_fit)) c_fit = s.c;
    int n = 0;
    for (const TdepEntry &s : kTdepShapes)
        if (s.c == c_fit && n < max_out) out[n++] = Shape{kKindRay, s.c, s.w, s.minb};
    return n;
}

// The shape without tuning. The bins across the lanes take a ray per 8 lanes and walk it serially
// (1.5-2 us per 8 cells of a lone warp), so they need rays to fill the chip: from 2048 rays on with
// 64 bins or more, from 4096 on with 32 to 63, and not with fewer (per chunk of 8 cells the kernel
// spends as much beside the slots as 45 bins cost). us, cells across / bins across the lanes, full rank, 24 temperatures:
//   79 bins: 256x64x32 52.2 / 51.7, 128x64x32 38 / 29, 512x64x32 110 / 95, 512x64x24 77 / 95,
//            1000x64x32 211 / 179, 1000x64x16 112 / 178, 256x128x128 306 / 186, 64x256x256 567 / 164;
//   32 bins: 256x64x48 37.5 / 43.9, 256x64x64 46.1 / 44.0, 256x128x128 135 / 119;
//   128 bins: 256x64x32 77 / 63;  16 bins: 256x64x64 31.4 / 39.6, 100x64x64 19.4 / 19.3.
// Below, of the register caps of the fewest cells per lane the wider (the bin-pair form:
// 256x128x16 64.6 -> 51.9).
Shape tdep_default(int nr, long long nrays, int n_active)
{
    Shape ts[16];
    const int n = tdep_shapes(nr, ts, 16);
    const bool bins = n_active >= 32 && nrays >= (n_active >= 64 ? 2048 : 4096);
    Shape best{kKindRay, 0, 0, 0};
    for (int i = 0; i < n; ++i) {
        if ((ts[i].min_blocks == 1) != bins) continue;
        if (best.cells_per_lane == 0 || ts[i].min_blocks < best.min_blocks) best = ts[i];
    }
    return best;
}

cudaError_t launch_tdep(Shape s, const TraceArgs &args, const float2 *kt2, const float *tg, int n_t,
                        cudaStream_t stream, unsigned *grid_out)
{
    const TdepTab t{kt2, tg, n_t};
    for (const TdepEntry &e : kTdepShapes)
        if (e.c == s.cells_per_lane && e.w == s.warps && (s.min_blocks == 0 || e.minb == s.min_blocks) &&
            32 * e.c >= args.nr)
            return e.fn(args, t, stream, grid_out);
    return cudaErrorInvalidValue;
}

cudaError_t launch_build_tdep(int n_active, int nnu_pad, int n_t, const double *kappa_t, const int *order,
                              float2 *kt2, cudaStream_t stream)
{
    const int n = nnu_pad * n_t;
    k_build_tdep<<<(n + 255) / 256, 256, 0, stream>>>(n_active, nnu_pad, n_t, kappa_t, order, kt2);
    return cudaGetLastError();
}

}  // namespace rt
