// Warp-per-ray form of the frequency-dependent tracer (Kuiper et al. 2010,
// Sect. 2.2-2.3, 3.3.4), for grids whose rays fill most of 32 P C cells (P = 1 or 2
// warps per ray): the body of rt_ray.cuh over all rays of one grid, then the CTA's
// energy partial. Persistent: the grid holds (SMs x resident CTAs) CTAs that stride
// over the rays.
#include "rt_ray.cuh"

namespace rt {
namespace {

// The fewest lanes per ray that still hold the ray: 8, 16 or 32 (G C >= nr), else two
// warps per ray (ray_warps_per_ray).
template <int C, int W, int MODE, int MINB, bool TW = false, bool LUT = false>
cudaError_t launch_ray(const TraceArgs &a, unsigned, cudaStream_t stream, unsigned *grid_out, unsigned max_grid)
{
    if ((a.n_tw > 0) != TW || (a.lut != nullptr) != LUT) return cudaErrorInvalidValue;
    if (8 * C >= a.nr) return launch_ray_g<C, W, MODE, MINB, 8, 1, TW, LUT>(a, stream, grid_out, max_grid);
    if (16 * C >= a.nr) return launch_ray_g<C, W, MODE, MINB, 16, 1, TW, LUT>(a, stream, grid_out, max_grid);
    if (32 * C >= a.nr) return launch_ray_g<C, W, MODE, MINB, 32, 1, TW, LUT>(a, stream, grid_out, max_grid);
    if constexpr (C <= 8) {
        if (64 * C >= a.nr) return launch_ray_g<C, W, MODE, MINB, 32, 2, TW, LUT>(a, stream, grid_out, max_grid);
    }
    return cudaErrorInvalidValue;
}

struct RayEntry {
    int precision, c, w, minb;
    cudaError_t (*fn)(const TraceArgs &, unsigned, cudaStream_t, unsigned *, unsigned);
};

#define RT_RAY(P, C, W, MB) {P, C, W, MB, &launch_ray<C, W, P, MB>}
const RayEntry kRayShapes[] = {
    RT_RAY(RT_FP32_KAHAN, 2, 4, 8),  RT_RAY(RT_FP32_KAHAN, 4, 4, 8),  RT_RAY(RT_FP32_KAHAN, 6, 4, 8),
    RT_RAY(RT_FP32_KAHAN, 8, 4, 6),  RT_RAY(RT_FP32_KAHAN, 8, 4, 8),  RT_RAY(RT_FP32_KAHAN, 12, 4, 5),
    RT_RAY(RT_FP32_KAHAN, 16, 4, 3), RT_RAY(RT_FP32_KAHAN, 16, 4, 4), RT_RAY(RT_FP32_PLAIN, 4, 4, 8),
    RT_RAY(RT_FP32_PLAIN, 8, 4, 6),  RT_RAY(RT_FP32_PLAIN, 16, 4, 4),
};
// shapes compiled with the column weight of a separable kappa(nu, T) table
#define RT_RAYW(P, C, W, MB) {P, C, W, MB, &launch_ray<C, W, P, MB, true>}
const RayEntry kRayShapesTW[] = {
    RT_RAYW(RT_FP32_KAHAN, 4, 4, 8),  RT_RAYW(RT_FP32_KAHAN, 8, 4, 6), RT_RAYW(RT_FP32_KAHAN, 16, 4, 4),
    RT_RAYW(RT_FP32_PLAIN, 8, 4, 6),  RT_RAYW(RT_FP32_PLAIN, 16, 4, 4),
};
#undef RT_RAYW
// shapes compiled with the lookup-table comparator
#define RT_RAYL(P, C, W, MB) {P, C, W, MB, &launch_ray<C, W, P, MB, false, true>}
const RayEntry kRayShapesLUT[] = {
    RT_RAYL(RT_FP32_KAHAN, 4, 4, 8), RT_RAYL(RT_FP32_KAHAN, 8, 4, 6), RT_RAYL(RT_FP32_KAHAN, 16, 4, 4),
    RT_RAYL(RT_FP32_PLAIN, 8, 4, 6), RT_RAYL(RT_FP32_PLAIN, 16, 4, 4),
};
#undef RT_RAYL
#undef RT_RAY

}  // namespace

int ray_shapes(int precision, int nr, Shape *out, int max_out)
{
    int n = 0;
    for (const RayEntry &s : kRayShapes)
        if (s.precision == precision && ray_warps_per_ray(s.c, nr) > 0 && n < max_out)
            out[n++] = Shape{kKindRay, s.c, s.w, s.minb};
    return n;
}

int ray_shapes_tw(int precision, int nr, Shape *out, int max_out)
{
    int n = 0;
    for (const RayEntry &s : kRayShapesTW)
        if (s.precision == precision && ray_warps_per_ray(s.c, nr) > 0 && n < max_out)
            out[n++] = Shape{kKindRay, s.c, s.w, s.minb};
    return n;
}

int ray_shapes_lut(int precision, int nr, Shape *out, int max_out)
{
    int n = 0;
    for (const RayEntry &s : kRayShapesLUT)
        if (s.precision == precision && ray_warps_per_ray(s.c, nr) > 0 && n < max_out)
            out[n++] = Shape{kKindRay, s.c, s.w, s.minb};
    return n;
}

// The warp-per-ray shape of a context that was not autotuned; false where the tile kernel serves it
// better (rays beyond 512 cells, few of them) or no such shape applies. Timed over 79 bins,
// tau550 = 0.1 to 100, nr 64 to 4096, 32 to 131072 rays:
//   - a lane's fixed work and the whole-warp decisions want many cells per lane, masked lanes want
//     few: the cost is cells held / nr, weighted per shape (256x128x256, tau550 = 10: C = 8 62 us,
//     C = 16 65, C = 4 with two warps per ray 99; 384x128x128, tau550 = 1: C = 12 32 us, C = 6 with
//     two warps 48, C = 16 46);
//   - grids that do not give every SM eight warps (32 with C = 16) are latency-bound: the fewest
//     cells per lane (64x32x1: C = 2 7.3 us, C = 8 7.5, C = 16 9.3). With the line at two warps per SM
//     a seventh of 1200 small cases (nr 48 to 512, 24 to 32768 rays, 32 to 128 bins, tau550 = 0.3 to 30)
//     was more than 5 % slower than the fewest cells whose lanes are 3/4 full, up to 26 %; so 1.8 % of
//     them, and the mean distance from the best shape is 1.5 % in place of 3.6 (one line at four, eight,
//     sixteen warps: 2.5, 1.7, 2.6 %). us, before / so: 128x24x32, 128 bins, tau550 = 30 10.4 / 8.5;
//     256x24x21, the same 10.4 / 8.5; 432x24x14, 79 bins, tau550 = 0.3 7.8 / 6.5; 432x24x170, 128 bins,
//     tau550 = 30 28.9 / 25.2;
//   - longer rays: the chunked form, which needs some 1500 rays to fill the SMs (1024x128x16:
//     31 us against the tiles' 58; 1024x16x16: tiles 22 us).
bool ray_default(int precision, int nr, long long nrays, bool tw, Shape *out)
{
    Shape s[32];
    const int n = tw ? ray_shapes_tw(precision, nr, s, 32) : ray_shapes(precision, nr, s, 32);
    if (n < 1) {
        if (tw || precision == RT_FP64 || nrays < 1536) return false;
        const int m = ray_shapes_mc(precision, nr, s, 32);
        for (int i = 0; i < m; ++i)
            if (s[i].cells_per_lane == 16 && s[i].min_blocks == 4) {
                *out = s[i];
                return true;
            }
        return false;
    }
    auto weight = [](int c) { return c <= 2 ? 2.1 : c <= 4 ? 1.3 : c <= 6 ? 1.35 : c <= 12 ? 1.0 : 1.07; };
    int bi = 0;
    double best = 0.0;
    for (int i = 0; i < n; ++i) {
        const int c = s[i].cells_per_lane, held = ray_cells_held(c, nr);
        double cost = (double)held / nr * weight(c) * (held > 32 * c ? 1.15 : 1.0);  // two warps per ray
        if (nrays * held < (c == 16 ? 4864LL : 1216LL) * 32 * c) cost = 100.0 + c;
        // of one shape's register caps the first but for the two of C = 16 (4 CTAs per SM)
        if (i == 0 || cost < best || (cost == best && c == 16 && s[bi].cells_per_lane == 16)) {
            best = cost;
            bi = i;
        }
    }
    *out = s[bi];
    return true;
}

cudaError_t launch_ray_shape(int precision, Shape s, const TraceArgs &args, cudaStream_t stream,
                             unsigned *grid_out, unsigned max_grid)
{
    if (s.kind == kKindRayChunked) return launch_ray_mc_shape(precision, s, args, stream, grid_out, max_grid);
    const bool tw = args.n_tw > 0, lut = args.lut != nullptr;
    const RayEntry *tab = lut ? kRayShapesLUT : (tw ? kRayShapesTW : kRayShapes);
    const int ntab = lut  ? (int)(sizeof(kRayShapesLUT) / sizeof(RayEntry))
                     : tw ? (int)(sizeof(kRayShapesTW) / sizeof(RayEntry))
                          : (int)(sizeof(kRayShapes) / sizeof(RayEntry));
    for (int k = 0; k < ntab; ++k) {
        const RayEntry &e = tab[k];
        if (e.precision == precision && e.c == s.cells_per_lane && e.w == s.warps &&
            (s.min_blocks == 0 || e.minb == s.min_blocks) && ray_warps_per_ray(e.c, args.nr) > 0)
            return e.fn(args, 0, stream, grid_out, max_grid);
    }
    return cudaErrorInvalidValue;
}

}  // namespace rt
