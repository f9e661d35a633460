// proposal_rays.cuh -- the rays of the proposal kernels' tiles (2 rays x 64 bins): box clips and bin centres.
#pragma once

#include "df64.cuh"
#include "dvgo_internal.cuh"

namespace dvgo {

constexpr int kPropBins = 64;

// Box clip of one ray as the encoding uses it: entry t0, bin width w = (t_exit - t_enter) / 64 and
// direction as double-float values of the FP64 clip, the origin, and whether the ray hits the box.
struct ClipDf {
    Df t0, w, dn[3];
    float o[3];
    int hit;        // 0; 1; 3: and its origin or exit lies further out than kDfReach
};
// Coordinates and distances up to which double-float positions do for the FP32 network: 2^5 x 2^12 x 2^-47 =
// 2^-30 in an encoded argument.
constexpr double kDfReach = 4096.0;

// Box clips (FP64, as in the renderer) of the rays of the CTA's tiles k0 .. k0 + 63 (its k-th tile
// is blockIdx.x + k gridDim.x, rays 2 tile and 2 tile + 1), one ray per thread (the first 128).
// Clipping per ray instead of per tile keeps the FP64 work (1/64 of the FP32 rate on this GPU) off the
// tile loop.
__device__ __forceinline__ void clip_tile_rays(int R, const float *ro, const float *rd, const double mn[3],
                                               const double mx[3], double t_near, double t_far, int k0, ClipDf *cl) {
    const int tid = threadIdx.x;
    const long long tile = blockIdx.x + (long long)(k0 + (tid >> 1)) * gridDim.x, r = 2 * tile + (tid & 1);
    ClipDf c;
    c.t0 = c.w = c.dn[0] = c.dn[1] = c.dn[2] = Df{0.0f, 0.0f};
    c.o[0] = c.o[1] = c.o[2] = 0.0f;
    c.hit = 0;
    if (r < R) {
        const double o[3] = {(double)ro[3 * r], (double)ro[3 * r + 1], (double)ro[3 * r + 2]};
        const double d[3] = {(double)rd[3 * r], (double)rd[3 * r + 1], (double)rd[3 * r + 2]};
        const Clip q = slab_clip(o, d, mn, mx, t_near, t_far);
        c.hit = q.hi > q.lo;
        if (c.hit) {
            if (fmax(q.hi, fmax(fabs(o[0]), fmax(fabs(o[1]), fabs(o[2])))) > kDfReach) c.hit = 3;
            c.t0 = df_from_double(q.lo);
            c.w = df_from_double(__dmul_rn(__dsub_rn(q.hi, q.lo), 1.0 / kPropBins));   // exact: a power of two
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                c.dn[a] = df_from_double(q.dn[a]);
                c.o[a] = ro[3 * r + a];
            }
        }
    }
    cl[tid] = c;
}

// Distance of the centre of a bin, and the position there on axis a, as double-float values.
__device__ __forceinline__ Df bin_centre(const ClipDf &c, int bin) {
    return df_add(c.t0, df_mul_f(c.w, (float)bin + 0.5f));
}
__device__ __forceinline__ Df bin_position(const ClipDf &c, Df tb, int a) {
    return df_add(Df{c.o[a], 0.0f}, df_mul(tb, c.dn[a]));
}

}  // namespace dvgo
