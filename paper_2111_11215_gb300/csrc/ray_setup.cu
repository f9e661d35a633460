// ray_setup.cu -- per-ray clipping and sample counting, and the workspace layout.
//
// Sec. 4.2 (fine-stage points sampling): the near and far bounds of every ray become the two
// ends of its intersection with the grid's bounding box (the near bound stays put when the
// origin is inside).  Eq. coarse_sample / Supp. A: samples are equally spaced by the step and
// shifted by the per-ray jitter p.  With a normalised direction the count is the number of k >= 0
// with t_enter + (k + p) * step < t_exit.
//
// The count is an integer decided by floating point, so it is computed in FP64 with every
// operation a separately rounded IEEE operation (__dadd_rn & co. keep nvcc from contracting
// them into FMAs):
//   len   = sqrt((dx*dx + dy*dy) + dz*dz),   dn = d / len
//   per axis with dn != 0: t1 = (min - o) / dn, t2 = (max - o) / dn, lo = max(lo, min(t1, t2)),
//                          hi = min(hi, max(t1, t2));  starting from lo = t_near, hi = t_far
//   per axis with dn == 0 and o outside the slab: empty
//   n = ceil((hi - lo) / step - p) when hi > lo, capped at ceil(|max - min| / step) + 1.

#include "dvgo_internal.cuh"

namespace dvgo {

namespace {

// Thread per ray.  Every ray owns cap sample slots (the workspace is sized for the longest ray), so a
// ray's first slot is ray * cap and no scan of the counts runs before the sample passes: one scan block
// took 14 us for 8,192 rays and 97 us for 65,536.  Bound by the FP64 pipe (2 lanes a clock per SM), hence
// the divisions by known reciprocals (div_by) and no position that the sampling in use does not read.
// Records and encodings are written from registers, 16 bytes a store: staging them through shared memory
// would give whole-line stores, but the set-up runs beside the feature-grid Adam, whose loads take the
// SM's whole L1, and a block with shared memory then waits for the Adam to end (152 us instead of 20).
// Set-up and scan before, set-up alone now (events around the launches): 8,192 rays 32 -> 13 us, 65,536
// rays 126 -> 27 us.
constexpr int kSetupThreads = 64;

__global__ void __launch_bounds__(kSetupThreads) ray_setup_kernel(RenderArgs A, const float *__restrict__ rays_o,
                                                                   const float *__restrict__ rays_d,
                                                                   const float *__restrict__ jitter, double3 bmin,
                                                                   double3 bmax, double3 scale, double t_near,
                                                                   double t_far, double step, double inv_step,
                                                                   double cap, int n_expl) {
    const int r = blockIdx.x * kSetupThreads + threadIdx.x;
    if (r == 0) {
        A.hdr->flags = 0;
        A.hdr->n_kept = 0;
        A.hdr->done = 0u;
        A.hdr->loss_acc = 0.0;
        A.hdr->aux = (A.target && (A.w_pt != 0.0f || A.w_bg != 0.0f)) ? 1 : 0;
        A.hdr->xcache = A.xcache != nullptr ? 1 : 0;
        const bool fine = A.rayk != nullptr;
        const auto at = [&](const void *p) {
            return fine ? (unsigned long long)(static_cast<const char *>(p) - reinterpret_cast<const char *>(A.hdr)) : 0ull;
        };
        A.hdr->n_rays = fine ? A.R : 0;
        A.hdr->cap = A.cap;
        A.hdr->texit_at = at(A.texit);
        A.hdr->rayk_at = at(A.rayk);
        A.hdr->rchunk_at = at(A.rchunk);
        A.hdr->stau_at = at(A.stau);
    }
    if (r >= A.R) return;
    double o[3] = {(double)rays_o[3 * r], (double)rays_o[3 * r + 1], (double)rays_o[3 * r + 2]};
    double d[3] = {(double)rays_d[3 * r], (double)rays_d[3 * r + 1], (double)rays_d[3 * r + 2]};
    double mn[3] = {bmin.x, bmin.y, bmin.z}, mx[3] = {bmax.x, bmax.y, bmax.z};
    double sc[3] = {scale.x, scale.y, scale.z};
    double p = jitter ? (double)jitter[r] : 0.5;

    const Clip cl = slab_clip(o, d, mn, mx, t_near, t_far);
    const double lo = cl.lo, hi = cl.hi;
    alignas(16) RayRec rec;
    int n = 0;
    if (hi > lo) {
        double q = div_by(__dsub_rn(hi, lo), step, inv_step);
        q = __dsub_rn(q, p);
        double c = ceil(q);
        if (c > cap) c = cap;
        n = c > 0.0 ? (int)c : 0;
        if (n_expl >= 0) n = n_expl;   // explicit samples: all or nothing
    }
    const bool uniform = n_expl < 0;
    const double t_first = uniform ? fma(p, step, lo) : lo;   // t of sample 0 of the uniform stepping
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double uo = __dmul_rn(__dsub_rn(o[a], mn[a]), sc[a]);
        rec.e[a] = __dmul_rn(cl.dn[a], sc[a]);
        rec.dir[a] = (float)cl.dn[a];
        // fixed-point values only where they are used: in range for any sample inside the box
        const long long u = n > 0 ? to_fx(fma(t_first, rec.e[a], uo)) : 0;
        rec.uefx[a] = uniform ? 0 : u;
        rec.u0fx[a] = uniform ? u : 0;
        rec.dfx[a] = uniform && n > 0 ? to_fx(step * rec.e[a]) : 0;
    }
    rec.t_enter = lo;
    rec.p = (float)p;
    rec.n = n;
    rec.off = cl.ok ? r * A.cap : -1;
    const ulonglong2 *w = reinterpret_cast<const ulonglong2 *>(&rec);
    ulonglong2 *g = reinterpret_cast<ulonglong2 *>(A.rays + r);
#pragma unroll
    for (int k = 0; k < (int)sizeof(RayRec) / 16; ++k) g[k] = w[k];
    if (A.texit) A.texit[r] = hi;
    if (A.pe) {
        // positional encoding of the normalised direction (fine-stage MLP input, Supp. A, k_d = 4):
        // [d, sin(2^k d_c) (c-major), cos(2^k d_c) (c-major)]
        float pe[kPeStride];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            pe[a] = rec.dir[a];
#pragma unroll
            for (int k = 0; k < 4; ++k) sincosf(ldexpf(rec.dir[a], k), &pe[3 + a * 4 + k], &pe[15 + a * 4 + k]);
        }
#pragma unroll
        for (int k = 27; k < kPeStride; ++k) pe[k] = 0.0f;
        float4 *gp = reinterpret_cast<float4 *>(A.pe + (size_t)r * kPeStride);
#pragma unroll
        for (int k = 0; k < kPeStride / 4; ++k)
            gp[k] = make_float4(pe[4 * k], pe[4 * k + 1], pe[4 * k + 2], pe[4 * k + 3]);
    }
}

}  // namespace

void launch_ray_setup(const RenderArgs &A, const float *rays_o, const float *rays_d, const float *jitter,
                      const dvgo_params &p, const dvgo_grid_desc &g, long long cap, cudaStream_t s) {
    double3 bmin = make_double3(g.xyz_min[0], g.xyz_min[1], g.xyz_min[2]);
    double3 bmax = make_double3(g.xyz_max[0], g.xyz_max[1], g.xyz_max[2]);
    double3 sc = make_double3((double)(g.nx - 1) / (bmax.x - bmin.x), (double)(g.ny - 1) / (bmax.y - bmin.y),
                              (double)(g.nz - 1) / (bmax.z - bmin.z));
    const int blocks = (A.R + kSetupThreads - 1) / kSetupThreads;
    ProfScope ps_(DVGO_K_RAY_SETUP, s);
    ray_setup_kernel<<<blocks, kSetupThreads, 0, s>>>(A, rays_o, rays_d, jitter, bmin, bmax, sc, (double)p.t_near,
                                                      (double)p.t_far, (double)p.step, 1.0 / (double)p.step,
                                                      (double)cap, A.ts ? A.n_expl : -1);
}

WsLayout ws_layout(int R, long long max_samples, int mode, bool xcache, size_t mask_words) {
    auto up = [](size_t x) { return (x + 255) & ~(size_t)255; };
    WsLayout L;
    memset(&L, 0, sizeof(L));
    size_t o = 0;
    const size_t n = (size_t)(R > 0 ? R : 1);
    L.header = o; o += up(sizeof(WsHeader));
    L.rays = o; o += up(sizeof(RayRec) * n);
    L.rayout = o; o += up(sizeof(float4) * n);
    const size_t S = (size_t)(max_samples > 0 ? max_samples : 1);
    if (mode == DVGO_MODE_FINE) {
        L.pe = o; o += up(sizeof(float) * kPeStride * n);
        L.texit = o; o += up(sizeof(double) * n);
        L.rayk = o; o += up(sizeof(int4) * n);
        L.rchunk = o; o += up(sizeof(RayChunk) * n * chunks_per_ray((long long)(S / n)));
        L.stau = o; o += up(sizeof(float) * S);
        L.scol = o; o += up(sizeof(float4) * S);
        L.sgrad = o; o += up(sizeof(float4) * S);
        L.kept = o; o += up(sizeof(int2) * S);
    }
    // last; counted in total, so the allocation-free forward's static scratch includes it even
    // though that forward (no auxiliary losses) never writes it
    L.rtarget = o; o += up(sizeof(float4) * n);
    if (xcache && mode == DVGO_MODE_FINE) {   // 128 kept samples per tile, a 16 KiB panel each
        o = (o + 1023) & ~(size_t)1023;
        L.xcache = o;
        o += (size_t)16384 * ((S + 127) / 128);
    }
    L.need = o;
    if (mask_words > 0 && mode == DVGO_MODE_FINE) { o = up(o); L.mask = o; o += up(sizeof(unsigned) * mask_words); }
    L.total = o;
    L.max_samples = max_samples;
    return L;
}

}  // namespace dvgo
