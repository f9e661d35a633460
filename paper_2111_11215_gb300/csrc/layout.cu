// layout.cu -- grid storage: element counts, the copy between the canonical channel-last layout and
// the packed one (4x4x4 bricks, Morton order inside a brick) with FP32 / BF16 conversion (one
// thread per (lattice point, channel) of the source lattice), and the trilinear resize of
// progressive scaling (Sec. 4.2; a block per chunk of destination rows).

#include <cuda_bf16.h>

#include "df64.cuh"
#include "dvgo_internal.cuh"

namespace dvgo {

namespace {

long long lattice_points(const dvgo_grid_desc &g) {
    if (g.layout == DVGO_LAYOUT_PACKED)
        return (long long)((g.nx + 3) / 4) * ((g.ny + 3) / 4) * ((g.nz + 3) / 4) * 64;
    return (long long)g.nx * g.ny * g.nz;
}

template <typename TIn, typename TOut>
__device__ __forceinline__ TOut convert(TIn v);
template <> __device__ __forceinline__ float convert<float, float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 convert<float, __nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }
template <> __device__ __forceinline__ float convert<__nv_bfloat16, float>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <> __device__ __forceinline__ __nv_bfloat16 convert<__nv_bfloat16, __nv_bfloat16>(__nv_bfloat16 v) { return v; }

template <typename TIn, typename TOut>
__global__ void __launch_bounds__(256) pack_kernel(const TIn *__restrict__ in, TOut *__restrict__ out, int nx, int ny,
                                                   int nz, int C, int src_packed, int dst_packed) {
    const long long n = (long long)nx * ny * nz * C;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
        const int ch = (int)(t % C);
        const long long p = t / C;
        const int k = (int)(p % nz), j = (int)((p / nz) % ny), i = (int)(p / ((long long)ny * nz));
        const long long si = grid_index(i, j, k, ny, nz, src_packed != 0) * C + ch;
        const long long di = grid_index(i, j, k, ny, nz, dst_packed != 0) * C + ch;
        out[di] = convert<TIn, TOut>(in[si]);
    }
}

template <typename TIn, typename TOut>
void launch_pack(const dvgo_grid_desc &s, const void *in, const dvgo_grid_desc &d, void *out, cudaStream_t st) {
    const long long n = (long long)s.nx * s.ny * s.nz * s.channels;
    long long blocks = (n + 255) / 256;
    if (blocks > (long long)num_sms() * 16) blocks = (long long)num_sms() * 16;
    if (blocks < 1) blocks = 1;
    pack_kernel<TIn, TOut><<<(unsigned)blocks, 256, 0, st>>>(static_cast<const TIn *>(in), static_cast<TOut *>(out),
                                                             s.nx, s.ny, s.nz, s.channels,
                                                             s.layout == DVGO_LAYOUT_PACKED, d.layout == DVGO_LAYOUT_PACKED);
}

struct Axis3 {
    double v[3];
};

// Trilinear resize.  A destination point's position is clamped into the source box and turned into
// a source lattice coordinate per axis, u = (x - min) / (max - min) (n - 1), i0 = clamp(floor(u), 0,
// n - 2), f = u - i0, in FP64 (the interpolation of Sec. 3 Eq. interp); weights and sums then carry
// two FP32 words each (df64.cuh), and the result is rounded once to FP32.
//
// FP64 runs at 1/64 of the FP32 rate here, so only the per-axis coordinates use it: a block owns a
// chunk of up to kResizeZ destination points of one z range for up to kResizeRows (i, j) rows, and
// forms the coordinates of its z points and of its rows once.  Per row it (1) sums the four source
// rows around (i, j) into one row of two-word values in shared memory -- every source value is read
// once per row, coalesced along z and channels -- and (2) interpolates that row along z.  When the
// destination's z spacing is more than twice the source's, the source points between the wanted pairs
// would be summed for nothing, so stage 1 then forms just the two points of each destination point.
// The two-word sum of products keeps ~2^-46 of the largest term.  127^3 -> 160^3, density and 12
// channels (320 MB in and out): 3414 us with FP64 sums, 290 us so.
constexpr int kResizeThreads = 256;
constexpr int kResizeZ = 256;       // destination points per chunk, at most
constexpr int kResizeRows = 64;     // rows per block, at most
constexpr int kResizeElems = 2560;  // two-word source values per row and chunk (two buffers of 20 KB)
constexpr int kResizeCh = 64;       // channels per block

struct AxisPos {
    int i0;
    Df w[2];   // weights of i0 and i0 + 1
};

__device__ __forceinline__ AxisPos axis_pos(int i, int dn, double dmin, double dmax, int sn, double smin, double smax) {
    double x = dmin + (double)i * (dmax - dmin) / (double)(dn - 1);
    x = fmin(fmax(x, smin), smax);
    const double u = (x - smin) / (smax - smin) * (double)(sn - 1);
    const double fl = fmin(fmax(floor(u), 0.0), (double)(sn - 2));
    AxisPos p;
    p.i0 = (int)fl;
    p.w[0] = df_from_double(1.0 - (u - fl));
    p.w[1] = df_from_double(u - fl);
    return p;
}

// (s, c) += w v: the product and the sum error-free, the errors gathered in c (compensated dot
// product of Ogita, Rump and Oishi, 2005).
__device__ __forceinline__ void dot_add(float &s, float &c, Df w, float v) {
    const float p = __fmul_rn(w.hi, v);
    const float e = __fmaf_rn(w.lo, v, __fmaf_rn(w.hi, v, -p));
    const Df t = df_two_sum(s, p);
    s = t.hi;
    c = __fadd_rn(c, __fadd_rn(t.lo, e));
}

struct ResizeArgs {
    const float *in;
    float *out;
    int C, sn[3], dn[3], s_packed, d_packed;
    Axis3 dmin, dmax, smin, smax;
    int zlen, rows_per_block, pairs;   // destination points per chunk; rows per block; stage 1 per pair
    unsigned zchunks, cchunks;         // chunks along z and of the channels (blockIdx.x = (rows, z, channels))
};

__global__ void __launch_bounds__(kResizeThreads) resize_kernel(ResizeArgs A) {
    __shared__ float2 comb[2][kResizeElems];
    __shared__ Df zw[kResizeZ][2];
    __shared__ short zi[kResizeZ];             // first of the two entries of comb of a z point
    __shared__ int zsrc[kResizeZ];             // source index of a z point
    __shared__ Df rw[kResizeRows][4];          // weights of the four source rows (x bit, y bit)
    __shared__ int rij[kResizeRows][2];
    const int tid = threadIdx.x;
    const unsigned cb = blockIdx.x % A.cchunks, zb = (blockIdx.x / A.cchunks) % A.zchunks;
    const int z0 = (int)zb * A.zlen, zn = min(A.zlen, A.dn[2] - z0);
    const int ch0 = (int)cb * kResizeCh, cc = min(kResizeCh, A.C - ch0);
    const long long nrows = (long long)A.dn[0] * A.dn[1];
    const long long r0 = (long long)(blockIdx.x / A.cchunks / A.zchunks) * A.rows_per_block;
    const int rn = (int)min((long long)A.rows_per_block, nrows - r0);
    for (int k = tid; k < zn; k += kResizeThreads) {
        const AxisPos p = axis_pos(z0 + k, A.dn[2], A.dmin.v[2], A.dmax.v[2], A.sn[2], A.smin.v[2], A.smax.v[2]);
        zsrc[k] = p.i0;
        zw[k][0] = p.w[0];
        zw[k][1] = p.w[1];
    }
    for (int r = tid; r < rn; r += kResizeThreads) {
        const long long row = r0 + r;
        const int i = (int)(row / A.dn[1]), j = (int)(row - (long long)i * A.dn[1]);
        const AxisPos px = axis_pos(i, A.dn[0], A.dmin.v[0], A.dmax.v[0], A.sn[0], A.smin.v[0], A.smax.v[0]);
        const AxisPos py = axis_pos(j, A.dn[1], A.dmin.v[1], A.dmax.v[1], A.sn[1], A.smin.v[1], A.smax.v[1]);
        rij[r][0] = px.i0;
        rij[r][1] = py.i0;
#pragma unroll
        for (int q = 0; q < 4; ++q) rw[r][q] = df_mul(px.w[q >> 1], py.w[q & 1]);
    }
    __syncthreads();
    const int kbase = zsrc[0];
    for (int k = tid; k < zn; k += kResizeThreads) zi[k] = (short)(A.pairs ? 2 * k : zsrc[k] - kbase);
    // entries of a row: the source span of the chunk, or two per destination point
    const int ne = (A.pairs ? 2 * zn : zsrc[zn - 1] - kbase + 2) * cc;
    const int nd = zn * cc;
    const unsigned inv = (unsigned)((0x100000000ull + cc - 1) / cc);   // el / cc = el inv >> 32 (el < 2^15; cc > 1)
    auto split = [&](int el, int &k, int &ch) {
        k = cc == 1 ? el : (int)__umulhi((unsigned)el, inv);
        ch = el - k * cc;
    };
    __syncthreads();
    int buf = 0;
    for (int r = 0; r < rn; ++r, buf ^= 1) {
        const int si = rij[r][0], sj = rij[r][1];
        Df w[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) w[q] = rw[r][q];
        if (!A.s_packed && !A.pairs && cc == A.C) {   // the four source rows are contiguous: no index arithmetic
            const float *p0 = A.in + (((long long)si * A.sn[1] + sj) * A.sn[2] + kbase) * A.C;
            const long long dy = (long long)A.sn[2] * A.C, dx = dy * A.sn[1];
#pragma unroll 2
            for (int el = tid; el < ne; el += kResizeThreads) {
                float s = 0.0f, c = 0.0f;
                const float v0 = __ldg(p0 + el), v1 = __ldg(p0 + dy + el), v2 = __ldg(p0 + dx + el),
                            v3 = __ldg(p0 + dx + dy + el);
                dot_add(s, c, w[0], v0);
                dot_add(s, c, w[1], v1);
                dot_add(s, c, w[2], v2);
                dot_add(s, c, w[3], v3);
                comb[buf][el] = make_float2(s, c);
            }
        } else {
            for (int el = tid; el < ne; el += kResizeThreads) {
                int e, ch;
                split(el, e, ch);
                const int k = A.pairs ? zsrc[e >> 1] + (e & 1) : kbase + e;
                float s = 0.0f, c = 0.0f;
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    dot_add(s, c, w[q],
                            __ldg(A.in + grid_index(si + (q >> 1), sj + (q & 1), k, A.sn[1], A.sn[2], A.s_packed != 0) * A.C +
                                  ch0 + ch));
                comb[buf][el] = make_float2(s, c);
            }
        }
        __syncthreads();   // (the next row writes the other buffer, so one barrier a row is enough)
        const long long row = r0 + r;
        const int i = (int)(row / A.dn[1]), j = (int)(row - (long long)i * A.dn[1]);
        float *po = A.out + ((long long)row * A.dn[2] + z0) * A.C;
        for (int el = tid; el < nd; el += kResizeThreads) {
            int k, ch;
            split(el, k, ch);
            const float2 a = comb[buf][zi[k] * cc + ch], b = comb[buf][(zi[k] + 1) * cc + ch];
            const Df wa = zw[k][0], wb = zw[k][1];
            const float pa = __fmul_rn(wa.hi, a.x), pb = __fmul_rn(wb.hi, b.x);
            const float ea = __fmaf_rn(wa.lo, a.x, __fmaf_rn(wa.hi, a.y, __fmaf_rn(wa.hi, a.x, -pa)));
            const float eb = __fmaf_rn(wb.lo, b.x, __fmaf_rn(wb.hi, b.y, __fmaf_rn(wb.hi, b.x, -pb)));
            const Df t = df_two_sum(pa, pb);
            // an infinite or NaN sum is the result (its error terms are NaN)
            const float v = isfinite(t.hi) ? __fadd_rn(t.hi, __fadd_rn(t.lo, __fadd_rn(ea, eb))) : t.hi;
            if (!A.d_packed && cc == A.C) po[el] = v;
            else A.out[grid_index(i, j, z0 + k, A.dn[1], A.dn[2], A.d_packed != 0) * A.C + ch0 + ch] = v;
        }
    }
}

bool desc_ok(const dvgo_grid_desc *g) {
    return g && g->nx >= 2 && g->ny >= 2 && g->nz >= 2 && g->channels >= 1 &&
           (g->layout == DVGO_LAYOUT_CANONICAL || g->layout == DVGO_LAYOUT_PACKED) &&
           (g->dtype == DVGO_DTYPE_F32 || g->dtype == DVGO_DTYPE_BF16);
}

}  // namespace

}  // namespace dvgo

using namespace dvgo;

extern "C" {

size_t dvgo_grid_elements(const dvgo_grid_desc *g) {
    if (!desc_ok(g)) return 0;
    return (size_t)lattice_points(*g) * (size_t)g->channels;
}

int dvgo_pack_grid(const dvgo_grid_desc *src, const void *in, const dvgo_grid_desc *dst, void *out, void *stream) {
    if (!desc_ok(src) || !desc_ok(dst) || !in || !out) return DVGO_ERR_INVALID_ARG;
    if (src->nx != dst->nx || src->ny != dst->ny || src->nz != dst->nz || src->channels != dst->channels)
        return DVGO_ERR_INVALID_ARG;
    for (int a = 0; a < 3; ++a)
        if (src->xyz_min[a] != dst->xyz_min[a] || src->xyz_max[a] != dst->xyz_max[a]) return DVGO_ERR_INVALID_ARG;
    if (in == out) return DVGO_ERR_INVALID_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const size_t out_bytes = dvgo_grid_elements(dst) * (dst->dtype == DVGO_DTYPE_BF16 ? 2 : 4);
    {
        ProfScope ps_(DVGO_K_AUX, s);
        if (dst->layout == DVGO_LAYOUT_PACKED) cudaMemsetAsync(out, 0, out_bytes, s);   // padding points
        const bool sb = src->dtype == DVGO_DTYPE_BF16, db = dst->dtype == DVGO_DTYPE_BF16;
        if (!sb && !db) launch_pack<float, float>(*src, in, *dst, out, s);
        else if (!sb && db) launch_pack<float, __nv_bfloat16>(*src, in, *dst, out, s);
        else if (sb && !db) launch_pack<__nv_bfloat16, float>(*src, in, *dst, out, s);
        else launch_pack<__nv_bfloat16, __nv_bfloat16>(*src, in, *dst, out, s);
    }
    return cudaGetLastError() == cudaSuccess ? DVGO_OK : DVGO_ERR_CUDA;
}

int dvgo_resize_grid(const dvgo_grid_desc *src, const float *in, const dvgo_grid_desc *dst, float *out, void *stream) {
    if (!desc_ok(src) || !desc_ok(dst) || !in || !out || in == out) return DVGO_ERR_INVALID_ARG;
    if (src->dtype != DVGO_DTYPE_F32 || dst->dtype != DVGO_DTYPE_F32 || src->channels != dst->channels)
        return DVGO_ERR_INVALID_ARG;
    for (int a = 0; a < 3; ++a)
        if (!isfinite(src->xyz_min[a]) || !isfinite(src->xyz_max[a]) || !(src->xyz_max[a] > src->xyz_min[a]) ||
            !isfinite(dst->xyz_min[a]) || !isfinite(dst->xyz_max[a]) || !(dst->xyz_max[a] > dst->xyz_min[a]))
            return DVGO_ERR_INVALID_ARG;
    if (dvgo_grid_elements(src) >= (1ull << 31) || dvgo_grid_elements(dst) >= (1ull << 31)) return DVGO_ERR_UNSUPPORTED;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    ResizeArgs A;
    A.in = in;
    A.out = out;
    A.C = src->channels;
    const int sn[3] = {src->nx, src->ny, src->nz}, dn[3] = {dst->nx, dst->ny, dst->nz};
    for (int a = 0; a < 3; ++a) {
        A.sn[a] = sn[a];
        A.dn[a] = dn[a];
        A.dmin.v[a] = dst->xyz_min[a];
        A.dmax.v[a] = dst->xyz_max[a];
        A.smin.v[a] = src->xyz_min[a];
        A.smax.v[a] = src->xyz_max[a];
    }
    A.s_packed = src->layout == DVGO_LAYOUT_PACKED;
    A.d_packed = dst->layout == DVGO_LAYOUT_PACKED;
    // source points per destination point along z; up to 2 the whole span of a chunk is summed
    const double ratio = (A.dmax.v[2] - A.dmin.v[2]) / (dn[2] - 1) / ((A.smax.v[2] - A.smin.v[2]) / (sn[2] - 1));
    A.pairs = ratio > 2.0;
    const int cc = A.C < kResizeCh ? A.C : kResizeCh;
    // a chunk of zlen points spans at most (zlen - 1) ratio + 3 source points (two more for the rounding)
    const double fit = A.pairs ? (kResizeElems / cc) / 2.0 : (kResizeElems / cc - 5) / (ratio < 1e-3 ? 1e-3 : ratio);
    A.zlen = fit < kResizeZ ? (int)fit : kResizeZ;
    if (A.zlen > dn[2]) A.zlen = dn[2];
    const long long zchunks = (dn[2] + A.zlen - 1) / A.zlen, cchunks = (A.C + kResizeCh - 1) / kResizeCh;
    const long long rows = (long long)dn[0] * dn[1];
    // 4 blocks per SM in one wave where the rows allow it: the per-block coordinates are paid once
    long long rpb = (rows * zchunks * cchunks + num_sms() * 4 - 1) / (num_sms() * 4);
    A.rows_per_block = (int)(rpb < 1 ? 1 : (rpb > kResizeRows ? kResizeRows : rpb));
    A.zchunks = (unsigned)zchunks;
    A.cchunks = (unsigned)cchunks;
    const unsigned blocks = (unsigned)((rows + A.rows_per_block - 1) / A.rows_per_block * zchunks * cchunks);
    {
        ProfScope ps_(DVGO_K_AUX, s);
        if (dst->layout == DVGO_LAYOUT_PACKED) cudaMemsetAsync(out, 0, dvgo_grid_elements(dst) * sizeof(float), s);
        resize_kernel<<<blocks, kResizeThreads, 0, s>>>(A);
    }
    return cudaGetLastError() == cudaSuccess ? DVGO_OK : DVGO_ERR_CUDA;
}

}  // extern "C"
