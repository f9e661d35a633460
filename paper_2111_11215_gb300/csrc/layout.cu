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

// Trilinear resize.  A destination point's position is clamped into the source box and turned into
// a source lattice coordinate per axis, u = (x - min) / (max - min) (n - 1), i0 = clamp(floor(u), 0,
// n - 2), f = u - i0, in FP64 (the interpolation of Sec. 3 Eq. interp); weights and sums then carry
// two FP32 words each (df64.cuh), and the result is rounded once to FP32.
//
// FP64 runs at 1/64 of the FP32 rate here, so only the per-axis coordinates use it: a block owns a
// chunk of up to kResizeZ destination points of one z range for up to kResizeRows consecutive rows (i, j), and
// forms the coordinates of its z points and rows once.  It walks along the rows and keeps the two source rows
// around it, already interpolated along x (two-word values in shared memory: every source value is read
// once per plane pair and block, coalesced along z and channels); per destination row (1) a source row that
// is new is interpolated along x, (2) the two are interpolated along y, (3) the result along z.  When the
// destination's z spacing is more than twice the source's, the source points between the wanted pairs
// would be summed for nothing, so the rows then hold just the two points of each destination point.
// The two-word sums of products keep ~2^-46 of the largest term.  127^3 -> 160^3, density and 12
// channels (320 MB in and out): 3414 us with FP64 sums, 248 us so (200 us of it
// the features: FMA pipe 30 %, ALU 26 %, barriers between the three short passes of a row).
constexpr int kResizeZ = 256;       // destination points per chunk, at most
constexpr int kResizeRows = 64;     // rows per block, at most
constexpr int kResizeElems = 2048;  // two-word source values per row and chunk, at most
constexpr int kResizeCh = 64;       // channels per block

struct ResizeAxis {
    double dmin, dspan, dinv, smin, smax, sspan, sinv;   // dinv = 1 / (dn - 1), sinv = 1 / sspan
    int dn, sn;
};

struct AxisPos {
    int i0;
    Df w[2];   // weights of i0 and i0 + 1
};

// (div_by: the correctly rounded quotients)
__device__ __forceinline__ AxisPos axis_pos(int i, const ResizeAxis &a) {
    double x = a.dmin + div_by((double)i * a.dspan, (double)(a.dn - 1), a.dinv);
    x = fmin(fmax(x, a.smin), a.smax);
    const double u = div_by(x - a.smin, a.sspan, a.sinv) * (double)(a.sn - 1);
    const double fl = fmin(fmax(floor(u), 0.0), (double)(a.sn - 2));
    AxisPos p;
    p.i0 = (int)fl;
    p.w[0] = df_from_double(1.0 - (u - fl));
    p.w[1] = df_from_double(u - fl);
    return p;
}

// w0 v0 + w1 v1 of two-word weights and FP32 values / two-word values: products and sums error-free, the
// errors gathered in the low word (compensated dot product of Ogita, Rump and Oishi, 2005).
__device__ __forceinline__ float2 lerp_f(Df w0, float v0, Df w1, float v1) {
    const float p0 = __fmul_rn(w0.hi, v0), p1 = __fmul_rn(w1.hi, v1);
    const float e0 = __fmaf_rn(w0.lo, v0, __fmaf_rn(w0.hi, v0, -p0)), e1 = __fmaf_rn(w1.lo, v1, __fmaf_rn(w1.hi, v1, -p1));
    const Df t = df_two_sum(p0, p1);
    return make_float2(t.hi, __fadd_rn(t.lo, __fadd_rn(e0, e1)));
}
__device__ __forceinline__ float2 lerp_df(Df w0, float2 v0, Df w1, float2 v1) {
    const float p0 = __fmul_rn(w0.hi, v0.x), p1 = __fmul_rn(w1.hi, v1.x);
    const float e0 = __fmaf_rn(w0.lo, v0.x, __fmaf_rn(w0.hi, v0.y, __fmaf_rn(w0.hi, v0.x, -p0)));
    const float e1 = __fmaf_rn(w1.lo, v1.x, __fmaf_rn(w1.hi, v1.y, __fmaf_rn(w1.hi, v1.x, -p1)));
    const Df t = df_two_sum(p0, p1);
    return make_float2(t.hi, __fadd_rn(t.lo, __fadd_rn(e0, e1)));
}

struct ResizeArgs {
    const float *in;
    float *out;
    int C, s_packed, d_packed;
    ResizeAxis ax[3];
    int zlen, rows_per_block, pairs;   // destination points per chunk; rows per block; rows of point pairs
    unsigned zchunks, cchunks;         // blockIdx.x = (rows, z, channels)
    int elems;                         // two-word values of a row buffer (a multiple of 4)
    int walkers;                       // row walkers per block, of 256 / walkers threads
};

// V: 4 where the channels are a multiple of 4 in canonical grids on 16-byte boundaries (a thread takes four
// channels of a point: one index computation, 16-byte accesses), else 1.
template <int V>
__global__ void __launch_bounds__(256) resize_kernel(ResizeArgs A) {
    extern __shared__ __align__(16) float2 s_rows[];   // per walker: rowx[2][elems], comb[elems]
    __shared__ __align__(16) Df zw[kResizeZ][2];
    __shared__ short zi[kResizeZ];             // first of the two entries of a row of a z point
    __shared__ int zsrc[kResizeZ];             // source index of a z point
    __shared__ Df yw[kResizeRows][2], xw[kResizeRows][2];
    __shared__ int yj[kResizeRows], xi[kResizeRows];
    const int nt = blockDim.x / A.walkers, walker = threadIdx.x / nt, tid = threadIdx.x - walker * nt;
    unsigned b = blockIdx.x;
    const unsigned cb = b % A.cchunks;
    b /= A.cchunks;
    const unsigned zb = b % A.zchunks;
    b /= A.zchunks;
    const int dny = A.ax[1].dn, dnz = A.ax[2].dn, sny = A.ax[1].sn, snz = A.ax[2].sn;
    // rows (i, j) in order, whatever plane they are in
    const long long rb0 = (long long)b * A.rows_per_block * A.walkers;
    const int z0 = (int)zb * A.zlen, zn = min(A.zlen, dnz - z0);
    const int ch0 = (int)cb * kResizeCh, cc = min(kResizeCh, A.C - ch0);
    const int rb = (int)min((long long)A.rows_per_block * A.walkers, (long long)A.ax[0].dn * dny - rb0);   // the block's rows; this walker's
    const int r0 = walker * A.rows_per_block, rn = min(rb, r0 + A.rows_per_block);
    for (int k = threadIdx.x; k < zn; k += blockDim.x) {
        const AxisPos p = axis_pos(z0 + k, A.ax[2]);
        zsrc[k] = p.i0;
        zw[k][0] = p.w[0];
        zw[k][1] = p.w[1];
    }
    for (int r = threadIdx.x; r < rb; r += blockDim.x) {
        const int i = (int)((rb0 + r) / dny);
        const AxisPos p = axis_pos((int)(rb0 + r - (long long)i * dny), A.ax[1]), q = axis_pos(i, A.ax[0]);
        yj[r] = p.i0;
        yw[r][0] = p.w[0];
        yw[r][1] = p.w[1];
        xi[r] = q.i0;
        xw[r][0] = q.w[0];
        xw[r][1] = q.w[1];
    }
    __syncthreads();
    const int kbase = zsrc[0];
    for (int k = threadIdx.x; k < zn; k += blockDim.x) zi[k] = (short)(A.pairs ? 2 * k : zsrc[k] - kbase);
    // entries of a row: the source span of the chunk, or two per destination point
    const int ne = (A.pairs ? 2 * zn : zsrc[zn - 1] - kbase + 2) * cc;
    const int nd = zn * cc;
    const int cv = cc / V;   // channel groups of a point
    const unsigned inv = (unsigned)((0x100000000ull + cv - 1) / cv);   // el / cv = el inv >> 32 (el < 2^15; cv > 1)
    auto split = [&](int el, int &k, int &ch) {
        k = cv == 1 ? el : (int)__umulhi((unsigned)el, inv);
        ch = (el - k * cv) * V;
    };
    // the walker's threads meet at a barrier of their own
    auto sync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(1 + walker), "r"(nt) : "memory"); };
    float2 *base = s_rows + (size_t)walker * 3 * A.elems, *comb = base + 2 * A.elems;
    // V two-word values at el (V = 4: two 16-byte accesses)
    auto load = [](const float2 *p, float2 (&v)[V]) {
        if constexpr (V == 4) {
            const float4 a = reinterpret_cast<const float4 *>(p)[0], c = reinterpret_cast<const float4 *>(p)[1];
            v[0] = make_float2(a.x, a.y);
            v[1] = make_float2(a.z, a.w);
            v[2] = make_float2(c.x, c.y);
            v[3] = make_float2(c.z, c.w);
        } else {
            v[0] = *p;
        }
    };
    auto store = [](float2 *p, const float2 (&v)[V]) {
        if constexpr (V == 4) {
            reinterpret_cast<float4 *>(p)[0] = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
            reinterpret_cast<float4 *>(p)[1] = make_float4(v[2].x, v[2].y, v[3].x, v[3].y);
        } else {
            *p = v[0];
        }
    };
    // source row sj interpolated along x, into the buffer of its parity
    auto row_x = [&](int r, int sj) {
        const int si = xi[r];
        const Df wx0 = xw[r][0], wx1 = xw[r][1];
        float2 *row = base + (sj & 1) * A.elems;
        if (V == 4 || (!A.s_packed && !A.pairs && cc == A.C)) {   // contiguous: no index arithmetic
            const float *p0 = A.in + (((long long)si * sny + sj) * snz + kbase) * A.C;
            const float *p1 = p0 + (long long)sny * snz * A.C;
#pragma unroll 2
            for (int el = tid * V; el < ne; el += nt * V) {
                float2 v[V];
                if constexpr (V == 4) {
                    const float4 a = __ldg(reinterpret_cast<const float4 *>(p0 + el)), c = __ldg(reinterpret_cast<const float4 *>(p1 + el));
                    v[0] = lerp_f(wx0, a.x, wx1, c.x);
                    v[1] = lerp_f(wx0, a.y, wx1, c.y);
                    v[2] = lerp_f(wx0, a.z, wx1, c.z);
                    v[3] = lerp_f(wx0, a.w, wx1, c.w);
                } else {
                    v[0] = lerp_f(wx0, __ldg(p0 + el), wx1, __ldg(p1 + el));
                }
                store(row + el, v);
            }
        } else {
            for (int el = tid; el < ne; el += nt) {
                int e, ch;
                split(el, e, ch);
                const int k = A.pairs ? zsrc[e >> 1] + (e & 1) : kbase + e;
                row[el] = lerp_f(wx0, __ldg(A.in + grid_index(si, sj, k, sny, snz, A.s_packed != 0) * A.C + ch0 + ch), wx1,
                                 __ldg(A.in + grid_index(si + 1, sj, k, sny, snz, A.s_packed != 0) * A.C + ch0 + ch));
            }
        }
    };
    __syncthreads();
    int have = -1;   // rows have and have + 1 of plane `plane` are in place
    long long plane = -1;
    for (int r = r0; r < rn; ++r) {
        const int sj = yj[r];
        const long long row = rb0 + r, i = row / dny;
        if (sj != have || i != plane) {   // (the rows' last readers are past the barrier below)
            if (sj != have + 1 || have < 0 || i != plane) row_x(r, sj);
            row_x(r, sj + 1);
            have = sj;
            plane = i;
        }
        sync();
        const Df wy0 = yw[r][0], wy1 = yw[r][1];
        const float2 *ra = base + (sj & 1) * A.elems, *rc = base + ((sj + 1) & 1) * A.elems;
#pragma unroll 2
        for (int el = tid * V; el < ne; el += nt * V) {
            float2 u[V], w[V];
            load(ra + el, u);
            load(rc + el, w);
#pragma unroll
            for (int q = 0; q < V; ++q) u[q] = lerp_df(wy0, u[q], wy1, w[q]);
            store(comb + el, u);
        }
        sync();
        const int j = (int)(row - i * dny);
        float *po = A.out + (row * dnz + z0) * A.C;
#pragma unroll 2
        for (int el = tid; el < nd / V; el += nt) {
            int k, ch;
            split(el, k, ch);
            const int e = zi[k] * cc + ch;
            const Df w0 = zw[k][0], w1 = zw[k][1];
            float2 u[V], w[V];
            float v[V];
            load(comb + e, u);
            load(comb + e + cc, w);
#pragma unroll
            for (int q = 0; q < V; ++q) {
                u[q] = lerp_df(w0, u[q], w1, w[q]);
                // an infinite or NaN sum is the result (its error terms are NaN)
                v[q] = isfinite(u[q].x) ? __fadd_rn(u[q].x, u[q].y) : u[q].x;
            }
            if constexpr (V == 4) {
                reinterpret_cast<float4 *>(po)[el] = make_float4(v[0], v[1], v[2], v[3]);
            } else {
                if (!A.d_packed && cc == A.C) po[el] = v[0];
                else A.out[grid_index((int)i, j, z0 + k, dny, dnz, A.d_packed != 0) * A.C + ch0 + ch] = v[0];
            }
        }
        // the next row's x pass writes row buffers that nobody reads before its barrier; comb is read here
        // and written after that barrier
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
        ResizeAxis &x = A.ax[a];
        x.dmin = dst->xyz_min[a];
        x.dspan = (double)dst->xyz_max[a] - dst->xyz_min[a];
        x.dn = dn[a];
        x.dinv = 1.0 / (double)(dn[a] - 1);
        x.smin = src->xyz_min[a];
        x.smax = src->xyz_max[a];
        x.sspan = x.smax - x.smin;
        x.sinv = 1.0 / x.sspan;
        x.sn = sn[a];
    }
    A.s_packed = src->layout == DVGO_LAYOUT_PACKED;
    A.d_packed = dst->layout == DVGO_LAYOUT_PACKED;
    // source points per destination point along z; up to 2 the whole span of a chunk is summed
    const double ratio = A.ax[2].dspan / (dn[2] - 1) / (A.ax[2].sspan / (sn[2] - 1));
    A.pairs = ratio > 2.0;
    const int cc = A.C < kResizeCh ? A.C : kResizeCh;
    // a chunk of zlen points spans at most (zlen - 1) ratio + 3 source points (two more for the rounding)
    const double fit = A.pairs ? (kResizeElems / cc) / 2.0 : (kResizeElems / cc - 5) / (ratio < 1e-3 ? 1e-3 : ratio);
    A.zlen = fit < kResizeZ ? (int)fit : kResizeZ;
    if (A.zlen > dn[2]) A.zlen = dn[2];
    const double span = A.pairs ? 2.0 * A.zlen : (A.zlen - 1) * ratio + 5.0;
    A.elems = (int)span * cc < kResizeElems ? ((int)span * cc + 3) & ~3 : kResizeElems;
    A.zchunks = (unsigned)((dn[2] + A.zlen - 1) / A.zlen);
    A.cchunks = (unsigned)((A.C + kResizeCh - 1) / kResizeCh);
    const bool v4 = !A.s_packed && !A.d_packed && !A.pairs && A.C <= kResizeCh && A.C % 4 == 0 &&
                    ((reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out)) & 15u) == 0;
    // A short row leaves threads of a block idle, so it gets a quarter of them and the block walks four runs of
    // rows at once (the z coordinates, FP64, are then formed once for the four; for long rows two runs of 128
    // threads were slower, 252 us against 200: their row buffers let fewer warps onto an SM).  Rows are dealt
    // out so that one wave of four blocks per SM takes them all where they fit (with whole planes per
    // block, 640 blocks on 608 places took two waves).
    A.walkers = A.elems > 768 ? 1 : 4;
    const size_t smem = (size_t)A.walkers * 3 * A.elems * sizeof(float2);
    const long long per = (long long)A.zchunks * A.cchunks, rows = (long long)dn[0] * dn[1];
    const long long slots = (long long)num_sms() * 4 * A.walkers;
    long long rpw = (rows * per + slots - 1) / slots;
    const int most = kResizeRows / A.walkers;
    A.rows_per_block = (int)(rpw < 2 ? 2 : (rpw > most ? most : rpw));
    const long long rpb = (long long)A.rows_per_block * A.walkers;
    const unsigned blocks = (unsigned)((rows + rpb - 1) / rpb * per);
    {
        ProfScope ps_(DVGO_K_AUX, s);
        if (dst->layout == DVGO_LAYOUT_PACKED) cudaMemsetAsync(out, 0, dvgo_grid_elements(dst) * sizeof(float), s);
        auto kern = v4 ? resize_kernel<4> : resize_kernel<1>;
        ensure_smem(reinterpret_cast<const void *>(kern), 4 * 3 * 768 * (int)sizeof(float2));
        kern<<<blocks, 256, smem, s>>>(A);
    }
    return cudaGetLastError() == cudaSuccess ? DVGO_OK : DVGO_ERR_CUDA;
}

}  // extern "C"
