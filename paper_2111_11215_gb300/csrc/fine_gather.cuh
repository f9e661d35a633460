// fine_gather.cuh -- what the producers of the tensor-core colour kernels share: placing a kept sample
// from its ray's record, the trilinear gather of its 12 features (Sec. 4.2 Eq. fine_queries_rgb), and the
// scatter of a tile's feature gradients.
#pragma once

#include "dvgo_internal.cuh"

namespace dvgo {

// The ray data a producer needs to place a sample, fetched a tile ahead: uniform steps, the first
// sample and the per-step increment (fixed point); explicit samples, the entry point (fixed point),
// the direction in lattice units (FP64 bits) and t_enter; and the ray's first sample slot.
struct RayPre {
    long long f0[3], f1[3];
    double t_enter;
    int off;
};

__device__ __forceinline__ RayPre ray_pre(const RenderArgs &A, int ray) {
    RayPre p;
    const RayRec &r = A.rays[ray];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        p.f0[a] = A.ts ? r.uefx[a] : r.u0fx[a];
        p.f1[a] = A.ts ? __double_as_longlong(r.e[a]) : r.dfx[a];
    }
    p.t_enter = A.ts ? r.t_enter : 0.0;
    p.off = r.off;
    return p;
}

// sample_cell() from prefetched ray data (the same arithmetic).
__device__ __forceinline__ Cell cell_pre(const RenderArgs &A, const RayPre &p, int ray, int k, float &dt) {
    long long u[3];
    if (A.ts) {
        const double t = (double)A.ts[(long long)ray * A.n_expl + k];
        dt = A.dts[(long long)ray * A.n_expl + k];
#pragma unroll
        for (int a = 0; a < 3; ++a) u[a] = p.f0[a] + to_fx((t - p.t_enter) * __longlong_as_double(p.f1[a]));
    } else {
        dt = A.step;
#pragma unroll
        for (int a = 0; a < 3; ++a) u[a] = p.f0[a] + (long long)k * p.f1[a];
    }
    return cell_from_fx(u, A.nx, A.ny, A.nz);
}

// v[0:12] += the trilinear interpolation of the feature grid in cell c.
template <typename FeatT, bool PK>
__device__ __forceinline__ void gather_features(const RenderArgs &A, const Cell &c, float *v) {
    constexpr int FEAT = 12;
#pragma unroll
    for (int q = 0; q < 4; ++q) {   // corner pairs (x bit, y bit) with z = 0, 1 adjacent
        const int qa = q << 1;
        const long long idx0 = corner_index(c, qa, A.ny, A.nz, PK);
        const float w0 = corner_weight(c, qa), w1 = corner_weight(c, qa | 1);
        const FeatT *g = static_cast<const FeatT *>(A.cgrid) + idx0 * FEAT;
        // the z + 1 corner: the next point in the canonical layout, located in the packed one
        const FeatT *gz = PK ? static_cast<const FeatT *>(A.cgrid) +
                                         corner_index(c, qa | 1, A.ny, A.nz, true) * FEAT
                                   : g + FEAT;
        if constexpr (sizeof(FeatT) == 4) {
            const float4 *g4 = reinterpret_cast<const float4 *>(g), *gz4 = reinterpret_cast<const float4 *>(gz);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const float4 a = __ldg(g4 + k), bb = __ldg(gz4 + k);
                v[4 * k + 0] += w0 * a.x + w1 * bb.x;
                v[4 * k + 1] += w0 * a.y + w1 * bb.y;
                v[4 * k + 2] += w0 * a.z + w1 * bb.z;
                v[4 * k + 3] += w0 * a.w + w1 * bb.w;
            }
        } else if constexpr (!PK) {
            // canonical BF16: the pair is 48 contiguous bytes at offset 0 or 8 mod 16 (the grid is
            // 16-byte aligned, a point is 24 bytes): three aligned 16-byte loads from the pair's
            // 16-byte granule and, at offset 8, one 8-byte load for its last word pair -- no byte
            // outside the grid (at offset 8 the first 8 bytes loaded belong to the point before)
            const uintptr_t ad = reinterpret_cast<uintptr_t>(g);
            const uint4 *q = reinterpret_cast<const uint4 *>(ad & ~(uintptr_t)15);
            const bool off8 = (ad & 15u) != 0u;
            const uint4 q0 = __ldg(q), q1 = __ldg(q + 1), q2 = __ldg(q + 2);
            const uint2 q3 = off8 ? __ldg(reinterpret_cast<const uint2 *>(q + 3)) : make_uint2(0u, 0u);
            const uint32_t wd[14] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w,
                                     q2.x, q2.y, q2.z, q2.w, q3.x, q3.y};
#pragma unroll
            for (int m = 0; m < 6; ++m) {   // channels 2m, 2m + 1 of the corners z (word m) and z + 1
                uint32_t ua = off8 ? wd[m + 2] : wd[m], ub = off8 ? wd[m + 8] : wd[m + 6];
                const float2 a = __bfloat1622float2(*reinterpret_cast<__nv_bfloat162 *>(&ua));
                const float2 bz = __bfloat1622float2(*reinterpret_cast<__nv_bfloat162 *>(&ub));
                v[2 * m + 0] += w0 * a.x + w1 * bz.x;
                v[2 * m + 1] += w0 * a.y + w1 * bz.y;
            }
        } else {
            const uint2 *g2 = reinterpret_cast<const uint2 *>(g), *gz2 = reinterpret_cast<const uint2 *>(gz);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                uint2 a = __ldg(g2 + k), bb = __ldg(gz2 + k);
                const float2 a0 = __bfloat1622float2(*reinterpret_cast<__nv_bfloat162 *>(&a.x));
                const float2 a1 = __bfloat1622float2(*reinterpret_cast<__nv_bfloat162 *>(&a.y));
                const float2 b0 = __bfloat1622float2(*reinterpret_cast<__nv_bfloat162 *>(&bb.x));
                const float2 b1 = __bfloat1622float2(*reinterpret_cast<__nv_bfloat162 *>(&bb.y));
                v[4 * k + 0] += w0 * a0.x + w1 * b0.x;
                v[4 * k + 1] += w0 * a0.y + w1 * b0.y;
                v[4 * k + 2] += w0 * a1.x + w1 * b1.x;
                v[4 * k + 3] += w0 * a1.y + w1 * b1.y;
            }
        }
    }
}

// A row of a tile as the scatter needs it: the offsets inside its lattice cell (a little below 0 or above 1 on
// the rim of the box) and the cell (cell_base; kNoCell for a padding row, which come last in a tile).  A packed
// cell_base with i0 >= 1024 is negative too; kNoCell would be i0 = 2047, and i0 <= 2046.
constexpr int kNoCell = -1;
__device__ __forceinline__ float4 row_place(const RenderArgs &A, const Cell &c, bool live, bool packed) {
    return make_float4(c.fx, c.fy, c.fz, __int_as_float(live ? cell_base(c, A.ny, A.nz, packed) : kNoCell));
}

// *p += v (four floats, 16-byte aligned, in global memory), where `on` is not zero.
__device__ __forceinline__ void red_add4_if(unsigned on, float *p, const float4 &v) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.u32 p, %5, 0;\n\t"
        "@p red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};\n\t}\n" ::"l"(p),
        "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(on)
        : "memory");
}

// How many cells apart two cells (cell_base) are along each axis, when that is at most one each: then true.
// Flat indices: a pair of cells further apart never has the difference of one that is not, because k0 <= nz - 2
// and j0 <= ny - 2.
template <bool PK>
__device__ __forceinline__ bool cells_adjacent(int cb, int cbn, int ny, int nz, int &dx, int &dy, int &dz) {
    if (PK) {
        dx = (int)((unsigned)cbn >> 21) - (int)((unsigned)cb >> 21);
        dy = ((cbn >> 10) & 2047) - ((cb >> 10) & 2047);
        dz = (cbn & 1023) - (cb & 1023);
        return abs(dx) <= 1 && abs(dy) <= 1 && abs(dz) <= 1;
    }
    const int nyz = ny * nz;
    int d = cbn - cb;
    dx = (d > (nyz >> 1)) - (d < -(nyz >> 1));
    d -= dx * nyz;
    dy = (d > (nz >> 1)) - (d < -(nz >> 1));
    dz = d - dy * nz;
    return abs(dz) <= 1;
}

// A warp's table of 8 rows: by corner parity (x, y, z), the weight and the grid index of the corner.  (The
// ninth column keeps the rows' writes off each other's banks.)
constexpr int kScatterRows = 8;
struct ScatterTab {
    float2 at[kScatterRows][9];
};

// Producer warp: add the feature gradients of its 32 rows of a tile (*de(row, k): channels 4 k .. 4 k + 3 of a
// row) to the grid.  Rows are in kept order, so consecutive samples of a ray sit in consecutive rows; rows
// whose samples lie in one lattice cell share all eight corners, and of a cell and the next along a ray four
// corners are the same as a rule: a corner is added to the grid when the ray has left it.
// place: the tile's table of rows (row_place); all 32 lanes call.
// A lane holds 16 bytes of the corner with the lane's parities (the eight lanes of an (x, y) pair have the
// six pieces of its two z corners, two are idle): a corner that the next cell shares is the same lane's, so
// sums never move between lanes, and a reduction of the warp touches at most four runs of 96 bytes.
// Measured, all SMs reducing: a 16-byte reduction of 32 scattered rows takes an SM 174 clocks, one of four
// runs with 24 lanes 31, with the 12 lanes that move on as a rule 18.  A row to a lane kept the load/store unit
// busy for most of a tile (colour backward of 65,536 rays at 256^3, BF16: 11.6 -> 10.6 ms with a row to a
// warp, all eight corners); handing shared sums on by shuffles cost a chain of 200 clocks a row.
template <bool PK, typename De>
__device__ __forceinline__ void scatter_rows(const RenderArgs &A, const float4 *place, De de, ScatterTab &tab, int row) {
    constexpr int FEAT = 12, NB = 4;
    constexpr unsigned ALL = 0xffffffffu;
    const int lane = row & 31, r0 = row - lane;
    const int px = lane >> 4, py = (lane >> 3) & 1, piece = lane & 7;
    const int pz = piece >= 3 ? 1 : 0, k = piece < 6 ? piece - 3 * pz : 0;
    const int col = 4 * px + 2 * py + pz;
    unsigned flush;   // bit j: my sum leaves for the grid after row j
    const float4 mine = place[row];
    const unsigned live = __ballot_sync(ALL, __float_as_int(mine.w) != kNoCell);
    const int n = __popc(live);
    unsigned odd_x, odd_y, odd_z;   // bit j: the base corner of row j's cell is odd along the axis
    {
        const unsigned cb = (unsigned)__float_as_int(mine.w), t = cb / (unsigned)A.nz;
        odd_x = __ballot_sync(ALL, (PK ? cb >> 21 : t / (unsigned)A.ny) & 1u);
        odd_y = __ballot_sync(ALL, (PK ? cb >> 10 : t % (unsigned)A.ny) & 1u);
        odd_z = __ballot_sync(ALL, (PK ? cb : cb - t * (unsigned)A.nz) & 1u);
    }
    {
        const int cb = __float_as_int(mine.w), cbn = __shfl_down_sync(ALL, cb, 1);
        int dx, dy, dz;
        bool adj = cells_adjacent<PK>(cb, cbn, A.ny, A.nz, dx, dy, dz);
        adj = adj && lane < 31 && cbn != kNoCell;
        const unsigned xp = __ballot_sync(ALL, dx > 0), xm = __ballot_sync(ALL, dx < 0);
        const unsigned yp = __ballot_sync(ALL, dy > 0), ym = __ballot_sync(ALL, dy < 0);
        const unsigned zp = __ballot_sync(ALL, dz > 0), zm = __ballot_sync(ALL, dz < 0);
        // bit j: my corner of row j's cell is the upper one along the axis
        const unsigned ux = odd_x ^ (px ? ALL : 0u), uy = odd_y ^ (py ? ALL : 0u), uz = odd_z ^ (pz ? ALL : 0u);
        const unsigned left = (xp & ~ux) | (xm & ux) | (yp & ~uy) | (ym & uy) | (zp & ~uz) | (zm & uz);
        flush = live & ~(__ballot_sync(ALL, adj) & ~left);
        if (piece >= 6) flush = 0u;
    }
    float *base = A.grad_cgrid + 4 * k;
    float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll 1
    for (int j0 = 0; j0 < n; j0 += kScatterRows) {
        __syncwarp();
        {
            // four lanes a row, one for each pair of (y, z) parities
            const int j = j0 + (lane & 7), by = ((lane >> 4) ^ (odd_y >> j)) & 1, bz = ((lane >> 3) ^ (odd_z >> j)) & 1;
            const float4 f = place[r0 + j];
            const int cb = __float_as_int(f.w), ix = (odd_x >> j) & 1;
            const float wy = by ? f.y : 1.0f - f.y, wz = bz ? f.z : 1.0f - f.z;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int bx = q ^ ix;
                const float w = (bx ? f.x : 1.0f - f.x) * wy * wz;
                const unsigned idx = (unsigned)corner_from_base(cb, bx, by, bz, A.ny, A.nz, PK);
                tab.at[lane & 7][4 * q + (lane >> 3)] = make_float2(w, __uint_as_float(idx));
            }
        }
        __syncwarp();
#pragma unroll 1
        for (int j = 0; j < kScatterRows && j0 + j < n; j += NB, flush >>= NB) {   // (rows from n on add nothing)
            float4 e[NB];
            float2 t[NB];
#pragma unroll
            for (int u = 0; u < NB; ++u) {
                e[u] = *de(r0 + j0 + j + u, k);
                t[u] = tab.at[j + u][col];
            }
#pragma unroll
            for (int u = 0; u < NB; ++u) {
                acc = make_float4(fmaf(t[u].x, e[u].x, acc.x), fmaf(t[u].x, e[u].y, acc.y),
                                  fmaf(t[u].x, e[u].z, acc.z), fmaf(t[u].x, e[u].w, acc.w));
                const bool out = (flush & (1u << u)) != 0u;
                red_add4_if(out, base + (size_t)__float_as_uint(t[u].y) * FEAT, acc);
                if (out) acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            }
        }
    }
    __syncwarp();   // the tables may be overwritten
}

}  // namespace dvgo
