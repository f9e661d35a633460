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

// Producer: add a tile's feature gradients (de(row, k): channels 4 k .. 4 k + 3 of a row) to the grid.  Rows
// are in kept order, so consecutive samples of a ray sit in consecutive rows; rows whose samples lie
// in one lattice cell share all eight corners, and the last row of such a run adds the whole run's
// weighted de with one set of reductions (the run's other rows add nothing).
// slot (-1: padding row), cbase and frac: the tile's per-row tables.
// kParts: the corners are taken in that many turns (two halve the 96 accumulator registers).
template <bool PK, int kParts = 1, typename De>
__device__ __forceinline__ void scatter_row(const RenderArgs &A, const int *slot, const int *cbase,
                                            const float (*frac)[3], De de, int row) {
    constexpr int TM = 128, FEAT = 12, NQ = 8 / kParts;
    if (slot[row] < 0) return;
    const int cb = cbase[row];
    if (row + 1 < TM && slot[row + 1] >= 0 && cbase[row + 1] == cb) return;
#pragma unroll
    for (int part = 0; part < kParts; ++part) {
        float4 acc[NQ][3];
#pragma unroll
        for (int q = 0; q < NQ; ++q) acc[q][0] = acc[q][1] = acc[q][2] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        for (int j = row; j >= 0 && slot[j] >= 0 && cbase[j] == cb; --j) {
            const float4 e0 = de(j, 0), e1 = de(j, 1), e2 = de(j, 2);
            const float fx = frac[j][0], fy = frac[j][1], fz = frac[j][2];
#pragma unroll
            for (int i = 0; i < NQ; ++i) {
                const int q = part * NQ + i;
                const float w = (((q >> 2) & 1) ? fx : 1.0f - fx) * (((q >> 1) & 1) ? fy : 1.0f - fy) *
                                ((q & 1) ? fz : 1.0f - fz);
                acc[i][0] = make_float4(fmaf(w, e0.x, acc[i][0].x), fmaf(w, e0.y, acc[i][0].y),
                                        fmaf(w, e0.z, acc[i][0].z), fmaf(w, e0.w, acc[i][0].w));
                acc[i][1] = make_float4(fmaf(w, e1.x, acc[i][1].x), fmaf(w, e1.y, acc[i][1].y),
                                        fmaf(w, e1.z, acc[i][1].z), fmaf(w, e1.w, acc[i][1].w));
                acc[i][2] = make_float4(fmaf(w, e2.x, acc[i][2].x), fmaf(w, e2.y, acc[i][2].y),
                                        fmaf(w, e2.z, acc[i][2].z), fmaf(w, e2.w, acc[i][2].w));
            }
        }
#pragma unroll
        for (int i = 0; i < NQ; ++i) {
            const int q = part * NQ + i;
            const long long idx = corner_from_base(cb, (q >> 2) & 1, (q >> 1) & 1, q & 1, A.ny, A.nz, PK);
            float4 *g = reinterpret_cast<float4 *>(A.grad_cgrid + idx * FEAT);
            atomicAdd(g + 0, acc[i][0]);
            atomicAdd(g + 1, acc[i][1]);
            atomicAdd(g + 2, acc[i][2]);
        }
    }
}

}  // namespace dvgo
