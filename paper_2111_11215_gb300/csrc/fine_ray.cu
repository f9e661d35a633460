// fine_ray.cu -- the per-ray kernels of the fine-stage render (Sec. 4.2).
//
// fine_density:   warp per ray.  For each sample k of the ray: position; optionally the
//                 known-free-space test on the coarse grid (Sec. 4.2), which removes the sample
//                 before any fine query; density gather, sigma_ddot = interp(x, V_density)
//                 (Eq. fine_queries_densities), tau_k = softplus(sigma_ddot + b) * dt_k
//                 (Eq. density_activation, post-activation), removed when
//                 alpha_k = 1 - exp(-tau_k) < tau_f (Sec. 4.2 free space skipping).
//                 Kept samples are packed in order at the front of the ray's slots, and every 32 samples that
//                 hold one leave a record (RayChunk): the passes after it walk these records alone,
//                 which under the skips are a few per cent of all; the samples are also appended to the
//                 batch's list for the colour kernel (one atomic per 64 samples, order along the ray kept).
//                 A record keeps its samples in their lanes and the optical depth in front of them, so every
//                 sum over a ray is associated as without the skips: weights, colours and dL/do carry
//                 the same bits whatever was left out (scanning the packed samples moved the last bit of a
//                 quarter of the weights, which flipped BF16 roundings of dL/do).
//                 Early ray termination: a sample where T_k = exp(-(sum_{j<k} tau_j)) is exactly 0 in
//                 FP32 has weight 0 and no gradient through it, so it and the rest of the ray are
//                 not kept (nor queried), and T_K is exactly 0.
// empty_cells:    one bit per lattice cell that says whether a sample in it can reach tau_f: the
//                 interpolated raw density is at most the largest of its corners (plus rounding), and
//                 alpha rises with it.  The density pass reads that bit before anything else and
//                 neither gathers nor activates the samples of empty cells.
// fine_composite: warp per ray.  T_k = exp(-sum_{j<k} tau_j), w_k = T_k alpha_k,
//                 C_hat = sum w_k c_k + T_K bg (Eq. volume_rendering), loss (Eq. photo_loss).
// fine_comp_bwd:  warp per ray.  dC/dc_k = w_k -> stored for the colour backward;
//                 dC/dtau_k = T_{k+1} c_k - S_k with S_k = sum_{j>k} w_j c_j + T_K bg, evaluated as
//                 D_k = sum_{j>=k} T_{j+1} (c_j - c_{j+1}) (c_K = bg), which follows from
//                 D_k - D_{k+1} = T_{k+1} (c_k - c_{k+1}) and D_{K-1} = T_K (c_{K-1} - bg); the sum
//                 is taken from the back of the ray, so no large terms cancel when the colour in
//                 front of a surface matches the colour behind it.  dT_K/dtau_k = -T_K;
//                 dtau/dsigma_ddot = dt sigmoid(sigma_ddot + b) = dt (1 - exp(-tau/dt));
//                 the density gradient is scattered to the 8 corners (runs of lanes that share a
//                 corner are summed before one atomic).

#include <limits.h>

#include "dvgo_internal.cuh"

namespace dvgo {

namespace {

constexpr unsigned FULL = 0xffffffffu;

// A warp takes 32 cells along k of kMaskRows consecutive rows j of one plane i and walks along j with the
// maximum of the planes i and i + 1 of the last row in registers: two loads a row and lane (four with the
// column past the word), unrolled so that several rows' loads are in flight.  A cell whose corners
// include an infinity or NaN counts as occupied.  The bound on the interpolation: weights are formed in
// FP32 (their products sum to 1 within 8 ulp), so it exceeds the largest corner by less than 2^-19 of the
// largest magnitude.  160^3: 13 us (47 us with a warp per word and no reuse along j).
constexpr int kMaskRows = 16;
template <bool PK>
__global__ void __launch_bounds__(256) empty_cells_kernel(RenderArgs A) {
    const int lane = threadIdx.x & 31;
    const int jt = (A.ny - 1 + kMaskRows - 1) / kMaskRows;   // row blocks of a plane
    const int w = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int wk = w % A.mask_wpr, jb = (w / A.mask_wpr) % jt, i = w / (A.mask_wpr * jt);
    if (i >= A.nx - 1) return;
    const int k = min(wk * 32 + lane, A.nz - 1), ke = min(wk * 32 + 32, A.nz - 1);
    // largest value and magnitude sum of the points (i, j), (i + 1, j) at k
    const float *plane = A.density + (size_t)i * A.ny * A.nz;   // canonical
    const int next = A.ny * A.nz;
    auto column = [&](int j, int kk, float &mx, float &mag) {
        const float a = __ldg(PK ? A.density + packed_index(i, j, kk, A.ny, A.nz) : plane + j * A.nz + kk);
        const float b = __ldg(PK ? A.density + packed_index(i + 1, j, kk, A.ny, A.nz) : plane + next + j * A.nz + kk);
        mx = fmaxf(a, b);
        mag = fabsf(a) + fabsf(b);   // NaN and infinities carry through
    };
    const int j0 = jb * kMaskRows;
    float mx, mag, mxe, mage;
    column(j0, k, mx, mag);
    column(j0, ke, mxe, mage);
#pragma unroll 4
    for (int jj = 0; jj < kMaskRows; ++jj) {
        const int j = j0 + jj, jn = min(j + 1, A.ny - 1);
        float mx1, mag1, mxe1, mage1;
        column(jn, k, mx1, mag1);
        column(jn, ke, mxe1, mage1);
        const float m = fmaxf(mx, mx1), g = mag + mag1;
        float mn = __shfl_down_sync(FULL, m, 1), gn = __shfl_down_sync(FULL, g, 1);
        if (lane == 31) {
            mn = fmaxf(mxe, mxe1);
            gn = mage + mage1;
        }
        const bool empty = fmaf(g + gn, 0x1p-19f, fmaxf(m, mn)) < A.mask_thr;   // false for NaN and infinities
        const unsigned occ = __ballot_sync(FULL, !empty);
        if (lane == 0 && j < A.ny - 1) A.mask[((long long)i * A.ny + j) * A.mask_wpr + wk] = occ;
        mx = mx1;
        mag = mag1;
        mxe = mxe1;
        mage = mage1;
    }
}

// Optical depth of a sample at lattice coordinate u with step length dt, 0 and kept = false when it is
// removed.
template <bool kFreeSpace, int kOrder>
__device__ __forceinline__ float sample_tau(const RenderArgs &A, const long long u[3], float dt, bool &kept) {
    kept = false;
    if (kFreeSpace && known_free(A, u)) return 0.0f;   // known free space: no fine query
    const Cell c = cell_from_fx(u, A.nx, A.ny, A.nz);
    float tau;
    if (kOrder == DVGO_ACT_POST) {
        float s = 0.0f;
#pragma unroll
        for (int q = 0; q < 8; ++q)
            s = fmaf(corner_weight(c, q), __ldg(A.density + corner_index(c, q, A.ny, A.nz, A.packed)), s);
        tau = softplusf(s + A.shift_b) * dt;
    } else {
        float v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = __ldg(A.density + corner_index(c, q, A.ny, A.nz, A.packed));
        tau = tau_pre_in(kOrder, c, v, A.shift_b, dt);
    }
    kept = !(-expm1f(-tau) < A.tau_f);
    return kept ? tau : 0.0f;
}

// Whether a sample's cell can hold alpha >= tau_f (empty_cells).
__device__ __forceinline__ bool cell_occupied(const RenderArgs &A, const long long u[3]) {
    const int i = min(max((int)(u[0] >> kFxBits), 0), A.nx - 2), j = min(max((int)(u[1] >> kFxBits), 0), A.ny - 2);
    const int k = min(max((int)(u[2] >> kFxBits), 0), A.nz - 2);
    return (__ldg(A.mask + ((long long)i * A.ny + j) * A.mask_wpr + (k >> 5)) >> (k & 31)) & 1u;
}

// Specialised on the known-free-space test, the activation order, the sampling and the cell mask
// (uniform per launch), so the default configuration carries none of them.  A warp walks its ray two
// 32-sample chunks at a time: the optical depths of both chunks are formed first (their density loads
// in flight together), then the chunks are scanned in order, and one atomic reserves the kept-list slots
// of both.
// 128-thread blocks: the pass runs beside the feature-grid Adam of the other stream (3 x 256
// threads x 56 registers per SM), next to which three of them fit per SM where one 256-thread
// block does.
constexpr int kDensityThreads = 128;
template <bool kFreeSpace, int kOrder, bool kExpl, bool kMask>
__global__ void __launch_bounds__(kDensityThreads) fine_density_kernel(RenderArgs A) {
    int lane = threadIdx.x & 31;
    int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int r = warp; r < A.R; r += nwarps) {
        const RayRec rr = A.rays[r];
        flag_bad_ray(A, rr, lane);
        float carry = 0.0f;          // optical depth before this chunk
        int nk = 0, nrec = 0, kend = INT_MAX;
        RayChunk *recs = A.rchunk + (size_t)r * A.nchunk;
        long long u[3];              // uniform steps: lattice coordinate of sample base + lane
        if (!kExpl)
#pragma unroll
            for (int a = 0; a < 3; ++a) u[a] = rr.u0fx[a] + (long long)lane * rr.dfx[a];
        for (int base = 0; base < rr.n; base += 64) {
            float tau[2] = {0.0f, 0.0f};
            bool kept[2] = {false, false};
            if (kMask) {
                bool occ[2];
                long long v[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) v[a] = u[a] + 32 * rr.dfx[a];
                occ[0] = base + lane < rr.n && cell_occupied(A, u);
                occ[1] = base + 32 + lane < rr.n && cell_occupied(A, v);
                const bool any = __any_sync(FULL, occ[0] || occ[1]);
                if (any) {
                    if (occ[0]) tau[0] = sample_tau<kFreeSpace, kOrder>(A, u, A.step, kept[0]);
                    if (occ[1]) tau[1] = sample_tau<kFreeSpace, kOrder>(A, v, A.step, kept[1]);
                }
#pragma unroll
                for (int a = 0; a < 3; ++a) u[a] += 64 * rr.dfx[a];
                if (!any) {
                    if (expf(-carry) != 0.0f) continue;
                    kend = base;
                    break;
                }
            } else {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int k = base + 32 * h + lane;
                    if (k >= rr.n) continue;
                    float dt;
                    long long v[3];
                    if (kExpl) {   // sample_fx's explicit branch, without the run-time test
                        const double t = (double)A.ts[(long long)r * A.n_expl + k];
                        dt = A.dts[(long long)r * A.n_expl + k];
#pragma unroll
                        for (int a = 0; a < 3; ++a) v[a] = rr.uefx[a] + to_fx((t - rr.t_enter) * rr.e[a]);
                    } else {
                        dt = A.step;
#pragma unroll
                        for (int a = 0; a < 3; ++a) v[a] = u[a] + (32 * h) * rr.dfx[a];
                    }
                    tau[h] = sample_tau<kFreeSpace, kOrder>(A, v, dt, kept[h]);
                }
                if (!kExpl)
#pragma unroll
                    for (int a = 0; a < 3; ++a) u[a] += 64 * rr.dfx[a];
            }
            unsigned m[2];
            float pre[2];
            bool done = false;       // the ray is terminated: T = 0 from here on
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                // T_k; exactly 0 -> terminated (the scan sees tau of lanes below only)
                const float incl = warp_incl_scan(tau[h], lane);
                float excl = __shfl_up_sync(FULL, incl, 1);
                if (lane == 0) excl = 0.0f;
                const bool dead = done || expf(-(carry + excl)) == 0.0f;
                if (dead) kept[h] = false;
                const unsigned end = __ballot_sync(FULL, (dead || isinf(tau[h])) && base + 32 * h + lane < rr.n);
                pre[h] = carry;
                if (!done) {
                    if (end) {
                        kend = base + 32 * h + __ffs(end) - 1;
                        done = true;
                    }
                    carry += __shfl_sync(FULL, incl, 31);
                }
                m[h] = __ballot_sync(FULL, kept[h]);
            }
            const int cnt0 = __popc(m[0]), cnt = cnt0 + __popc(m[1]);
            int base_slot = 0;
            if (lane == 0 && cnt) base_slot = atomicAdd(&A.hdr->n_kept, cnt);
            base_slot = __shfl_sync(FULL, base_slot, 0);
            const unsigned below = (1u << lane) - 1u;
            const int pos[2] = {__popc(m[0] & below), cnt0 + __popc(m[1] & below)};
#pragma unroll
            for (int h = 0; h < 2; ++h)
                if (kept[h]) {
                    const int j = nk + pos[h], k = base + 32 * h + lane;
                    A.stau[(size_t)rr.off + j] = tau[h];
                    A.kept[base_slot + pos[h]] = make_int2(j | k << 16, r);
                }
            if (lane == 0 && m[0]) recs[nrec] = RayChunk{m[0], pre[0], base / 32, nk};
            nrec += m[0] ? 1 : 0;
            if (lane == 0 && m[1]) recs[nrec] = RayChunk{m[1], pre[1], base / 32 + 1, nk + cnt0};
            nrec += m[1] ? 1 : 0;
            nk += cnt;
            if (done) break;
        }
        if (lane == 0) A.rayk[r] = make_int4(nrec, kend, __float_as_int(kend != INT_MAX ? 0.0f : expf(-carry)), nk);
    }
}

__device__ void finish_loss_fine(const RenderArgs &A, float part) {
    __shared__ float red[32];
    __shared__ bool last;
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    part = warp_sum(part);
    if (lane == 0) red[wid] = part;
    __syncthreads();
    if (threadIdx.x == 0) {
        float s = 0.0f;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += red[i];
        atomicAdd(&A.hdr->loss_acc, (double)s);
        __threadfence();
        unsigned prev = atomicAdd(&A.hdr->done, 1u);
        last = (prev == gridDim.x - 1);
    }
    __syncthreads();
    if (last && threadIdx.x == 0 && A.loss_out) {
        __threadfence();
        const double tot = atomicAdd(&A.hdr->loss_acc, 0.0);
        A.loss_out[0] = A.R > 0 ? (float)(tot / (double)A.R) : 0.0f;
    }
}

// Block sizes: two rays per block where nothing joins the warps, so that a block's slots are free when
// its two rays are done (rays differ in length by an order of magnitude: fine_comp_bwd 68 -> 64 us for
// 1.38 M samples, 30 -> 27 us for 0.31 M).  The forward with a loss takes eight: its blocks end in two
// atomics on one address each (18 us with two rays a block, 12 us with eight, 8,192 rays).
constexpr int kRayThreads = 64, kLossThreads = 256;
__global__ void __launch_bounds__(kLossThreads) fine_composite_kernel(RenderArgs A) {
    int lane = threadIdx.x & 31;
    int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int nwarps = (gridDim.x * blockDim.x) >> 5;
    float loss_part = 0.0f;
    const bool aux = A.target && (A.w_pt != 0.0f || A.w_bg != 0.0f);
    for (int r = warp; r < A.R; r += nwarps) {
        const int4 rk = A.rayk[r];
        const size_t off = (size_t)r * A.cap;
        float tg[3] = {0.0f, 0.0f, 0.0f};
        if (aux)
            for (int ch = 0; ch < 3; ++ch) tg[ch] = A.target[3 * r + ch];
        float acc[3] = {0.0f, 0.0f, 0.0f}, pt = 0.0f;
        for (int c0 = 0; c0 < rk.x; c0 += 32) {
            const int nc = min(32, rk.x - c0);
            RayChunk mine;
            if (lane < nc) mine = A.rchunk[(size_t)r * A.nchunk + c0 + lane];
#pragma unroll 2
            for (int c = 0; c < nc; ++c) {
                const unsigned m = __shfl_sync(FULL, mine.mask, c);
                const float pre = __shfl_sync(FULL, mine.pre, c);
                const int first = __shfl_sync(FULL, mine.first, c);
                float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if ((m >> lane) & 1u) v = A.scol[off + first + __popc(m & ((1u << lane) - 1u))];
                const float incl = warp_incl_scan(v.w, lane);
                float excl = __shfl_up_sync(FULL, incl, 1);
                if (lane == 0) excl = 0.0f;
                const float w = expf(-(pre + excl)) * -expm1f(-v.w);
                acc[0] = fmaf(w, v.x, acc[0]);
                acc[1] = fmaf(w, v.y, acc[1]);
                acc[2] = fmaf(w, v.z, acc[2]);
                const float e0 = v.x - tg[0], e1 = v.y - tg[1], e2 = v.z - tg[2];
                pt = fmaf(w, fmaf(e0, e0, fmaf(e1, e1, e2 * e2)), pt);   // per-point rgb loss
            }
        }
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) acc[ch] = warp_sum(acc[ch]);
        if (aux) pt = warp_sum(pt);
        if (lane == 0) {
            const float TK = __int_as_float(rk.z);
            float rgb[3];
            for (int ch = 0; ch < 3; ++ch) rgb[ch] = fmaf(TK, A.bg[ch], acc[ch]);
            for (int ch = 0; ch < 3; ++ch) A.rgb_out[3 * r + ch] = rgb[ch];
            if (A.tfinal_out) A.tfinal_out[r] = TK;
            A.rayout[r] = make_float4(rgb[0], rgb[1], rgb[2], TK);
            if (A.target) {
                for (int ch = 0; ch < 3; ++ch) {
                    float e = rgb[ch] - A.target[3 * r + ch];
                    loss_part = fmaf(e, e, loss_part);
                    if (A.dloss_out) A.dloss_out[3 * r + ch] = 2.0f * e / (float)A.R;
                }
            }
            if (aux) {
                loss_part += A.w_pt * pt + A.w_bg * bg_entropy(TK);
                A.rtarget[r] = make_float4(tg[0], tg[1], tg[2], 0.0f);
            }
        }
    }
    if (A.target) finish_loss_fine(A, loss_part);
}

template <int kOrder>
__global__ void __launch_bounds__(kRayThreads) fine_comp_bwd_kernel(RenderArgs A) {
    const int lane = threadIdx.x & 31;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int r = warp; r < A.R; r += nwarps) {
        const int4 rk = A.rayk[r];
        if (rk.x == 0) continue;   // no kept sample
        const RayRec rr = A.rays[r];
        const float TK = A.rayout[r].w;
        const float g[3] = {A.grad_rgb[3 * r], A.grad_rgb[3 * r + 1], A.grad_rgb[3 * r + 2]};
        // auxiliary losses of the forward: the background entropy enters through T_K, the
        // per-point rgb loss adds 2 w_pt w_k (c_k - C) / R to dL/dc_k
        const bool aux = A.hdr->aux != 0;
        float4 tg = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (aux) tg = A.rtarget[r];
        const float gT = (A.grad_tfinal ? A.grad_tfinal[r] : 0.0f) +
                         (aux ? A.w_bg * bg_entropy_dT(TK) / (float)A.R : 0.0f);
        const float kpt = aux ? 2.0f * A.w_pt / (float)A.R : 0.0f;
        // back to front: D_k = dC/dtau_k as a suffix sum of T_{j+1} (c_j - c_{j+1}), the colour of a sample that
        // is not kept being 0
        float Dc[3] = {0.0f, 0.0f, 0.0f};
        float cnext[3] = {A.bg[0], A.bg[1], A.bg[2]};   // colour after the chunk's last sample
        float Tnext = TK;                               // T in front of it
        int inext = (rr.n + 31) >> 5;                   // the chunk handled before this one
        RayChunk mine;
        for (int ci = rk.x - 1; ci >= 0; --ci) {
            if (ci == rk.x - 1 || (ci & 31) == 31) {
                const int q = (ci & ~31) + lane;
                if (q < rk.x) mine = A.rchunk[(size_t)r * A.nchunk + q];
            }
            const unsigned m = __shfl_sync(FULL, mine.mask, ci & 31);
            const float pre = __shfl_sync(FULL, mine.pre, ci & 31);
            const int chunk = __shfl_sync(FULL, mine.index, ci & 31), first = __shfl_sync(FULL, mine.first, ci & 31);
            if (chunk + 1 < inext) {   // chunks without a kept sample in between: the step from 0 to the colour after them
#pragma unroll
                for (int ch = 0; ch < 3; ++ch) {
                    Dc[ch] += Tnext * (0.0f - cnext[ch]);
                    cnext[ch] = 0.0f;
                }
            }
            inext = chunk;
            const int k = chunk * 32 + lane;
            const bool valid = k < rr.n, kept = (m >> lane) & 1u;
            const size_t slot = (size_t)rr.off + first + __popc(m & ((1u << lane) - 1u));
            float4 sv = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (kept) sv = A.scol[slot];
            const float tau = sv.w;
            const float cc[3] = {sv.x, sv.y, sv.z};
            const float incl = warp_incl_scan(tau, lane);
            float excl = __shfl_up_sync(FULL, incl, 1);
            if (lane == 0) excl = 0.0f;
            const float T = expf(-(pre + excl));
            const float T1 = k >= rk.y ? 0.0f : expf(-(pre + incl));   // (rk.y: the first terminated sample)
            const float w = T * -expm1f(-tau);
            Tnext = expf(-pre);
            float D[3];
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) {
                float cn = __shfl_down_sync(FULL, cc[ch], 1);
                if (lane == 31 || k + 1 >= rr.n) cn = (k + 1 >= rr.n) ? A.bg[ch] : cnext[ch];
                float X = valid ? T1 * (cc[ch] - cn) : 0.0f;
                float sx = warp_suffix_scan(X, lane);
                D[ch] = Dc[ch] + sx;
                Dc[ch] += __shfl_sync(FULL, sx, 0);
                cnext[ch] = __shfl_sync(FULL, cc[ch], 0);
            }
            float dtau = -gT * TK;
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) dtau = fmaf(g[ch], D[ch], dtau);
            // kept samples have tau > 0 or an exactly-zero sigmoid factor
            const bool act = kept && tau > 0.0f;
            Cell c;
            c.i0 = c.j0 = c.k0 = 0;
            c.fx = c.fy = c.fz = 0.0f;
            float dz = 0.0f, dt = 0.0f;
            if (kept) {
                c = sample_cell(A, rr, r, k, dt);
                dz = act ? dtau * dt * -expm1f(-tau / dt) : 0.0f;   // post: dt sigmoid(z) = dt (1 - e^{-tau/dt})
                // for the colour backward: dL/dc_k through the sigmoid, dL/do = dL/dc c (1 - c)
                const float gc[3] = {fmaf(kpt * w, cc[0] - tg.x, g[0] * w), fmaf(kpt * w, cc[1] - tg.y, g[1] * w),
                                     fmaf(kpt * w, cc[2] - tg.z, g[2] * w)};
                A.sgrad[slot] = make_float4(0.0f, gc[0] * cc[0] * (1.0f - cc[0]), gc[1] * cc[1] * (1.0f - cc[1]),
                                            gc[2] * cc[2] * (1.0f - cc[2]));
            }
            // Runs of lanes in the same cell share all 8 corners (corner q of two samples is the
            // same point exactly when their cells are), so one segmentation serves every corner;
            // the 8 segmented sums run side by side and stop after the warp's longest run.
            const Seg sg = make_seg(act ? cell_base(c, A.ny, A.nz, A.packed) : -1 - lane, lane);
            int run = lane - sg.first + 1;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) run = max(run, __shfl_xor_sync(FULL, run, o));
            int idx[8];
            float gq[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                idx[q] = (int)corner_index(c, q, A.ny, A.nz, A.packed);
                if (kOrder == DVGO_ACT_POST) {
                    gq[q] = dz * corner_weight(c, q);
                } else {
                    gq[q] = act ? dtau * dtau_dv_pre_in(kOrder, c, q, __ldg(A.density + idx[q]), A.shift_b, dt, tau)
                                : 0.0f;
                }
            }
            for (int o = 1; o < run; o <<= 1) {
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const float n = __shfl_up_sync(FULL, gq[q], o);
                    if (lane - o >= sg.first) gq[q] += n;
                }
            }
#pragma unroll
            for (int q = 0; q < 8; ++q)   // the run's last lane adds its total; terminated samples add 0
                if (act && sg.tail && gq[q] != 0.0f) atomicAdd(A.grad_density + idx[q], gq[q]);
        }
    }
}

// Blocks for one warp per ray, up to 128 warps per SM in the grid, then the warps stride.
int warp_grid(int R, int warps_per_block) {
    int want = (R + warps_per_block - 1) / warps_per_block;
    int cap = num_sms() * 128 / warps_per_block;
    if (want > cap) want = cap;
    return want < 1 ? 1 : want;
}

}  // namespace

void launch_empty_cells(const RenderArgs &A, cudaStream_t s) {
    ProfScope ps_(DVGO_K_AUX, s);
    const long long warps = (long long)(A.nx - 1) * ((A.ny - 1 + kMaskRows - 1) / kMaskRows) * A.mask_wpr;
    if (A.packed) empty_cells_kernel<true><<<(unsigned)((warps + 7) / 8), 256, 0, s>>>(A);
    else empty_cells_kernel<false><<<(unsigned)((warps + 7) / 8), 256, 0, s>>>(A);
}

template <int kOrder>
static void launch_density_order(const RenderArgs &A, cudaStream_t s) {
    const int g = warp_grid(A.R, kDensityThreads / 32);
    const bool fs = A.fs_density != nullptr;
    if (A.ts) {
        if (fs) fine_density_kernel<true, kOrder, true, false><<<g, kDensityThreads, 0, s>>>(A);
        else fine_density_kernel<false, kOrder, true, false><<<g, kDensityThreads, 0, s>>>(A);
    } else if (A.mask) {
        if (fs) fine_density_kernel<true, kOrder, false, true><<<g, kDensityThreads, 0, s>>>(A);
        else fine_density_kernel<false, kOrder, false, true><<<g, kDensityThreads, 0, s>>>(A);
    } else {
        if (fs) fine_density_kernel<true, kOrder, false, false><<<g, kDensityThreads, 0, s>>>(A);
        else fine_density_kernel<false, kOrder, false, false><<<g, kDensityThreads, 0, s>>>(A);
    }
}

void launch_fine_density(const RenderArgs &A, cudaStream_t s) {
    ProfScope ps_(DVGO_K_FINE_DENSITY, s);
    if (A.act_order == DVGO_ACT_PRE) launch_density_order<DVGO_ACT_PRE>(A, s);
    else if (A.act_order == DVGO_ACT_IN) launch_density_order<DVGO_ACT_IN>(A, s);
    else launch_density_order<DVGO_ACT_POST>(A, s);
}

void launch_fine_composite_fwd(const RenderArgs &A, cudaStream_t s) {
    {
        ProfScope ps_(DVGO_K_FINE_COMPOSITE, s);
        const int t = A.target ? kLossThreads : kRayThreads;
        fine_composite_kernel<<<warp_grid(A.R, t / 32), t, 0, s>>>(A);
    }
}
void launch_fine_composite_bwd(const RenderArgs &A, cudaStream_t s) {
    {
        ProfScope ps_(DVGO_K_FINE_COMP_BWD, s);
        const dim3 g(warp_grid(A.R, kRayThreads / 32));
        if (A.act_order == DVGO_ACT_PRE) fine_comp_bwd_kernel<DVGO_ACT_PRE><<<g, kRayThreads, 0, s>>>(A);
        else if (A.act_order == DVGO_ACT_IN) fine_comp_bwd_kernel<DVGO_ACT_IN><<<g, kRayThreads, 0, s>>>(A);
        else fine_comp_bwd_kernel<DVGO_ACT_POST><<<g, kRayThreads, 0, s>>>(A);
    }
}

}  // namespace dvgo
