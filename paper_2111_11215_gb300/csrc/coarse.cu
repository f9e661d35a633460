// coarse.cu -- coarse-stage render (Sec. 4.1): density grid + view-invariant colour grid.
//
// One warp per ray, 32 consecutive samples per iteration.  Per sample:
//   sigma_ddot = interp(x, V_density)                      (Eq. coarse_queries_densities)
//   sigma = softplus(sigma_ddot + b), tau = sigma * dt       (Eq. density_activation, post-activation)
//   alpha = 1 - exp(-tau); removed when alpha < tau_f        (Eq. density_2_alpha, Sec. 4.2 skipping)
//   c = interp(x, V_rgb) (optionally sigmoid)                (Eq. coarse_queries)
// Compositing keeps the optical depth prefix sum: T_k = exp(-sum_{j<k} tau_j), w_k = T_k alpha_k,
// C_hat = sum w_k c_k + T_K bg (Eq. volume_rendering).  The prefix is a warp scan per chunk plus a
// running carry, which keeps T exact to FP32 rounding of the sum even over hundreds of samples.
//
// Backward (recomputes the forward chunk by chunk, stores nothing per sample in memory):
//   dC/dc_k = w_k,  dC/dtau_k = T_{k+1} c_k - S_k,  S_k = sum_{j>k} w_j c_j + T_K bg,
//   dT_K/dtau_k = -T_K,  dtau_k/dsigma_ddot = dt * sigmoid(sigma_ddot + b) = dt (1 - e^{-tau/dt});
// gradients are scattered to the 8 lattice corners with weights equal to the trilinear weights,
// summed first over runs of lanes that lie in the same cell.
//
// Both kernels are bound by the latency of a ray's serial chain of chunks (ncu: 12-24 % of the warp
// slots active, IPC 0.75), and rays differ in length by an order of magnitude, so blocks are two
// warps: a block's slots are free as soon as its two rays are done (with eight rays a block, half of
// the forward's stall cycles were warps waiting at the loss reduction's barrier).  100^3, 8192 rays,
// 858 k samples: forward 74 -> 58 us, backward 254 -> 101 us.

#include "dvgo_internal.cuh"

namespace dvgo {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int kCoarseThreads = 64;

struct CoarseSample {
    Cell cell;
    float tau;    // optical depth (0 when removed)
    float c[3];   // emitted colour
};

template <int kOrder>
__device__ __forceinline__ CoarseSample coarse_sample(const RenderArgs &A, const RayRec &rr, int ray, int k) {
    CoarseSample S;
    float dt;
    S.cell = sample_cell(A, rr, ray, k, dt);
    const float *rgb = static_cast<const float *>(A.cgrid);
    float s = 0.0f, col[3] = {0.0f, 0.0f, 0.0f}, v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        long long idx = corner_index(S.cell, q, A.ny, A.nz, A.packed);
        float w = corner_weight(S.cell, q);
        v[q] = __ldg(A.density + idx);
        s = fmaf(w, v[q], s);
        const float *cp = rgb + idx * 3;
        col[0] = fmaf(w, __ldg(cp + 0), col[0]);
        col[1] = fmaf(w, __ldg(cp + 1), col[1]);
        col[2] = fmaf(w, __ldg(cp + 2), col[2]);
    }
    S.tau = kOrder == DVGO_ACT_POST ? softplusf(s + A.shift_b) * dt : tau_pre_in(kOrder, S.cell, v, A.shift_b, dt);
    if (-expm1f(-S.tau) < A.tau_f) S.tau = 0.0f;
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) S.c[ch] = A.rgb_act ? sigmoidf_(col[ch]) : col[ch];
    return S;
}

// Block-level loss reduction: every block adds its partial sum; the last block to finish
// writes loss_out = sum / R.
__device__ void finish_loss(const RenderArgs &A, float part) {
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

template <int kOrder>
__global__ void __launch_bounds__(kCoarseThreads) coarse_fwd_kernel(RenderArgs A) {
    int lane = threadIdx.x & 31;
    int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int nwarps = (gridDim.x * blockDim.x) >> 5;
    float loss_part = 0.0f;
    const bool aux = A.target && (A.w_pt != 0.0f || A.w_bg != 0.0f);
    for (int r = warp; r < A.R; r += nwarps) {
        const RayRec rr = A.rays[r];
        flag_bad_ray(A, rr, lane);
        float tg[3] = {0.0f, 0.0f, 0.0f};
        if (aux)
            for (int ch = 0; ch < 3; ++ch) tg[ch] = A.target[3 * r + ch];
        float carry = 0.0f, acc[3] = {0.0f, 0.0f, 0.0f}, pt = 0.0f;
        for (int base = 0; base < rr.n; base += 32) {
            int k = base + lane;
            CoarseSample S;
            S.tau = 0.0f;
            S.c[0] = S.c[1] = S.c[2] = 0.0f;
            if (k < rr.n) S = coarse_sample<kOrder>(A, rr, r, k);
            float incl = warp_incl_scan(S.tau, lane);
            float excl = __shfl_up_sync(FULL, incl, 1);
            if (lane == 0) excl = 0.0f;
            float T = expf(-(carry + excl));
            float w = T * -expm1f(-S.tau);
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) {
                acc[ch] = fmaf(w, S.c[ch], acc[ch]);
                const float e = S.c[ch] - tg[ch];
                pt = fmaf(w * e, e, pt);          // per-point rgb loss
            }
            carry += __shfl_sync(FULL, incl, 31);
        }
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) acc[ch] = warp_sum(acc[ch]);
        if (aux) pt = warp_sum(pt);
        if (lane == 0) {
            float TK = expf(-carry);
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
    if (A.target) finish_loss(A, loss_part);
}

// Optical depth of one sample (density gather only), with the removal rule.
template <int kOrder>
__device__ __forceinline__ float coarse_tau(const RenderArgs &A, const RayRec &rr, int ray, int k) {
    float dt;
    Cell c = sample_cell(A, rr, ray, k, dt);
    float s = 0.0f, v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        v[q] = __ldg(A.density + corner_index(c, q, A.ny, A.nz, A.packed));
        s = fmaf(corner_weight(c, q), v[q], s);
    }
    float tau = kOrder == DVGO_ACT_POST ? softplusf(s + A.shift_b) * dt : tau_pre_in(kOrder, c, v, A.shift_b, dt);
    return (-expm1f(-tau) < A.tau_f) ? 0.0f : tau;
}

// Backward: pass 1 (front to back) recomputes every sample's optical depth (kept in shared memory,
// cap floats per warp) and the depth before every chunk; pass 2 (back to front) gathers the colours
// again and evaluates dC/dtau_k as the suffix sum D_k = sum_{j>=k} T_{j+1} (c_j - c_{j+1}) with c_K =
// bg (from D_k - D_{k+1} = T_{k+1}(c_k - c_{k+1}) and D_{K-1} = T_K (c_{K-1} - bg)), which avoids the
// cancellation of T_{k+1} c_k - S_k.  Two samples share a corner q exactly when their cells are the
// same, so one segmentation of the warp serves the 8 corners x 4 channels; the segmented sums run side
// by side and stop after the warp's longest run (half-voxel steps: one or two rounds instead of five).
template <int kOrder>
__global__ void __launch_bounds__(kCoarseThreads) coarse_bwd_kernel(RenderArgs A, int cap) {
    extern __shared__ float s_dyn[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    float *s_pre = s_dyn + wib * (cap + kMaxChunks), *s_tau = s_pre + kMaxChunks;
    int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int nwarps = (gridDim.x * blockDim.x) >> 5;
    const float *rgb = static_cast<const float *>(A.cgrid);
    for (int r = warp; r < A.R; r += nwarps) {
        const RayRec rr = A.rays[r];
        if (rr.n == 0) continue;
        const int nch = (rr.n + 31) >> 5;
        const float TK = A.rayout[r].w;
        const float g[3] = {A.grad_rgb[3 * r], A.grad_rgb[3 * r + 1], A.grad_rgb[3 * r + 2]};
        // auxiliary losses of the forward: the background entropy enters through T_K, the
        // per-point rgb loss adds 2 w_pt w_k (c_k - C) / R to dL/dc_k
        const bool aux = A.hdr->aux != 0;
        float4 tg = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (aux) tg = A.rtarget[r];
        const float tgc[3] = {tg.x, tg.y, tg.z};
        const float gT = (A.grad_tfinal ? A.grad_tfinal[r] : 0.0f) +
                         (aux ? A.w_bg * bg_entropy_dT(TK) / (float)A.R : 0.0f);
        const float kpt = aux ? 2.0f * A.w_pt / (float)A.R : 0.0f;
        float carry = 0.0f;
        for (int ci = 0; ci < nch; ci += 2) {   // two chunks' density loads in flight
            float tau[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int k = (ci + h) * 32 + lane;
                tau[h] = k < rr.n ? coarse_tau<kOrder>(A, rr, r, k) : 0.0f;
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int k = (ci + h) * 32 + lane;
                if (k < rr.n) s_tau[k] = tau[h];
                if (lane == 0 && ci + h < nch) s_pre[ci + h] = carry;
                carry += __shfl_sync(FULL, warp_incl_scan(tau[h], lane), 31);
            }
        }
        __syncwarp();
        float Dc[3] = {0.0f, 0.0f, 0.0f};
        float cnext[3] = {A.bg[0], A.bg[1], A.bg[2]};
        for (int ci = nch - 1; ci >= 0; --ci) {
            const int k = ci * 32 + lane;
            const bool valid = k < rr.n;
            const float tau = valid ? s_tau[k] : 0.0f;
            Cell cell;
            cell.i0 = cell.j0 = cell.k0 = 0;
            cell.fx = cell.fy = cell.fz = 0.0f;
            float dt = 0.0f, c[3] = {0.0f, 0.0f, 0.0f};
            int idx[8];
            if (valid) cell = sample_cell(A, rr, r, k, dt);
#pragma unroll
            for (int q = 0; q < 8; ++q) idx[q] = (int)corner_index(cell, q, A.ny, A.nz, A.packed);
            if (valid) {
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const float w = corner_weight(cell, q);
                    const float *cp = rgb + (long long)idx[q] * 3;
#pragma unroll
                    for (int ch = 0; ch < 3; ++ch) c[ch] = fmaf(w, __ldg(cp + ch), c[ch]);
                }
                if (A.rgb_act)
#pragma unroll
                    for (int ch = 0; ch < 3; ++ch) c[ch] = sigmoidf_(c[ch]);
            }
            const float pre = s_pre[ci];
            float incl = warp_incl_scan(tau, lane);
            float excl = __shfl_up_sync(FULL, incl, 1);
            if (lane == 0) excl = 0.0f;
            const float T1 = expf(-(pre + incl));
            const float w = expf(-(pre + excl)) * -expm1f(-tau);
            float dtau = -gT * TK;
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) {
                float cn = __shfl_down_sync(FULL, c[ch], 1);
                if (lane == 31 || k + 1 >= rr.n) cn = (k + 1 >= rr.n) ? A.bg[ch] : cnext[ch];
                const float sx = warp_suffix_scan(valid ? T1 * (c[ch] - cn) : 0.0f, lane);
                dtau = fmaf(g[ch], Dc[ch] + sx, dtau);
                Dc[ch] += __shfl_sync(FULL, sx, 0);
                cnext[ch] = __shfl_sync(FULL, c[ch], 0);
            }
            // kept samples have tau > 0 (or NaN) or exactly zero factors below; removed ones have tau = 0
            const bool act = valid && !(tau <= 0.0f);
            const float dz = act ? dtau * dt * -expm1f(-tau / dt) : 0.0f;
            float dc[3];
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) {
                float gc = g[ch] * w + kpt * w * (c[ch] - tgc[ch]);
                if (A.rgb_act) gc *= c[ch] * (1.0f - c[ch]);
                dc[ch] = act ? gc : 0.0f;
            }
            const Seg sg = make_seg(act ? cell_base(cell, A.ny, A.nz, A.packed) : -1 - lane, lane);
            int run = lane - sg.first + 1;
            run = __reduce_max_sync(FULL, run);
            float gq[8][4];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const float cw = corner_weight(cell, q);
                gq[q][0] = dz * cw;
                if (kOrder != DVGO_ACT_POST)
                    gq[q][0] = act ? dtau * dtau_dv_pre_in(kOrder, cell, q, __ldg(A.density + idx[q]), A.shift_b, dt, tau)
                                   : 0.0f;
#pragma unroll
                for (int ch = 0; ch < 3; ++ch) gq[q][1 + ch] = dc[ch] * cw;
            }
            for (int o = 1; o < run; o <<= 1) {
                const bool add = lane - o >= sg.first;
#pragma unroll
                for (int q = 0; q < 8; ++q)
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        const float n = __shfl_up_sync(FULL, gq[q][v], o);
                        if (add) gq[q][v] += n;
                    }
            }
            if (act && sg.tail) {
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    atomicAdd(A.grad_density + idx[q], gq[q][0]);
                    float *gc = A.grad_cgrid + (long long)idx[q] * 3;
#pragma unroll
                    for (int ch = 0; ch < 3; ++ch) atomicAdd(gc + ch, gq[q][1 + ch]);
                }
            }
        }
        __syncwarp();
    }
}

// Two rays per block; every ray has its own warp up to 64 blocks (128 rays) per SM in the grid, then the warps stride.
int coarse_grid(int R) {
    const int want = (R + 1) / 2, cap = num_sms() * 64;
    return want > cap ? cap : (want < 1 ? 1 : want);
}

}  // namespace

void launch_coarse_fwd(const RenderArgs &A, cudaStream_t s) {
    ProfScope ps_(DVGO_K_COARSE_FWD, s);
    const int g = coarse_grid(A.R);
    if (A.act_order == DVGO_ACT_PRE) coarse_fwd_kernel<DVGO_ACT_PRE><<<g, kCoarseThreads, 0, s>>>(A);
    else if (A.act_order == DVGO_ACT_IN) coarse_fwd_kernel<DVGO_ACT_IN><<<g, kCoarseThreads, 0, s>>>(A);
    else coarse_fwd_kernel<DVGO_ACT_POST><<<g, kCoarseThreads, 0, s>>>(A);
}

void launch_coarse_bwd(const RenderArgs &A, cudaStream_t s) {
    ProfScope ps_(DVGO_K_COARSE_BWD, s);
    const int g = coarse_grid(A.R);
    // the longest ray's optical depths per warp (at most kMaxSamplesPerRay: 16 KB a block)
    const int cap = A.cap;
    const size_t smem = sizeof(float) * (kCoarseThreads / 32) * (cap + kMaxChunks);
    if (A.act_order == DVGO_ACT_PRE) coarse_bwd_kernel<DVGO_ACT_PRE><<<g, kCoarseThreads, smem, s>>>(A, cap);
    else if (A.act_order == DVGO_ACT_IN) coarse_bwd_kernel<DVGO_ACT_IN><<<g, kCoarseThreads, smem, s>>>(A, cap);
    else coarse_bwd_kernel<DVGO_ACT_POST><<<g, kCoarseThreads, smem, s>>>(A, cap);
}

}  // namespace dvgo
