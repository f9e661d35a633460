// proposal.cu -- learned sample proposal: per-ray weight histograms (labels), the proposal MLP
// forward / backward (softmax cross-entropy), and inverse-CDF sampling of explicit samples.
//
// The paper renders with uniform steps and leaves hierarchical sampling to future work (Supp. B,
// step-size ablation); this proposal is the library's addition.  Definitions:
//   bins:     n_bins equal bins of the clipped interval [t_enter, t_exit] of each ray;
//   labels:   h_b = sum of the compositing weights w_k = T_k alpha_k of the samples whose t_k
//             falls in bin b, divided by sum_k w_k (uniform when that sum is below 1e-4), from a
//             uniform-step fine forward (Eq. volume_rendering);
//   network:  the bin centre x_b = o + t_b d is encoded as [x, sin(2^k x_c), cos(2^k x_c)]
//             (k < 6, c-major), then 39 -> 64 -> 64 -> 64 -> 1 with ReLU gives a logit per bin and
//             p = softmax over the bins; loss = -(1/R) sum_r sum_b h_rb log p_rb (rays that miss
//             the box contribute nothing);
//   sampling: q_b = (1 - eta) p_b + eta / n_bins, Q its CDF; sample j at u_j = (j + jit) / n * Q_nb
//             lies in the bin with Q_b <= u_j < Q_{b+1}, at t = t0 + (b + (u_j - Q_b) / q_b) w;
//             dt_j = t_{j+1} - t_j and, for the last sample, w Q_nb / (n q_b).
// The bin of a quantile (labels) is decided in FP64 with separately rounded operations, in the
// order written above.  Sampling runs in double-float arithmetic (below): its CDF, quantiles and
// sample positions carry ~48 significant bits, so a sample's bin can differ from the exact one
// only where its quantile lies within ~1e-14 of a bin edge -- where t is continuous across the
// edge -- and t, dt come out as the FP32 roundings of the exact values to within an ulp.

#include <math.h>

#include "dvgo_internal.cuh"
#include "proposal_rays.cuh"

namespace dvgo {

namespace {

constexpr int NB = kPropBins;      // bins
constexpr int NFQ = 6;             // PE frequencies on the bin centre
constexpr int PIN = 3 + 6 * NFQ;   // 39
constexpr int PK0 = PIN + 1;       // 40 with the bias column
constexpr int PW = 64;             // width
constexpr int PTM = 128;           // rows per tile = 2 rays x 64 bins
constexpr int PNT = 256;
constexpr int PLD = PTM + 4;       // activation row stride (feature-major storage)

struct BoxD {
    double mn[3], mx[3];
    double t_near, t_far;
};

BoxD make_box(const dvgo_params &p, const dvgo_grid_desc &g) {
    BoxD b;
    for (int a = 0; a < 3; ++a) {
        b.mn[a] = g.xyz_min[a];
        b.mx[a] = g.xyz_max[a];
    }
    b.t_near = p.t_near;
    b.t_far = p.t_far;
    return b;
}

__device__ __forceinline__ Clip clip_ray(const BoxD &B, const float *ro, const float *rd, int r) {
    const double o[3] = {(double)ro[3 * r], (double)ro[3 * r + 1], (double)ro[3 * r + 2]};
    const double d[3] = {(double)rd[3 * r], (double)rd[3 * r + 1], (double)rd[3 * r + 2]};
    return slab_clip(o, d, B.mn, B.mx, B.t_near, B.t_far);
}

// ---------------------------------------------------------------------------------------------
// Labels: per-ray histogram of compositing weights over n_bins bins (warp per ray)
// ---------------------------------------------------------------------------------------------

__global__ void __launch_bounds__(256) weight_bins_kernel(RenderArgs A, int nbins, float *labels) {
    __shared__ float bins[8][128];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    // the state lies where the forward's own parameters put it
    const WsHeader &H = *A.hdr;
    const char *base = reinterpret_cast<const char *>(A.hdr);
    const double *texit = reinterpret_cast<const double *>(base + H.texit_at);
    const int4 *rayk = reinterpret_cast<const int4 *>(base + H.rayk_at);
    const RayChunk *rchunk = reinterpret_cast<const RayChunk *>(base + H.rchunk_at);
    const float *stau = reinterpret_cast<const float *>(base + H.stau_at);
    const int n_rays = H.n_rays, cap = H.cap, nchunk = chunks_per_ray(cap);
    for (int r = warp; r < A.R; r += nwarps) {
        if (r >= n_rays) {   // not a ray of the forward
            for (int b = lane; b < nbins; b += 32) labels[(size_t)r * nbins + b] = 1.0f / nbins;
            continue;
        }
        const RayRec rr = A.rays[r];
        const double t0 = rr.t_enter, t1 = texit[r];
        // bin of sample k: floor((t_k - t_enter) / (t_exit - t_enter) nbins), t_k - t_enter = (k + p) step
        const double bin_scale = __ddiv_rn(__dmul_rn((double)A.step, (double)nbins), __dsub_rn(t1, t0));
        for (int b = lane; b < nbins; b += 32) bins[wib][b] = 0.0f;
        __syncwarp();
        float wsum = 0.0f;
        const int nrec = rayk[r].x;   // chunks with a kept sample; the other samples have weight 0
        const size_t off = (size_t)r * cap;
        for (int c = 0; c < nrec; ++c) {
            const RayChunk ch = rchunk[(size_t)r * nchunk + c];
            const bool kept = (ch.mask >> lane) & 1u;
            const float tau = kept ? stau[off + ch.first + __popc(ch.mask & ((1u << lane) - 1u))] : 0.0f;
            const float incl = warp_incl_scan(tau, lane);
            float excl = __shfl_up_sync(0xffffffffu, incl, 1);
            if (lane == 0) excl = 0.0f;
            const float w = expf(-(ch.pre + excl)) * -expm1f(-tau);
            if (kept) {
                const int k = ch.index * 32 + lane;
                int b = (int)floor(__dmul_rn(__dadd_rn((double)k, (double)rr.p), bin_scale));
                b = b < 0 ? 0 : (b >= nbins ? nbins - 1 : b);
                atomicAdd(&bins[wib][b], w);
            }
            wsum += warp_sum(w);
        }
        __syncwarp();
        const bool uniform = wsum < 1e-4f;
        for (int b = lane; b < nbins; b += 32)
            labels[(size_t)r * nbins + b] = uniform ? 1.0f / nbins : bins[wib][b] / wsum;
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------------------------
// Proposal MLP (FP32 SIMT), tiles of 2 rays x 64 bins
// ---------------------------------------------------------------------------------------------

struct PropArgs {
    int R;
    BoxD box;
    const float *ro, *rd, *labels;
    const float *w0, *b0, *w1, *b1, *w2, *b2, *w3, *b3;
    float *probs, *loss, *grad;
};

struct PropSmem {
    float w0[PK0 * PW];     // rows 0..38 = W0, row 39 = b0
    float w1[PW * PW], w2[PW * PW];
    float w1t[PW * PW], w2t[PW * PW];   // transposed copies for the backward
    float b1[PW], b2[PW], w3[PW];
    float b3[4];              // [0] used; 4 floats keep the following arrays 16-byte aligned
    float xt[PK0 * PLD];    // inputs, feature-major
    float h0[PW * PLD], h1[PW * PLD], h2[PW * PLD];
    alignas(16) float logit[PTM];
    alignas(16) float dlog[PTM];
    ClipDf clip[PTM];       // rays of the CTA's current 64 tiles
};

__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ void st4(float *p, float4 v) { *reinterpret_cast<float4 *>(p) = v; }

// acc[i][j] = sum_k InT[k][4 ty + i] W[k][col(j)] + bias for 128 rows x 64 outputs, one FMA chain over k
// per value.  Thread (ty, tx) = (t >> 3, t & 7): rows 4 ty .. +3, outputs 4 tx .. +3 and 32 + 4 tx .. +3, so
// that each 16-byte load of a warp is one pass over the banks.
__device__ __forceinline__ int out_col(int tx, int j) { return j < 4 ? 4 * tx + j : 28 + 4 * tx + j; }

template <int K>
__device__ __forceinline__ void ptile_gemm(const float *InT, const float *W, const float *bias, float (&acc)[4][8]) {
    const int ty = threadIdx.x >> 3, tx = threadIdx.x & 7;
    const int r0 = 4 * ty;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const float b = bias ? bias[out_col(tx, j)] : 0.0f;
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i][j] = b;
    }
#pragma unroll 8
    for (int k = 0; k < K; ++k) {
        const float4 a = ld4(InT + k * PLD + r0);
        const float4 x0 = ld4(W + k * PW + 4 * tx), x1 = ld4(W + k * PW + 32 + 4 * tx);
        const float av[4] = {a.x, a.y, a.z, a.w};
        const float bv[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
    }
}

// OutT = relu(acc).
__device__ __forceinline__ void store_relu(const float (&acc)[4][8], float *OutT) {
    const int ty = threadIdx.x >> 3, tx = threadIdx.x & 7;
#pragma unroll
    for (int j = 0; j < 8; ++j)
        st4(OutT + out_col(tx, j) * PLD + 4 * ty,
            make_float4(fmaxf(acc[0][j], 0.0f), fmaxf(acc[1][j], 0.0f), fmaxf(acc[2][j], 0.0f), fmaxf(acc[3][j], 0.0f)));
}

// OutT = acc [H > 0].
__device__ __forceinline__ void store_masked(const float (&acc)[4][8], const float *HT, float *OutT) {
    const int ty = threadIdx.x >> 3, tx = threadIdx.x & 7;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int o = out_col(tx, j) * PLD + 4 * ty;
        const float4 h = ld4(HT + o);
        st4(OutT + o, make_float4(h.x > 0.0f ? acc[0][j] : 0.0f, h.y > 0.0f ? acc[1][j] : 0.0f,
                                  h.z > 0.0f ? acc[2][j] : 0.0f, h.w > 0.0f ? acc[3][j] : 0.0f));
    }
}

// g[i][j] += sum_r HT[kq + 32 i][r] DT[nq + 8 j][r], thread (kq, nq) = (t >> 3, t & 7), and gb +=
// sum_r DT[nq + 8 w][r] with w the warp (kept by its lanes kq % 4 == 0).  The strided outputs put the
// eight rows a warp reads at once in different banks (with eight neighbouring rows per thread every
// load was eight-way conflicted, and the weight gradients took most of the backward).
__device__ __forceinline__ void weight_grad(const float *HT, const float *DT, float (&g)[2][8], float &gb) {
    const int kq = threadIdx.x >> 3, nq = threadIdx.x & 7, warp = threadIdx.x >> 5;
#pragma unroll 2
    for (int r = 0; r < PTM; r += 4) {
        const float4 a0 = ld4(HT + kq * PLD + r), a1 = ld4(HT + (kq + 32) * PLD + r);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float4 d = ld4(DT + (nq + 8 * j) * PLD + r);
            g[0][j] = fmaf(a0.x, d.x, fmaf(a0.y, d.y, fmaf(a0.z, d.z, fmaf(a0.w, d.w, g[0][j]))));
            g[1][j] = fmaf(a1.x, d.x, fmaf(a1.y, d.y, fmaf(a1.z, d.z, fmaf(a1.w, d.w, g[1][j]))));
            if (j == warp) gb += (d.x + d.y) + (d.z + d.w);
        }
    }
}

// sin / cos of the double-float argument a, reduced by 2 pi in double-float arithmetic (2 pi = 6.28318548... -
// 1.7484556e-7) and evaluated in FP32.  The argument and its reduction are each off by up to 2^-47 of what they are
// formed from, which is far below an FP32 rounding of the result up to kDfReach; beyond it encode_row_fp64.  The
// reduction in FP64, 18 per row, had the FP64 pipe busy for 17 us a tile.
__device__ __forceinline__ void sincos_reduced(Df a, float *s, float *c) {
    const Df two_pi = {6.283185482025146484375f, -1.74845553146951715e-7f};
    const float n = rintf(a.hi * 0.15915494f);
    const Df red = df_add(a, df_neg(df_mul_f(two_pi, n)));
    sincosf(red.hi, s, c);
}

// The same part of an input row with positions and argument reductions in FP64, for rays that reach further
// out than kDfReach.
__device__ __noinline__ void encode_row_fp64(const PropArgs &P, int r, int bin, int part, int row, float *xt) {
    const Clip c = clip_ray(P.box, P.ro, P.rd, r);
    const double tb = __dadd_rn(c.lo, __ddiv_rn(__dmul_rn((double)bin + 0.5, __dsub_rn(c.hi, c.lo)), (double)NB));
    const double two_pi = 6.283185307179586;
#pragma unroll 1
    for (int a = 0; a < 3; ++a) {
        const double x = __dadd_rn((double)P.ro[3 * r + a], __dmul_rn(tb, c.dn[a]));
        if (part == 0) xt[a * PLD + row] = (float)x;
        for (int k = 3 * part; k < 3 * part + 3; ++k) {
            const double arg = ldexp(x, k);
            float sv, cv;
            sincosf((float)fma(-rint(arg / two_pi), two_pi, arg), &sv, &cv);
            xt[(3 + a * NFQ + k) * PLD + row] = sv;
            xt[(3 + 3 * NFQ + a * NFQ + k) * PLD + row] = cv;
        }
    }
}

template <bool BWD>
__global__ void __launch_bounds__(PNT, 1) proposal_kernel(PropArgs P) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    PropSmem &S = *reinterpret_cast<PropSmem *>(smem_raw);
    const int tid = threadIdx.x;
    for (int i = tid; i < PK0 * PW; i += PNT) {
        const int k = i / PW, j = i % PW;
        S.w0[i] = k < PIN ? P.w0[k * PW + j] : P.b0[j];
    }
    for (int i = tid; i < PW * PW; i += PNT) {
        const int k = i / PW, j = i % PW;
        S.w1[i] = P.w1[i];
        S.w2[i] = P.w2[i];
        if (BWD) {
            S.w1t[j * PW + k] = P.w1[i];
            S.w2t[j * PW + k] = P.w2[i];
        }
    }
    if (tid < PW) {
        S.b1[tid] = P.b1[tid];
        S.b2[tid] = P.b2[tid];
        S.w3[tid] = P.w3[tid];
    }
    if (tid == 0) S.b3[0] = P.b3[0];
    // weight-gradient accumulators (backward)
    float g1[2][8], g2[2][8], g0[10], g3 = 0.0f, gb1 = 0.0f, gb2 = 0.0f, gb3 = 0.0f;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) g1[i][j] = g2[i][j] = 0.0f;
#pragma unroll
    for (int i = 0; i < 10; ++i) g0[i] = 0.0f;
    const float invR = 1.0f / (float)P.R;

    const int ntiles = (P.R + 1) / 2;
    int kt = 0;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++kt) {
        __syncthreads();
        if (kt % 64 == 0) {
            if (tid < PTM)
                clip_tile_rays(P.R, P.ro, P.rd, P.box.mn, P.box.mx, P.box.t_near, P.box.t_far, kt, S.clip);
            __syncthreads();
        }
        // encode the bin centres: 2 threads per row
        {
            const int row = tid >> 1, part = tid & 1;
            const ClipDf &cl = S.clip[2 * (kt % 64) + (row >> 6)];
            Df x[3] = {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}};
            if (cl.hit) {
                const Df tb = bin_centre(cl, row & 63);
#pragma unroll
                for (int a = 0; a < 3; ++a) x[a] = bin_position(cl, tb, a);
            }
            if (part == 0) S.xt[PIN * PLD + row] = 1.0f;
            // part 0: positions and k = 0..2, part 1: k = 3..5 for every axis
            if (cl.hit & 2) {
                encode_row_fp64(P, 2 * tile + (row >> 6), row & 63, part, row, S.xt);
            } else {
                if (part == 0)
#pragma unroll
                    for (int a = 0; a < 3; ++a) S.xt[a * PLD + row] = x[a].hi;
#pragma unroll
                for (int a = 0; a < 3; ++a)
#pragma unroll
                    for (int kk = 0; kk < 3; ++kk) {
                        const int k = 3 * part + kk;
                        const float p2 = (float)(1 << k);
                        float sv, cv;
                        sincos_reduced(Df{x[a].hi * p2, x[a].lo * p2}, &sv, &cv);
                        S.xt[(3 + a * NFQ + k) * PLD + row] = sv;
                        S.xt[(3 + 3 * NFQ + a * NFQ + k) * PLD + row] = cv;
                    }
            }
        }
        __syncthreads();
        float acc[4][8];
        ptile_gemm<PK0>(S.xt, S.w0, nullptr, acc);
        store_relu(acc, S.h0);
        __syncthreads();
        ptile_gemm<PW>(S.h0, S.w1, S.b1, acc);
        store_relu(acc, S.h1);
        __syncthreads();
        ptile_gemm<PW>(S.h1, S.w2, S.b2, acc);
        if (BWD) store_relu(acc, S.h2);
        {   // output layer: each thread's eight columns, then the eight threads of a row group
            const int ty = tid >> 3, tx = tid & 7;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float o = 0.0f;
#pragma unroll
                for (int j = 0; j < 8; ++j) o = fmaf(fmaxf(acc[i][j], 0.0f), S.w3[out_col(tx, j)], o);
                o += __shfl_xor_sync(0xffffffffu, o, 1);
                o += __shfl_xor_sync(0xffffffffu, o, 2);
                o += __shfl_xor_sync(0xffffffffu, o, 4);
                if (tx == i) S.logit[4 * ty + i] = o + S.b3[0];
            }
        }
        __syncthreads();
        // softmax per ray (warp 0: ray 0, warp 1: ray 1), loss, dlogit
        if (tid < 64) {
            const int rl = tid >> 5, lane = tid & 31, r = 2 * tile + rl;
            if (r < P.R) {
                const float l0 = S.logit[64 * rl + lane], l1 = S.logit[64 * rl + lane + 32];
                float m = fmaxf(l0, l1);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
                const float e0 = expf(l0 - m), e1 = expf(l1 - m);
                const float z = warp_sum(e0 + e1);
                float p0 = e0 / z, p1 = e1 / z;
                const bool hit = S.clip[2 * (kt % 64) + rl].hit != 0;
                if (!hit) p0 = p1 = 1.0f / NB;
                if (!BWD && P.probs) {
                    P.probs[(size_t)r * NB + lane] = p0;
                    P.probs[(size_t)r * NB + lane + 32] = p1;
                }
                float d0 = 0.0f, d1 = 0.0f;
                if (P.labels && hit) {
                    const float h0 = P.labels[(size_t)r * NB + lane], h1 = P.labels[(size_t)r * NB + lane + 32];
                    if (!BWD && P.loss) {
                        float lr = 0.0f;
                        if (h0 > 0.0f) lr -= h0 * logf(p0);
                        if (h1 > 0.0f) lr -= h1 * logf(p1);
                        lr = warp_sum(lr);
                        if (lane == 0) atomicAdd(P.loss, lr * invR);
                    }
                    d0 = (p0 - h0) * invR;
                    d1 = (p1 - h1) * invR;
                }
                S.dlog[64 * rl + lane] = d0;
                S.dlog[64 * rl + lane + 32] = d1;
            } else {
                S.dlog[64 * rl + lane] = 0.0f;
                S.dlog[64 * rl + lane + 32] = 0.0f;
            }
        }
        if (!BWD) continue;
        __syncthreads();
        // output layer: dW3 += H2^T dlogit, db3 += sum dlogit, and dZ2 = dlogit w3^T [H2 > 0] over H2: unit
        // t >> 2, every fourth group of four rows
        {
            const int f = tid >> 2, part = tid & 3;
            const float w3 = S.w3[f];
            float a = 0.0f;
#pragma unroll
            for (int r = 4 * part; r < PTM; r += 16) {
                const float4 h = ld4(S.h2 + f * PLD + r), d = ld4(S.dlog + r);
                a = fmaf(h.x, d.x, fmaf(h.y, d.y, fmaf(h.z, d.z, fmaf(h.w, d.w, a))));
                if (f == 0) gb3 += (d.x + d.y) + (d.z + d.w);
                st4(S.h2 + f * PLD + r, make_float4(h.x > 0.0f ? d.x * w3 : 0.0f, h.y > 0.0f ? d.y * w3 : 0.0f,
                                                    h.z > 0.0f ? d.z * w3 : 0.0f, h.w > 0.0f ? d.w * w3 : 0.0f));
            }
            g3 += a;
        }
        __syncthreads();
        weight_grad(S.h1, S.h2, g2, gb2);              // dW2 += H1^T dZ2, db2 += sum dZ2
        ptile_gemm<PW>(S.h2, S.w2t, nullptr, acc);     // dH1 = dZ2 W2^T
        __syncthreads();                               // all reads of H1 (dW2) and dZ2 done
        store_masked(acc, S.h1, S.h1);                 // dZ1 over H1
        __syncthreads();
        weight_grad(S.h0, S.h1, g1, gb1);              // dW1 += H0^T dZ1, db1 += sum dZ1
        ptile_gemm<PW>(S.h1, S.w1t, nullptr, acc);
        store_masked(acc, S.h0, S.h2);                 // dZ0 over h2 (free now)
        __syncthreads();
        // [dW0 | db0] += X^T dZ0 : thread: output n = t & 63, inputs 10 (t >> 6) .. +9
        {
            const int n = tid & 63, kq = tid >> 6;
            for (int r = 0; r < PTM; r += 4) {
                const float4 d = ld4(S.h2 + n * PLD + r);
#pragma unroll
                for (int i = 0; i < 10; ++i) {
                    const float4 a = ld4(S.xt + (10 * kq + i) * PLD + r);
                    g0[i] = fmaf(a.x, d.x, fmaf(a.y, d.y, fmaf(a.z, d.z, fmaf(a.w, d.w, g0[i]))));
                }
            }
        }
    }
    if (!BWD) return;
    // flush: grad = w0 | b0 | w1 | b1 | w2 | b2 | w3 | b3
    float *G0 = P.grad, *GB0 = G0 + PIN * PW, *G1 = GB0 + PW, *GB1 = G1 + PW * PW, *G2 = GB1 + PW, *GB2 = G2 + PW * PW;
    float *G3 = GB2 + PW, *GB3 = G3 + PW;
    {
        const int kq = tid >> 3, nq = tid & 7, warp = tid >> 5;
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                atomicAdd(G1 + (kq + 32 * i) * PW + nq + 8 * j, g1[i][j]);
                atomicAdd(G2 + (kq + 32 * i) * PW + nq + 8 * j, g2[i][j]);
            }
        if ((kq & 3) == 0) {
            atomicAdd(GB1 + nq + 8 * warp, gb1);
            atomicAdd(GB2 + nq + 8 * warp, gb2);
        }
        const int n = tid & 63, k0 = 10 * (tid >> 6);
#pragma unroll
        for (int i = 0; i < 10; ++i) {
            const int k = k0 + i;
            if (k < PIN) atomicAdd(G0 + k * PW + n, g0[i]);
            else if (k == PIN) atomicAdd(GB0 + n, g0[i]);
        }
    }
    g3 += __shfl_xor_sync(0xffffffffu, g3, 1);
    g3 += __shfl_xor_sync(0xffffffffu, g3, 2);
    gb3 += __shfl_xor_sync(0xffffffffu, gb3, 1);
    gb3 += __shfl_xor_sync(0xffffffffu, gb3, 2);
    if ((tid & 3) == 0) atomicAdd(G3 + (tid >> 2), g3);
    if (tid == 0) atomicAdd(GB3, gb3);
}

// ---------------------------------------------------------------------------------------------
// Inverse-CDF sampling.  FP64 runs at 1/64 of the FP32 rate on this GPU, so everything past the
// box clip is double-float arithmetic (df64.cuh).
// ---------------------------------------------------------------------------------------------

constexpr int kPdfThreads = 64;
constexpr int kPdfMaxBins = 128;

// A warp takes `group` consecutive rays: its lanes clip one ray each (FP64, one pass of the pipe for all of
// them), then the warp samples the rays one after the other -- the CDF is a warp scan over the bins
// (ceil(nb / 32) consecutive ones per lane), every lane places its own samples by a binary search over
// the lanes' CDF values, and rows are read and written coalesced.  No shared memory: the kernel runs
// beside the HBM-bound Adam, whose loads in flight take the SM's whole L1.  With a thread per ray (serial
// sums and merge, strided rows) 8,192 rays of 64 bins and 48 samples took 42 us, now
// 30 (events around the launch).
template <int kPer>   // bins per lane
__global__ void __launch_bounds__(kPdfThreads) sample_pdf_kernel(int R, BoxD B, const float *ro, const float *rd,
                                                                 const float *probs, int nb, int ns,
                                                                 const float *jitter, float eta, float *t_out,
                                                                 float *dt_out, int group) {
    const int lane = threadIdx.x & 31;
    const int r0 = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * group;
    if (r0 >= R) return;
    const int rn = min(group, R - r0);
    Df t0l = {0.0f, 0.0f}, wl = {0.0f, 0.0f};
    float jitl = 0.5f;
    bool hitl = false;
    if (lane < rn) {
        const Clip c = clip_ray(B, ro, rd, r0 + lane);
        hitl = c.hi > c.lo;
        if (hitl) {
            t0l = df_from_double(c.lo);
            wl = df_from_double(__ddiv_rn(__dsub_rn(c.hi, c.lo), (double)nb));
        }
        if (jitter) jitl = jitter[r0 + lane];
    }
    const float nbf = (float)nb, nsf = (float)ns;
    const Df one_m_eta = df_two_sum(1.0f, -eta);
    const Df eta_nb = df_div_n(Df{eta, 0.0f}, nbf);
    auto shfl = [](Df v, int src) {
        return Df{__shfl_sync(0xffffffffu, v.hi, src), __shfl_sync(0xffffffffu, v.lo, src)};
    };
    const int last_lane = (nb - 1) / kPer;
    for (int i = 0; i < rn; ++i) {
        const size_t r = (size_t)r0 + i;
        float *to = t_out + r * ns, *dto = dt_out + r * ns;
        if (!__shfl_sync(0xffffffffu, (int)hitl, i)) {
            for (int j = lane; j < ns; j += 32) to[j] = dto[j] = 0.0f;
            continue;
        }
        const Df t0 = shfl(t0l, i), w = shfl(wl, i);
        const float jit = __shfl_sync(0xffffffffu, jitl, i);
        // q of this lane's bins and their sum; exclusive scan over the lanes
        Df q[kPer], Q[kPer], sum = {0.0f, 0.0f};
#pragma unroll
        for (int m = 0; m < kPer; ++m) {
            const int b = lane * kPer + m;
            q[m] = Df{0.0f, 0.0f};
            if (b < nb) q[m] = df_add(df_mul_f(one_m_eta, __ldg(probs + r * nb + b)), eta_nb);
            Q[m] = sum;
            sum = df_add(sum, q[m]);
        }
        Df incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const Df up = {__shfl_up_sync(0xffffffffu, incl.hi, o), __shfl_up_sync(0xffffffffu, incl.lo, o)};
            if (lane >= o) incl = df_add(up, incl);
        }
        const Df Qtot = shfl(incl, 31);
        Df excl = {__shfl_up_sync(0xffffffffu, incl.hi, 1), __shfl_up_sync(0xffffffffu, incl.lo, 1)};
        if (lane == 0) excl = Df{0.0f, 0.0f};
#pragma unroll
        for (int m = 0; m < kPer; ++m) Q[m] = m == 0 ? excl : df_add(excl, Q[m]);   // CDF at the start of bin lane kPer + m
        Df carry = {0.0f, 0.0f};   // t of the last sample of the chunk before
        for (int base = 0; base < ns; base += 32) {
            const int j = base + lane;   // (lanes past the end place a sample that is not written)
            const Df u = df_mul(df_div_n(df_two_sum((float)j, jit), nsf), Qtot);
            int s = 0;                   // the last lane whose first bin starts at or before u
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const int c = s + o;
                const Df Qc = shfl(Q[0], c & 31);
                if (c <= last_lane && df_le(Qc, u)) s = c;
            }
            int b = s * kPer;
            Df Qb = shfl(Q[0], s), qb = shfl(q[0], s);
#pragma unroll
            for (int m = 1; m < kPer; ++m) {
                const Df Qm = shfl(Q[m], s), qm = shfl(q[m], s);
                if (s * kPer + m < nb && df_le(Qm, u)) {
                    b = s * kPer + m;
                    Qb = Qm;
                    qb = qm;
                }
            }
            // (a lane's last bin ends where the scan starts the next lane, 1e-15 off its own sum: a bin of
            // probability 0 may be met there, and the fraction leave [0, 1].  Below the first bin and above the last
            // a jitter outside [0, 1) extrapolates; a NaN among the probabilities, or none above 0, gives NaN.)
            float frac = __fdiv_rn(df_add(u, df_neg(Qb)).hi, qb.hi);
            if (qb.hi == 0.0f && Qtot.hi > 0.0f) frac = 0.0f;
            if (b > 0 && frac < 0.0f) frac = 0.0f;
            if (b < nb - 1 && frac > 1.0f) frac = 1.0f;
            const Df t = df_add(t0, df_mul(df_two_sum((float)b, frac), w));
            const Df tn = {__shfl_down_sync(0xffffffffu, t.hi, 1), __shfl_down_sync(0xffffffffu, t.lo, 1)};
            if (j < ns) to[j] = t.hi;
            if (lane == 0 && base > 0) dto[base - 1] = df_add(t, df_neg(carry)).hi;
            if (j == ns - 1)   // last step: the bin width over n times the bin's normalised probability
                dto[j] = __fdiv_rn(w.hi, __fdiv_rn(__fmul_rn(nsf, qb.hi), Qtot.hi));
            else if (j < ns && lane < 31)
                dto[j] = df_add(tn, df_neg(t)).hi;
            carry = shfl(t, 31);
        }
    }
}

}  // namespace

int launch_proposal_fwd_tc(const dvgo_params &p, const dvgo_grid_desc &g, const dvgo_proposal_mlp &m, int R,
                           const float *ro, const float *rd, const float *labels, float *probs, float *loss,
                           cudaStream_t s);
int launch_proposal_bwd_tc(const dvgo_params &p, const dvgo_grid_desc &g, const dvgo_proposal_mlp &m, int R,
                           const float *ro, const float *rd, const float *labels, float *grad, cudaStream_t s);

}  // namespace dvgo

using namespace dvgo;

extern "C" {

int dvgo_weight_bins(const dvgo_params *p, const dvgo_grid_desc *dd, int n_rays, int n_bins, const void *workspace,
                     size_t ws_bytes, float *labels_out, void *stream) {
    if (!p || !dd || n_rays < 0 || n_bins < 1 || n_bins > 128 || !workspace || (n_rays > 0 && !labels_out))
        return DVGO_ERR_INVALID_ARG;
    if (p->mode != DVGO_MODE_FINE || !(p->step > 0.0f)) return DVGO_ERR_UNSUPPORTED;
    if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return DVGO_ERR_WORKSPACE;
    if (n_rays == 0) return DVGO_OK;
    dvgo_params q = *p;
    q.tau_f = 0.0f;   // (what a render with tau_f cannot do without)
    const size_t need = dvgo_workspace_size(&q, dd, n_rays, nullptr);
    if (need == 0) return DVGO_ERR_INVALID_ARG;
    if (ws_bytes < need) return DVGO_ERR_WORKSPACE;
    const WsLayout L = ws_layout(n_rays, 0, DVGO_MODE_FINE);   // (header and ray records: the same in every layout)
    RenderArgs A;
    memset(&A, 0, sizeof(A));
    char *b = static_cast<char *>(const_cast<void *>(workspace));
    A.R = n_rays;
    A.step = p->step;
    A.hdr = reinterpret_cast<WsHeader *>(b + L.header);
    A.rays = reinterpret_cast<RayRec *>(b + L.rays);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int blocks = (n_rays + 7) / 8;
    if (blocks > num_sms() * 16) blocks = num_sms() * 16;
    {
        ProfScope ps_(DVGO_K_WEIGHT_BINS, s);
        weight_bins_kernel<<<blocks, 256, 0, s>>>(A, n_bins, labels_out);
    }
    return cudaGetLastError() == cudaSuccess ? DVGO_OK : DVGO_ERR_CUDA;
}

static int proposal_launch(bool bwd, const dvgo_params *p, const dvgo_grid_desc *dd, const dvgo_proposal_desc *pd,
                           const dvgo_proposal_mlp *m, int n_rays, const float *rays_o, const float *rays_d,
                           const float *labels, float *probs_out, float *loss_out, float *grad, void *stream) {
    if (!p || !dd || !pd || !m || n_rays < 0) return DVGO_ERR_INVALID_ARG;
    if (!m->w0 || !m->b0 || !m->w1 || !m->b1 || !m->w2 || !m->b2 || !m->w3 || !m->b3) return DVGO_ERR_INVALID_ARG;
    if (pd->n_bins != NB || pd->n_freq != NFQ || pd->width != PW) return DVGO_ERR_UNSUPPORTED;
    if (pd->precision != DVGO_MLP_FP32 && pd->precision != DVGO_MLP_BF16) return DVGO_ERR_INVALID_ARG;
    if (n_rays > 0 && (!rays_o || !rays_d)) return DVGO_ERR_INVALID_ARG;
    if (bwd && (!labels || !grad)) return DVGO_ERR_INVALID_ARG;
    if (!bwd && n_rays > 0 && !probs_out) return DVGO_ERR_INVALID_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (loss_out && !bwd) cudaMemsetAsync(loss_out, 0, sizeof(float), s);
    if (n_rays == 0) return cudaGetLastError() == cudaSuccess ? DVGO_OK : DVGO_ERR_CUDA;
    if (!bwd && pd->precision == DVGO_MLP_BF16)
        return launch_proposal_fwd_tc(*p, *dd, *m, n_rays, rays_o, rays_d, labels, probs_out,
                                      labels ? loss_out : nullptr, s);
    if (bwd && pd->precision == DVGO_MLP_BF16)
        return launch_proposal_bwd_tc(*p, *dd, *m, n_rays, rays_o, rays_d, labels, grad, s);
    PropArgs P;
    P.R = n_rays;
    P.box = make_box(*p, *dd);
    P.ro = rays_o;
    P.rd = rays_d;
    P.labels = labels;
    P.w0 = m->w0; P.b0 = m->b0; P.w1 = m->w1; P.b1 = m->b1; P.w2 = m->w2; P.b2 = m->b2; P.w3 = m->w3; P.b3 = m->b3;
    P.probs = probs_out;
    P.loss = bwd ? nullptr : (labels ? loss_out : nullptr);
    P.grad = grad;
    void (*kern)(PropArgs) = bwd ? proposal_kernel<true> : proposal_kernel<false>;
    ensure_smem(reinterpret_cast<const void *>(kern), (int)sizeof(PropSmem));
    int ntiles = (n_rays + 1) / 2;
    int blocks = ntiles < num_sms() ? ntiles : num_sms();
    {
        ProfScope ps_(bwd ? DVGO_K_PROPOSAL_BWD : DVGO_K_PROPOSAL_FWD, s);
        kern<<<blocks, PNT, sizeof(PropSmem), s>>>(P);
    }
    return cudaGetLastError() == cudaSuccess ? DVGO_OK : DVGO_ERR_CUDA;
}

int dvgo_proposal_fwd(const dvgo_params *p, const dvgo_grid_desc *dd, const dvgo_proposal_desc *pd,
                      const dvgo_proposal_mlp *m, int n_rays, const float *rays_o, const float *rays_d,
                      const float *labels, float *probs_out, float *loss_out, void *stream) {
    return proposal_launch(false, p, dd, pd, m, n_rays, rays_o, rays_d, labels, probs_out, loss_out, nullptr, stream);
}

int dvgo_proposal_bwd(const dvgo_params *p, const dvgo_grid_desc *dd, const dvgo_proposal_desc *pd,
                      const dvgo_proposal_mlp *m, int n_rays, const float *rays_o, const float *rays_d,
                      const float *labels, float *grad_mlp, void *stream) {
    return proposal_launch(true, p, dd, pd, m, n_rays, rays_o, rays_d, labels, nullptr, nullptr, grad_mlp, stream);
}

int dvgo_sample_pdf(const dvgo_params *p, const dvgo_grid_desc *dd, int n_rays, const float *rays_o,
                    const float *rays_d, const float *probs, int n_bins, int n_samples, const float *jitter,
                    float eta, float *t_out, float *dt_out, void *stream) {
    if (!p || !dd || n_rays < 0 || n_bins < 1 || n_bins > kPdfMaxBins || n_samples < 1 ||
        n_samples > (1 << 24) || !(eta >= 0.0f && eta <= 1.0f))
        return DVGO_ERR_INVALID_ARG;
    if (n_rays > 0 && (!rays_o || !rays_d || !probs || !t_out || !dt_out)) return DVGO_ERR_INVALID_ARG;
    if (n_rays == 0) return DVGO_OK;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    {
        ProfScope ps_(DVGO_K_SAMPLE_PDF, s);
        // rays per warp: about eight warps per SM, so that the FP64 clips are shared by many rays and the
        // serial part stays short (8,192 rays: seven)
        int group = (n_rays + num_sms() * 8 - 1) / (num_sms() * 8);
        group = group < 1 ? 1 : (group > 32 ? 32 : group);
        const int warps = (n_rays + group - 1) / group, blocks = (warps + kPdfThreads / 32 - 1) / (kPdfThreads / 32);
        const BoxD box = make_box(*p, *dd);
        auto kern = n_bins <= 32 ? sample_pdf_kernel<1> : (n_bins <= 64 ? sample_pdf_kernel<2> : sample_pdf_kernel<4>);
        kern<<<blocks, kPdfThreads, 0, s>>>(n_rays, box, rays_o, rays_d, probs, n_bins, n_samples, jitter, eta, t_out,
                                            dt_out, group);
    }
    return cudaGetLastError() == cudaSuccess ? DVGO_OK : DVGO_ERR_CUDA;
}

}  // extern "C"
