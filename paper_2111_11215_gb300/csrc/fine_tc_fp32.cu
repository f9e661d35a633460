// fine_tc_fp32.cu -- forward colour queries of the fine stage with the FP32 MLP, on the tensor cores.
//
// Same function as the FP32 contract asks (Sec. 4.2 Eq. fine_queries_rgb, Supp. A: 39 inputs, or 72 with
// PE(x, 5); two hidden layers of 128 with ReLU, sigmoid output).  Every FP32 operand x is written as
// three BF16 numbers x = hi + mid + lo, each the rounding to nearest of what the ones before leave (24
// significand bits in all, so the sum is x exactly unless lo falls below the smallest BF16), and a
// product of two operands as the six BF16 products hi hi, hi mid, mid hi, mid mid, hi lo, lo hi; the
// three left out are below 2^-25 of it.  tcgen05 MMAs accumulate in FP32, cutting what falls below the
// accumulator's last bit, so the small products go first, into an accumulator of their own size, and the
// 128-wide contraction keeps two accumulators (64 inputs each) that are added with rounding.  Colours
// and gradients are as close to FP64 as with the FP32 FMA chains (rgb 3.4e-8 relative either way).
//
// Bound: six MMAs for each FP32 one still leave the CUDA cores' FP32 rate (128 FMA a clock per SM, of
// which the SIMT kernel before reached 45 %) far behind.  1.38 M samples at 160^3: 1806 us there, 376 us here.
//
// Persistent CTAs of 384 threads walk tiles of M = 128 kept samples, thread r (mod 128) of a warpgroup
// owning row r (TMEM lane r).  Warps 8-11 gather the next tile's input rows and split them into shared
// memory; warps 0-7 (two per row, 64 columns each) issue the MMAs (thread 0) and run the epilogues:
//   Z1 = X W1 (bias in a constant-1 column) -> H1 = relu(Z1), split, to tensor memory (the next A operand)
//   -> Z2 = H1 W2 -> o = relu(Z2 + b2) W3 + b3 on the CUDA cores -> c = sigmoid(o).
// Layer 1 of the next tile runs while the last epilogue does.  Shared memory: W2 split 96 KB, W1 and X
// split 48 KB each (64 KB with PE(x)) as 16-column blocks in 128-byte-swizzled panels (tc_helpers.cuh).
// TMEM columns: Z1 [0, 128), then H1 hi / mid / lo [0, 192) over it; Z2 [192, 320) and [320, 448).
//
// An infinity has no such split (inf, then inf - inf), nor has a value that rounds to one in BF16.  A tile with an
// input, or a launch with weights, of a size from which the hidden layers could get there is evaluated in
// plain FP32 instead (rows_fp32, about the time of the CUDA-core kernel).

#include "dvgo_internal.cuh"
#include "fine_gather.cuh"
#include "tc_helpers.cuh"

namespace dvgo {

namespace {

using namespace tc;

constexpr int TM = 128, NC = 256, NP = 128;
constexpr int HID = 128, FEAT = 12, NFX = 5;
constexpr int PX = FEAT + 3 + 6 * 4;   // 39: first input of the PE(x) block
constexpr uint32_t COL_Z1 = 0, COL_H1 = 0, COL_Z2 = 192, NCOLS = 512;

template <bool PEX>
struct SplitDims {
    static constexpr int IN = PX + (PEX ? 3 + 6 * NFX : 0);   // inputs; column IN is the constant 1 (bias)
    static constexpr int KB = (IN + 1 + 15) / 16;             // 16-column blocks of a split: 3 or 5
    static constexpr int PANELS = (3 * KB + 3) / 4;           // of the three splits, block s KB + kb in order
    static constexpr int AUX = 3 * KB;                        // a block left over in the last panel: (W3, b2)
    static_assert(AUX < 4 * PANELS, "a free block for the output layer");
};

struct SplitSmall {
    float part[TM][3];   // the second half-row's share of the output layer
    float xmax[2][NP / 32];   // largest feature (and position) magnitude of a producer warp's rows, tile i in [i & 1]
    int wmax;                 // largest weight magnitude (float bits)
    uint64_t full, empty, mma, fin;
    uint32_t tmem_base;
    int abort;
    float b3[4];
};

template <bool PEX>
constexpr size_t split_smem() {
    return (size_t)(6 + 2 * SplitDims<PEX>::PANELS) * kPanelBytes + sizeof(SplitSmall) + 1023;
}
static_assert(split_smem<true>() <= 232448, "one CTA per SM (227 KB of shared memory)");

// Barrier among the 256 consumer threads.
__device__ __forceinline__ void consumer_sync() {
    fence_before();
    asm volatile("bar.sync 1, 256;" ::: "memory");
    fence_after();
}

// The input row of a kept sample (its cell and ray), the constant 1 last.
template <typename FeatT, bool PEX, bool PK>
__device__ __forceinline__ void input_row(const RenderArgs &A, const Cell &c, int ray, float *v) {
    gather_features<FeatT, PK>(A, c, v);
    const float4 *pe = reinterpret_cast<const float4 *>(A.pe + (size_t)ray * kPeStride);
#pragma unroll
    for (int k = 0; k < 7; ++k) {
        const float4 q4 = __ldg(pe + k);
        const float q[4] = {q4.x, q4.y, q4.z, q4.w};
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (4 * k + j < 27) v[FEAT + 4 * k + j] = q[j];
    }
    if constexpr (PEX) {
        // PE(x) of the world-space sample position: [x (3), sin(2^k x_c) (15), cos(2^k x_c) (15)]
        float xv[3];
        cell_world(A, c, xv);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            v[PX + a] = xv[a];
            pe_axis<NFX>(xv[a], v + PX + 3 + a * NFX, v + PX + 3 + 3 * NFX + a * NFX);
        }
    }
    v[SplitDims<PEX>::IN] = 1.0f;
}

// The MLP of a tile's rows in plain FP32, for inputs or weights whose split would leave the finite range: thread
// (row, half) takes kept sample e (-1: none) and 64 units of each layer, the hidden layer between them passes
// through the row's first 128 TMEM columns (ta), the share of the output layer is added to o.  All consumers call.
template <typename FeatT, bool PEX, bool PK>
__device__ __noinline__ void rows_fp32(const RenderArgs &A, int e, uint32_t ta, int hc, float (&o)[3]) {
    constexpr int NI = SplitDims<PEX>::IN + 1;
    float x[NI];
#pragma unroll
    for (int k = 0; k < NI; ++k) x[k] = 0.0f;
    if (e >= 0) {
        const int2 kv = A.kept[e];
        float dt;
        const Cell c = sample_cell(A, A.rays[kv.y], kv.y, kv.x >> 16, dt);
        input_row<FeatT, PEX, PK>(A, c, kv.y, x);
    }
#pragma unroll 1
    for (int u = 64 * hc; u < 64 * hc + 64; u += 8) {
        float z[8] = {};
        uint32_t h[8];
#pragma unroll
        for (int k = 0; k < NI; ++k)
#pragma unroll
            for (int j = 0; j < 8; ++j) z[j] = fmaf(x[k], __ldg((k < NI - 1 ? A.w1 + k * HID : A.b1) + u + j), z[j]);
#pragma unroll
        for (int j = 0; j < 8; ++j) h[j] = __float_as_uint(fmaxf(z[j], 0.0f));
        tmem_st8(ta + u, h);
    }
    tmem_wait_st();
    consumer_sync();
#pragma unroll 1
    for (int u = 64 * hc; u < 64 * hc + 64; u += 8) {
        float z[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) z[j] = __ldg(A.b2 + u + j);
#pragma unroll 1
        for (int k = 0; k < HID; k += 16) {
            float h[16];
            tmem_ld16(ta + k, h);
#pragma unroll
            for (int q = 0; q < 16; ++q)
#pragma unroll
                for (int j = 0; j < 8; ++j) z[j] = fmaf(h[q], __ldg(A.w2 + (k + q) * HID + u + j), z[j]);
        }
#pragma unroll
        for (int j = 0; j < 8; ++j)
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) o[ch] = fmaf(fmaxf(z[j], 0.0f), __ldg(A.w3 + 3 * (u + j) + ch), o[ch]);
    }
    consumer_sync();   // the columns are read: the next tile's first layer may take them
}

template <typename FeatT, bool PEX, bool PK>
__global__ void __launch_bounds__(NC + NP, 1) fine_colour_fwd_split_kernel(RenderArgs A) {
    using D = SplitDims<PEX>;
    constexpr int KB = D::KB;
    const int n_kept = A.hdr->n_kept;
    const int ntiles = (n_kept + TM - 1) / TM;
    if ((int)blockIdx.x >= ntiles) return;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *w2t = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    unsigned char *w1t = w2t + 6 * kPanelBytes, *xs = w1t + D::PANELS * kPanelBytes;
    SplitSmall &S = *reinterpret_cast<SplitSmall *>(xs + D::PANELS * kPanelBytes);
    const int tid = threadIdx.x, warp = tid >> 5;
    if (tid == 0) {
        mbar_init(&S.full, NP);
        mbar_init(&S.empty, 1);
        mbar_init(&S.mma, 1);
        mbar_init(&S.fin, 1);
        S.abort = 0;
        S.wmax = 0;
    }
    if (warp == 0) tmem_alloc(&S.tmem_base, NCOLS);
    // barriers initialised: the producers gather the first tile while the consumers stage the weights
    fence_before();
    __syncthreads();
    fence_after();
    bool ok = true;
    uint32_t mphase = 0;

    if (tid >= NC) {
        // ------------------------------- producers -------------------------------
        const int row = tid - NC;
        auto kept_at = [&](int t) -> int2 {
            const int e = t * TM + row;
            return (t < ntiles && e < n_kept) ? A.kept[e] : make_int2(-1, -1);
        };
        int2 kv = kept_at(blockIdx.x);
        RayPre rp = kv.y >= 0 ? ray_pre(A, kv.y) : RayPre{};
        int i = 0;
        for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++i) {
            const int2 kv_next = kept_at(tile + gridDim.x);
            float v[16 * KB], xmax = 0.0f;
#pragma unroll
            for (int k = 0; k < 16 * KB; ++k) v[k] = 0.0f;
            if (kv.y >= 0) {
                float dt;
                const Cell c = cell_pre(A, rp, kv.y, kv.x >> 16, dt);
                input_row<FeatT, PEX, PK>(A, c, kv.y, v);
#pragma unroll
                for (int k = 0; k < FEAT; ++k) xmax = fmaxf(xmax, fabsf(v[k]));
                if constexpr (PEX)
#pragma unroll
                    for (int a = 0; a < 3; ++a) xmax = fmaxf(xmax, fabsf(v[PX + a]));
            }
            rp = kv_next.y >= 0 ? ray_pre(A, kv_next.y) : RayPre{};
            kv = kv_next;
            if (i >= 1) ok = __all_sync(0xffffffffu, mbar_wait(&S.empty, (i - 1) & 1, A.wait_ns));
            if (!ok) break;
#pragma unroll
            for (int c = 0; c < 2 * KB; ++c) {
                uint4 q[3];
                split8(v + 8 * c, q);
#pragma unroll
                for (int s = 0; s < 3; ++s) *split_chunk<KB>(xs, s, row, c) = q[s];
            }
            xmax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(xmax)));
            if ((row & 31) == 0) S.xmax[i & 1][row >> 5] = xmax;
            fence_async_smem();
            // (testing aid: one arrival withheld on a chosen tile makes the consumers' wait run out)
            if (!(row == 0 && tile + 1 == A.withhold_tile)) mbar_arrive(&S.full);
        }
        if (!ok) atomicExch(&S.abort, 1);
    } else {
        // ------------------------------- consumers -------------------------------
        // W1^T | b1 and W2^T split: (unit n, 8 input columns) per thread and turn
        float wmax = 0.0f;
        for (int t = tid; t < HID * (2 * KB + 16); t += NC) {
            const int n = t & (HID - 1), c = t >> 7;
            float v[8];
            uint4 q[3];
            if (c < 2 * KB) {
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int k = 8 * c + j;
                    v[j] = k < D::IN ? A.w1[k * HID + n] : (k == D::IN ? A.b1[n] : 0.0f);
                    wmax = fmaxf(wmax, fabsf(v[j]));
                }
                split8(v, q);
#pragma unroll
                for (int s = 0; s < 3; ++s) *split_chunk<KB>(w1t, s, n, c) = q[s];
            } else {
                const int c2 = c - 2 * KB;   // 0-15
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    v[j] = A.w2[(8 * c2 + j) * HID + n];
                    wmax = fmaxf(wmax, fabsf(v[j]));
                }
                split8(v, q);
#pragma unroll
                for (int s = 0; s < 3; ++s)
                    *reinterpret_cast<uint4 *>(w2t + (2 * s + (c2 >> 3)) * kPanelBytes + panel_offset(n, (c2 & 7) * 8)) = q[s];
            }
        }
        unsigned char *aux = w1t + (D::AUX >> 2) * kPanelBytes;   // per unit (W3 row, b2), 16 bytes in the free block
        constexpr int aux_col = (D::AUX & 3) * 16;
        if (tid < HID)
            *reinterpret_cast<float4 *>(aux + panel_offset(tid, aux_col)) =
                make_float4(A.w3[3 * tid], A.w3[3 * tid + 1], A.w3[3 * tid + 2], A.b2[tid]);
        if (tid < 3) S.b3[tid] = A.b3[tid];
        if (tid < HID) wmax = fmaxf(wmax, fabsf(A.b2[tid]));
        wmax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(wmax)));
        if ((tid & 31) == 0) atomicMax(&S.wmax, __float_as_int(wmax));
        fence_async_smem();
        consumer_sync();
        // Inputs up to which no operand leaves the finite BF16 range: the hidden layers are at most 128 M (73 M X + 1) <
        // 1e4 M^2 X for weights up to M and inputs up to X (both taken as 1 at least).  Above, or with an infinity among
        // them, the split would make NaN of what FP32 arithmetic can turn into a number: rows_fp32.
        const float wm = fmaxf(__int_as_float(S.wmax), 1.0f), xlimit = wm <= 1e17f ? 1e34f / (wm * wm) : -1.0f;

        const int r = tid & (TM - 1), hc = tid >> 7;
        const uint32_t tb = S.tmem_base;
        const uint32_t idesc = idesc_bf16(128, 128, 0, 0);
        // the six products, smallest first: split of A, split of B
        constexpr int PA[6] = {0, 2, 1, 0, 1, 0}, PB[6] = {2, 0, 1, 1, 0, 0};
        // waits of a warp as one; the verdicts of the warps meet at the last barrier of a tile (barrier_all)
        auto wait = [&](uint64_t *bar, uint32_t par) {
            if (ok) ok = __all_sync(0xffffffffu, mbar_wait(bar, par, A.wait_ns));
            fence_after();
        };
        auto wait_mma = [&]() {
            wait(&S.mma, mphase);
            mphase ^= 1;
        };
        auto issue_layer1 = [&]() {
            const uint64_t x = desc_kmajor(smem_u32(xs), 0), w = desc_kmajor(smem_u32(w1t), 0);
#pragma unroll
            for (int p = 0; p < 6; ++p)
#pragma unroll
                for (int kk = 0; kk < KB; ++kk)
                    mma(tb + COL_Z1, x + kstep(PA[p] * KB + kk), w + kstep(PB[p] * KB + kk), idesc, (p | kk) != 0);
            commit(&S.mma);
        };
        int i = 0;
        wait(&S.full, 0);
        if (ok && tid == 0) issue_layer1();
        for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++i) {
            // this row's sample slot and optical depth, needed at the end
            const int e = tile * TM + r;
            int slot = -1;
            float tau = 0.0f;
            if (hc == 0 && e < n_kept) {
                const int2 kv = A.kept[e];
                slot = kv.y * A.cap + (kv.x & 0xffff);
                tau = __ldg(A.stau + slot);
            }
            wait_mma();
            if (ok && tid == 0) mbar_arrive(&S.empty);   // X is free
            const float *xm = S.xmax[i & 1];
            const bool split = fmaxf(fmaxf(xm[0], xm[1]), fmaxf(xm[2], xm[3])) <= xlimit;   // (the same for all)
            float o[3] = {0.0f, 0.0f, 0.0f};
            if (hc == 0) {
                o[0] = S.b3[0];
                o[1] = S.b3[1];
                o[2] = S.b3[2];
            }
            if (split) {
                // ---- epilogue 1: H1 = relu(Z1), split, over Z1 (read whole before any is overwritten) ----
                {
                    float z[2][32];
                    tmem_ld32(taddr(tb, warp, COL_Z1 + 64 * hc), z[0]);
                    tmem_ld32(taddr(tb, warp, COL_Z1 + 64 * hc + 32), z[1]);
                    consumer_sync();
#pragma unroll
                    for (int g = 0; g < 2; ++g) {
                        uint32_t w[3][16];
#pragma unroll
                        for (int k = 0; k < 32; k += 8) {
                            float v[8];
                            uint4 q[3];
#pragma unroll
                            for (int j = 0; j < 8; ++j) v[j] = fmaxf(z[g][k + j], 0.0f);
                            split8(v, q);
#pragma unroll
                            for (int s = 0; s < 3; ++s) {
                                w[s][k / 2] = q[s].x;
                                w[s][k / 2 + 1] = q[s].y;
                                w[s][k / 2 + 2] = q[s].z;
                                w[s][k / 2 + 3] = q[s].w;
                            }
                        }
#pragma unroll
                        for (int s = 0; s < 3; ++s) tmem_st16(taddr(tb, warp, COL_H1 + 64 * s + 32 * hc + 16 * g), w[s]);
                    }
                    tmem_wait_st();
                    consumer_sync();
                }
                // ---- layer 2: Z2 = H1 W2, A = H1 from TMEM; inputs 0-63 and 64-127 in accumulators of their own ----
                if (ok && tid == 0) {
                    const uint64_t w = desc_kmajor(smem_u32(w2t), 0);
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int p = 0; p < 6; ++p)
#pragma unroll
                            for (int kk = 4 * h; kk < 4 * h + 4; ++kk)
                                mma_ts(tb + COL_Z2 + 128u * h, tb + COL_H1 + 64u * PA[p] + 8u * kk,
                                       w + 2 * PB[p] * kPanelStep + kstep(kk), idesc, p > 0 || kk > 4 * h);
                    commit(&S.mma);
                }
                wait_mma();
            } else {
                rows_fp32<FeatT, PEX, PK>(A, ok && e < n_kept ? e : -1, taddr(tb, warp, 0), hc, o);
            }
            // ---- layer 1 of the next tile, beside the last epilogue ----
            if (tile + (int)gridDim.x < ntiles) {
                wait(&S.full, (i + 1) & 1);
                if (ok && tid == 0) issue_layer1();
            }
            if (split) {
                // ---- epilogue 2: relu(Z2 + b2) W3, my 64 columns; the two halves of a row join ----
#pragma unroll 1
                for (int g = 0; g < 2; ++g) {
                    const int col = 64 * hc + 32 * g;
                    float za[32], zb[32];
                    tmem_ld32(taddr(tb, warp, COL_Z2 + col), za);
                    tmem_ld32(taddr(tb, warp, COL_Z2 + 128 + col), zb);
#pragma unroll
                    for (int k = 0; k < 32; ++k) {
                        const float4 w = *reinterpret_cast<const float4 *>(aux + panel_offset(col + k, aux_col));
                        const float h = fmaxf(za[k] + zb[k] + w.w, 0.0f);
                        o[0] = fmaf(h, w.x, o[0]);
                        o[1] = fmaf(h, w.y, o[1]);
                        o[2] = fmaf(h, w.z, o[2]);
                    }
                }
            }
            if (hc == 1) {
                S.part[r][0] = o[0];
                S.part[r][1] = o[1];
                S.part[r][2] = o[2];
            }
            fence_before();
            ok = barrier_all(1, NC, ok);
            fence_after();
            if (!ok) break;
            if (slot >= 0)
                A.scol[slot] = make_float4(sigmoidf_(o[0] + S.part[r][0]), sigmoidf_(o[1] + S.part[r][1]),
                                           sigmoidf_(o[2] + S.part[r][2]), tau);
        }
        if (!ok) atomicExch(&S.abort, 1);
    }

    fence_before();
    __syncthreads();
    fence_after();
    if (S.abort != 0) {
        if (tid == 0) {
            atomicOr(&A.hdr->flags, 2);
            commit(&S.fin);   // MMAs may still be running: all that were issued are complete before TMEM is freed (bounded)
            mbar_wait(&S.fin, 0, A.wait_ns);
        }
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 0) tmem_dealloc(S.tmem_base, NCOLS);
}

template <typename FeatT, bool PEX, bool PK>
void launch_split(const RenderArgs &A, cudaStream_t s) {
    auto kern = fine_colour_fwd_split_kernel<FeatT, PEX, PK>;
    constexpr int bytes = (int)split_smem<PEX>();
    ensure_smem(reinterpret_cast<const void *>(kern), bytes);
    ProfScope ps_(DVGO_K_FINE_COLOUR_FWD, s);
    kern<<<num_sms(), NC + NP, bytes, s>>>(A);
}

}  // namespace

void launch_fine_colour_fwd_fp32(const RenderArgs &A, cudaStream_t s) {
    const bool bf = A.cdtype == DVGO_DTYPE_BF16, pex = A.nfreq_pos > 0;
    if (A.packed) {
        if (bf && pex) launch_split<__nv_bfloat16, true, true>(A, s);
        else if (bf) launch_split<__nv_bfloat16, false, true>(A, s);
        else if (pex) launch_split<float, true, true>(A, s);
        else launch_split<float, false, true>(A, s);
    } else {
        if (bf && pex) launch_split<__nv_bfloat16, true, false>(A, s);
        else if (bf) launch_split<__nv_bfloat16, false, false>(A, s);
        else if (pex) launch_split<float, true, false>(A, s);
        else launch_split<float, false, false>(A, s);
    }
}

}  // namespace dvgo
