// fine_tc_fp32_bwd.cu -- backward of the fine stage's colour queries with the FP32 MLP of 39 inputs, on the
// tensor cores (the 72-input form is fine_simt.cu: its operands do not fit beside the weights).
//
// Arithmetic as in fine_tc_fp32.cu: every FP32 operand is the exact sum of three BF16 numbers, every
// contraction the six products that matter with FP32 accumulation, the smallest first.  Weight
// gradients leave their TMEM accumulator after every tile and are summed over the tiles in registers, with
// rounding (an accumulator that lived through all tiles would lose a part in 10^4 to the tensor core's
// truncation).  Within a tile the same truncation cuts every product off at the last bit of the running sum,
// always towards 0: with one accumulator of 128 samples for hi x hi, dW1 and dW2 were 2e-6 off where an FP32
// chain is 4e-7 off (samples of a proposal, weights over many orders of magnitude).  So hi x hi of dW1 and
// dW2 goes to four accumulators of 32 samples, that of dH1 and de to two of 64 units; they join with rounding.
// Errors against FP64 over 40 drawn steps, relative to the CUDA-core kernel's: MLP gradients 0.70, feature
// gradients 0.87 (geometric means).  A ReLU unit within rounding of zero is decided by the plain FP32 FMA
// chain over its inputs (exact_z1 / exact_z2, the order of the SIMT kernel), so the gradients do not hang
// on which arithmetic recomputed the hidden layers.
//
// Bound: the serial chain of a tile -- nine MMA batches and, between them, three epilogues that split 16 k values
// each on two warps per scheduler; shared memory (weights and 64 KB of activations) leaves no room for a
// second tile beside it.  160^3, 8,192 rays, 1.38 M samples: 4610 us on the CUDA cores (45 % of their FP32
// rate), 1320 us here, 18.6 us a tile, the tensor pipe active for 35 % of it (1240 us and 38 % with one
// accumulator for hi x hi of each weight gradient).
//
// Per tile of M = 128 kept samples, with dout = dL/do from the compositing backward; activations are kept
// transposed (TMEM lane = hidden unit, column = sample), so that a thread owns a unit: the sums over the
// samples of db2 and dW3 stay in its registers, and the activations are directly the A operand, from
// tensor memory, of the weight gradients:
//   Z1^T = W1^T X^T                 A = W1 (shared), B = X (shared)
//   Z2^T = W2^T H1^T                A = W2 (shared), B = H1^T (shared, a third at a time)
//   dZ2 = (dout W3^T) [Z2 > 0], dW3 += H2^T dout, db2 += sum dZ2      (CUDA cores)
//   dW2 += H1^T dZ2                 A = H1^T (TMEM), B = dZ2^T (shared, a third at a time)
//   dH1^T = W2 dZ2^T                A = W2 (shared, read MN-major), B = dZ2^T
//   dZ1 = dH1 [Z1 > 0]
//   de = dZ1 W1[0:12]^T             A = dZ1^T (shared, read MN-major), B = W1 (read MN-major)
//   [dW1 | db1]^T += dZ1^T X        A = dZ1^T (TMEM), B = X (staged again; mid | lo and hi | mid side by side)
// Shared memory: W2 split 96 KB, W1 split 48 KB, and a pool of 64 KB that holds X, then pairs of
// 32 KB thirds of the activations, then X again.  Warps 0-7 consume (thread (n, half): unit n = t mod 128,
// samples 64 half .. +63), warps 8-11 gather X, stage it twice and scatter the feature gradients of the
// tile before.  TMEM columns: activations' split [0, 192); layer accumulator [192, 320); dW2 [320, 448) and, over
// H1's mid and lo thirds, [64, 192), then the second half of dH1 [320, 448); dZ2's hi third, then de [448, 512) and
// [400, 448); dW1's six accumulators [192, 480) over them.

#include "dvgo_internal.cuh"
#include "fine_gather.cuh"
#include "tc_helpers.cuh"

namespace dvgo {

namespace {

using namespace tc;

constexpr unsigned FULL = 0xffffffffu;
constexpr int TM = 128, NC = 256, NP = 128;
constexpr int HID = 128, FEAT = 12, IN = 39, XK = 40;   // column IN of X is the constant 1 (bias)
constexpr int KB = 3;                                   // 16-column blocks of X and W1 per split
constexpr uint32_t T_ACT = 0, T_DW2B = 64, T_Z = 192, T_DW2 = 320, T_DW1 = 192, T_DE = 448, T_DE2 = 400, T_HI = 448, NCOLS = 512;
constexpr int DW1 = 16 * KB;                            // columns of a dW1 accumulator

struct BwdSmall {
    alignas(16) float dout[3][TM];   // dL/do
    alignas(16) float xmax[TM];      // largest input magnitude of the row (0: padding row)
    float gmax[TM / 16];             // the same of 16 rows
    float4 de[TM][3];      // feature gradients of a tile
    float4 place[2][TM];
    ScatterTab tab[NP / 32];
    uint64_t full, empty, mma_a, mma_b, fin;
    uint32_t tmem_base;
    int abort;
    int s1max;             // largest absolute row sum of W1^T | b1 (float bits)
};

constexpr int kPoolPanels = 4;
constexpr size_t kBwdSmem = (size_t)(6 + 3 + kPoolPanels) * kPanelBytes + sizeof(BwdSmall) + 1023;
static_assert(kBwdSmem <= 232448, "one CTA per SM (227 KB of shared memory)");

__device__ __forceinline__ void consumer_sync() {
    fence_before();
    asm volatile("bar.sync 1, 256;" ::: "memory");
    fence_after();
}
// Operands written by the consumers become visible to the tensor core, then the consumers sync.
__device__ __forceinline__ void publish() {
    fence_async_smem();
    consumer_sync();
}

// The input row of kept sample e, bit for bit as the SIMT kernel forms it: lane l holds inputs l and 32 + l
// (input 39: the constant 1).  All lanes of the warp take part.
template <typename FeatT, bool PK>
__device__ __noinline__ float2 exact_inputs(const RenderArgs &A, int e) {
    const int lane = threadIdx.x & 31, q = lane & 3;
    const int2 kv = A.kept[e];
    float dt;
    const Cell c = sample_cell(A, A.rays[kv.y], kv.y, kv.x >> 16, dt);
    const FeatT *g0 = static_cast<const FeatT *>(A.cgrid) + corner_index(c, 2 * q, A.ny, A.nz, PK) * FEAT;
    const FeatT *g1 = static_cast<const FeatT *>(A.cgrid) + corner_index(c, 2 * q + 1, A.ny, A.nz, PK) * FEAT;
    const float w0 = corner_weight(c, 2 * q), w1 = corner_weight(c, 2 * q + 1);
    float x0 = 0.0f;
#pragma unroll
    for (int ch = 0; ch < FEAT; ++ch) {
        float f = fmaf(w0, (float)g0[ch], w1 * (float)g1[ch]);
        f += __shfl_xor_sync(FULL, f, 1);
        f += __shfl_xor_sync(FULL, f, 2);
        if (lane == ch) x0 = f;
    }
    const float *pe = A.pe + (size_t)kv.y * kPeStride;
    if (lane >= FEAT) x0 = pe[lane - FEAT];
    return make_float2(x0, lane < 7 ? pe[20 + lane] : (lane == 7 ? 1.0f : 0.0f));
}

// z of a unit of layer 1 / layer 2 at kept sample e: FMA chains in input order (the bias last / first).
template <typename FeatT, bool PK>
__device__ __noinline__ float exact_z1(const RenderArgs &A, int e, int unit) {
    const int lane = threadIdx.x & 31;
    const float2 x = exact_inputs<FeatT, PK>(A, e);
    const float w0 = A.w1[lane * HID + unit],
                w1 = lane < 7 ? A.w1[(32 + lane) * HID + unit] : (lane == 7 ? A.b1[unit] : 0.0f);
    float z = 0.0f;
#pragma unroll 8
    for (int k = 0; k < 32; ++k) z = fmaf(__shfl_sync(FULL, x.x, k), __shfl_sync(FULL, w0, k), z);
#pragma unroll
    for (int k = 0; k < 8; ++k) z = fmaf(__shfl_sync(FULL, x.y, k), __shfl_sync(FULL, w1, k), z);
    return z;
}

template <typename FeatT, bool PK>
__device__ __noinline__ float exact_z2(const RenderArgs &A, int e, int unit) {
    const int lane = threadIdx.x & 31;
    const float2 x = exact_inputs<FeatT, PK>(A, e);
    float h[4] = {0.0f, 0.0f, 0.0f, 0.0f}, w[4];
    for (int k0 = 0; k0 < XK; k0 += 8) {   // eight inputs' weights in flight
        float r[8][4];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float *row = k0 + j < IN ? A.w1 + (k0 + j) * HID : A.b1;
#pragma unroll
            for (int i = 0; i < 4; ++i) r[j][i] = row[lane + 32 * i];
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float xk = k0 < 32 ? __shfl_sync(FULL, x.x, k0 + j) : __shfl_sync(FULL, x.y, j);
#pragma unroll
            for (int i = 0; i < 4; ++i) h[i] = fmaf(xk, r[j][i], h[i]);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        h[i] = fmaxf(h[i], 0.0f);
        w[i] = A.w2[(lane + 32 * i) * HID + unit];
    }
    float z = A.b2[unit];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll 8
        for (int l = 0; l < 32; ++l) z = fmaf(__shfl_sync(FULL, h[i], l), __shfl_sync(FULL, w[i], l), z);
    return z;
}

// The signs of the units within rounding of zero, decided by the FMA chains: amb marks this lane's among
// samples e0 .. e0 + 15 (bit k), on holds the bits z > 0 (sample k in bit 15 - k) and is returned corrected.  All
// lanes of the warp take part.
template <typename FeatT, bool PK, int kLayer>
__device__ __noinline__ uint32_t resolve(const RenderArgs &A, int e0, int unit, uint32_t amb, uint32_t on) {
    const int lane = threadIdx.x & 31;
    for (unsigned any = __ballot_sync(FULL, amb != 0u); any; any = __ballot_sync(FULL, amb != 0u)) {
        const int src = __ffs(any) - 1, k = __ffs(__shfl_sync(FULL, amb, src)) - 1, u = __shfl_sync(FULL, unit, src);
        const float z = kLayer == 1 ? exact_z1<FeatT, PK>(A, e0 + k, u) : exact_z2<FeatT, PK>(A, e0 + k, u);
        if (lane == src) {
            amb &= amb - 1u;
            const uint32_t bit = 0x8000u >> k;
            on = z > 0.0f ? on | bit : on & ~bit;
        }
    }
    return on;
}
__device__ __forceinline__ bool off(uint32_t on, int k) { return !((on >> (15 - k)) & 1u); }

// Splits 16 consecutive samples of this thread's unit (row n, samples 64 hc + 16 g ..): the three terms as
// packed pairs (for TMEM) in w, and the chosen ones into the half panels lo / mid (row = unit).
__device__ __forceinline__ void split16(const float *v, uint32_t (&w)[3][8]) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        uint4 q[3];
        split8(v + 8 * c, q);
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            w[s][4 * c] = q[s].x;
            w[s][4 * c + 1] = q[s].y;
            w[s][4 * c + 2] = q[s].z;
            w[s][4 * c + 3] = q[s].w;
        }
    }
}
__device__ __forceinline__ void store16(unsigned char *half_panel, int n, int g, const uint32_t (&w)[8]) {
#pragma unroll
    for (int c = 0; c < 2; ++c)
        *reinterpret_cast<uint4 *>(half_panel + panel_offset(n, 16 * g + 8 * c)) =
            make_uint4(w[4 * c], w[4 * c + 1], w[4 * c + 2], w[4 * c + 3]);
}

// dL/do of four consecutive samples.
__device__ __forceinline__ void load_dout(const BwdSmall &S, int s, float (&d)[3][4]) {
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) *reinterpret_cast<float4 *>(d[ch]) = *reinterpret_cast<const float4 *>(&S.dout[ch][s]);
}

template <typename FeatT, bool PK>
__global__ void __launch_bounds__(NC + NP, 1) fine_colour_bwd_split_kernel(RenderArgs A) {
    const int n_kept = A.hdr->n_kept;
    const int ntiles = (n_kept + TM - 1) / TM;
    if ((int)blockIdx.x >= ntiles) return;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *w2t = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    unsigned char *w1t = w2t + 6 * kPanelBytes, *pool = w1t + 3 * kPanelBytes;
    BwdSmall &S = *reinterpret_cast<BwdSmall *>(pool + kPoolPanels * kPanelBytes);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        mbar_init(&S.full, NP);
        mbar_init(&S.empty, 1);
        mbar_init(&S.mma_a, 1);
        mbar_init(&S.mma_b, 1);
        mbar_init(&S.fin, 1);
        S.abort = 0;
        S.s1max = 0;
    }
    if (warp == 0) tmem_alloc(&S.tmem_base, NCOLS);
    fence_before();
    __syncthreads();
    fence_after();
    bool ok = true;
    uint32_t pa = 0, pb = 0;   // phases of mma_a and mma_b

    if (tid >= NC) {
        // ------------------------------- producers -------------------------------
        // 384 x 168 registers at launch = 256 x 192 + 128 x 120
        asm volatile("setmaxnreg.dec.sync.aligned.u32 120;");
        const int row = tid - NC;
        struct Row {
            uint4 q[XK / 8][3];   // the input row's three terms, 8 columns a chunk
            float d[3], xmax;
            int slot, ray;        // slot < 0: padding row
            Cell c;
        };
        // Placing a sample takes two dependent loads (list, ray record); done while the consumers work on the
        // tile before, with the corners' lines fetched towards the SM, it leaves one short load for the gather.
        auto place = [&](int t, Row &w) {
            const int e = t * TM + row;
            w.slot = -1;
            w.ray = 0;
            w.c.i0 = w.c.j0 = w.c.k0 = 0;
            w.c.fx = w.c.fy = w.c.fz = 0.0f;
            if (t >= ntiles || e >= n_kept) return;
            const int2 kv = A.kept[e];
            const RayPre rp = ray_pre(A, kv.y);
            float dt;
            w.c = cell_pre(A, rp, kv.y, kv.x >> 16, dt);
            w.slot = rp.off + (kv.x & 0xffff);
            w.ray = kv.y;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const FeatT *g = static_cast<const FeatT *>(A.cgrid) + corner_index(w.c, 2 * q, A.ny, A.nz, PK) * FEAT;
                const FeatT *h = static_cast<const FeatT *>(A.cgrid) + corner_index(w.c, 2 * q + 1, A.ny, A.nz, PK) * FEAT;
                asm volatile("prefetch.global.L1 [%0];" ::"l"(g));
                asm volatile("prefetch.global.L1 [%0];" ::"l"(h + FEAT - 1));
            }
            asm volatile("prefetch.global.L1 [%0];" ::"l"(A.sgrad + w.slot));
            asm volatile("prefetch.global.L1 [%0];" ::"l"(A.pe + (size_t)kv.y * kPeStride));
        };
        auto gather = [&](Row &w) {
            float v[XK];
#pragma unroll
            for (int k = 0; k < XK; ++k) v[k] = 0.0f;
            w.d[0] = w.d[1] = w.d[2] = w.xmax = 0.0f;
            if (w.slot >= 0) {
                const float4 g = A.sgrad[w.slot];
                gather_features<FeatT, PK>(A, w.c, v);
                const float4 *pe = reinterpret_cast<const float4 *>(A.pe + (size_t)w.ray * kPeStride);
#pragma unroll
                for (int k = 0; k < 7; ++k) {
                    const float4 q4 = __ldg(pe + k);
                    const float q[4] = {q4.x, q4.y, q4.z, q4.w};
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (4 * k + j < 27) v[FEAT + 4 * k + j] = q[j];
                }
                v[IN] = 1.0f;
                w.xmax = 1.0f;
#pragma unroll
                for (int k = 0; k < FEAT; ++k) w.xmax = fmaxf(w.xmax, fabsf(v[k]));
                w.d[0] = g.y;
                w.d[1] = g.z;
                w.d[2] = g.w;
            }
#pragma unroll
            for (int c8 = 0; c8 < XK / 8; ++c8) split8(v + 8 * c8, w.q[c8]);
        };
        // the terms side by side, 48 columns each: mid, lo from the first panel's start, hi, mid from the third's
        auto stage = [&](const Row &w) {
#pragma unroll
            for (int c = 0; c < 2 * KB; ++c) {
                const uint4 z = make_uint4(0u, 0u, 0u, 0u);
                const uint4 hi = c < XK / 8 ? w.q[c][0] : z, mid = c < XK / 8 ? w.q[c][1] : z, lo = c < XK / 8 ? w.q[c][2] : z;
                *split_chunk<KB>(pool, 0, row, c) = mid;
                *split_chunk<KB>(pool, 1, row, c) = lo;
                *split_chunk<KB>(pool + 2 * kPanelBytes, 0, row, c) = hi;
                *split_chunk<KB>(pool + 2 * kPanelBytes, 1, row, c) = mid;
            }
        };
        auto scatter_tile = [&](int t) {
            scatter_rows<PK>(A, S.place[t], [&](int r, int k) { return &S.de[r][k]; }, S.tab[row >> 5], row);
        };
        Row cur;
        place(blockIdx.x, cur);
        gather(cur);
        int i = 0;
        for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++i) {
            // the pool is free once the tile before is done (second release of a tile)
            // (the warp leaves as one: the scatter is a warp's work)
            if (i > 0) ok = __all_sync(0xffffffffu, mbar_wait(&S.empty, 1, A.wait_ns));
            if (!ok) break;
            stage(cur);
            const int t = i & 1;
            S.place[t][row] = row_place(A, cur.c, cur.slot >= 0, PK);
            S.dout[0][row] = cur.d[0];
            S.dout[1][row] = cur.d[1];
            S.dout[2][row] = cur.d[2];
            S.xmax[row] = cur.xmax;
            float gm = cur.xmax;
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) gm = fmaxf(gm, __shfl_xor_sync(FULL, gm, o));
            if ((row & 15) == 0) S.gmax[row >> 4] = gm;
            fence_async_smem();
            // (testing aid: one arrival withheld on a chosen tile makes the consumers' wait run out)
            if (!(row == 0 && tile + 1 == A.withhold_tile)) mbar_arrive(&S.full);
            // de of the tile before is in place: written before the consumers' release that this thread
            // has just waited for
            if (i > 0) scatter_tile(t ^ 1);
            place(tile + gridDim.x, cur);
            ok = __all_sync(0xffffffffu, mbar_wait(&S.empty, 0, A.wait_ns));
            if (!ok) break;
            stage(cur);   // again, for dW1
            fence_async_smem();
            mbar_arrive(&S.full);
            gather(cur);
        }
        if (ok && i > 0) {
            ok = __all_sync(0xffffffffu, mbar_wait(&S.empty, 1, A.wait_ns));
            if (ok) scatter_tile((i - 1) & 1);
        }
        if (!ok) atomicExch(&S.abort, 1);
    } else {
        // ------------------------------- consumers -------------------------------
        asm volatile("setmaxnreg.inc.sync.aligned.u32 192;");
        const int n = tid & (HID - 1), hc = tid >> 7;
        // W1^T | b1 and W2^T split: (unit, 8 input columns) per thread and turn
        for (int t = tid; t < HID * (2 * KB + 16); t += NC) {
            const int u = t & (HID - 1), c = t >> 7;
            float v[8];
            uint4 q[3];
            if (c < 2 * KB) {
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int k = 8 * c + j;
                    v[j] = k < IN ? A.w1[k * HID + u] : (k == IN ? A.b1[u] : 0.0f);
                }
                split8(v, q);
#pragma unroll
                for (int s = 0; s < 3; ++s)
                    *split_chunk<KB>(w1t, s, u, c) = q[s];
                if (c < 2)   // the features' columns once more, their three terms side by side in the free blocks
#pragma unroll
                    for (int s = 0; s < 3; ++s)
                        *reinterpret_cast<uint4 *>(w1t + 2 * kPanelBytes + panel_offset(u, 16 * (1 + s) + 8 * c)) = q[s];
            } else {
                const int c2 = c - 2 * KB;   // 0-15
#pragma unroll
                for (int j = 0; j < 8; ++j) v[j] = A.w2[(8 * c2 + j) * HID + u];
                split8(v, q);
#pragma unroll
                for (int s = 0; s < 3; ++s)
                    *reinterpret_cast<uint4 *>(w2t + (2 * s + (c2 >> 3)) * kPanelBytes + panel_offset(u, (c2 & 7) * 8)) = q[s];
            }
        }
        const float w30 = A.w3[3 * n], w31 = A.w3[3 * n + 1], w32 = A.w3[3 * n + 2], b2 = A.b2[n];
        const float nb2 = __fsub_rn(0.0f, b2);   // (+0 for a bias of 0)
        // Where a unit's sign is looked at again: 2^-23 of a bound on the sum of magnitudes behind z (more than
        // ten times the usual difference of the two arithmetics), for inputs of magnitude 1.
        float s1 = fabsf(A.b1[n]), s2 = 0.0f;
        for (int k = 0; k < IN; ++k) s1 += fabsf(A.w1[k * HID + n]);
        for (int k = 0; k < HID; ++k) s2 += fabsf(A.w2[k * HID + n]);
        atomicMax(&S.s1max, __float_as_int(s1));
        publish();
        const float eps1 = 0x1p-23f * s1, eps2 = 0x1p-23f * (0.25f * __int_as_float(S.s1max) * s2 + fabsf(b2));

        const uint32_t tb = S.tmem_base;
        const uint32_t w1_ = smem_u32(w1t), w2_ = smem_u32(w2t), pool_ = smem_u32(pool);
        unsigned char *buf0 = pool + hc * kPanelBytes, *buf1 = pool + (2 + hc) * kPanelBytes;   // this thread's halves
        const uint32_t b0_ = pool_, b1_ = pool_ + 2 * kPanelBytes;
        const uint32_t id_z1 = idesc_bf16(128, 128, 0, 0), id_z2 = idesc_bf16(128, 128, 0, 1),
                       id_dh = idesc_bf16(128, 128, 1, 1);
        constexpr int PA[6] = {0, 2, 1, 0, 1, 0}, PB[6] = {2, 0, 1, 1, 0, 0};   // the six products, small first
        // Waits of a warp as one.  The verdicts of the warps meet at the last barrier of a tile (barrier_all): until
        // then a warp whose wait ran out keeps the others company at their barriers.
        auto wait = [&](uint64_t *bar, uint32_t par) {
            if (ok) ok = __all_sync(FULL, mbar_wait(bar, par, A.wait_ns));
            fence_after();
        };
        auto wait_a = [&]() {
            wait(&S.mma_a, pa);
            pa ^= 1;
        };
        auto wait_b = [&]() {
            wait(&S.mma_b, pb);
            pb ^= 1;
        };
        // MMA batches over a third of an activation held in the pool at b_ (thread 0).  Descriptors are a base
        // and steps of the address field (16-byte units), so that an MMA costs the issuing thread two adds.
        auto z2_batch = [&](uint32_t b_, int sa, bool first) {   // Z2^T (+)= W2[sa] H1^T
            const uint64_t a = desc_kmajor(w2_ + 2u * sa * kPanelBytes, 0), b = desc_mnmajor(b_, 0);
#pragma unroll
            for (int kk = 0; kk < 8; ++kk)
                mma(tb + T_Z, a + kstep(kk), b + mnstep(kk), id_z2, !first || kk > 0);
        };
        auto dh_batch = [&](uint32_t b_, int sa, bool first) {   // dH1^T (+)= W2[sa] dZ2^T
            const uint64_t a = desc_mnmajor(w2_ + 2u * sa * kPanelBytes, 0), b = desc_mnmajor(b_, 0);
#pragma unroll
            for (int kk = 0; kk < 8; ++kk) mma(tb + T_Z, a + mnstep(kk), b + mnstep(kk), id_dh, !first || kk > 0);
        };
        auto dw2_batch = [&](uint32_t b_, int sa, bool first) {  // dW2 (+)= H1^T[sa] dZ2
            const uint64_t b = desc_kmajor(b_, 0);
#pragma unroll
            for (int kk = 0; kk < 8; ++kk)
                mma_ts(tb + T_DW2, tb + T_ACT + 64u * sa + 8u * kk, b + kstep(kk), id_z1, !first || kk > 0);
        };
        // hi x hi of dW2, k-steps 4 r .. + 3 (dZ2's hi third in b0): two to an accumulator
        auto dw2_hi = [&](int r) {
            const uint64_t b = desc_kmajor(b0_, 0);
#pragma unroll
            for (int kk = 4 * r; kk < 4 * r + 4; ++kk)
                mma_ts(tb + (kk & 2 ? T_DW2B : T_DW2), tb + T_ACT + 8u * kk, b + kstep(kk), id_z1,
                       (kk & 1) || (r == 0 && !(kk & 2)));
            commit(&S.mma_b);
        };
        // [de hi | de mid | de lo] (+)= dZ1 [W1 hi | W1 mid | W1 lo]^T, the first `terms` of W1 (16 columns each; an
        // MMA this narrow costs the same for 16 columns as for 48).  The three parts join in FP32; of dZ1's hi third,
        // which comes last, units 64-127 go to an accumulator of their own.
        auto de_batch = [&](uint32_t b_, int terms, bool first, bool hi) {
            const uint64_t a = desc_mnmajor(b_, 0), b = desc_mnmajor(w1_ + 2 * kPanelBytes + 32u, 0);
            const uint32_t id = idesc_bf16(128, 16 * terms, 1, 1);
#pragma unroll
            for (int kk = 0; kk < 8; ++kk)
                mma(tb + (hi && kk >= 4 ? T_DE2 : T_DE), a + mnstep(kk), b + mnstep(kk), id, hi ? kk != 4 : (!first || kk > 0));
        };
        // copies a hi third from TMEM columns `from` into the pool's first buffer
        auto stage_hi = [&](uint32_t from) {
#pragma unroll 1
            for (int g = 0; g < 2; ++g) {
                float v[16];
                tmem_ld16(taddr(tb, warp, from + 32 * hc + 16 * g), v);
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    *reinterpret_cast<uint4 *>(buf0 + panel_offset(n, 32 * g + 8 * c)) =
                        make_uint4(__float_as_uint(v[4 * c]), __float_as_uint(v[4 * c + 1]), __float_as_uint(v[4 * c + 2]),
                                   __float_as_uint(v[4 * c + 3]));
            }
        };

        float acc2[64], acc1[24], a3[3] = {0.0f, 0.0f, 0.0f}, ab2 = 0.0f, ab3[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int j = 0; j < 64; ++j) acc2[j] = 0.0f;
#pragma unroll
        for (int j = 0; j < 24; ++j) acc1[j] = 0.0f;
        for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
            wait(&S.full, 0);
            if (ok && tid == 0) {
                const uint64_t a = desc_kmajor(w1_, 0), b = desc_kmajor(pool_, 0);
#pragma unroll
                for (int p = 0; p < 6; ++p)
#pragma unroll
                    for (int kk = 0; kk < KB; ++kk)
                        mma(tb + T_Z, a + kstep(PA[p] * KB + kk), b + (PB[p] == 0 ? 2 * kPanelStep : 0) + kstep((PB[p] == 2 ? KB : 0) + kk),
                            id_z1, (p | kk) != 0);
                commit(&S.mma_a);
            }
            if (hc == 0) {
#pragma unroll
                for (int ch = 0; ch < 3; ++ch) ab3[ch] += S.dout[ch][n];
            }
            wait_a();
            // ---- epilogue 1: H1 = relu(Z1), split: TMEM (A of dW2), lo and mid into the pool ----
            // Which units are on (z > 0): 16 samples a word, sample k in bit 15 - k.  The sign of 0 - z is set just
            // there: not for a zero of either sign (a unit whose weights are all 0) nor for a NaN.
            uint32_t m1[4], m2[2];
            float zz[32];
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                tmem_ld32(taddr(tb, warp, T_Z + 64 * hc + 32 * half), zz);
                bool near = false;   // a unit within rounding of zero
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    uint32_t on = 0;
                    float low = 0x1p127f;
#pragma unroll
                    for (int k = 0; k < 16; ++k) {
                        on = __funnelshift_l(__float_as_uint(__fsub_rn(0.0f, zz[16 * q + k])), on, 1);
                        low = fminf(low, fabsf(zz[16 * q + k]));
                    }
                    m1[2 * half + q] = on;
                    near |= low < eps1 * S.gmax[4 * hc + 2 * half + q];
                }
                if (ok && __any_sync(FULL, near)) {
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const int k0 = 64 * hc + 32 * half + 16 * q;
                        uint32_t amb = 0;
#pragma unroll
                        for (int k = 0; k < 16; ++k)
                            amb |= (fmaf(-eps1, S.xmax[k0 + k], fabsf(zz[16 * q + k])) < 0.0f ? 1u : 0u) << k;
                        m1[2 * half + q] = resolve<FeatT, PK, 1>(A, tile * TM + k0, n, amb, m1[2 * half + q]);
                    }
                }
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int g = 2 * half + q;
                    float z[16];
#pragma unroll
                    for (int k = 0; k < 16; ++k) z[k] = fmaxf(zz[16 * q + k], 0.0f);
                    uint32_t w[3][8];
                    split16(z, w);
                    store16(buf0, n, g, w[2]);
                    store16(buf1, n, g, w[1]);
#pragma unroll
                    for (int t = 0; t < 3; ++t) tmem_st8(taddr(tb, warp, T_ACT + 64 * t + 32 * hc + 8 * g), w[t]);
                }
            }
            tmem_wait_st();
            publish();
            // ---- layer 2 ----
            if (ok && tid == 0) {
                z2_batch(b0_, 0, true);
                commit(&S.mma_a);
                z2_batch(b1_, 1, false);
                z2_batch(b1_, 0, false);
                commit(&S.mma_b);
            }
            wait_a();
            stage_hi(T_ACT);
            publish();
            if (ok && tid == 0) {
                z2_batch(b0_, 2, false);
                z2_batch(b0_, 1, false);
                z2_batch(b0_, 0, false);
                commit(&S.mma_a);
            }
            wait_b();
            wait_a();
            // ---- epilogue 2: dZ2, dW3, db2 (a tile's sums first, then the running ones) ----
            float t3[3] = {0.0f, 0.0f, 0.0f}, tb2 = 0.0f;
            // (dL/do of a sample is read once for both: a read of four samples' takes the load unit four clocks a
            // warp, and reading it for h, for dZ2 and again for dZ2's hi third took it 4,600 clocks of a tile; so did
            // xmax of every sample 1,000.  1482 -> 1245 us at 1.38 M samples.)
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                tmem_ld32(taddr(tb, warp, T_Z + 64 * hc + 32 * half), zz);
                bool near = false;
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    uint32_t on = 0;
                    float low = 0x1p127f;
#pragma unroll
                    for (int k = 0; k < 16; k += 4) {
                        float d[3][4];
                        load_dout(S, 64 * hc + 32 * half + 16 * q + k, d);
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            float &z = zz[16 * q + k + j];
                            const float v = __fsub_rn(nb2, z), h = fmaxf(-v, 0.0f);   // v = -(z + b2), rounded alike
                            on = __funnelshift_l(__float_as_uint(v), on, 1);
                            low = fminf(low, fabsf(v));
                            t3[0] = fmaf(h, d[0][j], t3[0]);
                            t3[1] = fmaf(h, d[1][j], t3[1]);
                            t3[2] = fmaf(h, d[2][j], t3[2]);
                            z = fmaf(d[2][j], w32, fmaf(d[1][j], w31, d[0][j] * w30));   // dH2
                        }
                    }
                    m2[q] = on;
                    near |= low < eps2 * S.gmax[4 * hc + 2 * half + q];
                }
                if (ok && __any_sync(FULL, near)) {
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const int k0 = 64 * hc + 32 * half + 16 * q;
                        float z[16];
                        tmem_ld16(taddr(tb, warp, T_Z + k0), z);
                        uint32_t amb = 0;
#pragma unroll
                        for (int k = 0; k < 16; ++k)
                            amb |= (fmaf(-eps2, S.xmax[k0 + k], fabsf(z[k] + b2)) < 0.0f ? 1u : 0u) << k;
                        m2[q] = resolve<FeatT, PK, 2>(A, tile * TM + k0, n, amb, m2[q]);
                    }
                }
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int g = 2 * half + q;
                    float z[16];
#pragma unroll
                    for (int k = 0; k < 16; ++k) z[k] = off(m2[q], k) ? 0.0f : zz[16 * q + k];
#pragma unroll
                    for (int k = 0; k < 16; k += 4) tb2 += (z[k] + z[k + 1]) + (z[k + 2] + z[k + 3]);
                    uint32_t w[3][8];
                    split16(z, w);
                    store16(buf0, n, g, w[2]);
                    store16(buf1, n, g, w[1]);
                    tmem_st8(taddr(tb, warp, T_HI + 32 * hc + 8 * g), w[0]);   // until the pool has room for it
                }
            }
            tmem_wait_st();
            ab2 += tb2;
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) a3[ch] += t3[ch];
            publish();
            // ---- dW2 and dH1 ----
            if (ok && tid == 0) {
                dw2_batch(b0_, 0, true);
                dh_batch(b0_, 0, true);
                commit(&S.mma_a);
                dw2_batch(b1_, 1, false);
                dw2_batch(b1_, 0, false);
                dh_batch(b1_, 1, false);
            }
            wait_a();
            stage_hi(T_HI);
            publish();
            if (ok && tid == 0) {
                dw2_batch(b0_, 2, false);
                dw2_batch(b0_, 1, false);
                commit(&S.mma_b);
                dh_batch(b1_, 0, false);
            }
            wait_b();   // H1's mid and lo thirds have been read: room for a second accumulator of dW2
            if (ok && tid == 0) {
                dw2_hi(0);
                dh_batch(b0_, 2, false);
            }
            // hi x hi of dH1 last: units 0-63 on top of the small products, 64-127 in an accumulator of their own
            // (dW2's, read by then)
            const uint64_t dh_a = desc_mnmajor(w2_, 0), dh_b = desc_mnmajor(b0_, 0);
#pragma unroll
            for (int r = 0; r < 2; ++r) {   // this tile's dW2, beside the MMAs of dH1
                wait_b();
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    float v[16], u[16];
                    tmem_ld16x2(taddr(tb, warp, T_DW2 + 64 * hc + 16 * g), v, taddr(tb, warp, T_DW2B + 64 * hc + 16 * g), u);
#pragma unroll
                    for (int k = 0; k < 16; ++k) acc2[16 * g + k] += v[k] + u[k];
                }
                consumer_sync();
                if (ok && tid == 0) {
                    if (r == 0) {
                        dw2_hi(1);
                        dh_batch(b0_, 1, false);
                    }
#pragma unroll
                    for (int kk = 4 * r; kk < 4 * r + 4; ++kk)
                        mma(tb + (r == 0 ? T_Z : T_DW2), dh_a + mnstep(kk), dh_b + mnstep(kk), id_dh, kk != 4);
                    if (r == 1) commit(&S.mma_a);
                }
            }
            wait_a();
            // ---- epilogue 3: dZ1 = dH1 [Z1 > 0], split: TMEM (A of dW1), lo and mid into the pool ----
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                float z[16], z2[16];
                tmem_ld16(taddr(tb, warp, T_Z + 64 * hc + 16 * g), z);
                tmem_ld16(taddr(tb, warp, T_DW2 + 64 * hc + 16 * g), z2);
#pragma unroll
                for (int k = 0; k < 16; ++k) z[k] = off(m1[g], k) ? 0.0f : z[k] + z2[k];
                uint32_t w[3][8];
                split16(z, w);
                store16(buf0, n, g, w[2]);
                store16(buf1, n, g, w[1]);
#pragma unroll
                for (int s = 0; s < 3; ++s) tmem_st8(taddr(tb, warp, T_ACT + 64 * s + 32 * hc + 8 * g), w[s]);
            }
            tmem_wait_st();
            publish();
            // ---- de ----
            if (ok && tid == 0) {
                de_batch(b1_, 3, true, false);    // the mid term (with all of W1's, so that it starts all three parts)
                de_batch(b0_, 1, false, false);   // lo
                commit(&S.mma_a);
            }
            wait_a();
            stage_hi(T_ACT);
            publish();
            if (ok && tid == 0) {
                de_batch(b0_, 3, false, true);
                commit(&S.mma_a);
            }
            wait_a();
            if (ok && tid == 0) mbar_arrive(&S.empty);   // the pool is free for X
            float de[16];
            if (hc == 0) {   // lane = sample here
                float d1[16], d2[16];
                tmem_ld16x2(taddr(tb, warp, T_DE + 16), d1, taddr(tb, warp, T_DE2 + 16), d2);
#pragma unroll
                for (int k = 0; k < FEAT; ++k) de[k] = d1[k] + d2[k];
                tmem_ld16x2(taddr(tb, warp, T_DE + 32), d1, taddr(tb, warp, T_DE2 + 32), d2);
#pragma unroll
                for (int k = 0; k < FEAT; ++k) de[k] += d1[k] + d2[k];
                tmem_ld16x2(taddr(tb, warp, T_DE), d1, taddr(tb, warp, T_DE2), d2);
#pragma unroll
                for (int k = 0; k < FEAT; ++k) de[k] += d1[k] + d2[k];
                fence_before();
                asm volatile("bar.sync 2, 128;" ::: "memory");   // (dW1's accumulators take these columns)
                fence_after();
            }
            // (X staged again: the producers are also done with the de of the tile before)
            wait(&S.full, 1);
            // ---- dW1: the small products in two accumulators side by side, hi x hi in four of its own ----
            if (ok && tid == 0) {
                const uint64_t ml = desc_mnmajor(pool_, 0), hm = desc_mnmajor(pool_ + 2 * kPanelBytes, 0);
                const uint32_t id = idesc_bf16(128, DW1, 0, 1), id2 = idesc_bf16(128, 2 * DW1, 0, 1);
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) mma_ts(tb + T_DW1, tb + T_ACT + 8u * kk, ml + mnstep(kk), id2, kk != 0);
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) mma_ts(tb + T_DW1, tb + T_ACT + 64u + 8u * kk, hm + mnstep(kk), id2, 1u);
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) mma_ts(tb + T_DW1 + DW1, tb + T_ACT + 128u + 8u * kk, hm + mnstep(kk), id, 1u);
#pragma unroll
                for (int kk = 0; kk < 8; ++kk)
                    mma_ts(tb + T_DW1 + DW1 * (2 + kk / 2), tb + T_ACT + 8u * kk, hm + mnstep(kk), id, kk & 1);
                commit(&S.mma_a);
            }
            if (hc == 0) {
#pragma unroll
                for (int k = 0; k < 3; ++k) S.de[n][k] = make_float4(de[4 * k], de[4 * k + 1], de[4 * k + 2], de[4 * k + 3]);
            }
            wait_a();
            {   // columns 24 hc ..
                float t[24], v[24];
                const uint32_t from = taddr(tb, warp, T_DW1 + 24 * hc);
                tmem_ld24(from, t);
#pragma unroll
                for (int q = 1; q < 6; ++q) {
                    tmem_ld24(from + DW1 * q, v);
#pragma unroll
                    for (int k = 0; k < 24; ++k) t[k] += v[k];
                }
#pragma unroll
                for (int k = 0; k < 24; ++k) acc1[k] += t[k];
            }
            fence_before();
            ok = barrier_all(1, NC, ok);   // de written, TMEM reads done
            fence_after();
            if (!ok) break;
            if (tid == 0) mbar_arrive(&S.empty);   // the tile is done
        }
        if (!ok) {
            atomicExch(&S.abort, 1);
        } else {
            // grad_mlp = w1 | b1 | w2 | b2 | w3 | b3
            float *gW1 = A.grad_mlp, *gB1 = gW1 + IN * HID, *gW2 = gB1 + HID, *gB2 = gW2 + HID * HID;
            float *gW3 = gB2 + HID, *gB3 = gW3 + HID * 3;
#pragma unroll
            for (int j = 0; j < 64; ++j) atomicAdd(gW2 + n * HID + 64 * hc + j, acc2[j]);
#pragma unroll
            for (int j = 0; j < 24; ++j) {
                const int c = 24 * hc + j;
                if (c < IN) atomicAdd(gW1 + c * HID + n, acc1[j]);
                else if (c == IN) atomicAdd(gB1 + n, acc1[j]);
            }
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) ab3[ch] = warp_sum(ab3[ch]);
            // one sum a CTA: the halves of a unit and the warps of db3 join in the pool, which is free
            float4 *half = reinterpret_cast<float4 *>(pool), *rows = half + HID;
            if (hc == 1) half[n] = make_float4(a3[0], a3[1], a3[2], ab2);
            if (lane == 0 && warp > 0 && hc == 0) rows[warp] = make_float4(ab3[0], ab3[1], ab3[2], 0.0f);
            consumer_sync();
            if (hc == 0) {
                const float4 o = half[n];
                atomicAdd(gW3 + 3 * n, a3[0] + o.x);
                atomicAdd(gW3 + 3 * n + 1, a3[1] + o.y);
                atomicAdd(gW3 + 3 * n + 2, a3[2] + o.z);
                atomicAdd(gB2 + n, ab2 + o.w);
            }
            if (tid == 0) {
                const float4 r1 = rows[1], r2 = rows[2], r3 = rows[3];
                atomicAdd(gB3, (ab3[0] + r1.x) + (r2.x + r3.x));
                atomicAdd(gB3 + 1, (ab3[1] + r1.y) + (r2.y + r3.y));
                atomicAdd(gB3 + 2, (ab3[2] + r1.z) + (r2.z + r3.z));
            }
        }
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

template <typename FeatT, bool PK>
void launch_split_bwd(const RenderArgs &A, cudaStream_t s) {
    auto kern = fine_colour_bwd_split_kernel<FeatT, PK>;
    ensure_smem(reinterpret_cast<const void *>(kern), (int)kBwdSmem);
    ProfScope ps_(DVGO_K_FINE_COLOUR_BWD, s);
    kern<<<num_sms(), NC + NP, kBwdSmem, s>>>(A);
}

}  // namespace

void launch_fine_colour_bwd_fp32(const RenderArgs &A, cudaStream_t s) {
    const bool bf = A.cdtype == DVGO_DTYPE_BF16;
    if (A.nfreq_pos > 0) launch_fine_colour_bwd_simt(A, s);
    else if (A.packed) {
        if (bf) launch_split_bwd<__nv_bfloat16, true>(A, s);
        else launch_split_bwd<float, true>(A, s);
    } else {
        if (bf) launch_split_bwd<__nv_bfloat16, false>(A, s);
        else launch_split_bwd<float, false>(A, s);
    }
}

}  // namespace dvgo
