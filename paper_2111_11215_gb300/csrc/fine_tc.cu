// fine_tc.cu -- colour queries of the fine stage with the BF16 tensor-core MLP (tcgen05, sm_103a).
//
// Same function as fine_tc_fp32.cu and fine_tc_fp32_bwd.cu (Sec. 4.2 Eq. fine_queries_rgb, Supp. A: 12 features + PE(d, 4)
// = 39 inputs, or 72 with PE(x, 5) appended; two hidden layers of 128 with ReLU, sigmoid output)
// with the two 128-wide layers
// and all weight-gradient contractions on the 5th-generation tensor cores: BF16 operands in
// shared memory (128-byte swizzled panels, see tc_helpers.cuh), FP32 accumulators in TMEM, MMAs
// issued by one thread, completion signalled through mbarriers.  The 128 -> 3 output layer, the
// sigmoid and the element-wise steps run on the CUDA cores in the epilogues.
//
// Persistent CTAs walk tiles of M = 128 kept samples.  Warps 8-15 (producers, two sets)
// gather the next tile -- features at the 8 lattice corners, the ray's direction encoding, the
// bias column -- into one of two X panels, and in the backward also scatter the feature gradients
// of the tile that last used that panel.  The forward stores every finished X panel (16 KiB, as
// swizzled in shared memory) in the workspace (one bulk copy per tile); the backward loads it back
// with one bulk copy instead of gathering again (tile t holds the same kept samples in both: the
// kept list is the forward's), so its producers only form the per-row tables, dL/dc and the PE(x)
// tail.  Warps 0-7 (consumers)
// run the epilogues and, in the forward, issue the MMAs.  full[b] / empty[b] mbarriers hand the X
// panels over; every wait is bounded.
//
// The backward is a chain of MMA batches and epilogues.  Waiting for each batch as a whole, with one
// thread of an epilogue issuing it, a tile took 11,700 clocks, of which the MMAs are 3,500.  So a warp of
// its own (warp 16) issues them: what the next epilogue waits for first, the weight gradients behind it, and
// the next tile's layer 1 before this tile's last batch; dZ1 goes over H2, not H1, so that its epilogue
// need not wait for dW2, and the next tile's first epilogue runs during dW1.  The consumers hold no barrier
// among themselves: a warp waits for MMA batches only and signals the issuing warp.  65,536 rays at 256^3
// (284,928 tiles): 11.55 -> 7.33 ms, the scatter's new form (fine_gather.cuh) included, 6.87 ms with two producer
// sets (the scatter was 4,800 of a producer's 7,400 clocks a tile); 310,320 samples: 121 -> 84 -> 77 us.  What
// bounds it now: the consumers' chain of three epilogues and three MMA batches, 7,000 clocks a tile.
//
// Inputs beyond the 64 columns of the X panel (PE(x) entries 24-32 of the 72-input row) live in a
// "tail panel" that also holds W3: columns 0-15 W3 (3 used), 16-31 / 32-47 the tail of X buffer 0 /
// 1, 48-63 the tail rows of W1 (transposed).  Layer 1 adds one K = 16 MMA over the tails; the
// backward adds dW1_tail^T += dZ1^T X_tail (an MN-major operand that starts 32 or 64 bytes into
// the swizzled rows).
//
// Forward per tile:  X[128x64] (features, PE(d), [PE(x)], 1) -> Z1 = X W1|b1 -> H1 = relu(Z1) -> Z2 = H1 W2
//                    -> H2 = relu(Z2 + b2) -> O = H2 W3 (N = 16, 3 used) -> c = sigmoid(O + b3).
// Backward per tile (recomputes layers 1 and 2; the colour c is the one the forward stored in the
// sample record, so layer 3 is not recomputed), with dL/dc from the compositing backward:
//   dout = dL/dc c (1 - c)                                        (producers; epilogue, BF16 panel)
//   dH2 = dout W3^T;  dZ2 = dH2 [Z2 + b2 > 0]                      (MMA, epilogue)
//   dH1 = dZ2 W2^T;  [dW2^T | db2] += dZ2^T [H1 | dout];  dW3 += H2^T dout   (MMAs; dout's
//   column 3 is 1, so one N = 144 MMA gives dW2^T and db2)
//   dZ1 = dH1 [Z1 > 0]                                             (epilogue)
//   de = dZ1 W1[0:16]^T;  [dW1 | db1]^T += dZ1^T X                 (MMAs)
//   de[0:12] -> shared memory -> scattered to the feature grid by the producers
// TMEM columns: Z1 / O / dH2 [0,128), Z2 / dH1 [128,256), [dW2^T | db2] [256,400), dW1^T [400,464),
// dW3 [464,480), de [480,496), dW1_tail^T [496,512).  The weight-gradient accumulators live in TMEM for
// the whole launch and are added to global memory once per CTA.

#include <stddef.h>

#include "dvgo_internal.cuh"
#include "fine_gather.cuh"
#include "tc_helpers.cuh"

namespace dvgo {

namespace {

using namespace tc;

constexpr int TM = 128;
constexpr int NC = 256;        // consumer threads: warp w owns TMEM lanes 32 (w % 4).., columns 64 (w / 4)..
constexpr int NP = 128;        // producer threads of one set (one sample row each)
// producer sets: set p fills X buffer p with every other tile, so that two tiles are gathered (in the backward
// also scattered) at once
constexpr int kProdSets = 2;
// the backward has one more warp, which issues the MMAs
template <bool BWD>
constexpr int kThreads = NC + NP * kProdSets + (BWD ? 32 : 0);   // 544 / 512
constexpr int HID = 128;
constexpr int FEAT = 12;
constexpr int NF = 4;
constexpr int NFX = 5;
constexpr int PX = FEAT + 3 + 6 * NF;   // 39: first input of the PE(x) block

// Input row of the two widths: IN inputs, NMAIN of them in the X panel, the first-layer bias as
// the constant-1 column BIAS of the X panel, NTAIL inputs in the tail panel.
template <bool PEX>
struct TcDims {
    static constexpr int IN = PX + (PEX ? 3 + 6 * NFX : 0);   // 39 or 72
    static constexpr int NMAIN = PEX ? 63 : IN;
    static constexpr int BIAS = NMAIN;
    static constexpr int NTAIL = IN - NMAIN;                  // 0 or 9
};

constexpr uint32_t COL_Z1 = 0, COL_Z2 = 128, COL_DW2T = 256, COL_DW1 = 400, COL_DW3 = 464,
                   COL_DE = 480, COL_DW1T = 496;

// Small per-CTA state, padded to a multiple of 1024 bytes so that the panels after it stay
// aligned to the 128-byte-swizzle atom.
struct alignas(1024) SmallTC {
    float b2[HID];
    float b3[4];
    float db3[4];
    // per-row tables of a tile.  Forward: the sample slot (-1 for padding rows), a ring of 4 (tile i in
    // entry i % 4; a group may still read its entry when its X buffer is handed back).  Backward: what the
    // scatter of tile i needs, which runs after tile i + 2 is placed
    union {
        int slot[4][TM];
        float4 place[4][TM];
    };
    ScatterTab tab[kProdSets * NP / 32];   // backward
    float dc[2][TM][3];       // dL/dc (backward)
    uint64_t full[2], empty[2];
    uint64_t mma[2];          // forward: the MMAs of consumer group 0 / 1
    uint64_t stop[2];         // forward: all MMAs of a group that gave up
    // backward.  xl: the bulk load of X panel b from the forward's copy; z1, z2, dh, de: MMA batches
    // complete; ev[e]: consumers have finished epilogue e; fin: every MMA of the launch complete; sc: the
    // de of a tile of X buffer b has been scattered
    uint64_t xl[2], z1, z2, dh, de, ev[4], fin, sc[2];
    uint32_t tmem_base;
    int abort;
};

struct SmemTC {
    unsigned char w1t[kPanelBytes];       // W1|b1 transposed: row = hidden unit, 64 input columns
    unsigned char w2t[2 * kPanelBytes];   // W2 transposed: row = output unit, 128 input columns
    unsigned char tp[kPanelBytes];        // tail panel: row = hidden unit / sample; W3 in columns 0-2,
                                          // X tails in 16-31 / 32-47, W1 tail in 48-63
    unsigned char x[2][kPanelBytes];      // X (double-buffered): row = sample
    // The backward's consumers hold no barrier among themselves; a buffer is rewritten once the MMA batches they
    // wait for were the last to read it: H1 (read by layer 2 and dW2) after the next tile's z1; H2 (read by
    // dW3) by dZ1 after dh, dZ1 (read by de and dW1) by the next H2 after the next z2; dZ2 (read by dH1 and dW2)
    // after the next z2.  The forward keeps its hidden layers in tensor memory.
    unsigned char h1[2 * kPanelBytes];    // H1
    // backward: columns 0-15: [dout_r, dout_g, dout_b, 1, ...] (MMA operand); bytes 32-79 and 80-127
    // of every row (16-byte chunks 2-4 and 5-7): de[0:12] in FP32 for X buffer 0 and 1.  It follows
    // H1 directly, so [H1 | dout] is one MN-major operand of N = 144 (panels 16 KiB apart)
    unsigned char dout[kPanelBytes];
    unsigned char h2[2 * kPanelBytes];    // H2, then dZ1
    SmallTC sm;
    // backward only (the forward allocates the struct up to here)
    unsigned char dz2[2 * kPanelBytes];   // dZ2
};
static_assert(offsetof(SmemTC, dout) == offsetof(SmemTC, h1) + 2 * kPanelBytes, "[H1 | dout] must be contiguous");

constexpr size_t smem_bytes(bool bwd) { return (bwd ? sizeof(SmemTC) : offsetof(SmemTC, dz2)) + 1024; }
static_assert(smem_bytes(true) <= 232448, "the backward must fit one CTA per SM (227 KB of shared memory)");

// 16-byte chunk k (0-2) of the de[0:12] slot of X buffer b in row r of the dout panel.
__device__ __forceinline__ float4 *de_slot(unsigned char *dout, int b, int r, int k) {
    return reinterpret_cast<float4 *>(dout + panel_offset(r, 8 * (2 + 3 * b + k)));
}

// Producer: gather sample row `row` of a tile (kept entry kv, kv.y < 0 for a padding row; its ray's
// prefetched data rp) into X panel b (and its tail) and the per-row tables.
template <typename FeatT, bool BWD, bool PEX, bool PK>
__device__ __forceinline__ void produce_row(const RenderArgs &A, SmemTC &S, int b, int t, int2 kv,
                                            const RayPre &rp, const float4 &gc, int row, bool cached) {
    // cached (backward): the X panel arrives by bulk copy; only the tables, dL/dc and the tail here
    using D = TcDims<PEX>;
    float v[64], tail[16];
#pragma unroll
    for (int i = 0; i < 64; ++i) v[i] = 0.0f;
#pragma unroll
    for (int i = 0; i < 16; ++i) tail[i] = 0.0f;
    int slot = -1;
    float4 place = make_float4(0.0f, 0.0f, 0.0f, __int_as_float(kNoCell));
    float d0 = 0.0f, d1 = 0.0f, d2 = 0.0f;
    if (kv.y >= 0) {
        float dt;
        const Cell c = cell_pre(A, rp, kv.y, kv.x >> 16, dt);
        slot = rp.off + (kv.x & 0xffff);
        if (BWD) {
            place = row_place(A, c, true, PK);
            // dout = dL/dc c (1 - c), formed by the compositing backward with the forward's colour c
            d0 = gc.y;
            d1 = gc.z;
            d2 = gc.w;
        }
        if (!cached) gather_features<FeatT, PK>(A, c, v);
        const float4 *pe = reinterpret_cast<const float4 *>(A.pe + (size_t)kv.y * kPeStride);
#pragma unroll
        for (int k = 0; k < (cached ? 0 : 7); ++k) {
            const float4 q4 = __ldg(pe + k);
            if (4 * k + 0 < 27) v[FEAT + 4 * k + 0] = q4.x;
            if (4 * k + 1 < 27) v[FEAT + 4 * k + 1] = q4.y;
            if (4 * k + 2 < 27) v[FEAT + 4 * k + 2] = q4.z;
            if (4 * k + 3 < 27) v[FEAT + 4 * k + 3] = q4.w;
        }
        if constexpr (PEX) {
            // PE(x) of the world-space sample position: [x (3), sin(2^k x_c) (15), cos(2^k x_c) (15)]
            float xv[3], pe[3 + 6 * NFX];
            cell_world(A, c, xv);
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                pe[a] = xv[a];
                pe_axis<NFX>(xv[a], pe + 3 + a * NFX, pe + 3 + 3 * NFX + a * NFX);
            }
#pragma unroll
            for (int j = 0; j < D::NMAIN - PX; ++j) v[PX + j] = pe[j];
#pragma unroll
            for (int j = 0; j < D::NTAIL; ++j) tail[j] = pe[D::NMAIN - PX + j];
        }
        v[D::BIAS] = 1.0f;
    }
    if (!cached) {
#pragma unroll
        for (int c = 0; c < 64; c += 8) panel_store8(S.x[b], row, c, v + c);
    }
    if constexpr (PEX) {
        panel_store8(S.tp, row, 16 * (1 + b), tail);
        panel_store8(S.tp, row, 16 * (1 + b) + 8, tail + 8);
    }
    if (!BWD) S.sm.slot[t][row] = slot;
    if (BWD) {
        S.sm.place[t][row] = place;
        S.sm.dc[b][row][0] = d0;
        S.sm.dc[b][row][1] = d1;
        S.sm.dc[b][row][2] = d2;
    }
}

template <typename FeatT, bool BWD, bool PEX, bool PK>
__global__ void __launch_bounds__(kThreads<BWD>, 1) fine_colour_tc_kernel(RenderArgs A) {
    using D = TcDims<PEX>;
    extern __shared__ unsigned char smem_raw[];
    SmemTC &S = *reinterpret_cast<SmemTC *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int tid = threadIdx.x, warp = tid >> 5;
    constexpr uint32_t NCOLS = 512;   // backward: activations + weight gradients; forward: 256 per consumer group

    if (tid == 0) {
        mbar_init(&S.sm.full[0], NP);
        mbar_init(&S.sm.full[1], NP);
        mbar_init(&S.sm.empty[0], BWD ? 4 : 1);
        mbar_init(&S.sm.empty[1], BWD ? 4 : 1);
        mbar_init(&S.sm.mma[0], 1);
        mbar_init(&S.sm.mma[1], 1);
        mbar_init(&S.sm.stop[0], 1);
        mbar_init(&S.sm.stop[1], 1);
        if (BWD) {
            mbar_init(&S.sm.xl[0], 1);
            mbar_init(&S.sm.xl[1], 1);
            mbar_init(&S.sm.z1, 1);
            mbar_init(&S.sm.z2, 1);
            mbar_init(&S.sm.dh, 1);
            mbar_init(&S.sm.de, 1);
            for (int e = 0; e < 4; ++e) mbar_init(&S.sm.ev[e], NC / 32);
            mbar_init(&S.sm.fin, 1);
            mbar_init(&S.sm.sc[0], NP);
            mbar_init(&S.sm.sc[1], NP);
        }
        S.sm.abort = 0;
    }
    if (warp == 0) tmem_alloc(&S.sm.tmem_base, NCOLS);
    // barriers initialised and TMEM allocated: the producers start gathering the first tile while
    // consumer warps 0-3 stage the weights (published to the consumers and the tensor core below)
    fence_before();
    __syncthreads();
    fence_after();
    if (tid < TM) {
        // weights: row n = tid of W1^T (64 input columns, bias in column BIAS), of W2^T and of the
        // tail panel (W3, and with PE(x) the tail rows of W1)
        float v[64];
#pragma unroll
        for (int k = 0; k < 64; ++k) v[k] = k < D::NMAIN ? A.w1[k * HID + tid] : (k == D::BIAS ? A.b1[tid] : 0.0f);
#pragma unroll
        for (int c = 0; c < 64; c += 8) panel_store8(S.w1t, tid, c, v + c);
#pragma unroll
        for (int pnl = 0; pnl < 2; ++pnl) {
#pragma unroll
            for (int k = 0; k < 64; ++k) v[k] = A.w2[(pnl * 64 + k) * HID + tid];
#pragma unroll
            for (int c = 0; c < 64; c += 8) panel_store8(S.w2t + pnl * kPanelBytes, tid, c, v + c);
        }
#pragma unroll
        for (int k = 0; k < 64; ++k)
            v[k] = k < 3 ? A.w3[3 * tid + k]
                         : ((k >= 48 && k - 48 < D::NTAIL) ? A.w1[(D::NMAIN + k - 48) * HID + tid] : 0.0f);
        // only the weight columns (0-15: W3, 48-63: W1 tail): columns 16-47 hold the X tails, which
        // the producers are already writing
        panel_store8(S.tp, tid, 0, v);
        panel_store8(S.tp, tid, 8, v + 8);
        panel_store8(S.tp, tid, 48, v + 48);
        panel_store8(S.tp, tid, 56, v + 56);
        if (BWD) {
#pragma unroll
            for (int k = 0; k < 64; ++k) v[k] = 0.0f;
#pragma unroll
            for (int c = 0; c < 64; c += 8) panel_store8(S.dout, tid, c, v + c);
        }
        S.sm.b2[tid] = A.b2[tid];
        if (tid < 3) S.sm.b3[tid] = A.b3[tid];
        if (tid < 4) S.sm.db3[tid] = 0.0f;
    }
    if (tid < NC || tid >= NC + NP * kProdSets) {   // weights staged: all that issue MMAs may use them
        fence_async_smem();
        fence_before();
        asm volatile("bar.sync 1, %0;" ::"n"(NC + (BWD ? 32 : 0)) : "memory");
        fence_after();
    }

    const int n_kept = A.hdr->n_kept;
    const int ntiles = (n_kept + TM - 1) / TM;
    // backward: reload the X panels the forward stored (the workspace has room and the forward that
    // filled it stored them); otherwise gather them again
    const bool cached = BWD && A.xcache != nullptr && A.hdr->xcache != 0;
    bool ok = true;
    int ntile_mine = 0;

    if (tid >= NC && tid < NC + NP * kProdSets) {
        // ------------------------------- producers -------------------------------
        // Set pset takes the CTA's tiles i = pset, pset + nsets, ... (X buffer i & 1).  Software-
        // pipelined a tile deep: while producing a tile, a producer already has its set's next tile's
        // kept entry and fetches that tile's ray data and the kept entry of the tile after, so that
        // only the corner-feature loads of a tile wait on memory when it is produced.
        constexpr int nsets = kProdSets;
        const int row = (tid - NC) & (NP - 1), pset = (tid - NC) / NP;
        const int stride = nsets * (int)gridDim.x;
        auto kept_at = [&](int t) -> int2 {
            const int e = t * TM + row;
            return (t < ntiles && e < n_kept) ? A.kept[e] : make_int2(-1, -1);
        };
        auto scatter_tile = [&](int j) {   // the CTA's tile j
            scatter_rows<PK>(A, S.sm.place[j & 3], [&](int r, int k) { return de_slot(S.dout, j & 1, r, k); },
                             S.sm.tab[warp - NC / 32], row);
        };
        auto dldo_at = [&](const int2 &kv, const RayPre &rp) -> float4 {
            return (BWD && kv.y >= 0) ? A.sgrad[rp.off + (kv.x & 0xffff)] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        };
        const int tile0 = (int)blockIdx.x + pset * (int)gridDim.x;
        int2 kv_cur = kept_at(tile0);
        RayPre rp_cur = kv_cur.y >= 0 ? ray_pre(A, kv_cur.y) : RayPre{};
        float4 gc_cur = dldo_at(kv_cur, rp_cur);
        int2 kv_next = kept_at(tile0 + stride);
        int nload[2] = {0, 0};   // row 0, backward: bulk loads issued into X panel 0 / 1
        int i = pset;
        for (int tile = tile0; tile < ntiles; tile += stride, i += nsets) {
            const int b = i & 1;
            const RayPre rp_next = kv_next.y >= 0 ? ray_pre(A, kv_next.y) : RayPre{};
            const int2 kv_after = kept_at(tile + 2 * stride);
            if (i >= 2) ok = mbar_wait(&S.sm.empty[b], ((i >> 1) - 1) & 1, A.wait_ns);
            // (the warp leaves as one: the scatter is a warp's work)
            if (__any_sync(0xffffffffu, !ok)) {
                ok = false;
                break;
            }
            if (__any_sync(0xffffffffu, *(volatile int *)&S.sm.abort != 0)) break;
            if (cached && row == 0) {   // X panel b is free: the forward's copy of this tile's panel
                bulk_load(S.x[b], A.xcache + (size_t)tile * kPanelBytes, kPanelBytes, &S.sm.xl[b]);
                ++nload[b];
            }
            produce_row<FeatT, BWD, PEX, PK>(A, S, b, i & 3, kv_cur, rp_cur, gc_cur, row, cached);
            fence_async_smem();
            // (testing aid: one arrival withheld on a chosen tile makes the consumers' wait run out)
            if (!(row == 0 && tile + 1 == A.withhold_tile)) mbar_arrive(&S.sm.full[b]);
            if (BWD && i >= 2) {
                scatter_tile(i - 2);
                mbar_arrive(&S.sm.sc[b]);
            }
            gc_cur = dldo_at(kv_next, rp_next);
            kv_cur = kv_next;
            rp_cur = rp_next;
            kv_next = kv_after;
        }
        if (BWD && ok) {
            // the last tile: wait until the consumers are done with it, then scatter
            for (int j = i - nsets; j >= 0 && j < i && ok; j += nsets) {
                ok = __all_sync(0xffffffffu, mbar_wait(&S.sm.empty[j & 1], (j >> 1) & 1, A.wait_ns));
                if (ok && !__any_sync(0xffffffffu, *(volatile int *)&S.sm.abort != 0)) scatter_tile(j);
            }
        }
        // every bulk load issued has landed before the CTA can exit (bounded)
        for (int bb = 0; bb < 2; ++bb)
            if (nload[bb] > 0) mbar_wait(&S.sm.xl[bb], (nload[bb] - 1) & 1, A.wait_ns);
        if (!ok) atomicExch(&S.sm.abort, 1);
    } else if constexpr (!BWD) {
        // --------------------------- forward consumers: two groups ---------------------------
        // Group grp = warp / 4 takes every other tile of this CTA (the CTA's tiles i = grp, grp + 2,
        // ..., so always X buffer grp), so that one group's epilogues run while the other group's
        // MMAs do.  Thread r = tid % 128 owns row r (its TMEM lane) and all 128 columns; the group
        // has its own 256 TMEM columns, MMA barrier and named barrier (2 + grp, 128 threads).  The
        // hidden activations never go to shared memory: each epilogue writes them back to TMEM as
        // BF16 (two per column) and the next layer reads its A operand from there.  Columns:
        // Z1 at +0, then H1 at +0 (64 columns, over the Z1 values already read) and H2 at +64;
        // Z2 at +128, then O at +128.
        constexpr uint32_t F_H1 = 0, F_H2 = 64, F_Z2 = 128, F_O = 128;
        const int grp = warp >> 2, r = tid & (TM - 1);
        const uint32_t tb = S.sm.tmem_base + 256u * (uint32_t)grp;
        uint64_t *mbar = &S.sm.mma[grp];
        uint32_t mphase = 0;
        // waits of a warp as one; the verdicts of a group's warps meet at its last barrier of a tile (barrier_all)
        auto wait = [&](uint64_t *bar, uint32_t par) {
            if (ok) ok = __all_sync(0xffffffffu, mbar_wait(bar, par, A.wait_ns));
            fence_after();
        };
        auto wait_mma = [&]() {
            wait(mbar, mphase);
            mphase ^= 1;
        };
        auto group_sync = [&]() {
            fence_before();
            if (grp) asm volatile("bar.sync 3, 128;" ::: "memory");
            else asm volatile("bar.sync 2, 128;" ::: "memory");
            fence_after();
        };
        int i = grp;
        for (int tile = blockIdx.x + grp * gridDim.x; tile < ntiles; tile += 2 * gridDim.x, i += 2) {
            const int b = grp;
            uint32_t x_ = smem_u32(S.x[b]), w1t_ = smem_u32(S.w1t), w2t_ = smem_u32(S.w2t), w3p_ = smem_u32(S.tp);
            asm volatile("" : "+r"(x_), "+r"(w1t_), "+r"(w2t_), "+r"(w3p_));
            // (no abort-flag test here: the group's warps could read it on either side of its setting; a failed
            // producer leaves this wait unsatisfied for every thread of the group)
            wait(&S.sm.full[b], (i >> 1) & 1);
            if (!ok) {   // (the table may hold nothing yet)
                group_sync();
                group_sync();
                barrier_all(2 + grp, TM, false);
                break;
            }
            const int slot = S.sm.slot[i & 3][r];
            const float tau = slot >= 0 ? __ldg(A.stau + slot) : 0.0f;   // goes with the colour
            // ---- layer 1: Z1 = X W1 ----
            if (ok && r == 0) {
#pragma unroll 1
                for (int kk = 0; kk < 4; ++kk)
                    mma(tb + COL_Z1, desc_kmajor(x_, kk), desc_kmajor(w1t_, kk), idesc_bf16(128, 128, 0, 0), kk > 0);
                if (PEX)
                    mma(tb + COL_Z1, desc_kmajor(w3p_, 1 + b), desc_kmajor(w3p_, 3), idesc_bf16(128, 128, 0, 0), 1u);
                commit(mbar);
                if (A.xcache) bulk_store(A.xcache + (size_t)tile * kPanelBytes, S.x[b], kPanelBytes);   // for the backward
            }
            wait_mma();
            if (ok && r == 0) {   // X[b] is free once layer 1 and the copy have read it
                if (A.xcache) bulk_wait_read();
                mbar_arrive(&S.sm.empty[b]);
            }
            // ---- epilogue 1: H1 = relu(Z1), all 128 columns of my row, as BF16 into TMEM (32-column
            //      chunk g of Z1 becomes columns 16 g .. 16 g + 15, which chunks before g held) ----
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                float z[32];
                tmem_ld32(taddr(tb, warp, COL_Z1 + 32 * g), z);
                uint32_t h[16];
#pragma unroll
                for (int k = 0; k < 16; ++k) h[k] = relu_bf16(pack_bf16(z[2 * k], z[2 * k + 1]));
                tmem_st16(taddr(tb, warp, F_H1 + 16 * g), h);
            }
            tmem_wait_st();
            group_sync();
            // ---- layer 2: Z2 = H1 W2, A = H1 from TMEM ----
            if (ok && r == 0) {
#pragma unroll
                for (int kk = 0; kk < 8; ++kk)
                    mma_ts(tb + F_Z2, tb + F_H1 + 8u * (uint32_t)kk, desc_kmajor(w2t_, kk), idesc_bf16(128, 128, 0, 0),
                           kk > 0);
                commit(mbar);
            }
            wait_mma();
            // ---- epilogue 2: H2 = relu(Z2 + b2), as BF16 into TMEM ----
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                float z[32];
                tmem_ld32(taddr(tb, warp, F_Z2 + 32 * g), z);
                uint32_t h[16];
#pragma unroll
                for (int k = 0; k < 32; k += 4) {
                    const float4 bb = *reinterpret_cast<const float4 *>(&S.sm.b2[32 * g + k]);
                    h[k / 2] = relu_bf16(pack_bf16(z[k] + bb.x, z[k + 1] + bb.y));
                    h[k / 2 + 1] = relu_bf16(pack_bf16(z[k + 2] + bb.z, z[k + 3] + bb.w));
                }
                tmem_st16(taddr(tb, warp, F_H2 + 16 * g), h);
            }
            tmem_wait_st();
            group_sync();
            // ---- layer 3: O = H2 W3 (N = 16, columns 0-2 used), A = H2 from TMEM ----
            if (ok && r == 0) {
#pragma unroll
                for (int kk = 0; kk < 8; ++kk)
                    mma_ts(tb + F_O, tb + F_H2 + 8u * (uint32_t)kk, desc_mnmajor(w3p_, kk), idesc_bf16(128, 16, 0, 1),
                           kk > 0);
                commit(mbar);
            }
            wait_mma();
            float o[16];
            tmem_ld16(taddr(tb, warp, F_O), o);
            if (ok && slot >= 0)
                A.scol[slot] = make_float4(sigmoidf_(o[0] + S.sm.b3[0]), sigmoidf_(o[1] + S.sm.b3[1]),
                                           sigmoidf_(o[2] + S.sm.b3[2]), tau);
            fence_before();
            ok = barrier_all(2 + grp, TM, ok);   // TMEM and panel reads done before this group's next MMAs
            fence_after();
            if (!ok) break;
        }
        if (r == 0 && A.xcache) bulk_wait_all();   // the copies are complete before the kernel ends
        if (!ok) atomicExch(&S.sm.abort, 1);
    } else if (warp == (NC + NP * kProdSets) / 32) {
        // ------------------------------- MMA issue (backward) -------------------------------
        // One thread issues a tile's batches as their operands become ready, and the next tile's layer 1 as
        // soon as its X panel is there, so that it is complete when the consumers come to it:
        //   Z1(0) | Z2, dH2 | dW3 | dH1 | dW2, then Z1 of the next tile | de, dW1
        if ((tid & 31) == 0) {
            const uint32_t tb = S.sm.tmem_base;
            auto wait = [&](uint64_t *bar, uint32_t par) -> bool {
                ok = ok && mbar_wait(bar, par, A.wait_ns);
                fence_after();
                return ok;
            };
            // descriptors of k-step 0; the steps are constants added to them, so that a batch is issued
            // faster than the tensor core takes it
            const uint64_t x_k = desc_kmajor(smem_u32(S.x[0]), 0), x_m = desc_mnmajor(smem_u32(S.x[0]), 0);
            const uint64_t w1_k = desc_kmajor(smem_u32(S.w1t), 0), w1_m = desc_mnmajor(smem_u32(S.w1t), 0);
            const uint64_t w2_k = desc_kmajor(smem_u32(S.w2t), 0), w2_m = desc_mnmajor(smem_u32(S.w2t), 0);
            const uint64_t h1_k = desc_kmajor(smem_u32(S.h1), 0), h1_m = desc_mnmajor(smem_u32(S.h1), 0);
            const uint64_t h2_k = desc_kmajor(smem_u32(S.h2), 0), h2_m = desc_mnmajor(smem_u32(S.h2), 0);
            const uint64_t dz2_k = desc_kmajor(smem_u32(S.dz2), 0), dz2_m = desc_mnmajor(smem_u32(S.dz2), 0);
            const uint64_t do_k = desc_kmajor(smem_u32(S.dout), 0), do_m = desc_mnmajor(smem_u32(S.dout), 0);
            const uint64_t tp_k = desc_kmajor(smem_u32(S.tp), 0), tp_m = desc_mnmajor(smem_u32(S.tp), 0);
            auto layer1 = [&](int b) {   // Z1 = X W1; the X tail (k-step 1 + b of the tail panel) against the W1 tail
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                    mma(tb + COL_Z1, x_k + (b ? kPanelStep : 0) + kstep(kk), w1_k + kstep(kk), idesc_bf16(128, 128, 0, 0), kk > 0);
                if (PEX)
                    mma(tb + COL_Z1, tp_k + (b ? kstep(2) : kstep(1)), tp_k + kstep(3), idesc_bf16(128, 128, 0, 0), 1u);
                commit(&S.sm.z1);
            };
            bool early = false;   // this tile's layer 1 has been issued
            int i = 0;
            for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++i) {
                const int b = i & 1;
                const uint32_t par = i & 1, xpar = (i >> 1) & 1;
                const uint32_t acc_w = i > 0 ? 1u : 0u;   // first tile of this CTA initialises the accumulators
                if (!early) {
                    if (!wait(&S.sm.full[b], xpar) || (cached && !wait(&S.sm.xl[b], xpar))) break;
                    layer1(b);
                }
                // ---- layer 2: Z2 = H1 W2; and dH2 = dout W3^T (K = 16: dout's columns [dL/do, 1, 0 ...]
                //      against the tail panel's [W3, 0 ...]) into Z1's columns, which epilogue 1 has read ----
                if (!wait(&S.sm.ev[0], par)) break;
#pragma unroll
                for (int kk = 0; kk < 8; ++kk)
                    mma(tb + COL_Z2, h1_k + kstep(kk), w2_k + kstep(kk), idesc_bf16(128, 128, 0, 0), kk > 0);
                mma(tb + COL_Z1, do_k, tp_k, idesc_bf16(128, 128, 0, 0), 0u);
                commit(&S.sm.z2);
                // ---- dW3, while the consumers form dZ2 ----
                if (!wait(&S.sm.ev[1], par)) break;
#pragma unroll
                for (int kk = 0; kk < 8; ++kk)
                    mma(tb + COL_DW3, h2_m + mnstep(kk), do_m + mnstep(kk), idesc_bf16(128, 16, 1, 1),
                        acc_w | (kk > 0));
                // ---- dH1; then, while the consumers form dZ1 (over H2, which dW3 has read), dW2 ----
                if (!wait(&S.sm.ev[2], par)) break;
#pragma unroll
                for (int kk = 0; kk < 8; ++kk)
                    mma(tb + COL_Z2, dz2_k + kstep(kk), w2_m + mnstep(kk), idesc_bf16(128, 128, 0, 1), kk > 0);
                commit(&S.sm.dh);
#pragma unroll
                for (int kk = 0; kk < 8; ++kk)
                    mma(tb + COL_DW2T, dz2_m + mnstep(kk), h1_m + mnstep(kk), idesc_bf16(128, 144, 1, 1),
                        acc_w | (kk > 0));   // [dW2^T | db2]: B = [H1 | dout]
                // ---- the next tile's layer 1 (its columns were read with dH2), if its X panel comes first ----
                early = false;
                const bool more = tile + (int)gridDim.x < ntiles;
                const uint32_t npar = ((i + 1) >> 1) & 1;
                const uint64_t t0 = globaltimer();
                for (;;) {
                    if (more && !early && mbar_test(&S.sm.full[b ^ 1], npar) &&
                        (!cached || mbar_test(&S.sm.xl[b ^ 1], npar))) {
                        fence_after();
                        layer1(b ^ 1);
                        early = true;
                    }
                    if (mbar_test(&S.sm.ev[3], par)) break;
                    if (globaltimer() - t0 > A.wait_ns) {
                        ok = false;
                        break;
                    }
                }
                fence_after();
                if (!ok) break;
                // ---- de = dZ1 W1[0:16]^T and dW1 ----
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) {
                    mma(tb + COL_DE, h2_k + kstep(kk), w1_m + mnstep(kk), idesc_bf16(128, 16, 0, 1), kk > 0);
                    mma(tb + COL_DW1, h2_m + mnstep(kk), x_m + (b ? kPanelStep : 0) + mnstep(kk), idesc_bf16(128, 64, 1, 1),
                        acc_w | (kk > 0));
                    if (PEX)
                        mma(tb + COL_DW1T, h2_m + mnstep(kk), tp_m + (b ? 4u : 2u) + mnstep(kk),
                            idesc_bf16(128, 16, 1, 1), acc_w | (kk > 0));
                }
                commit(&S.sm.de);
            }
            if (!ok) atomicExch(&S.sm.abort, 1);
            commit(&S.sm.fin);   // every MMA is complete before the CTA goes on (bounded)
            mbar_wait(&S.sm.fin, 0, A.wait_ns);
        }
        __syncwarp();
    } else {
        // ------------------------------- consumers -------------------------------
        // thread: row r = 32 (warp % 4) + lane (its TMEM lane), column half hc = warp / 4.  A warp only ever
        // overwrites what the MMA batches it has waited for were the last to read, so the consumers need
        // no barrier among themselves.
        const int r = tid & (TM - 1), hc = tid >> 7;
        const uint32_t tb = S.sm.tmem_base;
        float db3_part[3] = {0.0f, 0.0f, 0.0f};
        int i = 0;
        auto wait = [&](uint64_t *bar, uint32_t par) -> bool {
            ok = __all_sync(0xffffffffu, mbar_wait(bar, par, A.wait_ns));
            fence_after();
            return ok;
        };
        auto signal = [&](uint64_t *bar) {   // my warp's operands are written and its accumulators read
            fence_async_smem();
            fence_before();
            __syncwarp();
            if ((tid & 31) == 0) mbar_arrive(bar);
        };
        // de[0:12] of tile j for the producers' scatter, when the tile that had the slot is scattered; X[j & 1] is
        // the producers' again
        auto stage_de = [&](int j) -> bool {
            if (!wait(&S.sm.de, j & 1) || (j >= 2 && !wait(&S.sm.sc[j & 1], ((j >> 1) - 1) & 1))) return false;
            float de[16];
            tmem_ld16(taddr(tb, warp, COL_DE), de);
            *de_slot(S.dout, j & 1, r, 0) = make_float4(de[0], de[1], de[2], de[3]);
            *de_slot(S.dout, j & 1, r, 1) = make_float4(de[4], de[5], de[6], de[7]);
            *de_slot(S.dout, j & 1, r, 2) = make_float4(de[8], de[9], de[10], de[11]);
            fence_before();
            __syncwarp();
            if ((tid & 31) == 0) mbar_arrive(&S.sm.empty[j & 1]);
            return true;
        };
        for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++i) {
            const int b = i & 1;
            const uint32_t par = i & 1;
            // (no abort-flag test: a failed producer leaves these waits unsatisfied for every thread)
            if (!wait(&S.sm.full[b], (i >> 1) & 1) || !wait(&S.sm.z1, par)) break;
            // ---- epilogue 1: H1 = relu(Z1), my 64 columns ----
            // (The epilogues are bound by the ALU pipe.  So the ReLU is taken, and its derivative looked up,
            // two values at a time on the BF16 operand: 5 ALU instructions a hidden unit and sample in
            // all, against 12 with FP32 compares, selects and a bit mask.  z > 0 and bf16(z) > 0 differ
            // only below 2^-134.)
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                float z[32];
                tmem_ld32(taddr(tb, warp, COL_Z1 + 64 * hc + 32 * g), z);
#pragma unroll
                for (int k = 0; k < 32; k += 8) *panel_chunk(S.h1 + hc * kPanelBytes, r, 32 * g + k) = pack8_relu(z + k);
            }
            // dout = dL/dc c (1 - c), formed by the producers, into the dout panel: the operand of
            // dH2 (issued with layer 2), of dW3 and, through its constant-1 column, of db2
            if (hc == 0) {
                const float d0 = S.sm.dc[b][r][0], d1 = S.sm.dc[b][r][1], d2 = S.sm.dc[b][r][2];
                db3_part[0] += d0;
                db3_part[1] += d1;
                db3_part[2] += d2;
                uint2 q;
                q.x = pack_bf16(d0, d1);
                q.y = pack_bf16(d2, 1.0f);
                *reinterpret_cast<uint2 *>(S.dout + panel_offset(r, 0)) = q;
            }
            signal(&S.sm.ev[0]);
            // ---- the tile before: its de, while layer 2 runs ----
            if (i > 0 && hc == 1 && !stage_de(i - 1)) break;
            // ---- epilogue 2: H2 = relu(Z2 + b2), then dZ2 = dH2 [Z2 + b2 > 0], my 64 columns ----
            if (!wait(&S.sm.z2, par)) break;
            uint4 hw[8];   // my row of H2, then of H1, for the ReLU's derivative
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                const int col = 64 * hc + 32 * g;
                float z[32];
                tmem_ld32(taddr(tb, warp, COL_Z2 + col), z);
#pragma unroll
                for (int k = 0; k < 32; k += 4) {
                    const float4 bb = *reinterpret_cast<const float4 *>(&S.sm.b2[col + k]);
                    z[k] += bb.x;
                    z[k + 1] += bb.y;
                    z[k + 2] += bb.z;
                    z[k + 3] += bb.w;
                }
#pragma unroll
                for (int k = 0; k < 32; k += 8) {
                    hw[4 * g + k / 8] = pack8_relu(z + k);
                    *panel_chunk(S.h2 + hc * kPanelBytes, r, 32 * g + k) = hw[4 * g + k / 8];
                }
            }
            signal(&S.sm.ev[1]);
            auto masked = [&](uint32_t col, unsigned char *dz) {   // dz = dh where h > 0
#pragma unroll
                for (int g = 0; g < 2; ++g) {
                    float z[32];
                    tmem_ld32(taddr(tb, warp, col + 64 * hc + 32 * g), z);
#pragma unroll
                    for (int k = 0; k < 32; k += 8)
                        *panel_chunk(dz + hc * kPanelBytes, r, 32 * g + k) = pack8_where(hw[4 * g + k / 8], z + k);
                }
            };
            masked(COL_Z1, S.dz2);
            signal(&S.sm.ev[2]);
            // ---- dZ1 = dH1 [Z1 > 0], over H2 ----
#pragma unroll
            for (int c = 0; c < 8; ++c) hw[c] = *panel_chunk(S.h1 + hc * kPanelBytes, r, 8 * c);
            if (!wait(&S.sm.dh, par)) break;
            masked(COL_Z2, S.h2);
            signal(&S.sm.ev[3]);
        }
        if (ok && i > 0) {   // the last tile's de; all wait for the last MMAs
            if (hc == 1) stage_de(i - 1);
            else wait(&S.sm.de, (i - 1) & 1);
        }
        ntile_mine = i;
        if (!ok) atomicExch(&S.sm.abort, 1);
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) {
            const float sum = warp_sum(db3_part[ch]);
            if ((tid & 31) == 0) atomicAdd(&S.sm.db3[ch], sum);
        }
    }

    fence_before();
    __syncthreads();
    fence_after();
    const bool failed = S.sm.abort != 0;
    if (failed) {
        if (tid == 0) atomicOr(&A.hdr->flags, 2);
        // forward: MMAs may still be running: all that were issued are complete before TMEM is freed (bounded)
        if (!BWD && (tid == 0 || tid == TM)) {
            commit(&S.sm.stop[tid / TM]);
            mbar_wait(&S.sm.stop[tid / TM], 0, A.wait_ns);
        }
    }
    if (BWD && !failed && tid < NC && ntile_mine > 0) {
        const uint32_t tb = S.sm.tmem_base;
        const int r = tid & (TM - 1), hc = tid >> 7;
        float *gW1 = A.grad_mlp, *gB1 = gW1 + D::IN * HID, *gW2 = gB1 + HID, *gB2 = gW2 + HID * HID;
        float *gW3 = gB2 + HID, *gB3 = gW3 + HID * 3;
        // dW2^T: lane = output unit r, columns = input units (64 per half); column 128 + 3 = db2
#pragma unroll 1
        for (int c = 0; c < 2; ++c) {
            const int col = 64 * hc + 32 * c;
            float v[32];
            tmem_ld32(taddr(tb, warp, COL_DW2T + col), v);
#pragma unroll
            for (int k = 0; k < 32; ++k) atomicAdd(gW2 + (col + k) * HID + r, v[k]);
        }
        // [dW1 | db1]^T: lane = hidden unit r, columns = X columns (BIAS = bias), 32 per half
        {
            float v[32];
            tmem_ld32(taddr(tb, warp, COL_DW1 + 32 * hc), v);
#pragma unroll
            for (int k = 0; k < 32; ++k) {
                const int kin = 32 * hc + k;
                if (kin < D::NMAIN) atomicAdd(gW1 + kin * HID + r, v[k]);
                else if (kin == D::BIAS) atomicAdd(gB1 + r, v[k]);
            }
        }
        if constexpr (PEX) {   // dW1 tail^T: columns = inputs NMAIN..IN-1
            float v[16];
            tmem_ld16(taddr(tb, warp, COL_DW1T), v);
            if (hc == 0)
#pragma unroll
                for (int t = 0; t < D::NTAIL; ++t) atomicAdd(gW1 + (D::NMAIN + t) * HID + r, v[t]);
        }
        float v[16];
        tmem_ld16(taddr(tb, warp, COL_DW3), v);
        if (hc == 0) {
            atomicAdd(gW3 + r * 3 + 0, v[0]);
            atomicAdd(gW3 + r * 3 + 1, v[1]);
            atomicAdd(gW3 + r * 3 + 2, v[2]);
        }
        tmem_ld16(taddr(tb, warp, COL_DW2T + 128), v);
        if (hc == 0) atomicAdd(gB2 + r, v[3]);
        if (tid < 3) atomicAdd(gB3 + tid, S.sm.db3[tid]);
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 0) tmem_dealloc(S.sm.tmem_base, NCOLS);
}

template <typename FeatT, bool BWD, bool PEX, bool PK>
void launch_tc(const RenderArgs &A, int kind, cudaStream_t s) {
    auto kern = fine_colour_tc_kernel<FeatT, BWD, PEX, PK>;
    const int bytes = (int)smem_bytes(BWD);
    ensure_smem(reinterpret_cast<const void *>(kern), bytes);
    ProfScope ps_(kind, s);
    kern<<<num_sms(), kThreads<BWD>, bytes, s>>>(A);
}

template <bool BWD>
void launch_tc_any(const RenderArgs &A, cudaStream_t s) {
    const int kind = BWD ? DVGO_K_FINE_COLOUR_BWD : DVGO_K_FINE_COLOUR_FWD;
    const bool bf = A.cdtype == DVGO_DTYPE_BF16, pex = A.nfreq_pos > 0;
    if (A.packed) {
        if (bf && pex) launch_tc<__nv_bfloat16, BWD, true, true>(A, kind, s);
        else if (bf) launch_tc<__nv_bfloat16, BWD, false, true>(A, kind, s);
        else if (pex) launch_tc<float, BWD, true, true>(A, kind, s);
        else launch_tc<float, BWD, false, true>(A, kind, s);
    } else {
        if (bf && pex) launch_tc<__nv_bfloat16, BWD, true, false>(A, kind, s);
        else if (bf) launch_tc<__nv_bfloat16, BWD, false, false>(A, kind, s);
        else if (pex) launch_tc<float, BWD, true, false>(A, kind, s);
        else launch_tc<float, BWD, false, false>(A, kind, s);
    }
}

}  // namespace

int launch_fine_colour_fwd_tc(const RenderArgs &A, cudaStream_t s) {
    launch_tc_any<false>(A, s);
    return DVGO_OK;
}

int launch_fine_colour_bwd_tc(const RenderArgs &A, cudaStream_t s) {
    launch_tc_any<true>(A, s);
    return DVGO_OK;
}

}  // namespace dvgo
