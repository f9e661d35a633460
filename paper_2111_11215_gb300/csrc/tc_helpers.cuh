// tc_helpers.cuh -- 5th-generation tensor core (tcgen05) building blocks for sm_103a, written as
// inline PTX: shared-memory matrix descriptors for the 128-byte-swizzled canonical layouts, the
// BF16 instruction descriptor, MMA issue (A from shared or from tensor memory) / commit, TMEM
// allocation, loads and stores, mbarriers with bounded waits, bulk copies.
//
// Operand tiles live in "panels": 128 rows x 128 bytes (64 BF16 values per row), 1024-byte
// aligned, with the 128-byte swizzle applied to every 8-row (1024-byte) group: the 16-byte chunk
// c of row r is stored at chunk c ^ (r & 7).  A matrix with more than 64 columns is a sequence of
// panels 16 KiB apart.  The same panel serves as a K-major operand (rows = M or N, columns = K)
// and as an MN-major operand (rows = K, columns = M or N); only the descriptor differs.
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

namespace dvgo {
namespace tc {

constexpr uint32_t kPanelBytes = 128 * 128;   // 128 rows x 128 bytes
constexpr uint32_t kGroupBytes = 1024;        // 8 rows x 128 bytes (one swizzle atom)

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Byte offset inside a panel of element (row, col) (BF16), with the 128-byte swizzle.
__device__ __forceinline__ uint32_t panel_offset(int row, int col) {
    uint32_t chunk = (uint32_t)(col >> 3) ^ (uint32_t)(row & 7);
    return (uint32_t)row * 128u + (chunk << 4) + (uint32_t)(col & 7) * 2u;
}

// Shared-memory matrix descriptor (tcgen05 format): start address, leading- and stride-
// dimension byte offsets, fixed version bits 0b001 at [46, 49), 128-byte swizzle mode (2) at
// [61, 64).
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// K-major operand (rows = M or N, K along the row), MMA k-step kk (16 BF16 = 32 bytes):
// panel = kk / 4, byte offset 32 (kk % 4) inside the swizzled row; 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t desc_kmajor(uint32_t base, int kk) {
    return sdesc(base + (uint32_t)(kk >> 2) * kPanelBytes + (uint32_t)(kk & 3) * 32u, 16u, kGroupBytes);
}

// MN-major operand (rows = K, M or N along the row, 64 per panel; panels 16 KiB apart),
// MMA k-step kk = 16 rows = two 8-row groups.
__device__ __forceinline__ uint64_t desc_mnmajor(uint32_t base, int kk) {
    return sdesc(base + (uint32_t)kk * 2u * kGroupBytes, kPanelBytes, kGroupBytes);
}

// What to add to a descriptor of k-step 0 for k-step kk (the address field counts 16-byte units), and for
// the next panel.
constexpr uint64_t kPanelStep = kPanelBytes >> 4;
__host__ __device__ constexpr uint64_t kstep(int kk) { return (uint64_t)(kk >> 2) * kPanelStep + (uint64_t)(kk & 3) * 2u; }
__host__ __device__ constexpr uint64_t mnstep(int kk) { return (uint64_t)kk * (2u * kGroupBytes >> 4); }

// Instruction descriptor, kind::f16: D = F32 (bits 4-5 = 1), A = B = BF16 (bits 7-9, 10-12 = 1),
// A / B major-ness (bit 15 / 16: 1 = MN-major), N >> 3 at bits 17-22, M >> 4 at bits 24-28.
__device__ __forceinline__ uint32_t idesc_bf16(int M, int N, int a_mn, int b_mn) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a_mn << 15) | ((uint32_t)b_mn << 16) |
           ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// D[tmem] (+)= A * B^T (single CTA), issued by one thread.
__device__ __forceinline__ void mma(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}

// D[tmem] (+)= A * B^T with A read from tensor memory: M = 128 rows on the 128 TMEM lanes, the
// k-step's 16 BF16 values of a row packed two per 32-bit column (lower index in the low half), so
// 8 consecutive columns starting at a_tmem; B from shared memory as in mma().
__device__ __forceinline__ void mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t idesc,
                                       uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}\n" ::"r"(d_tmem),
        "r"(a_tmem), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}

// Arrive once on the mbarrier when all previously issued MMAs of this thread complete.
__device__ __forceinline__ void commit(uint64_t *mbar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(mbar))
                 : "memory");
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// Makes generic-proxy shared-memory writes visible to the tensor core (async proxy).
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// TMEM allocation by one full warp; the base address is written to *dst (shared memory).
__device__ __forceinline__ void tmem_alloc(uint32_t *dst, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst)), "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t base, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(ncols) : "memory");
}

// 32 consecutive FP32 columns of this thread's TMEM lane (warp w reads lanes 32(w%4)..+31).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// Two runs of 16 columns, waited for once.
__device__ __forceinline__ void tmem_ld16x2(uint32_t ta, float (&v)[16], uint32_t tb, float (&u)[16]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%32];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%33];\n\t"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=&r"(r[0]), "=&r"(r[1]), "=&r"(r[2]), "=&r"(r[3]), "=&r"(r[4]), "=&r"(r[5]), "=&r"(r[6]), "=&r"(r[7]),
          "=&r"(r[8]), "=&r"(r[9]), "=&r"(r[10]), "=&r"(r[11]), "=&r"(r[12]), "=&r"(r[13]), "=&r"(r[14]), "=&r"(r[15]),
          "=&r"(r[16]), "=&r"(r[17]), "=&r"(r[18]), "=&r"(r[19]), "=&r"(r[20]), "=&r"(r[21]), "=&r"(r[22]), "=&r"(r[23]),
          "=&r"(r[24]), "=&r"(r[25]), "=&r"(r[26]), "=&r"(r[27]), "=&r"(r[28]), "=&r"(r[29]), "=&r"(r[30]), "=&r"(r[31])
        : "r"(ta), "r"(tb)
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        v[i] = __uint_as_float(r[i]);
        u[i] = __uint_as_float(r[16 + i]);
    }
}

__device__ __forceinline__ void tmem_ld24(uint32_t taddr, float (&v)[24]) {
    uint32_t r[24];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%24];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%16,%17,%18,%19,%20,%21,%22,%23}, [%25];\n\t"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=&r"(r[0]), "=&r"(r[1]), "=&r"(r[2]), "=&r"(r[3]), "=&r"(r[4]), "=&r"(r[5]), "=&r"(r[6]), "=&r"(r[7]),
          "=&r"(r[8]), "=&r"(r[9]), "=&r"(r[10]), "=&r"(r[11]), "=&r"(r[12]), "=&r"(r[13]), "=&r"(r[14]), "=&r"(r[15]),
          "=&r"(r[16]), "=&r"(r[17]), "=&r"(r[18]), "=&r"(r[19]), "=&r"(r[20]), "=&r"(r[21]), "=&r"(r[22]), "=&r"(r[23])
        : "r"(taddr), "r"(taddr + 16u)
        : "memory");
#pragma unroll
    for (int i = 0; i < 24; ++i) v[i] = __uint_as_float(r[i]);
}

// 16 consecutive 32-bit columns of this thread's TMEM lane from registers; the stores are
// complete (visible to a later MMA after a thread sync with the tcgen05 fences) once
// tmem_wait_st() returns.
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
            taddr),
        "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
        "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
        : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&v)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(v[0]), "r"(v[1]),
                 "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                 : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// TMEM address of (lane base of this warp, column).
__device__ __forceinline__ uint32_t taddr(uint32_t base, int warp, int col) {
    return base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)col;
}

__device__ __forceinline__ void mbar_init(uint64_t *mbar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(mbar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ uint64_t globaltimer() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Wait for the mbarrier phase with the given parity; gives up after limit_ns nanoseconds of the
// global timer (default 2 s) and returns false.
__device__ __forceinline__ bool mbar_wait(uint64_t *mbar, uint32_t parity,
                                          unsigned long long limit_ns = 2000000000ull) {
    uint32_t addr = smem_u32(mbar);
    uint64_t t0 = globaltimer();
    for (;;) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.b32 %0, 1, 0, p;\n\t}\n"
            : "=r"(done)
            : "r"(addr), "r"(parity)
            : "memory");
        if (done) return true;
        if (globaltimer() - t0 > limit_ns) return false;
    }
}

// Has the phase with the given parity completed?
__device__ __forceinline__ bool mbar_test(uint64_t *mbar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(smem_u32(mbar)), "r"(parity)
        : "memory");
    return done != 0;
}

// Barrier `id` of n threads (whole warps) that tells all of them whether ok held for every one.  Waits of a group of
// warps run out one by one: a warp whose wait did goes on to the group's next such barrier without
// waiting again or issuing anything, so that none is left alone at a barrier, which has no limit.
__device__ __forceinline__ bool barrier_all(int id, int n, bool ok) {
    uint32_t all;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 q, %3, 0;\n\t"
        "barrier.cta.red.and.pred p, %1, %2, q;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(all)
        : "r"(id), "r"(n), "r"((uint32_t)ok)
        : "memory");
    return all != 0;
}

__device__ __forceinline__ void mbar_arrive(uint64_t *mbar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(mbar)) : "memory");
}

// Bulk copies (cp.async.bulk, 16-byte aligned addresses, size a multiple of 16).  Shared ->
// global, tracked by the issuing thread's bulk groups: commit after the copy; wait_read before
// the source is overwritten, wait_all before the kernel exits.
__device__ __forceinline__ void bulk_store(void *gdst, const void *ssrc, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(gdst), "r"(smem_u32(ssrc)),
                 "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// Global -> shared, completing on an mbarrier: the issuing thread arrives on it with the expected
// byte count first (one of the barrier's arrivals).
__device__ __forceinline__ void bulk_load(void *sdst, const void *gsrc, uint32_t bytes, uint64_t *mbar) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(mbar)), "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(sdst)),
                 "l"(gsrc), "r"(bytes), "r"(smem_u32(mbar))
                 : "memory");
}

// v rounded to BF16 (to nearest, ties to even) and back to FP32.
__device__ __forceinline__ float bf16_round(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t *>(&v);
}

// Store 8 consecutive BF16 values (one 16-byte chunk) of row `row`, columns [col, col + 8).
__device__ __forceinline__ void panel_store8(unsigned char *panel, int row, int col, const float *v) {
    uint4 q;
    q.x = pack_bf16(v[0], v[1]);
    q.y = pack_bf16(v[2], v[3]);
    q.z = pack_bf16(v[4], v[5]);
    q.w = pack_bf16(v[6], v[7]);
    *reinterpret_cast<uint4 *>(panel + panel_offset(row, col)) = q;
}

// max(., 0) of two BF16 values (0 for a NaN, as fmaxf gives).
__device__ __forceinline__ uint32_t relu_bf16(uint32_t h) {
    uint32_t r;
    asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(h), "r"(0u));
    return r;
}

// 16-byte chunk of a panel: row, columns [col, col + 8).
__device__ __forceinline__ uint4 *panel_chunk(unsigned char *panel, int row, int col) {
    return reinterpret_cast<uint4 *>(panel + panel_offset(row, col));
}

// Eight values as BF16: max(v, 0); and v where h, a chunk of such values, is above 0, 0 elsewhere.
__device__ __forceinline__ uint4 pack8_relu(const float *v) {
    return make_uint4(relu_bf16(pack_bf16(v[0], v[1])), relu_bf16(pack_bf16(v[2], v[3])),
                      relu_bf16(pack_bf16(v[4], v[5])), relu_bf16(pack_bf16(v[6], v[7])));
}
__device__ __forceinline__ uint4 pack8_where(const uint4 &h, const float *v) {
    // h holds no negative values: adding 0x7fff sets the top bit of every half that is not 0, and the byte
    // permutation spreads it over the half
    auto where = [](uint32_t hw, float a, float b) {
        uint32_t m;
        asm("prmt.b32 %0, %1, 0, 0xbb99;" : "=r"(m) : "r"(hw + 0x7fff7fffu));
        return pack_bf16(a, b) & m;
    };
    return make_uint4(where(h.x, v[0], v[1]), where(h.y, v[2], v[3]), where(h.z, v[4], v[5]), where(h.w, v[6], v[7]));
}

// Eight FP32 values as three BF16 chunks of 16 bytes: hi, mid, lo.
__device__ __forceinline__ void split8(const float *v, uint4 (&q)[3]) {
    uint32_t w[3][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float a = v[2 * i], b = v[2 * i + 1];
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            w[s][i] = pack_bf16(a, b);
            a = __fsub_rn(a, __uint_as_float(w[s][i] << 16));
            b = __fsub_rn(b, __uint_as_float(w[s][i] & 0xffff0000u));
        }
    }
#pragma unroll
    for (int s = 0; s < 3; ++s) q[s] = make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
}

// A split operand of KB 16-column blocks a term: block (term s, kb) is number s KB + kb, four to a panel.
// 16-byte chunk c (columns 8 c ..) of row `row`, and what to add to a K-major descriptor for a block.
template <int KB>
__device__ __forceinline__ uint4 *split_chunk(unsigned char *base, int s, int row, int c) {
    const int q = s * KB + (c >> 1);
    return reinterpret_cast<uint4 *>(base + (q >> 2) * kPanelBytes + panel_offset(row, (q & 3) * 16 + (c & 1) * 8));
}

}  // namespace tc
}  // namespace dvgo
