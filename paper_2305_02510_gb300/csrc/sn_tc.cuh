// Blackwell (sm_103a) tensor-core building blocks shared by the kernels that
// run tcgen05 MMAs: shared-memory addresses, bounded mbarrier waits, 2-D TMA
// loads, the 128-byte-swizzle K-major matrix descriptor, instruction
// descriptors, MMA issue and commit, and TMEM loads and stores.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "sn_device.cuh"

namespace sn {

// Wall-clock limit of one mbarrier wait (nanoseconds of %globaltimer).
constexpr unsigned long long kWaitNs = 2000000000ull;

__device__ __forceinline__ uint32_t smem_addr(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n.reg .pred p;\n"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}

// Whether the phase of `parity` is complete, without waiting.
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n.reg .pred p;\n"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}

// Bounded wait for the phase of `parity`; false (status latched) on expiry or
// when another block has latched a status.
__device__ inline bool mbar_wait(uint32_t bar, uint32_t parity, Control *ctl) {
    unsigned long long t0 = 0;
    for (unsigned it = 0;; ++it) {
        if (mbar_try(bar, parity)) return true;
        if ((it & 255u) == 255u) {
            const unsigned long long now = global_timer_ns();
            if (t0 == 0) t0 = now;
            else if (now - t0 > kWaitNs) { atomicCAS(&ctl->status, 0, (int)SN_ETIMEOUT); return false; }
            if (ld_status(ctl) != 0) return false;
        }
    }
}

// Wait before shared memory or TMEM goes away, for a phase that copies or MMAs in
// flight will complete: bounded by the wall clock alone, whatever status is latched.
__device__ inline void mbar_drain(uint32_t bar, uint32_t parity) {
    unsigned long long t0 = 0;
    while (!mbar_try(bar, parity)) {
        const unsigned long long now = global_timer_ns();
        if (t0 == 0) t0 = now;
        else if (now - t0 > kWaitNs) return;
    }
}

// Both for a whole converged warp, with one answer for all its lanes.  Lanes that
// poll for themselves may disagree around a timeout or another block's status, some
// having seen the phase and others given up, and the warp-wide instructions that follow
// (elections, TMEM loads and stores) need all of them.  The votes also keep what
// follows uniform to the compiler: votes inside the polling loop, and a test behind the
// MMAs instead of before them, cost nothing (shared_res_kernel 864 us a run with lanes
// by themselves, 859 so, 974 with a vote after each lane's own wait).
__device__ __forceinline__ bool mbar_test_warp(uint32_t bar, uint32_t parity) {
    return __all_sync(0xffffffffu, mbar_test(bar, parity));
}
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, Control *ctl) {
    unsigned long long t0 = 0;
    for (unsigned it = 0;; ++it) {
        if (__all_sync(0xffffffffu, mbar_try(bar, parity))) return true;
        if ((it & 255u) == 255u) {
            const unsigned long long now = global_timer_ns();
            bool late = false;
            if (t0 == 0) t0 = now;
            else late = now - t0 > kWaitNs;
            if (late) atomicCAS(&ctl->status, 0, (int)SN_ETIMEOUT);
            if (__any_sync(0xffffffffu, late || ld_status(ctl) != 0)) return false;
        }
    }
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n"
        :: "r"(dst), "l"((uint64_t)map), "r"(x), "r"(y), "r"(bar) : "memory");
}

// Shared-memory matrix descriptor of a K-major tile with 128-byte swizzle:
// 8-row atoms of 128 B stacked every 1024 B (stride byte offset), start
// address in 16-byte units, descriptor version 1, layout SWIZZLE_128B (2).
__device__ __forceinline__ uint64_t umma_desc_sw128(uint32_t addr) {
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFFu);
    d |= (uint64_t)(16u >> 4) << 16;
    d |= (uint64_t)(1024u >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// The same swizzle for an MN-major tile of 16-bit elements (the operand's rows
// or columns contiguous, K in steps of 128 bytes): atoms of 64 MN elements x 8 K
// rows (1024 bytes) follow one another along K, the next 64 MN elements lie
// mn_stride bytes away.  A K step of 16 advances the address by 2048 bytes.
__device__ __forceinline__ uint64_t umma_desc_mn_sw128(uint32_t addr, uint32_t mn_stride) {
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFFu);
    d |= (uint64_t)(mn_stride >> 4) << 16;
    d |= (uint64_t)(1024u >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// Instruction descriptor of kind::f8f6f4: FP32 accumulator, A and B E4M3,
// both K-major, N = 128, M = 128.
__host__ __device__ constexpr uint32_t idesc_e4m3_f32(int m, int n) {
    return (1u << 4) | (0u << 7) | (0u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

// MMAs and commits are called by a whole converged warp and issued by the lane
// that elect.sync names (the same lane every time).  Called from a branch
// that one lane takes, their operands are not warp-uniform to the compiler: such
// an MMA took about 150 cycles to issue against 64 to run (128 x 128), and 95 to
// 125 with the election outside as a C++ branch; in this form the issue is hidden
// (66 to 72 cycles an MMA with one barrier look-ahead per four or eight).
__device__ __forceinline__ void mma_f8(uint32_t tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, int acc) {
    asm volatile(
        "{\n.reg .pred p, q;\nelect.sync _|q, 0xffffffff;\nsetp.ne.b32 p, %4, 0;\n"
        "@q tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n}\n"
        :: "r"(tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc));
}

// The four MMAs of a 128-byte K block with A in tensor memory (row = lane, four
// 8-bit elements of K per 32-bit column: an MMA of K = 32 takes 8 columns), and
// the commits of the block's two operand stages, under one election.
__device__ __forceinline__ void mma_f8_block_ta(uint32_t tmem, uint32_t ta, uint64_t bdesc, uint32_t idesc, int acc,
                                                uint32_t bar_a, uint32_t bar_b) {
    asm volatile(
        "{\n.reg .pred p, q, t;\n.reg .b32 a1, a2, a3;\n.reg .b64 b1, b2, b3;\n"
        "elect.sync _|q, 0xffffffff;\nsetp.ne.b32 p, %4, 0;\nsetp.eq.u32 t, 0, 0;\n"
        "add.u32 a1, %1, 8;\nadd.u32 a2, %1, 16;\nadd.u32 a3, %1, 24;\n"
        "add.u64 b1, %2, 2;\nadd.u64 b2, %2, 4;\nadd.u64 b3, %2, 6;\n"
        "@q tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], [%1], %2, %3, p;\n"
        "@q tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], [a1], b1, %3, t;\n"
        "@q tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], [a2], b2, %3, t;\n"
        "@q tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], [a3], b3, %3, t;\n"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%5];\n"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%6];\n}\n"
        :: "r"(tmem), "r"(ta), "l"(bdesc), "r"(idesc), "r"(acc), "r"(bar_a), "r"(bar_b) : "memory");
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("{\n.reg .pred q;\nelect.sync _|q, 0xffffffff;\n"
                 "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n"
                 :: "r"(bar) : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]),
          "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]),
          "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]),
          "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
}

// A 16-column TMEM load and the wait for it.
__device__ __forceinline__ void tmem_ld16(uint32_t ta, uint32_t (&a)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]), "=r"(a[7]),
          "=r"(a[8]), "=r"(a[9]), "=r"(a[10]), "=r"(a[11]), "=r"(a[12]), "=r"(a[13]), "=r"(a[14]),
          "=r"(a[15])
        : "r"(ta)
        : "memory");
}

// Two 16-column TMEM loads (this warp's lane quarter, one lane per thread)
// and the wait for both, in one statement so that no use of the registers
// can be scheduled before the wait.
__device__ __forceinline__ void tmem_ld16x2(uint32_t ta, uint32_t tb, uint32_t (&a)[16], uint32_t (&b)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%32];\n"
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%33];\n"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]), "=r"(a[7]),
          "=r"(a[8]), "=r"(a[9]), "=r"(a[10]), "=r"(a[11]), "=r"(a[12]), "=r"(a[13]), "=r"(a[14]),
          "=r"(a[15]), "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3]), "=r"(b[4]), "=r"(b[5]), "=r"(b[6]),
          "=r"(b[7]), "=r"(b[8]), "=r"(b[9]), "=r"(b[10]), "=r"(b[11]), "=r"(b[12]), "=r"(b[13]),
          "=r"(b[14]), "=r"(b[15])
        : "r"(ta), "r"(tb)
        : "memory");
}

// Three 8-column TMEM loads and the wait for all three.
__device__ __forceinline__ void tmem_ld8x3(uint32_t ta, uint32_t tb, uint32_t tc, uint32_t (&a)[8], uint32_t (&b)[8],
                                           uint32_t (&c)[8]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%24];\n"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8,%9,%10,%11,%12,%13,%14,%15}, [%25];\n"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%16,%17,%18,%19,%20,%21,%22,%23}, [%26];\n"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]), "=r"(a[7]),
          "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3]), "=r"(b[4]), "=r"(b[5]), "=r"(b[6]), "=r"(b[7]),
          "=r"(c[0]), "=r"(c[1]), "=r"(c[2]), "=r"(c[3]), "=r"(c[4]), "=r"(c[5]), "=r"(c[6]), "=r"(c[7])
        : "r"(ta), "r"(tb), "r"(tc)
        : "memory");
}

// Two 8-column TMEM stores and the wait for both.
__device__ __forceinline__ void tmem_st8x2(uint32_t ta, uint32_t tb, const uint32_t (&a)[8], const uint32_t (&b)[8]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%2,%3,%4,%5,%6,%7,%8,%9};\n"
        "tcgen05.st.sync.aligned.32x32b.x8.b32 [%1], {%10,%11,%12,%13,%14,%15,%16,%17};\n"
        "tcgen05.wait::st.sync.aligned;\n"
        :: "r"(ta), "r"(tb), "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]),
           "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]), "r"(b[7])
        : "memory");
}

// Two 16-column TMEM stores and the wait for both (the registers stay
// live until the stores have completed).
__device__ __forceinline__ void tmem_st16x2(uint32_t ta, uint32_t tb, const uint32_t (&a)[16],
                                            const uint32_t (&b)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17};\n"
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%1], "
        "{%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32,%33};\n"
        "tcgen05.wait::st.sync.aligned;\n"
        :: "r"(ta), "r"(tb), "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]),
           "r"(a[7]), "r"(a[8]), "r"(a[9]), "r"(a[10]), "r"(a[11]), "r"(a[12]), "r"(a[13]), "r"(a[14]),
           "r"(a[15]), "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]),
           "r"(b[7]), "r"(b[8]), "r"(b[9]), "r"(b[10]), "r"(b[11]), "r"(b[12]), "r"(b[13]), "r"(b[14]),
           "r"(b[15])
        : "memory");
}

// A 16-column TMEM store (this warp's lane quarter); tmem_st_wait waits for the
// stores issued before it.
__device__ __forceinline__ void tmem_st16(uint32_t ta, const uint32_t (&a)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};\n"
        :: "r"(ta), "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]),
           "r"(a[8]), "r"(a[9]), "r"(a[10]), "r"(a[11]), "r"(a[12]), "r"(a[13]), "r"(a[14]), "r"(a[15])
        : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory"); }

// Instruction descriptor of kind::f16 with BF16 A and B, FP32 accumulator,
// both K-major.
__host__ __device__ constexpr uint32_t idesc_bf16_f32(int m, int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

// The same with both operands MN-major.
__host__ __device__ constexpr uint32_t idesc_bf16_f32_mn(int m, int n) {
    return idesc_bf16_f32(m, n) | (1u << 15) | (1u << 16);
}

// Four MMAs of K = 16 under one election, the descriptors advancing by STEP
// 16-byte units (2: 32 bytes of a K-major row; 128: 16 rows of an MN-major tile).
// Descriptors put together for each MMA took the issuing warp about 100 cycles an
// MMA; a running sum from one descriptor costs next to nothing.
template <int STEP>
__device__ __forceinline__ void mma_bf16_x4(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t idesc, int acc) {
    asm volatile(
        "{\n.reg .pred p, q, t;\n.reg .b64 a1, a2, a3, b1, b2, b3;\n"
        "elect.sync _|q, 0xffffffff;\nsetp.ne.b32 p, %4, 0;\nsetp.eq.u32 t, 0, 0;\n"
        "add.u64 a1, %1, %5;\nadd.u64 a2, %1, %6;\nadd.u64 a3, %1, %7;\n"
        "add.u64 b1, %2, %5;\nadd.u64 b2, %2, %6;\nadd.u64 b3, %2, %7;\n"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], a1, b1, %3, t;\n"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], a2, b2, %3, t;\n"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], a3, b3, %3, t;\n}\n"
        :: "r"(tmem), "l"(ad), "l"(bd), "r"(idesc), "r"(acc), "n"(STEP), "n"(2 * STEP), "n"(3 * STEP));
}

}  // namespace sn
