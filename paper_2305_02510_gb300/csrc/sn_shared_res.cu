// The shared dense integer network (see sn_shared.cu) when every block holds
// one 128 x 128 tile of trains x post-neurons for the whole launch.
//
// What bounds the form of sn_shared.cu is not the tensor pipe but the bytes that
// each SM takes in and moves through shared memory: 32 KiB of operands per 128 pre-
// neurons, read again by the MMA (64 KiB through shared memory, at least 512
// cycles at 128 bytes a cycle; 680 measured, against 294 of the MMA).  Here the
// spike operand never touches shared memory: spikes travel as bits (a sixteenth
// of the FP8 bytes with their tags), and the warps that own the tile's rows
// expand them into tensor memory, from which the MMA takes its A operand.  Shared
// memory holds only weights, eight 16 KiB stages deep, loaded by TMA across the
// steps without a pause.
//
// A bit becomes the E4M3 byte 0x40 = 2.0: the word with the bits of 32 neurons
// gives eight operand words by a shift and a mask each, word c taking the bits
// 8 i + c (i = 0..3).  (The integer pipe is the busiest unit of these warps; at
// this bit position all but one of the shifts are left shifts, which run as
// multiplications on the other pipe.)  The weights are stored in that order of K
// (wt_res_pos), so the sums are the same integers, times two, exact in FP32.
//
// Sixteen warps own the rows: warp w the TMEM lane quarter w % 4 (a lane is a
// train), and for the state update the 32 columns 32 (w / 4).  The four warps of
// part w / 4 expand every fourth K block, always into operand stage w / 4 (so a
// stage's barrier is never more than one phase away from its waiter).  Warp 16
// issues the TMA loads, warp 17 the MMAs.  Between its K blocks a thread draws
// the Poisson input of its own train and columns; after the last MMA it applies
// the LIF rule to them (V and r stay in TMEM) and stores its spike word with the
// step's number beside it.  That is all a step's synchronisation: no grid
// barrier, the words of a K block are waited for where they are expanded, the
// block's own first.  A slot (two, by the step's parity) is stored again only
// after the words of the step between have come from every tile of these trains,
// and a tile stores a step's words after its K loop, so no reader is left.
// The words lie as they are read: [parity][K block][train][4].
//
// 8192 neurons x 256 trains (128 blocks), 40 steps: 1266 -> 857 us (31.6 -> 21.4 us
// a step).  No single part bounds it: left out one at a time, the weights' loads
// give 0.6 us of a step, the draws 0.9, the expansion's shifts 1.2, loads and draws
// together 1.9; the MMAs alone would take 8.  What is left is the chain from a stage
// that falls free over the waiting owners' stores back to the MMA (a vote in front of
// each MMA instead of behind it: 2.9 us), and the exchange of the words.
//
// TMEM: accumulator columns 0..127, V 128..255, r 256..383, four operand stages of
// 32 columns at 384.  Every wait is bounded as in sn_shared.cu.
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "sn_shared.cuh"
#include "sn_tc.cuh"

namespace sn {

namespace {

constexpr int kStagesW = 8;                    // weight stages in shared memory (a power of two)
constexpr int kStagesA = 4;                    // operand stages in TMEM
constexpr int kStageW = kTN * kTK;             // 16 KiB
constexpr int kOwners = 16;                    // warps that own rows
constexpr int kThreadsRes = 32 * (kOwners + 2);
constexpr uint32_t kVCol = 128, kRCol = 256, kACol = 384;
static_assert(kTM == 128 && kTN == 128 && kTK == 128, "a K block is the spike bits of one tile of neurons");

__device__ __forceinline__ ulonglong2 ld_words2(const unsigned long long *p) {
    ulonglong2 v;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p) : "memory");
    return v;
}

// The four spike words of each lane's row and a K block, once all carry `tag`.
// While some lane's are missing, the first such lane alone looks for its own and
// the others look again when it has them: polled by every lane, the words took
// most of the L2's bandwidth.  Bounded; false when it gave up.
__device__ __forceinline__ bool wait_words(const unsigned long long *src, unsigned tag, ulonglong2 &w01, ulonglong2 &w23,
                                           int lane, Control *ctl) {
    for (;;) {
        auto there = [&]() {
            return (unsigned)(w01.x >> 32) == tag && (unsigned)(w01.y >> 32) == tag && (unsigned)(w23.x >> 32) == tag &&
                   (unsigned)(w23.y >> 32) == tag;
        };
        const unsigned missing = __ballot_sync(0xffffffffu, !there());
        if (!missing) return true;
        bool ok = true;
        if (lane == __ffs(missing) - 1) {
            for (unsigned spins = 0, began = 0; !there();) {
                if ((++spins & 63u) == 0) {
                    const unsigned now = (unsigned)(global_timer_ns() >> 10);       // units of 1.024 us
                    if (spins == 64u) began = now;
                    if (ld_status(ctl) != 0) ok = false;
                    else if (now - began > (unsigned)(kWaitNs >> 10)) {
                        atomicCAS(&ctl->status, 0, (int)SN_ETIMEOUT);
                        ok = false;
                    }
                    if (!ok) break;
                }
                w01 = ld_words2(src);
                w23 = ld_words2(src + 2);
            }
        }
        if (!__all_sync(0xffffffffu, ok)) return false;
        if (!there()) {
            w01 = ld_words2(src);
            w23 = ld_words2(src + 2);
        }
    }
}

// lif_update_i32 in 32 bits: leak and reset are below 2^24 in magnitude, so the
// leak step cannot wrap (v > reset before a subtraction, v < reset before an
// addition), nor can acc + ext (at most 2^25); the last addition's overflow shows in
// the sign of `wrapped`.
__device__ __forceinline__ bool lif_update_small(int &v, int &rr, int in, const int4 &par, int &wrapped) {
    const int u = v > par.z ? max(v - par.y, par.z) : min(v + par.y, par.z);
    const int w = u + in;
    wrapped |= (u ^ w) & (in ^ w);
    const bool fire = w > par.x && rr == 0;
    v = fire ? par.z : w;
    rr = fire ? par.w : max(rr - 1, 0);
    return fire;
}

__global__ void __launch_bounds__(kThreadsRes, 1)
shared_res_kernel(const __grid_constant__ CUtensorMap tmW, SharedArgs a) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t fullW[kStagesW], emptyW[kStagesW], fullA[kStagesA], emptyA[kStagesA], accbar, accfree;
    __shared__ int4 sPar[kTN];                         // threshold, leak, reset, refractory
    __shared__ int sAmp[kTN];
    __shared__ __align__(16) unsigned sRate[kTN];
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t sbase = smem_addr(smem);
    const int m0 = (blockIdx.x % a.tiles_m) * kTM, n0 = (blockIdx.x / a.tiles_m) * kTN;

    if (threadIdx.x == 0) {
        auto init = [](uint64_t *b, int n) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" :: "r"(smem_addr(b)), "r"(n));
        };
        for (int s = 0; s < kStagesW; ++s) { init(&fullW[s], 1); init(&emptyW[s], 1); }
        for (int s = 0; s < kStagesA; ++s) { init(&fullA[s], 4); init(&emptyA[s], 1); }
        init(&accbar, 1);
        init(&accfree, kOwners);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        s_abort = 0;
    }
    if (warp == kOwners) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n"
                     :: "r"(smem_addr(&s_tmem)), "r"(512u));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    for (int c = threadIdx.x; c < kTN; c += kThreadsRes) {
        const int j = n0 + c;
        sPar[c] = make_int4(a.th[j], a.lk[j], a.rs[j], a.R[j]);
        sAmp[c] = a.pamp[j];
        sRate[c] = a.prate[j];
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = s_tmem;
    const int quarter = warp & 3, part = warp >> 2;
    const int row = m0 + quarter * 32 + lane;          // this thread's train
    const uint32_t trow = tmem + ((uint32_t)(quarter * 32) << 16);
    const int c0 = part * 32;                          // its 32 columns of the tile
    // the K blocks in a cycle from the block's own, which is there first
    const int kblocks = a.n / kTK, kb0 = n0 / kTK;
    unsigned issued = 0;                               // stages this thread has put through its ring
    unsigned long long my_spikes = 0;
    int wrapped = 0;                                   // negative: a state left int32

    if (warp < kOwners) {
        // the tile's state into TMEM for the whole launch
        for (int h = 0; h < 2; ++h) {
            const int c = c0 + h * 16;
            const int *Vp = a.V + (size_t)(n0 + c) * a.B + row;
            const int *rp = a.r + (size_t)(n0 + c) * a.B + row;
            uint32_t vv[16], rr[16];
#pragma unroll
            for (int q = 0; q < 16; ++q) {
                vv[q] = (uint32_t)__ldcg(Vp + (size_t)q * a.B);
                rr[q] = (uint32_t)__ldcg(rp + (size_t)q * a.B);
            }
            tmem_st16x2(trow + kVCol + c, trow + kRCol + c, vv, rr);
        }
        const unsigned long long key = a.pkey[row];
        const size_t part_words = (size_t)a.B * a.words;
        for (int s = 0; s < a.steps; ++s) {
            const int t = a.t0 + s;
            // words of step t - 1, stored by this launch with number s (or,
            // for its first step, prepared with number 0)
            const unsigned long long *words = a.bits + (size_t)((t + 1) & 1) * part_words + (size_t)row * 4;
            const unsigned tag = (unsigned)s;
            unsigned pb = 0;
            int drawn = 0;
            // four more of this thread's draws
            auto draw4 = [&]() {
                const uint4 thr = *(const uint4 *)(sRate + c0 + drawn);
                const unsigned j = (unsigned)(n0 + c0 + drawn), tt = (unsigned)t;
                pb |= ((unsigned)poisson_fires(key, tt, j, thr.x) | (unsigned)poisson_fires(key, tt, j + 1, thr.y) << 1 |
                       (unsigned)poisson_fires(key, tt, j + 2, thr.z) << 2 |
                       (unsigned)poisson_fires(key, tt, j + 3, thr.w) << 3) << drawn;
                drawn += 4;
            };
            auto block_words = [&](int i) {
                const int kb = kb0 + i >= kblocks ? kb0 + i - kblocks : kb0 + i;
                return words + (size_t)kb * 4 * a.B;
            };
            // this part's K blocks: those whose place in the launch's sequence of
            // stages is part modulo 4
            bool ok = true;
            int i = (part - (int)((unsigned)s * (unsigned)kblocks % kStagesA)) & (kStagesA - 1);
            ulonglong2 w01 = make_ulonglong2(0ull, 0ull), w23 = w01;
            if (i < kblocks) { w01 = ld_words2(block_words(i)); w23 = ld_words2(block_words(i) + 2); }
            for (; i < kblocks; i += kStagesA) {
                ok = wait_words(block_words(i), tag, w01, w23, lane, a.ctl);
                const unsigned y[4] = {(unsigned)w01.x, (unsigned)w01.y, (unsigned)w23.x, (unsigned)w23.y};
                if (i + kStagesA < kblocks) {
                    w01 = ld_words2(block_words(i + kStagesA));
                    w23 = ld_words2(block_words(i + kStagesA) + 2);
                }
                // expanded before the stage is free: only the stores are left then
                uint32_t e[2][16];
#pragma unroll
                for (int c = 0; c < 32; ++c) {
                    const unsigned x = y[c >> 3];
                    const int b = c & 7;
                    e[c >> 4][c & 15] = (b < 7 ? x << (6 - b) : x >> 1) & 0x40404040u;
                }
                // four draws a K block, while the MMAs of the others run
                if (drawn < 32) draw4();
                const unsigned round = ((unsigned)s * (unsigned)kblocks + (unsigned)i) / kStagesA;
                if (ok && round > 0) ok = mbar_wait_warp(smem_addr(&emptyA[part]), (round - 1) & 1u, a.ctl);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                tmem_st16(trow + kACol + (uint32_t)(part * 32), e[0]);
                tmem_st16(trow + kACol + (uint32_t)(part * 32 + 16), e[1]);
                tmem_st_wait();
                asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
                __syncwarp();
                if (lane == 0)
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" :: "r"(smem_addr(&fullA[part])) : "memory");
            }
            while (drawn < 32) draw4();
            if (!ok) { s_abort = 1; break; }
            if (!mbar_wait_warp(smem_addr(&accbar), (unsigned)s & 1u, a.ctl)) { s_abort = 1; break; }
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            unsigned bits = 0;
#pragma unroll 1
            for (int h = 0; h < 4; ++h) {
                const uint32_t col = (uint32_t)(c0 + 8 * h);
                uint32_t v[8], vv[8], rr[8];
                tmem_ld8x3(trow + col, trow + kVCol + col, trow + kRCol + col, v, vv, rr);
                if (h == 3) {
                    // the accumulator is read: the next step's MMAs may begin
                    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
                    __syncwarp();
                    if (lane == 0)
                        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" :: "r"(smem_addr(&accfree)) : "memory");
                }
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int c = c0 + 8 * h + q;
                    const int acc = __float2int_rn(__uint_as_float(v[q]) * 0.5f);
                    const int ext = ((pb >> (8 * h + q)) & 1u) ? sAmp[c] : 0;
                    const int4 par = sPar[c];
                    int vq = (int)vv[q], rq = (int)rr[q];
                    const bool fire = lif_update_small(vq, rq, acc + ext, par, wrapped);
                    vv[q] = (uint32_t)vq;
                    rr[q] = (uint32_t)rq;
                    bits |= (unsigned)fire << (8 * h + q);
                    if (q % 4 == 3) asm volatile("" ::: "memory");   // few parameters in registers at a time
                }
                tmem_st8x2(trow + kVCol + col, trow + kRCol + col, vv, rr);
            }
            const int word = (n0 + c0) >> 5;
            const unsigned long long tagged = ((unsigned long long)(unsigned)(s + 1) << 32) | bits;
            asm volatile("st.relaxed.gpu.global.u64 [%0], %1;"
                         :: "l"(a.bits + (size_t)(t & 1) * part_words + ((size_t)kb0 * a.B + row) * 4 + part), "l"(tagged) : "memory");
            a.raster[((size_t)(t % a.cap) * a.B + row) * a.words + word] = bits;
            my_spikes += (unsigned long long)__popc(bits);
        }
    } else if (warp == kOwners && lane == 0) {
        // weights, stage after stage, across the steps
        for (int s = 0; s < a.steps && !s_abort; ++s)
            for (int i = 0; i < kblocks; ++i, ++issued) {
                const int st = issued % kStagesW;
                const unsigned round = issued / kStagesW;
                if (round > 0 && !mbar_wait(smem_addr(&emptyW[st]), (round - 1) & 1u, a.ctl)) { s_abort = 1; break; }
                const uint32_t fb = smem_addr(&fullW[st]);
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" :: "r"(fb), "r"(kStageW) : "memory");
                const int kb = kb0 + i >= kblocks ? kb0 + i - kblocks : kb0 + i;
                tma_load_2d(sbase + st * kStageW, &tmW, kb * kTK, n0, fb);
            }
        // loads in flight land before the block's shared memory goes away
        for (unsigned i = issued > kStagesW ? issued - kStagesW : 0; i < issued; ++i)
            mbar_drain(smem_addr(&fullW[i % kStagesW]), (i / kStagesW) & 1u);
    } else if (warp == kOwners + 1) {
        // MMAs; the next barriers are looked at while those at hand run
        constexpr uint32_t idesc = idesc_e4m3_f32(kTM, kTN);
        const uint64_t wdesc = umma_desc_sw128(sbase);
        bool ready = false;
        for (int s = 0; s < a.steps; ++s) {
            if (s > 0 && !mbar_wait_warp(smem_addr(&accfree), (unsigned)(s - 1) & 1u, a.ctl)) { s_abort = 1; break; }
            int i = 0;
            for (; i < kblocks; ++i, ++issued) {
                const unsigned sw = issued % kStagesW, sa = issued % kStagesA;
                if (!ready && (!mbar_wait_warp(smem_addr(&fullW[sw]), (issued / kStagesW) & 1u, a.ctl) ||
                               !mbar_wait_warp(smem_addr(&fullA[sa]), (issued / kStagesA) & 1u, a.ctl))) {
                    s_abort = 1;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                mma_f8_block_ta(tmem, tmem + kACol + sa * 32, wdesc + sw * (kStageW / 16), idesc, i != 0,
                                smem_addr(&emptyA[sa]), smem_addr(&emptyW[sw]));
                const unsigned nx = issued + 1;
                ready = __all_sync(0xffffffffu, mbar_test(smem_addr(&fullW[nx % kStagesW]), (nx / kStagesW) & 1u) &
                                                    mbar_test(smem_addr(&fullA[nx % kStagesA]), (nx / kStagesA) & 1u));
            }
            if (i < kblocks) break;
            mma_commit(smem_addr(&accbar));
        }
        // MMAs issued complete before TMEM goes away
        for (unsigned i = issued > kStagesA ? issued - kStagesA : 0; i < issued; ++i)
            mbar_drain(smem_addr(&emptyA[i % kStagesA]), (i / kStagesA) & 1u);
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (warp < kOwners) {
        // the tile's state back to its neuron-major arrays
        for (int h = 0; h < 2; ++h) {
            const int c = c0 + h * 16;
            int *Vp = a.V + (size_t)(n0 + c) * a.B + row;
            int *rp = a.r + (size_t)(n0 + c) * a.B + row;
            uint32_t vv[16], rr[16];
            tmem_ld16x2(trow + kVCol + c, trow + kRCol + c, vv, rr);
#pragma unroll
            for (int q = 0; q < 16; ++q) {
                __stcg(Vp + (size_t)q * a.B, (int)vv[q]);
                __stcg(rp + (size_t)q * a.B, (int)rr[q]);
            }
        }
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    }
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (warp == kOwners)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" :: "r"(tmem), "r"(512u));
    if (wrapped < 0) atomicCAS(&a.ctl->status, 0, (int)SN_EOVERFLOW);
    if (my_spikes) {
        atomicAdd(&a.ctl->spikes, my_spikes);
        atomicAdd(&a.ctl->events, my_spikes * (unsigned long long)a.n);
    }
}

// Before a launch: every word's step number becomes 0 (a launch's own steps
// count from 1).
__global__ void shared_tags_kernel(unsigned long long *bits, long long count) {
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i < count) bits[i] &= 0xffffffffull;
}

constexpr size_t kResSmem = (size_t)kStagesW * kStageW + 1024;

}  // namespace

// Byte of pre-neuron i within its row of the weight operand.
int wt_res_pos(int i) { return (i & ~31) + 4 * (i & 7) + ((i >> 3) & 3); }

cudaError_t plan_shared_res(int n, int B, int *fits) {
    *fits = 0;
    int dev = 0, sms = 0, per = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    const void *f = (const void *)shared_res_kernel;
    if ((e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kResSmem)) != cudaSuccess) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, f, kThreadsRes, kResSmem)) != cudaSuccess) return e;
    // one block per SM: the whole of its TMEM
    *fits = per > 0 && (long long)(B / kTM) * (n / kTN) <= sms;
    return cudaSuccess;
}

cudaError_t launch_shared_res(const void *tmap_w, const SharedHostArgs &h, cudaStream_t s) {
    SharedArgs a = shared_args(h);
    const long long count = 2ll * a.B * a.words;
    shared_tags_kernel<<<(int)((count + 255) / 256), 256, 0, s>>>(a.bits, count);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    void *args[] = {(void *)tmap_w, (void *)&a};
    // cooperative: the blocks wait for one another's spikes, so all must be resident
    return cudaLaunchCooperativeKernel((const void *)shared_res_kernel, dim3(a.tiles), dim3(kThreadsRes), args, kResSmem, s);
}

}  // namespace sn
