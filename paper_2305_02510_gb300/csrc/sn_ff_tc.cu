// Tensor-core (tcgen05, BF16 operands, FP32 accumulation in TMEM) contractions
// of the feedforward network: the forward synaptic input and the backward's spike
// gradient (ff_tc_rows_kernel) and the weight gradient (ff_tc_dw_kernel).
// sn_ff.cu has the recurrences and the SIMT forms of these contractions.
//
// A delay-shifted contraction is a sum of plain GEMMs, one per delay d, with
// the weights restricted to the synapses of delay d (W_d = W masked by
// [D == d]) and the gradient or spike rows shifted by d steps (d * B rows):
//   gS[r][i] = sum_d sum_j gI[r + dB][j] W_d[i][j]
//   dW[i][j] = sum_d [D[i][j] = d] sum_r S[r - dB][i] gI[r][j]
// with r = t * B + b, rows outside [0, T * B) contributing zero (TMA fills
// coordinates outside a tensor with zeros).  FP32 weights and gradients enter
// as two-term BF16 splits x = hi + mid (about 16 significant bits), spikes as
// exact 0/1, and the cross products hi*hi + hi*mid + mid*hi are accumulated in
// FP32 (relative error near 2^-16 per product).
//
// The forward synaptic input I[r][j] = sum_d sum_i S[r - dB][i] W_d[i][j] multiplies
// 0/1 spikes by the three BF16 parts hi + mid + lo of every weight (an exact
// split), so every product is exact; one 64-input block of all delays at a time
// accumulates in TMEM, and the blocks are added in FP32 (round to nearest) in
// registers: only 48 MMA steps ever accumulate in TMEM.
//
// Warp 0 lane 0 issues TMA into rings of shared memory, warp 1 the MMAs; work
// items are taken by a persistent grid; every wait is bounded.

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "sn_internal.h"
#include "sn_tc.cuh"

namespace sn {

namespace {

constexpr int kT = 128;                         // tile rows (M) and columns (N)
constexpr int kKB = 64;                         // BF16 elements of K per stage (128 bytes)
constexpr int kStageA = kT * 128;               // 16 KiB
constexpr int kThreads = 256;
constexpr int kCPitch = kT + 4;                 // floats per staged output row

// Weight gradient: dW[i][j] = sum over the rows r of S[r - dB][i] gI[r][j], d the
// synapse's own delay.  One 128 x 128 tile per work item with four TMEM
// accumulators, one per delay; K is the rows, 64 a stage.  A stage holds both parts
// of the gradient tile and the spike tile shifted by each of the four delays (96
// KiB, 32 MMAs): the gradient is read once for the four delays (47 bytes a cycle
// into the SM at the MMAs' full rate; one delay at a time took 94, and the L2 gives
// about 53).  Both operands are taken as they lie, rows of K with the inputs or
// outputs contiguous (MN-major), so nothing is transposed for them.  What bounds it
// is shared memory: an MMA of 128 x 128 x 16 reads 8 KiB in its 64 cycles and 3 KiB
// are written for it, 86 cycles at 128 bytes a cycle (92 measured).  Separate rings
// for spike tiles and gradient, freed one by one, were slower (108: a barrier and a
// commit every 8 MMAs).  256 threads: warp 0 lane 0 TMA, warp 1 MMA, all eight the
// epilogue.  12,800 rows: 1024 x 1024 183 -> 152 us, 700 x 1024 130 -> 116 us, and the
// transposes (60 us) are gone.
constexpr int kDwSt = 2;
constexpr int kDwHalf = 64 * 128;               // 64 rows x 64 columns: one TMA box, 8 KiB
constexpr int kDwTile = 2 * kDwHalf;
constexpr int kDwStageBytes = 6 * kDwTile;

__global__ void __launch_bounds__(kThreads, 1) ff_tc_dw_kernel(const __grid_constant__ FfTcMaps maps, FfTcDwArgs a) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t full[kDwSt], empty[kDwSt], accbar;
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t sbase = smem_addr(smem);
    constexpr unsigned ncols = 512;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kDwSt; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" :: "r"(smem_addr(&full[s])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" :: "r"(smem_addr(&empty[s])));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" :: "r"(smem_addr(&accbar)));
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        s_abort = 0;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n"
                     :: "r"(smem_addr(&s_tmem)), "r"(ncols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = s_tmem;
    constexpr uint32_t idesc = idesc_bf16_f32_mn(kT, kT);
    unsigned g_prod = 0, g_mma = 0, items_done = 0;
    bool ready = false;                            // the next stage's operands are known to be there
    const int items = a.tiles_m * a.tiles_n * a.ksplit;

    bool live = true;                              // no wait of this block has given up (the same for all threads)
    for (int item = blockIdx.x; item < items && live; item += gridDim.x) {
        const int ks = item % a.ksplit, tile = item / a.ksplit;
        const int tm = tile % a.tiles_m, tn = tile / a.tiles_m;
        const int kb0 = (int)((long long)a.kblocks * ks / a.ksplit);
        const int kb1 = (int)((long long)a.kblocks * (ks + 1) / a.ksplit);
        if (warp == 0 && lane == 0) {
            for (int kb = kb0; kb < kb1; ++kb, ++g_prod) {
                const int st = g_prod % kDwSt;
                const unsigned round = g_prod / kDwSt;
                if (round > 0 && !mbar_wait(smem_addr(&empty[st]), (round - 1) & 1u, a.ctl)) { s_abort = 1; break; }
                const uint32_t fb = smem_addr(&full[st]);
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n"
                             :: "r"(fb), "r"(kDwStageBytes) : "memory");
                const uint32_t d0 = sbase + st * kDwStageBytes;
                // gradient parts, then the spikes 1 .. 4 steps earlier (rows
                // before the first and past the last are zeros)
                for (int q = 0; q < 2; ++q)
                    for (int h = 0; h < 2; ++h)
                        tma_load_2d(d0 + q * kDwTile + h * kDwHalf, &maps.m[1 + q], tn * kT + h * 64, kb * kKB, fb);
                for (int d = 1; d <= 4; ++d)
                    for (int h = 0; h < 2; ++h)
                        tma_load_2d(d0 + (1 + d) * kDwTile + h * kDwHalf, &maps.m[0], tm * kT + h * 64,
                                    kb * kKB - d * a.B, fb);
            }
        } else if (warp == 1) {
            for (int kb = kb0; kb < kb1; ++kb, ++g_mma) {
                const int st = g_mma % kDwSt;
                if (!ready && !mbar_wait_warp(smem_addr(&full[st]), (g_mma / kDwSt) & 1u, a.ctl)) { s_abort = 1; break; }
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                const uint64_t d0 = umma_desc_mn_sw128(sbase + st * kDwStageBytes, kDwHalf);
#pragma unroll
                for (int d = 0; d < 4; ++d) {
                    mma_bf16_x4<128>(tmem + d * kT, d0 + (2 + d) * (kDwTile / 16), d0, idesc, kb > kb0);
                    mma_bf16_x4<128>(tmem + d * kT, d0 + (2 + d) * (kDwTile / 16), d0 + kDwTile / 16, idesc, 1);
                }
                mma_commit(smem_addr(&empty[st]));
                ready = mbar_test_warp(smem_addr(&full[(g_mma + 1) % kDwSt]), ((g_mma + 1) / kDwSt) & 1u);
            }
            mma_commit(smem_addr(&accbar));
        }
        __syncwarp();
        if (!mbar_wait(smem_addr(&accbar), items_done & 1u, a.ctl)) s_abort = 1;
        ++items_done;
        __syncthreads();
        live = !s_abort;                           // (nobody sets it before the item's last barrier)
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        // epilogue: warps w and w + 4 read TMEM lane quarter w (tile rows), each
        // half of the columns, every element from its own delay's accumulator;
        // the values leave as coalesced rows through the (now idle) stages
        float *Cs = (float *)smem;                  // [128][kCPitch]
        const int quarter = warp & 3, half = warp >> 2;
        const int ml = quarter * 32 + lane, m = tm * kT + ml;
        for (int cc = 0; cc < 2; ++cc) {
            const int c0 = half * 64 + cc * 32;
            const int n0 = tn * kT + c0;
            float out[32];
#pragma unroll
            for (int q = 0; q < 32; ++q) out[q] = 0.0f;
            for (int d = 0; d < 4; ++d) {
                uint32_t v[32];
                tmem_ld32(tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(d * kT + c0), v);
                if (!live || kb1 == kb0 || m >= a.M) continue;
                const uint8_t *Dr = a.D + (size_t)m * a.N;
#pragma unroll
                for (int q = 0; q < 32; ++q)
                    if (n0 + q < a.N && Dr[n0 + q] == d + 1) out[q] = __uint_as_float(v[q]);
            }
            float4 *dst = (float4 *)(Cs + ml * kCPitch + c0);
#pragma unroll
            for (int q4 = 0; q4 < 8; ++q4)
                dst[q4] = make_float4(out[4 * q4], out[4 * q4 + 1], out[4 * q4 + 2], out[4 * q4 + 3]);
        }
        __syncthreads();
        if (live) {
            float *C = a.C + (size_t)ks * a.cstride;
            const int ncol = min(kT, a.N - tn * kT);
            for (int row = warp; row < kT; row += kThreads / 32) {
                const int mm = tm * kT + row;
                if (mm >= a.M) break;
                float *crow = C + (size_t)mm * a.N + tn * kT;
                const float *srow = Cs + row * kCPitch;
                for (int c = lane; c < ncol; c += 32) crow[c] = srow[c];
            }
        }
        // the staged tile was written and read through the generic proxy; the
        // next item's TMA (async proxy) reuses those bytes
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
        __syncthreads();
    }

    // drain: copies issued and MMAs committed complete before shared memory and
    // TMEM go away (bounded waits; no-ops when the phases have completed)
    if (warp == 0 && lane == 0) {
        for (unsigned i = g_prod > kDwSt ? g_prod - kDwSt : 0; i < g_prod; ++i)
            mbar_drain(smem_addr(&full[i % kDwSt]), (i / kDwSt) & 1u);
    }
    if (warp == 1 && lane == 0) {
        for (unsigned i = g_mma > kDwSt ? g_mma - kDwSt : 0; i < g_mma; ++i)
            mbar_drain(smem_addr(&empty[i % kDwSt]), (i / kDwSt) & 1u);
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" :: "r"(tmem), "r"(ncols));
}

// Forward synaptic input and spike gradient: C[r][n] = sum over the delays d, the
// K blocks kb and the products (A part, B part) of A[r + shift d][kb] B_d[n][kb].
//   forward (SG = false): A the spikes, shift -B, three B parts (hi, mid, lo);
//   spike gradient (SG): A parts hi, mid of the gradient, shift +B, B parts hi,
//   mid; products hi hi, hi mid, mid hi.
// A work item is H tiles of 128 rows x one tile of 128 columns.  Two row tiles share
// each weight tile: with one, the operands come in at 85 bytes a cycle at the MMAs'
// full rate, with two at 52 (forward) and 62 (the L2 gives an SM about 53).  What
// then bounds it is shared memory: 8 KiB read by an MMA in its 64 cycles and 3.4 (4)
// KiB written for it, 89 (94) cycles at 128 bytes a cycle; 92 and 94 measured.  The
// operands go through two rings, units of one A part (H tiles) and of one B part, so
// that each is freed as soon as its last MMA is done; the weights run one (kb, d)
// step ahead of the rows.
// A chunk of steps accumulates in TMEM (two buffers), and the drain warps add it
// into FP32 registers: the forward's chunk is one K block (all delays: 48 MMA steps
// in TMEM at most, a sequential sum over K blocks in round to nearest), the spike
// gradient's the whole item.  384 threads: warp 0 lane 0 TMA, warp 1 MMA, warps 4..11
// drain (warp w: TMEM lane quarter w % 4, columns 64 * ((w - 4) / 4) ..+63).
// A layer of at most 112 columns loads and multiplies only those (bn).
// (Two row tiles of the forward take the 168 registers that 384 threads leave and
// spill 44 bytes; its time is the MMAs'.)
// 12,800 rows, forward: 1024 x 1024 228 -> 202 us, 700 x 1024 161 -> 145; spike
// gradient: 1024 x 1024 282 -> 209, 1024 x 20 52 -> 33.
constexpr int kRowsThreads = 384;

template <int H, bool SG>
struct Rows {
    static constexpr int NA = SG ? 2 : 1, NB = SG ? 2 : 3;        // parts of a step
    static constexpr int RA = SG ? 4 : H == 2 ? 2 : 4;            // units in the rings
    static constexpr int RB = H == 2 ? (SG ? 5 : 9) : (SG ? 8 : 9);
    static constexpr int kUnitA = H * kStageA;
    static constexpr int kBytes = RA * kUnitA + RB * kStageA;
};

template <int H, bool SG>
__global__ void __launch_bounds__(kRowsThreads, 1) ff_tc_rows_kernel(const __grid_constant__ FfTcMaps maps, FfTcArgs a) {
    using R = Rows<H, SG>;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t fullA[R::RA], emptyA[R::RA], fullB[R::RB], emptyB[R::RB], accf[2], acce[2], mmas_done;
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t baseA = smem_addr(smem), baseB = baseA + R::RA * R::kUnitA;
    constexpr unsigned ncols = 2 * H * kT;

    if (threadIdx.x == 0) {
        auto init = [](uint64_t *b, int n) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" :: "r"(smem_addr(b)), "r"(n));
        };
        for (int q = 0; q < R::RA; ++q) { init(&fullA[q], 1); init(&emptyA[q], 1); }
        for (int q = 0; q < R::RB; ++q) { init(&fullB[q], 1); init(&emptyB[q], 1); }
        for (int q = 0; q < 2; ++q) { init(&accf[q], 1); init(&acce[q], 8); }
        init(&mmas_done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        s_abort = 0;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n"
                     :: "r"(smem_addr(&s_tmem)), "r"(ncols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = s_tmem;
    const int items = a.tiles_m * a.tiles_n, steps = 4 * a.kblocks;   // step s: K block s / 4, delay s % 4 + 1
    const int chunk = SG ? steps : 4, chunks = steps / chunk;
    unsigned ua = 0, ub = 0;                       // units this thread has put through (or taken from) the rings
    unsigned g_chunk = 0;                          // chunks issued, or drained
    bool live = true;                              // this warp's waits have all seen their phase

    if (warp == 0 && lane == 0) {
        const int bytesB = a.bn * 128;
        for (int item = blockIdx.x; item < items && !s_abort; item += gridDim.x) {
            const int tm = item % a.tiles_m, tn = item / a.tiles_m;
            auto loadA = [&](int s) {
                const int y = tm * H * kT + a.shift * (s % 4 + 1), x = s / 4 * kKB;
                for (int p = 0; p < R::NA; ++p, ++ua) {
                    const unsigned st = ua % R::RA, round = ua / R::RA;
                    if (round > 0 && !mbar_wait(smem_addr(&emptyA[st]), (round - 1) & 1u, a.ctl)) { s_abort = 1; return; }
                    const uint32_t fb = smem_addr(&fullA[st]);
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n"
                                 :: "r"(fb), "r"(R::kUnitA) : "memory");
                    for (int h = 0; h < H; ++h)
                        tma_load_2d(baseA + st * R::kUnitA + h * kStageA, &maps.m[p], x, y + h * kT, fb);
                }
            };
            auto loadB = [&](int s) {
                const int x = s / 4 * kKB;
                for (int p = 0; p < R::NB; ++p, ++ub) {
                    const unsigned st = ub % R::RB, round = ub / R::RB;
                    if (round > 0 && !mbar_wait(smem_addr(&emptyB[st]), (round - 1) & 1u, a.ctl)) { s_abort = 1; return; }
                    const uint32_t fb = smem_addr(&fullB[st]);
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n"
                                 :: "r"(fb), "r"(bytesB) : "memory");
                    tma_load_2d(baseB + st * kStageA, &maps.m[2], x, (s % 4 * R::NB + p) * a.part_rows + tn * kT, fb);
                }
            };
            loadB(0);
            for (int s = 0; s < steps && !s_abort; ++s) {
                loadA(s);
                if (s + 1 < steps && !s_abort) loadB(s + 1);
            }
        }
    } else if (warp == 1) {
        const uint32_t idesc = idesc_bf16_f32(kT, a.bn);
        const uint64_t descA = umma_desc_sw128(baseA), descB = umma_desc_sw128(baseB);
        // barriers are looked at while the MMAs in front of theirs run
        bool seenA = false, seenB = false;
        auto waitA = [&](unsigned u) {
            const bool ok = seenA || mbar_wait_warp(smem_addr(&fullA[u % R::RA]), (u / R::RA) & 1u, a.ctl);
            seenA = false;
            return ok;
        };
        auto waitB = [&](unsigned u) {
            const bool ok = seenB || mbar_wait_warp(smem_addr(&fullB[u % R::RB]), (u / R::RB) & 1u, a.ctl);
            seenB = false;
            return ok;
        };
        auto lookA = [&](unsigned u) { seenA = mbar_test_warp(smem_addr(&fullA[u % R::RA]), (u / R::RA) & 1u); };
        auto lookB = [&](unsigned u) { seenB = mbar_test_warp(smem_addr(&fullB[u % R::RB]), (u / R::RB) & 1u); };
        for (int item = blockIdx.x; item < items && live; item += gridDim.x)
            for (int c = 0; c < chunks; ++c, ++g_chunk) {
                const unsigned buf = g_chunk & 1u, use = g_chunk >> 1;
                if (use > 0 && !mbar_wait_warp(smem_addr(&acce[buf]), (use - 1) & 1u, a.ctl)) { live = false; break; }
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                const uint32_t tacc = tmem + buf * (H * kT);
                auto product = [&](unsigned u, unsigned v, int on) {
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                    const uint64_t dA = descA + u % R::RA * (R::kUnitA / 16), dB = descB + v % R::RB * (kStageA / 16);
#pragma unroll
                    for (int h = 0; h < H; ++h)
                        mma_bf16_x4<2>(tacc + h * kT, dA + h * (kStageA / 16), dB, idesc, on);
                };
                int s = 0;
                for (; s < chunk; ++s) {
                    const int on = s > 0;
                    if constexpr (!SG) {
                        if (!waitA(ua) || !waitB(ub)) break;
                        product(ua, ub, on);
                        mma_commit(smem_addr(&emptyB[ub % R::RB]));
                        lookB(ub + 1);
                        if (!waitB(ub + 1)) break;
                        product(ua, ub + 1, 1);
                        mma_commit(smem_addr(&emptyB[(ub + 1) % R::RB]));
                        lookB(ub + 2);
                        if (!waitB(ub + 2)) break;
                        product(ua, ub + 2, 1);
                        mma_commit(smem_addr(&emptyB[(ub + 2) % R::RB]));
                        mma_commit(smem_addr(&emptyA[ua % R::RA]));
                        lookA(ua + 1);
                        lookB(ub + 3);
                        ua += 1;
                        ub += 3;
                    } else {
                        if (!waitA(ua) || !waitB(ub)) break;
                        product(ua, ub, on);
                        lookB(ub + 1);
                        if (!waitB(ub + 1)) break;
                        product(ua, ub + 1, 1);
                        mma_commit(smem_addr(&emptyA[ua % R::RA]));
                        mma_commit(smem_addr(&emptyB[(ub + 1) % R::RB]));
                        lookA(ua + 1);
                        if (!waitA(ua + 1)) break;
                        product(ua + 1, ub, 1);
                        mma_commit(smem_addr(&emptyA[(ua + 1) % R::RA]));
                        mma_commit(smem_addr(&emptyB[ub % R::RB]));
                        lookA(ua + 2);
                        lookB(ub + 2);
                        ua += 2;
                        ub += 2;
                    }
                }
                if (s < chunk) { live = false; break; }
                mma_commit(smem_addr(&accf[buf]));
            }
        if (!live) s_abort = 1;
    } else if (warp >= 4) {
        const int quarter = warp & 3, half = (warp - 4) >> 2;
        bool ok = true;
        for (int item = blockIdx.x; item < items; item += gridDim.x) {
            const int tm = item % a.tiles_m, tn = item / a.tiles_m;
            float acc[H][64];
#pragma unroll
            for (int h = 0; h < H; ++h)
#pragma unroll
                for (int q = 0; q < 64; ++q) acc[h][q] = 0.0f;
            for (int c = 0; c < chunks; ++c, ++g_chunk) {
                const unsigned buf = g_chunk & 1u, use = g_chunk >> 1;
                ok = mbar_wait_warp(smem_addr(&accf[buf]), use & 1u, a.ctl);
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
#pragma unroll
                for (int h = 0; h < H; ++h)
#pragma unroll
                    for (int w = 0; w < 4; ++w) {
                        uint32_t v[16];
                        tmem_ld16(tmem + ((uint32_t)(quarter * 32) << 16) +
                                      (uint32_t)((buf * H + h) * kT + half * 64 + w * 16), v);
#pragma unroll
                        for (int q = 0; q < 16; ++q)
                            acc[h][w * 16 + q] = __fadd_rn(acc[h][w * 16 + q], __uint_as_float(v[q]));
                    }
                asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
                __syncwarp();
                if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" :: "r"(smem_addr(&acce[buf])) : "memory");
                if (!ok) break;
            }
            if (!ok) { s_abort = 1; break; }
            const int n0 = tn * kT + half * 64;
#pragma unroll
            for (int h = 0; h < H; ++h) {
                const int m = (tm * H + h) * kT + quarter * 32 + lane;
                if (m >= a.M) continue;
                float *crow = a.C + (size_t)m * a.ldc;
                if (n0 + 64 <= a.N && (a.ldc & 3) == 0) {
#pragma unroll
                    for (int q4 = 0; q4 < 16; ++q4)
                        *(float4 *)(crow + n0 + 4 * q4) =
                            make_float4(acc[h][4 * q4], acc[h][4 * q4 + 1], acc[h][4 * q4 + 2], acc[h][4 * q4 + 3]);
                } else {
#pragma unroll
                    for (int q = 0; q < 64; ++q)
                        if (n0 + q < a.N) crow[n0 + q] = acc[h][q];
                }
            }
        }
    }
    __syncwarp();

    // drain: copies issued and MMAs committed complete before shared memory and
    // TMEM go away (bounded waits; no-ops when the phases have completed)
    if (warp == 0 && lane == 0) {
        for (unsigned i = ua > R::RA ? ua - R::RA : 0; i < ua; ++i)
            mbar_drain(smem_addr(&fullA[i % R::RA]), (i / R::RA) & 1u);
        for (unsigned i = ub > R::RB ? ub - R::RB : 0; i < ub; ++i)
            mbar_drain(smem_addr(&fullB[i % R::RB]), (i / R::RB) & 1u);
    }
    if (warp == 1) {
        // every MMA issued: up to the last chunk's commit, or those of a step that a
        // failed wait cut short
        if (!live) mma_commit(smem_addr(&mmas_done));
        mbar_drain(smem_addr(live ? &accf[(g_chunk - 1) & 1u] : &mmas_done), live ? ((g_chunk - 1) >> 1) & 1u : 0u);
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" :: "r"(tmem), "r"(ncols));
}

// Weight parts: Wb[(d-1)*2 + s] = part s (hi, mid) of W_d ([rows_in][nout_p],
// rows_in = n_in rounded up to 128) for the backward; if Wf is given,
// Wf[(d-1)*3 + s] = part s (hi, mid, lo: hi + mid + lo = w exactly) of W_d
// transposed ([rows_out][nin_p]) for the forward.  Only each weight's own
// delay slot is written: the buffers are zeroed once when the context is
// set up and the delays never change, so every other slot stays zero.
// 32 x 32 tiles through shared memory (a grid-stride loop over tiles), so
// that both outputs leave as 64-byte row pieces.
__global__ void __launch_bounds__(256) ff_tc_weights_kernel(const float *__restrict__ W,
                                                            const uint8_t *__restrict__ D, int n_in, int n_out,
                                                            int nout_p, int rows_in, int nin_p, int rows_out,
                                                            __nv_bfloat16 *Wb, __nv_bfloat16 *Wf) {
    __shared__ __nv_bfloat16 sp[3][32][34];
    __shared__ uint8_t sd[32][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;      // 32 x 8
    const size_t bsz = (size_t)rows_in * nout_p, fsz = (size_t)rows_out * nin_p;
    const int ti = (n_in + 31) / 32, tj = (n_out + 31) / 32;
    const long long ntiles = (long long)ti * tj;
    for (long long tl = blockIdx.x; tl < ntiles; tl += gridDim.x) {
        const int i0 = (int)(tl / tj) * 32, j0 = (int)(tl % tj) * 32;
        for (int y = ty; y < 32; y += 8) {
            const int i = i0 + y, j = j0 + tx;
            if (i >= n_in || j >= n_out) continue;
            const size_t q = (size_t)i * n_out + j;
            const int d = D[q];
            const float w = W[q];
            const __nv_bfloat16 hi = __float2bfloat16_rn(w);
            const float r1 = __fsub_rn(w, __bfloat162float(hi));
            const __nv_bfloat16 mid = __float2bfloat16_rn(r1);
            if (Wb) {
                const size_t b = (size_t)i * nout_p + j;
                Wb[(size_t)((d - 1) * 2 + 0) * bsz + b] = hi;
                Wb[(size_t)((d - 1) * 2 + 1) * bsz + b] = mid;
            }
            sp[0][y][tx] = hi;
            sp[1][y][tx] = mid;
            sp[2][y][tx] = __float2bfloat16_rn(__fsub_rn(r1, __bfloat162float(mid)));
            sd[y][tx] = (uint8_t)d;
        }
        if (!Wf) continue;
        __syncthreads();
        for (int y = ty; y < 32; y += 8) {
            const int j = j0 + y, i = i0 + tx;
            if (i >= n_in || j >= n_out) continue;
            const int d = sd[tx][y];
            const size_t f = (size_t)j * nin_p + i;
#pragma unroll
            for (int part = 0; part < 3; ++part) Wf[(size_t)((d - 1) * 3 + part) * fsz + f] = sp[part][tx][y];
        }
        __syncthreads();
    }
}

// Spike bits [rows][words] -> 0/1 BF16 rows S [rows][nin_p] (padding stays zero).
__global__ void __launch_bounds__(256) ff_tc_spikes_kernel(const unsigned *__restrict__ bits, int rows, int n_in,
                                                           int words, int nin_p, __nv_bfloat16 *S) {
    const int r = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (r >= rows) return;
    const __nv_bfloat16 one = __float2bfloat16_rn(1.0f), zero = __float2bfloat16_rn(0.0f);
    for (int w = 0; w < words; ++w) {
        const unsigned b = __ldg(bits + (size_t)r * words + w);
        const int i = w * 32 + lane;
        if (i < n_in) S[(size_t)r * nin_p + i] = (b >> lane) & 1u ? one : zero;
    }
}

// Blocks for a grid-stride loop over 32 x 32 tiles: at most 1216 (eight per
// SM of a 152-SM part).
static int tile_grid(long long tiles) {
    const long long b = tiles < 1216 ? tiles : 1216;
    return (int)(b < 1 ? 1 : b);
}

}  // namespace

template <int H, bool SG>
static cudaError_t rows_launch(const FfTcMaps &maps, FfTcArgs args, int sms, cudaStream_t s) {
    const size_t smem = (size_t)Rows<H, SG>::kBytes + 1024;
    cudaError_t e = cudaFuncSetAttribute((const void *)ff_tc_rows_kernel<H, SG>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    args.tiles_m = (args.M + H * kT - 1) / (H * kT);
    args.tiles_n = (args.N + kT - 1) / kT;
    const int items = args.tiles_m * args.tiles_n;
    ff_tc_rows_kernel<H, SG><<<items < sms ? items : sms, kRowsThreads, smem, s>>>(maps, args);
    return cudaGetLastError();
}

cudaError_t ff_tc_rows(const FfTcMaps &maps, const FfTcArgs &args, bool spike_grad, cudaStream_t s) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    // two row tiles an item once single ones fill the SMs more than once: a
    // pair takes 1.2 to 1.3 times as long as a single one
    const long long singles = (long long)((args.M + kT - 1) / kT) * ((args.N + kT - 1) / kT);
    if (singles > sms)
        return spike_grad ? rows_launch<2, true>(maps, args, sms, s) : rows_launch<2, false>(maps, args, sms, s);
    return spike_grad ? rows_launch<1, true>(maps, args, sms, s) : rows_launch<1, false>(maps, args, sms, s);
}

cudaError_t ff_tc_dw(const FfTcMaps &maps, const FfTcDwArgs &args, cudaStream_t s) {
    static_assert(kT * kCPitch * 4 <= kDwSt * kDwStageBytes, "staged output tile fits the stage buffers");
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    const size_t smem = (size_t)kDwSt * kDwStageBytes + 1024;
    if ((e = cudaFuncSetAttribute((const void *)ff_tc_dw_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)smem)) != cudaSuccess)
        return e;
    const int items = args.tiles_m * args.tiles_n * args.ksplit;
    ff_tc_dw_kernel<<<items < sms ? items : sms, kThreads, smem, s>>>(maps, args);
    return cudaGetLastError();
}

cudaError_t ff_tc_weights(const float *W, const uint8_t *D, int n_in, int n_out, int nout_p, int rows_in,
                          void *Wb, int nin_p, int rows_out, void *Wf, cudaStream_t s) {
    ff_tc_weights_kernel<<<tile_grid((long long)((n_in + 31) / 32) * ((n_out + 31) / 32)), 256, 0, s>>>(
        W, D, n_in, n_out, nout_p, rows_in, nin_p, rows_out, (__nv_bfloat16 *)Wb, (__nv_bfloat16 *)Wf);
    return cudaGetLastError();
}

cudaError_t ff_tc_spikes(const unsigned *bits, int rows, int n_in, int words, int nin_p, void *S, cudaStream_t s) {
    ff_tc_spikes_kernel<<<(rows + 7) / 8, 256, 0, s>>>(bits, rows, n_in, words, nin_p, (__nv_bfloat16 *)S);
    return cudaGetLastError();
}

}  // namespace sn
