// Pull propagation in blocks of three timesteps (Section 2.1, second step of
// a timestep; Section 2.2: a spike reaches the post-neuron d steps later).
//
// A synapse of delay d >= 4 takes, for the steps T, T+1 and T+2 of a block,
// the spikes of its pre-neuron at T-d .. T+2-d: three neighbouring steps that
// are all known before the block begins.  So each block keeps, in shared
// memory, one word of HB bits per neuron of the network, its spikes by step
// (the newest at the bottom), and a synapse is loaded once and looked up once for
// three steps: one shared load and one shift give three bits, and three
// accumulators (one per step) take the weight.  Every list is in the order of
// sn_pull.cu (descending delay, then ascending pre and input index), so each
// step's float sum adds the same weights in the same order: the FP32 mirror's,
// bit for bit.
//
// Every block keeps the words up to date itself: the rows of three steps enter
// them at once (hist_advance).  Copying the words from one owner instead was
// measured slower (200 KB read by every block from the same L2 lines took
// 7,500 cycles a block of steps, and the words have to be fenced off).
//
// The list of a thread position (pin_perm as in sn_pull.cu) is split by delay
// into five regions, one after another in the store of its 32-position slice,
// entry q of lane l being half q % 2 of uint4 number (q / 2) * 32 + l of the
// region, {x, weight bits}:
//   0: d >= 7, looked up for the next block while this one runs
//   1: d = 4..6, looked up for the next block at the end of this one
//   2, 3, 4: d = 3, 2, 1, looked up per step in the rows of the last two steps
// Regions 0 and 1: x = (byte of the pre-neuron's word) << 5 | shift, shift =
// d - 7 or d - 4 (the bit of step T' + 2 - d, T' the next block's first step,
// when the words' lowest bit is step T' - 5 or T' - 2; the two steps before it
// are the next two bits).  Regions 2-4: x = (pre / 32) << 7 | pre % 32 as in
// sn_pull.cu, a bit of one row.
//
// Blocks meet without a barrier: each warp stores the spike word of its 32
// neurons with the step's number beside it (one 8-byte store), and every
// block reads all words of the row until each carries the step's number.
// That read is the only wait of a step (bounded, as the grid barrier's is);
// everything that does not need the newest row (regions 0-3, the raster, the
// external input of the next step) runs between the block's own store and
// that read.  Row t lies in slot t % kTagRows, so a launch that continues the last one
// finds its rows in their slots; any other has them written from the history first.  A
// row slot is reused after kTagRows steps; a block that has
// read all of row t knows that every block has stored it, so no block is
// more than one step ahead of another.
//
// What bounds it, at 100,000 neurons and 10^7 synapses of delays 1..16 (149
// blocks of 672 threads): nothing alone; the integer pipe (41 % busy), the shared-
// memory lookups (3.3 wavefronts each from bank conflicts; L1 55 %) and the latency
// of the L2 loads that each region begins with.  A step reads a synapse 0.44
// times instead of once: 200 steps 2.12 -> 1.53 ms (10.5 -> 7.2 us a step); 20,011
// neurons, 64 synapses each of delays 1..8, integer: 1.24 -> 0.69 ms (6.1 -> 3.2).
// A launch prepares its first sums by one pass over region 0 and one step of the loop:
// runs of a single step take 20.4 us at 20,000 neurons of 64 synapses, delays 1..16,
// and 49.5 at 100,000 of 100 (one step at a time: 29.8 and 49.5).
// Measured and left out: owning the neurons by thread position (no sum through
// shared memory, but 3 % slower), loading the second unit of the delay-1 lists
// ahead (spills: 12 % slower), reading the padding instead of testing each
// lane's list length (5 % slower).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "sn_pull.cuh"

namespace sn {
namespace {

// A neuron's summed input: float in list order, or int32 (the host takes this
// kernel only where no neuron's incoming weights sum to 2^31 in magnitude).
template <int MODE> struct BlockAcc;
template <> struct BlockAcc<SN_F32> : PullAcc<SN_F32> {};
template <> struct BlockAcc<SN_I32> {
    using T = int;
    static __device__ __forceinline__ T add(T acc, unsigned wbits) { return acc + (int)wbits; }
};

constexpr int kTagRows = 8;         // slots of the tagged spike rows (at least 5: see the kernel)
// Blocks of up to kPullNarrow threads have 80 registers a thread, wider ones 64;
// a unit (half of the double buffer) is 3 or 2 16-byte loads of two synapses
// each.  The narrow form may not spill: next to 228 KB of shared memory the L1 is
// too small, and 50 bytes of spills a thread cost 15 % of the step.  The wide one
// spills up to 40 bytes, and the host takes it by a stricter rule (block_store_wins).
template <int MAXT> constexpr int unit_of() { return MAXT <= kPullNarrow ? 3 : 2; }

constexpr int kCols = 3;            // 16-byte reads of a row a thread has in flight: words / 2 <= kCols * threads

// Layout of the words.  A column is the 32 neurons of a spike word; neuron n of
// it has the field f of word j in the column's piece p = n % 4, where n / 4 =
// f * V + j and a piece is V = HB / 4 words: with that order one nibble word
// (below) holds the new bits of a piece, four bits apart.  The eight pieces
// of the columns 2i and 2i + 1 (piece l = column % 2 * 4 + p) lie in the order
// (l + i) % 8 (HB = 8: (l + i / 2) % 8), so that the lanes of a warp, which take
// the pairs i, i + 1, ..., have no bank conflicts at any l.
__host__ __device__ constexpr int piece_slot(int i, int l, int hb) { return ((hb == 8 ? i >> 1 : i) + l) & 7; }

// Three rows (oldest first) enter the words of the column pair i.  The integer
// pipe bounds this (about 13 operations a piece), so the shift of a word is a
// multiplication (the other pipe).
template <int HB>
__device__ __forceinline__ void hist_advance(unsigned *s_h, int i, const uint2 (&r)[3]) {
    constexpr unsigned low3 = HB == 32 ? 0x00000007u : HB == 16 ? 0x00070007u : 0x07070707u;
    constexpr int V = HB / 4;
    unsigned *pair = s_h + (size_t)i * (2 * HB);
#pragma unroll
    for (int l = 0; l < 8; ++l) {
        const unsigned r2 = l < 4 ? r[2].x : r[2].y, r1 = l < 4 ? r[1].x : r[1].y, r0 = l < 4 ? r[0].x : r[0].y;
        const int p = l & 3;
        // nibble jj: steps newest (bit 0) to oldest of neuron 4 * jj + p
        const unsigned e = (__funnelshift_r(r2, r2, p) & 0x11111111u) | (__funnelshift_r(r1, r1, p - 1) & 0x22222222u) |
                           (__funnelshift_r(r0, r0, p - 2) & 0x44444444u);
        unsigned *w = pair + piece_slot(i, l, HB) * V;
        auto enter = [&](unsigned h, int j) { return ((h * 8u) & ~low3) | ((e >> (4 * j)) & low3); };
        if constexpr (HB == 8) {
            uint2 h = *(const uint2 *)w;
            h.x = enter(h.x, 0); h.y = enter(h.y, 1);
            *(uint2 *)w = h;
        } else {
#pragma unroll
            for (int q = 0; q < HB / 16; ++q) {
                uint4 h = ((const uint4 *)w)[q];
                h.x = enter(h.x, 4 * q); h.y = enter(h.y, 4 * q + 1);
                h.z = enter(h.z, 4 * q + 2); h.w = enter(h.w, 4 * q + 3);
                ((uint4 *)w)[q] = h;
            }
        }
    }
}

template <int HB> struct HistWord;
template <> struct HistWord<8> { using T = unsigned char; };
template <> struct HistWord<16> { using T = unsigned short; };
template <> struct HistWord<32> { using T = unsigned; };

template <int HB>
__device__ __forceinline__ unsigned hist_bits(const unsigned char *hist, unsigned x) {
    const unsigned h = *(const typename HistWord<HB>::T *)(hist + (x >> 5));
    return __funnelshift_r(h, 0u, x);
}

__device__ __forceinline__ bool row_bit(const unsigned char *row, unsigned x) {
    const unsigned w = *(const unsigned *)(row + (x >> 5));
    return __funnelshift_r(w, w, x) & 1u;
}

template <int P>
__device__ __forceinline__ void unit_load(uint4 (&e)[P], const uint4 *ent, int p0, int np) {
#pragma unroll
    for (int u = 0; u < P; ++u)
        e[u] = p0 + u < np ? __ldg(ent + (size_t)(p0 + u) * 32) : make_uint4(0u, 0u, 0u, 0u);
}

// test(x, weight bits) of the first `valid` pairs of a unit (the same for the
// whole warp), in list order.
template <int P, typename Test>
__device__ __forceinline__ void unit_all(const uint4 (&e)[P], Test test) {
#pragma unroll
    for (int u = 0; u < P; ++u) { test(e[u].x, e[u].y); test(e[u].z, e[u].w); }
}
template <int P, typename Test>
__device__ __forceinline__ void unit_part(const uint4 (&e)[P], int valid, Test test) {
#pragma unroll
    for (int u = 0; u < P; ++u)
        if (u < valid) { test(e[u].x, e[u].y); test(e[u].z, e[u].w); }
}

// The np pairs of one region (npmax the warp's largest), which begins `at`
// pairs after ent, in list order.  e0 holds the first P pairs on
// entry, and those of the region walked next (np_next pairs at at_next) on
// exit.
template <int P, typename Test>
__device__ __forceinline__ void region_loop(uint4 (&e0)[P], uint4 (&e1)[P], const uint4 *ent,
                                            int at, int np, int npmax, int at_next, int np_next, Test test) {
    // pairs p0 .. of the region: pull_load counts from its own base
    auto load = [&](uint4 (&e)[P], int p0) { unit_load(e, ent + (size_t)(at + p0) * 32, 0, np - p0); };
    int p0 = 0;
    for (; p0 + 2 * P < npmax; p0 += 2 * P) {
        load(e1, p0 + P);
        unit_all(e0, test);
        load(e0, p0 + 2 * P);
        unit_all(e1, test);
    }
    // the last pairs, at most 2P: only those before the warp's longest
    // list's end are tested
    const int rem = npmax - p0;
    if (rem > P) {
        load(e1, p0 + P);
        unit_all(e0, test);
        unit_load(e0, ent + (size_t)at_next * 32, 0, np_next);
        unit_part(e1, rem - P, test);
    } else {
        unit_part(e0, rem, test);
        unit_load(e0, ent + (size_t)at_next * 32, 0, np_next);
    }
}

__device__ __forceinline__ ulonglong2 ld_tagged2(const unsigned long long *p) {
    ulonglong2 v;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p) : "memory");
    return v;
}

// The tagged row of a step into shared memory, once every word carries `tag`.
// Bounded: false when another block latched a status or the wall-clock limit
// ran out (then SN_ETIMEOUT is latched).
__device__ __forceinline__ bool read_row(const unsigned long long *row, int words, unsigned tag, unsigned *dst,
                                         Control *ctl) {
    const unsigned long long *src = row + 2 * threadIdx.x;
    unsigned todo = 0, spins = 0, began = 0;
#pragma unroll
    for (int u = 0; u < kCols; ++u)
        if (2 * (int)(threadIdx.x + u * blockDim.x) < words) todo |= 1u << u;
    while (todo) {
        ulonglong2 v[kCols];
#pragma unroll
        for (int u = 0; u < kCols; ++u)
            if ((todo >> u) & 1u) v[u] = ld_tagged2(src + 2 * u * blockDim.x);
#pragma unroll
        for (int u = 0; u < kCols; ++u) {
            if (!((todo >> u) & 1u)) continue;
            const int i = threadIdx.x + u * blockDim.x;
            // the odd word past the row's end is never stored (and stays zero)
            if ((unsigned)(v[u].x >> 32) == tag && (2 * i + 1 >= words || (unsigned)(v[u].y >> 32) == tag)) {
                *(uint2 *)(dst + 2 * i) = make_uint2((unsigned)v[u].x, (unsigned)v[u].y);
                todo &= ~(1u << u);
            }
        }
        if (todo && (++spins & 63u) == 0) {
            // wall clock in units of 1.024 us
            const unsigned now = (unsigned)(global_timer_ns() >> 10);
            if (spins == 64u) began = now;
            if (ld_status(ctl) != 0) return false;
            if (now - began > (unsigned)(kBarrierTimeoutNs >> 10)) {
                atomicCAS(&ctl->status, 0, (int)SN_ETIMEOUT);
                return false;
            }
        }
    }
    return true;
}

template <int MODE, int HB, int MAXT>
__global__ void __launch_bounds__(MAXT, 1) pull_block_kernel(NetArgs a) {
    using V = typename Tr<MODE>::V;
    using Acc = typename BlockAcc<MODE>::T;
    using RA = typename Tr<MODE>::A;
    constexpr int kUnit = unit_of<MAXT>();
    extern __shared__ uint4 s_mem4[];
    // [words][HB] spike words (none when no delay exceeds 3; words rounded up
    // to a pair), two rows, sums
    // (sizes and offsets are arguments: not values to keep in registers)
    const int D = a.hD, W = a.words, Wp = a.wp, Wt = a.wt;
    const bool use_h = D > 3;
    unsigned *s_h = (unsigned *)s_mem4;
    unsigned *s_rows = (unsigned *)((unsigned char *)s_mem4 + a.rows_at);
    Acc *s_acc = (Acc *)((unsigned char *)s_mem4 + a.acc_at);
    const unsigned char *hist = (const unsigned char *)s_h;
    __shared__ int s_stop, s_fail, s_hdr[32][8];
    const int lane = threadIdx.x & 31;
    const int t0 = a.t0;

    const int bfirst = blockIdx.x * a.chunk;
    const int j = bfirst + threadIdx.x;
    const bool mine = j < a.n;
    const int pj = mine ? a.pin_perm[j] - bfirst : 0;   // the neuron (of this block) whose lists this thread sums
    const int wword = j >> 5;                           // this warp's spike word
    const bool word_lane = lane == 0 && wword < W;
    V v = 0;
    // pairs of each region of this position's list, 16 bits each (the host
    // takes this kernel only for lists that fit)
    unsigned np01 = 0, np23 = 0, np4 = 0;
    int rr = 0;
    unsigned thr = 0;
    const uint4 *ent = a.pin;
    if (mine) {
        v = ((const V *)a.V)[j];
        rr = a.r[j];
        thr = a.prate[j];
        auto pairs = [&](int g) { return (unsigned)(a.pin_len[(size_t)g * a.n + j] + 1) >> 1; };
        np01 = pairs(0) | pairs(1) << 16;
        np23 = pairs(2) | pairs(3) << 16;
        np4 = pairs(4);
        ent = a.pin + a.pin_off[j >> 5] + lane;
    }
    auto np = [&](int g) -> int {
        return g == 0 ? np01 & 0xffffu : g == 1 ? np01 >> 16 : g == 2 ? np23 & 0xffffu : g == 3 ? np23 >> 16 : np4;
    };
    // the warp's longest list in each region, and the pairs of the slice before
    // regions 2, 3 and 4: read from shared memory where they are needed
    // (registers are short, and a spill would go through an L1 that has no room)
    volatile int *hdr = s_hdr[threadIdx.x >> 5];
    {
        int at = 0;
        for (int g = 0; g < 5; ++g) {
            const int longest = __reduce_max_sync(0xffffffffu, np(g));
            if (lane == 0) { hdr[g] = longest; if (g >= 2) hdr[3 + g] = at; }
            at += longest;
        }
        __syncwarp();
    }

    // the spike rows of the steps before the launch, from the history
    auto hist_word = [&](int tau, int w) -> unsigned {
        return w < W && tau >= 0 && tau >= t0 - D ? __ldcg(a.hist + (size_t)(tau % D) * W + w) : 0u;
    };
    if (threadIdx.x == 0) { s_stop = 0; s_fail = 0; }
    for (int i = threadIdx.x; i < Wp; i += blockDim.x) {
        s_rows[((t0 - 3) & 1) * Wp + i] = hist_word(t0 - 3, i);
        s_rows[(t0 & 1) * Wp + i] = hist_word(t0 - 2, i);
    }
    if (use_h) {
        for (int i = threadIdx.x; i < (W + (W & 1)) * (HB / 4); i += blockDim.x) s_mem4[i] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
        // the words as of the block before the first one: steps up to t0 - 5
        for (int g = (D - 4 + 2) / 3 - 1; g >= 0; --g)
            for (int i = threadIdx.x; 2 * i < W; i += blockDim.x) {
                uint2 r[3];
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    const int tau = t0 - 7 - 3 * g + q;
                    r[q] = make_uint2(hist_word(tau, 2 * i), hist_word(tau, 2 * i + 1));
                }
                hist_advance<HB>(s_h, i, r);
            }
    }
    __syncthreads();

    RA *ring = (RA *)a.ring;
    unsigned fired = 0;                                 // spikes of this thread's neuron
    bool overflow = false;
    uint4 ea[kUnit], eb[kUnit];
    // a0: the sum of the step at hand; a1, a2: of the two steps after it in
    // its block; n0..n2: of the next block's three steps
    Acc a0 = 0, a1 = 0, a2 = 0, n0 = 0, n1 = 0, n2 = 0;
    V ext = 0;                                          // external input of the step at hand
    int k = 2;                                          // step within its block
    int rslot = t0 % a.cap, hslot = t0 % D;             // raster and history rows of the step at hand
    // the lists above delay 3 for a block of steps, from its words
    auto three = [&](unsigned x, unsigned w) {
        const unsigned bits = hist_bits<HB>(hist, x);
        if (bits & 4u) n0 = BlockAcc<MODE>::add(n0, w);
        if (bits & 2u) n1 = BlockAcc<MODE>::add(n1, w);
        if (bits & 1u) n2 = BlockAcc<MODE>::add(n2, w);
    };
    // region 0 for the first block of steps; the rest of what comes before step 0
    // is the last step of a block like any other's
    unit_load(ea, ent, 0, np(0));
    region_loop(ea, eb, ent, 0, np(0), hdr[0], 0, 0, three);
    for (int s = -1; s < a.steps; ++s) {
        const int t = t0 + s;
        const unsigned char *row_prev = (const unsigned char *)(s_rows + ((t - 1) & 1) * Wp);   // step t - 1
        if (s >= 0) {
            // the neuron's parameters come from the L2 while the sum runs:
            // registers are short (no spill may hit the small L1)
            V th = 0, lk = 0, rs = 0;
            int R = 0;
            if (mine) {
                th = __ldg((const V *)a.th + j);
                lk = __ldg((const V *)a.lk + j);
                rs = __ldg((const V *)a.rs + j);
                R = __ldg(a.R + j);
            }
            // delay 1: the row of step t - 1 (the first unit is loaded)
            auto one = [&](unsigned x, unsigned w) {
                if (row_bit(row_prev, x)) a0 = BlockAcc<MODE>::add(a0, w);
            };
            const int len = hdr[4];
            if (len > kUnit) {
                const uint4 *ent4 = ent + (size_t)hdr[7] * 32;
                unit_load(eb, ent4, kUnit, np(4));
                unit_all(ea, one);
                unit_part(eb, len - kUnit, one);
                for (int p0 = 2 * kUnit; p0 < len; p0 += kUnit) {
                    unit_load(ea, ent4, p0, np(4));
                    unit_all(ea, one);
                }
            } else {
                unit_part(ea, len, one);
            }
            if (mine) s_acc[pj] = a0;
            __syncthreads();
            bool fire = false;
            if (mine) {
                const Acc sum = s_acc[threadIdx.x];
                // input still pending in the ring from an earlier push run
                V ring_in = 0;
                if (t < a.ring_until) {
                    RA *slot = ring + (size_t)(t % a.D1) * a.n + j;
                    ring_in = Tr<MODE>::from_acc(*slot);
                    *slot = 0;
                }
                if constexpr (MODE == SN_F32) {
                    const float in = t < a.ring_until ? __fadd_rn(sum, ring_in) : sum;
                    fire = lif_update_f32(v, rr, in, ext, th, lk, rs, R);
                } else {
                    // the integrated state is checked against int32 before the threshold
                    const long long in = (long long)sum + ring_in;
                    long long u;
                    if (v > rs) { u = (long long)v - lk; u = u > rs ? u : rs; }
                    else if (v < rs) { u = (long long)v + lk; u = u < rs ? u : rs; }
                    else u = rs;
                    u += in;
                    u += ext;
                    if (u > 2147483647ll || u < -2147483648ll) overflow = true;
                    fire = (u > th) && (rr == 0);
                    if (fire) { u = rs; rr = R; }
                    else if (rr > 0) rr -= 1;
                    v = (int)u;
                }
            }
            const unsigned ball = __ballot_sync(0xffffffffu, fire);
            if (word_lane) {
                st_tagged(a.ptag + (size_t)(t & (kTagRows - 1)) * Wt + wword, (unsigned)t + 1u, ball);
                a.raster[(size_t)rslot * W + wword] = ball;
                // the history's row of the step before: its slot held row t - 1 - D,
                // which no block reads any more (every block has stored row t - 1)
                if (s > 0)
                    a.hist[(size_t)(hslot == 0 ? D - 1 : hslot - 1) * W + wword] = ((const unsigned *)row_prev)[wword];
            }
            rslot = rslot + 1 == a.cap ? 0 : rslot + 1;
            hslot = hslot + 1 == D ? 0 : hslot + 1;
            if (fire) fired += 1;
            if (overflow) atomicCAS(&a.ctl->status, 0, (int)SN_EOVERFLOW);
        }
        // the part of the lists above delay 3 walked now: half of region 0 for
        // the first two steps of a block, region 1 at its last
        const int len0 = hdr[0], halfA = (len0 + 1) >> 1;
        const int atA = k == 0 ? 0 : k == 1 ? halfA : len0;
        const int npA = k == 0 ? min(np(0), halfA) : k == 1 ? max(np(0) - halfA, 0) : np(1);
        const int npAmax = k == 0 ? halfA : k == 1 ? len0 - halfA : hdr[1];
        if (k != 2 && s >= 0) unit_load(ea, ent + (size_t)atA * 32, 0, npA);
        // ---- what does not need the row of step t
        int st = 0;
        if (threadIdx.x == 0 && s >= 0) st = ld_status(a.ctl);
        const bool more = s + 1 < a.steps;
        if (more) {
            // the thread's columns of row t - 3 enter the words below, the first
            // pair loaded ahead (its slot is stored again only at step t + 5,
            // when every block has passed here)
            const unsigned long long *tag3 = a.ptag + (size_t)((t - 3) & (kTagRows - 1)) * Wt;
            auto oldest = [&](int i) -> uint2 {
                if (2 * i >= W) return make_uint2(0u, 0u);
                const ulonglong2 x = ld_tagged2(tag3 + 2 * i);
                return make_uint2((unsigned)x.x, (unsigned)x.y);
            };
            uint2 old = make_uint2(0u, 0u);
            if (k == 2 && use_h) old = oldest(threadIdx.x);
            // external input of the next step
            ext = 0;
            if (mine) {
                const int tn = t + 1;
                if (tn < a.ev_nsteps) {
                    int lo = a.ev_off[tn], hi = a.ev_off[tn + 1];
                    const int end = hi;
                    while (lo < hi) {
                        const int mid = (lo + hi) >> 1;
                        if (a.ev_neuron[mid] < j) lo = mid + 1; else hi = mid;
                    }
                    if (lo < end && a.ev_neuron[lo] == j) ext = ((const V *)a.ev_val)[lo];
                }
                if (thr && poisson_fires(a.pkey, (unsigned)tn, (unsigned)j, thr)) {
                    const V amp = __ldg((const V *)a.pamp + j);
                    if (MODE == SN_F32) ext = __fadd_rn(ext, amp); else ext = ext + amp;
                }
            }
            const unsigned *row_pp = s_rows + (t & 1) * Wp;                 // step t - 2
            if (k == 2 && use_h) {
                // rows t - 3 .. t - 1 enter the words: the next block's view
#pragma unroll 1
                for (int i = threadIdx.x; 2 * i < W; i += blockDim.x) {
                    const uint2 r[3] = {old, *(const uint2 *)(row_pp + 2 * i),
                                        *(const uint2 *)((const unsigned *)row_prev + 2 * i)};
                    old = oldest(i + blockDim.x);
                    hist_advance<HB>(s_h, i, r);
                }
                __syncthreads();
            }
            if (k == 2) unit_load(ea, ent + (size_t)atA * 32, 0, npA);
            // delays above 3 of the next block's steps
            region_loop(ea, eb, ent, atA, npA, npAmax, k == 1 ? hdr[6] : hdr[5], k == 1 ? np(3) : np(2), three);
            if (k == 2) {
                // delay 3 of the next block's first two steps: rows t - 2, t - 1
                region_loop(ea, eb, ent, hdr[5], np(2), hdr[2], hdr[6], np(3), [&](unsigned x, unsigned w) {
                    if (row_bit((const unsigned char *)row_pp, x)) n0 = BlockAcc<MODE>::add(n0, w);
                    if (row_bit(row_prev, x)) n1 = BlockAcc<MODE>::add(n1, w);
                });
                a0 = n0; a1 = n1; a2 = n2;
                n0 = n1 = n2 = 0;
            } else {
                a0 = a1; a1 = a2;
                // delay 3 of this block's last step: row t - 1
                if (k == 0)
                    region_loop(ea, eb, ent, hdr[5], np(2), hdr[2], hdr[6], np(3), [&](unsigned x, unsigned w) {
                        if (row_bit(row_prev, x)) a1 = BlockAcc<MODE>::add(a1, w);
                    });
            }
            // delay 2 of the next step: row t - 1
            region_loop(ea, eb, ent, hdr[6], np(3), hdr[3], hdr[7], np(4), [&](unsigned x, unsigned w) {
                if (row_bit(row_prev, x)) a0 = BlockAcc<MODE>::add(a0, w);
            });
        }
        // ---- the row of step t, in place of row t - 2 (read in this phase
        // only when it ends a block)
        unsigned *row = s_rows + (t & 1) * Wp;
        if (k == 2) __syncthreads();
        if (s >= 0) {
            if (!read_row(a.ptag + (size_t)(t & (kTagRows - 1)) * Wt, W, (unsigned)t + 1u, row, a.ctl)) s_fail = 1;
        } else {
            for (int i = threadIdx.x; i < W; i += blockDim.x) row[i] = hist_word(t, i);
        }
        k = k == 2 ? 0 : k + 1;
        if (threadIdx.x == 0) s_stop = st;
        __syncthreads();
        if (s_stop | s_fail) break;
    }
    if (word_lane && !(s_stop | s_fail)) {
        const int t = t0 + a.steps - 1;
        a.hist[(size_t)(t % D) * W + wword] = s_rows[(t & 1) * Wp + wword];
    }
    unsigned long long my_spikes = fired, my_events = 0;
    if (mine) {
        ((V *)a.V)[j] = v;
        a.r[j] = rr;
        my_events = my_spikes * (unsigned long long)(a.rowptr[j + 1] - a.rowptr[j]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        my_spikes += __shfl_down_sync(0xffffffffu, my_spikes, o);
        my_events += __shfl_down_sync(0xffffffffu, my_events, o);
    }
    if (lane == 0 && my_spikes) {
        atomicAdd(&a.ctl->spikes, my_spikes);
        atomicAdd(&a.ctl->events, my_events);
    }
}


// The rows of the last kTagRows steps from the history into their slots (all of them:
// no number of a later step is left behind).
__global__ void pull_rows_kernel(NetArgs a) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x, q = i / a.wt, w = i % a.wt;
    if (q >= kTagRows) return;
    const int tau = a.t0 - kTagRows + q;
    const bool in = tau >= 0 && tau >= a.t0 - a.hD && w < a.words;
    a.ptag[(size_t)(tau & (kTagRows - 1)) * a.wt + w] =
        (unsigned long long)((unsigned)tau + 1u) << 32 | (in ? a.hist[(size_t)(tau % a.hD) * a.words + w] : 0u);
}

template <int HB, int MAXT>
const void *block_fn_of(int dtype) {
    return dtype == SN_F32 ? (const void *)pull_block_kernel<SN_F32, HB, MAXT>
                           : (const void *)pull_block_kernel<SN_I32, HB, MAXT>;
}

const void *block_fn(int dtype, int hb, int threads) {
    const bool wide = threads > kPullNarrow;
    switch (hb) {
        case 8: return wide ? block_fn_of<8, kPullMaxBlock>(dtype) : block_fn_of<8, kPullNarrow>(dtype);
        case 16: return wide ? block_fn_of<16, kPullMaxBlock>(dtype) : block_fn_of<16, kPullNarrow>(dtype);
        default: return wide ? block_fn_of<32, kPullMaxBlock>(dtype) : block_fn_of<32, kPullNarrow>(dtype);
    }
}

}  // namespace

// The blocked form of a pull plan (grid and chunk from plan_pull): *hb = the
// bits of a neuron's spike word (8, 16 or 32: delays up to hb + 4), 0 when
// the words, two rows and the sums do not fit a block's shared memory.
cudaError_t plan_pull_block(int n, int D, int dtype, int grid, int chunk, int *hb, size_t *smem) {
    *hb = 0;
    const int bits = D <= 12 ? 8 : D <= 20 ? 16 : D <= 36 ? 32 : 0;
    if (bits == 0 || grid < 2) return cudaSuccess;
    int dev = 0, optin = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    const size_t words = ((size_t)n + 31) / 32, wp = (words + 3) & ~(size_t)3;
    const size_t bytes = (D > 3 ? (words + (words & 1)) * bits * 4 : 0) + 2 * wp * 4 + (size_t)chunk * 4;
    if (bytes + 1100 > (size_t)optin || grid > sms || (words + 1) / 2 > (size_t)kCols * chunk) return cudaSuccess;
    const void *fn = block_fn(dtype, bits, chunk);
    if ((e = allow_all_smem(fn)) != cudaSuccess) return e;
    int p = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&p, fn, chunk, bytes)) != cudaSuccess) return e;
    if (p < 1) return cudaSuccess;
    *hb = bits;
    *smem = bytes;
    return cudaSuccess;
}

// Bytes of the tagged spike rows of a network of `words` spike words.
size_t pull_tag_bytes(int words) { return (size_t)kTagRows * ((words + 1) & ~1) * 8; }

// Byte of neuron pre's word in the blocked kernel's shared memory.
unsigned pull_hist_byte(unsigned pre, int hb) {
    const unsigned v = hb / 4, n = pre & 31u, jj = n >> 2, pair = pre >> 6;
    const unsigned l = (pre >> 5 & 1u) * 4 + (n & 3u);
    return (pair * 2 * hb + piece_slot((int)pair, (int)l, hb) * v + jj % v) * 4u + (jj / v) * (hb / 8);
}

// rows_live: the slots hold the last rows (the last launch of this kernel ended at
// step t0, and nothing has changed the history since).
cudaError_t launch_pull_block(NetArgs a, int dtype, int hb, int grid, size_t smem, bool rows_live, cudaStream_t s) {
    a.wp = (a.words + 3) & ~3;
    a.wt = (a.words + 1) & ~1;
    a.rows_at = a.hD > 3 ? a.wt * hb * 4 : 0;
    a.acc_at = a.rows_at + 2 * a.wp * 4;
    void *args[] = {(void *)&a};
    const void *fn = block_fn(dtype, hb, a.chunk);
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(s, &capture);
    if (e != cudaSuccess) return e;
    // (a graph may be launched again after something else has run)
    if (!rows_live || capture != cudaStreamCaptureStatusNone) {
        const int total = kTagRows * a.wt;
        pull_rows_kernel<<<(total + 255) / 256, 256, 0, s>>>(a);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    // cooperative: the blocks wait for one another's rows, so all must be resident
    return cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(a.chunk), args, smem, s);
}

}  // namespace sn
