// Batched simulation: thousands of independent networks of uneven size and
// heterogeneous parameters in one persistent launch.
//
// Each network runs all requested timesteps on one executor: a whole block
// for networks larger than the warp threshold, a single warp for the small
// ones (no block-wide barrier then, eight networks per block at a time).
// Blocks take networks from two atomic work queues, largest first, so the
// long networks start early and the short ones fill the tail.  The
// timestep is the same as in the single-network kernels (Section 2.1 order,
// strict threshold, clamped constant leak; delays through a ring of D+1
// pending-input slots with fixed-point accumulation).  A network's ring is
// copied into shared memory while it runs when it fits the block's arena.

#include <cuda_runtime.h>
#include <stdint.h>

#include "sn_device.cuh"
#include "sn_internal.h"

namespace sn {

constexpr int kWarps = kBatchBlock / 32;
constexpr int kListInts = kBatchMaxN;          // spiker list arena (ints) per block

template <int MODE>
struct BatchNet {
    using A = typename Tr<MODE>::A;
    using V = typename Tr<MODE>::V;
    int b, off, n, woff;
    unsigned long long key;
};

// Update of neuron j (local) of network nb at step t, in two halves so that a
// thread can issue the loads of several neurons before it uses any of them:
// batch_load reads the pending input, state and parameters; batch_finish
// clears the pending-input slot, adds the external input and applies the LIF
// rule (Section 2.1 order), storing the state.  Returns the spike.
template <int MODE>
struct NeuronIn {
    typename Tr<MODE>::A raw;
    typename Tr<MODE>::V v, th, lk, rs;
    int rr, R;
};

template <int MODE>
__device__ __forceinline__ void batch_load(const BatchArgs &a, const BatchNet<MODE> &nb, int j,
                                           const typename Tr<MODE>::A *slot, bool global_ring, NeuronIn<MODE> &in) {
    using V = typename Tr<MODE>::V;
    const int g = nb.off + j;
    in.raw = global_ring ? __ldcg(slot + j) : slot[j];
    in.v = ((const V *)a.V)[g];
    in.rr = a.r[g];
    in.th = __ldg((const V *)a.th + g);
    in.lk = __ldg((const V *)a.lk + g);
    in.rs = __ldg((const V *)a.rs + g);
    in.R = __ldg(a.R + g);
}

template <int MODE>
__device__ __forceinline__ bool batch_finish(const BatchArgs &a, const BatchNet<MODE> &nb, int t, int j,
                                             typename Tr<MODE>::A *slot, NeuronIn<MODE> &in, bool &overflow) {
    using V = typename Tr<MODE>::V;
    const int g = nb.off + j;
    slot[j] = 0;
    const V acc = Tr<MODE>::from_acc(in.raw);
    const V ext = external_input_at<MODE>(a.ev_off, a.ev_nsteps, a.ev_neuron, a.ev_val, a.prate, a.pamp,
                                          nb.key, t, g, j);
    bool fire;
    if constexpr (MODE == SN_F32)
        fire = lif_update_f32(in.v, in.rr, acc, ext, in.th, in.lk, in.rs, in.R);
    else
        fire = lif_update_i32(in.v, in.rr, acc, ext, in.th, in.lk, in.rs, in.R, overflow);
    ((V *)a.V)[g] = in.v;
    a.r[g] = in.rr;
    return fire;
}

// Neurons whose loads one thread issues together in the update phase.
constexpr int kUpdAhead = 8;

// Synapses of a row whose loads a lane issues together before their adds.
constexpr int kPushAhead = 8;

// Push of spiker i (local) of network nb: lanes stride the CSR row, each
// lane loading kPushAhead synapses before it issues their accumulates (the
// accumulates are fixed-point, so their order does not matter).
template <int MODE>
__device__ __forceinline__ long long batch_push(const BatchArgs &a, const BatchNet<MODE> &nb, int i, int cur,
                                                typename Tr<MODE>::A *ring, int lane) {
    const long long beg = a.rowptr[nb.off + i], end = a.rowptr[nb.off + i + 1];
    for (long long p0 = beg + lane; p0 < end; p0 += 32 * kPushAhead) {
        unsigned e[kPushAhead], w[kPushAhead];
#pragma unroll
        for (int u = 0; u < kPushAhead; ++u) {
            const long long p = p0 + 32 * u;
            e[u] = p < end ? __ldg(a.sidx + p) : 0u;
            w[u] = p < end ? __ldg(a.sw + p) : 0u;
        }
#pragma unroll
        for (int u = 0; u < kPushAhead; ++u) {
            if (p0 + 32 * u >= end) break;
            const int post = (int)(e[u] & 0xFFFu);
            int sl = cur + (int)(e[u] >> 12) + 1;
            if (sl >= a.D1) sl -= a.D1;
            atomicAdd(ring + (size_t)sl * nb.n + post, Tr<MODE>::to_acc(w[u]));
        }
    }
    return end - beg;
}

template <int MODE>
__device__ BatchNet<MODE> load_net(const BatchArgs &a, int b) {
    BatchNet<MODE> nb;
    nb.b = b;
    nb.off = a.net_off[b];
    nb.n = a.net_off[b + 1] - nb.off;
    nb.woff = a.word_off[b];
    nb.key = a.pkey[b];
    return nb;
}

// A load that stays where it is written: the compiler moves a plain load down
// into the guarded block of its accumulate, and the row's loads then wait for
// one another.
__device__ __forceinline__ unsigned ld_row_u16(const unsigned short *p, bool ok) {
    unsigned v;
    asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %2, 0;\n mov.u32 %0, 0;\n @q ld.global.nc.u16 %0, [%1];\n}"
                 : "=r"(v) : "l"(p), "r"((unsigned)ok));
    return v;
}
__device__ __forceinline__ unsigned ld_row_u32(const unsigned *p, bool ok) {
    unsigned v;
    asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %2, 0;\n mov.u32 %0, 0;\n @q ld.global.nc.u32 %0, [%1];\n}"
                 : "=r"(v) : "l"(p), "r"((unsigned)ok));
    return v;
}

// Fixed point (2^-32 units in 64 bits) to and from float, rounded to nearest
// even and saturating, bit for bit what the 64-bit conversions give.  Those are
// served at two lanes a cycle and SM (16 cycles a warp, measured); these take
// 32-bit ones and no branch: a conversion under a predicate costs its 16 cycles
// as well.  16 warps of an SM: 2.9 and 4.3 cycles a warp.
__device__ __forceinline__ unsigned long long fixed_from_float(float w) {
    const float m = fabsf(w);
    const int hi = __float2int_rz(m);
    // what is left is exact and below 1: one rounding, of the last product
    const unsigned lo = __float2uint_rn((m - __int2float_rn(hi)) * 4294967296.0f);
    unsigned long long u = ((unsigned long long)(unsigned)hi << 32) | lo;
    u = w < 0.0f ? 0ull - u : u;
    return m < 2147483648.0f ? u : w >= 2147483648.0f ? 0x7FFFFFFFFFFFFFFFull : 0x8000000000000000ull;
}
__device__ __forceinline__ float float_from_fixed(unsigned long long a) {
    const unsigned lo = (unsigned)a;
    const int hi = (int)(a >> 32);
    // two pieces of at most 24 bits, each exact, and one rounding of their sum.
    // From 2^48 on the lower piece is 23 bits above 2^16 and whether anything
    // lies below them, which is all the rounding needs to know.
    const bool big = (unsigned)(hi + 65536) >= 131072u;
    const int top = big ? hi >> 7 : (int)__funnelshift_r(lo, (unsigned)hi, 24);
    const unsigned mid = (__funnelshift_r(lo, (unsigned)hi, 16) & 0x7FFFFFu) * 2u + ((lo & 0xFFFFu) != 0u);
    const unsigned low = big ? mid : lo & 0xFFFFFFu;
    return __fmaf_rn(__int2float_rn(top), big ? 128.0f : 0.00390625f,
                     __uint2float_rn(low) * (big ? 7.62939453125e-06f : 2.3283064365386963e-10f));
}

template <int MODE>
__device__ __forceinline__ typename Tr<MODE>::A own_to_acc(unsigned wbits) {
    if constexpr (MODE == SN_F32) return fixed_from_float(__uint_as_float(wbits)); else return wbits;
}
template <int MODE>
__device__ __forceinline__ typename Tr<MODE>::V own_from_acc(typename Tr<MODE>::A a) {
    if constexpr (MODE == SN_F32) return float_from_fixed(a); else return (int)a;
}

// Adds to a 64-bit sum.  Shared memory has no 64-bit add, only a compare-and-swap
// loop; two 32-bit adds, the second with the first one's carry, give the same
// sum once both are in, and nobody reads it before the step's barrier.
__device__ __forceinline__ void add_shared(unsigned long long *p, unsigned long long x) {
    unsigned *q = (unsigned *)p;
    const unsigned lo = (unsigned)x, old = atomicAdd(q, lo);
    const unsigned hi = (unsigned)(x >> 32) + (old + lo < old ? 1u : 0u);
    if (hi) atomicAdd(q + 1, hi);
}
__device__ __forceinline__ void add_shared(unsigned *p, unsigned x) { atomicAdd(p, x); }

// All steps of a network of at most SLOTS * LANES neurons, by a block (LANES =
// 256) or a warp (32).  A step of the general form below is five dependent
// trips to memory: state and parameters, event range, row bounds, synapses, and
// the stores in between.  Here a thread keeps the state and the parameters of its
// neurons in registers, a spiker's list entry carries its row, and the external
// input of t + 1 is prepared while the first synapses of step t are on their way:
// one trip a step, 4.6 -> 2.5 us at 1021 neurons with two blocks an SM.  What bounds it now is the instruction
// issue of an SM's 16 warps (the draws' 64-bit multiplies, the rule, the synapses).
// A network of one neuron a thread at most takes SLOTS = 1: the rule and the draws of
// three empty slots made 2000 of 130 neurons 9 % slower than the general form (885 ->
// 961 us, 523 with one slot).
// `list` holds SLOTS * LANES rows and `rows` as many; `cnt` two counters, both
// zero.  (The row bounds lie in shared memory and the amplitudes, which few
// neurons need in a step, in global: at 128 registers a thread anything more
// spills, and with 28 KB of L1 left a spill is a trip to L2.)
constexpr int kOwn = 4;
static_assert(kListInts >= 4 * kOwn * kBatchBlock, "rows and list of a block (and of its warps)");

template <int MODE, int LANES, int SLOTS>
__device__ __forceinline__ void run_own(const BatchArgs &a, const BatchNet<MODE> &nb, typename Tr<MODE>::A *ring,
                                        bool global_ring, int tid, int2 *list, int2 *rows, int *cnt,
                                        unsigned long long &my_spikes, unsigned long long &my_events,
                                        bool &overflow) {
    using V = typename Tr<MODE>::V;
    using A = typename Tr<MODE>::A;
    const int lane = tid & 31, warp = tid >> 5;
    auto sync = [] { if (LANES == 32) __syncwarp(); else __syncthreads(); };
    V v[SLOTS], th[SLOTS], lk[SLOTS], rs[SLOTS], ext[SLOTS];
    int rr[SLOTS], R[SLOTS];
    unsigned thr[SLOTS];
    const long long base = a.rowptr[nb.off];
    const unsigned short *sidx = a.sidx + base;
    const unsigned *sw = a.sw + base;
#pragma unroll
    for (int u = 0; u < SLOTS; ++u) {
        const int j = u * LANES + tid, g = nb.off + j;
        thr[u] = 0;
        v[u] = th[u] = lk[u] = rs[u] = 0;
        rr[u] = R[u] = 0;
        if (j < nb.n) {
            v[u] = ((const V *)a.V)[g];
            rr[u] = a.r[g];
            th[u] = ((const V *)a.th)[g];
            lk[u] = ((const V *)a.lk)[g];
            rs[u] = ((const V *)a.rs)[g];
            R[u] = a.R[g];
            thr[u] = a.prate[g];
            // first synapse (from the network's first) and count; read by this thread alone
            const int b = (int)(a.rowptr[g] - base);
            rows[j] = make_int2(b, (int)(a.rowptr[g + 1] - base) - b);
        }
    }
    auto prepare = [&](int t) {
        const bool events = t < a.ev_nsteps && a.ev_off[t] < a.ev_off[t + 1];
#pragma unroll
        for (int u = 0; u < SLOTS; ++u) {
            const int j = u * LANES + tid;
            V x = 0;
            if (events && j < nb.n) {
                int lo = a.ev_off[t], hi = a.ev_off[t + 1];
                const int end = hi, g = nb.off + j;
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (a.ev_neuron[mid] < g) lo = mid + 1; else hi = mid;
                }
                if (lo < end && a.ev_neuron[lo] == g) x = ((const V *)a.ev_val)[lo];
            }
            if (thr[u] && poisson_fires(nb.key, (unsigned)t, (unsigned)j, thr[u])) {
                const V amp = __ldg((const V *)a.pamp + nb.off + j);
                if constexpr (MODE == SN_F32) x = __fadd_rn(x, amp); else x = x + amp;
            }
            ext[u] = x;
        }
    };
    prepare(a.t0);
    int cur = a.t0 % a.D1, at = a.t0 % a.cap;
    for (int s = 0; s < a.steps; ++s) {
        int *count = cnt + (s & 1);
        A *slot = ring + (size_t)cur * nb.n;
        unsigned *rrow = a.raster + (size_t)at * a.total_words + nb.woff;
        A raw[SLOTS];
        unsigned fired = 0;
#pragma unroll
        for (int u = 0; u < SLOTS; ++u) {
            const int j = u * LANES + tid;
            raw[u] = j < nb.n ? (global_ring ? __ldcg(slot + j) : slot[j]) : (A)0;
        }
        // the rules of all SLOTS neurons first, then their ballots: a neuron past
        // the network's end (no input, no draw, threshold 0) takes its turn too,
        // so that no branch parts one neuron's chain from the next
#pragma unroll
        for (int u = 0; u < SLOTS; ++u) {
            const V acc = own_from_acc<MODE>(raw[u]);
            bool fire;
            if constexpr (MODE == SN_F32)
                fire = lif_update_f32(v[u], rr[u], acc, ext[u], th[u], lk[u], rs[u], R[u]);
            else
                fire = lif_update_i32(v[u], rr[u], acc, ext[u], th[u], lk[u], rs[u], R[u], overflow);
            if (u * LANES + tid < nb.n) slot[u * LANES + tid] = 0;
            fired |= fire ? 1u << u : 0u;
        }
        int own = 0;                                       // spikers of the warp
#pragma unroll
        for (int u = 0; u < SLOTS; ++u) {
            const unsigned ball = __ballot_sync(0xffffffffu, (fired >> u) & 1u);
            const int wb = u * LANES + warp * 32;
            if (lane == 0 && wb < nb.n) rrow[wb >> 5] = ball;
            own += __popc(ball);
        }
        if (own) {
            int first = 0;
            if (LANES > 32) {
                if (lane == 0) first = atomicAdd(count, own);
                first = __shfl_sync(0xffffffffu, first, 0);
            }
#pragma unroll
            for (int u = 0; u < SLOTS; ++u) {
                const bool fire = (fired >> u) & 1u;
                const unsigned ball = __ballot_sync(0xffffffffu, fire);
                if (fire) list[first + __popc(ball & ((1u << lane) - 1u))] = rows[u * LANES + tid];
                first += __popc(ball);
            }
        }
        sync();
        const int k = LANES > 32 ? *count : own;
        if (tid == 0) {
            my_spikes += (unsigned long long)k;
            if (LANES > 32) cnt[(s & 1) ^ 1] = 0;
        }
        // the rows, 256 synapses at a time
        int q = warp, p = lane;
        int2 rw = q < k ? list[q] : make_int2(0, 0);
        unsigned e[kPushAhead], w[kPushAhead];
        auto load = [&] {
#pragma unroll
            for (int u = 0; u < kPushAhead; ++u) {
                const bool ok = p + 32 * u < rw.y;
                e[u] = ld_row_u16(sidx + rw.x + p + 32 * u, ok);
                w[u] = ld_row_u32(sw + rw.x + p + 32 * u, ok);
            }
        };
        if (q < k) load();
        if (s + 1 < a.steps) prepare(a.t0 + s + 1);
        while (q < k) {
#pragma unroll
            for (int u = 0; u < kPushAhead; ++u) {
                if (p + 32 * u < rw.y) {
                    const int post = (int)(e[u] & 0xFFFu);
                    int sl = cur + (int)(e[u] >> 12) + 1;
                    if (sl >= a.D1) sl -= a.D1;
                    A *to = ring + sl * nb.n + post;
                    if (global_ring) atomicAdd(to, own_to_acc<MODE>(w[u]));
                    else add_shared(to, own_to_acc<MODE>(w[u]));
                }
            }
            p += 32 * kPushAhead;
            if (p - lane >= rw.y) {
                if (lane == 0) my_events += (unsigned long long)rw.y;
                q += LANES / 32;
                p = lane;
                if (q < k) rw = list[q];
            }
            if (q < k) load();
        }
        sync();
        cur = cur + 1 < a.D1 ? cur + 1 : 0;
        at = at + 1 < a.cap ? at + 1 : 0;
    }
#pragma unroll
    for (int u = 0; u < SLOTS; ++u) {
        const int j = u * LANES + tid;
        if (j < nb.n) {
            ((V *)a.V)[nb.off + j] = v[u];
            a.r[nb.off + j] = rr[u];
        }
    }
}

// FORM 0: the general form; 1 and 2: every network takes run_own (batch_form), with 2
// the blocks' networks of one neuron a thread in an instantiation of theirs.  Kernels
// of their own: with the general form in one the registers of either spill (136 bytes;
// networks of 4096 neurons 1.7 times the time), and with the one-slot loop in it the
// others' are about 1 % slower (100 networks of 300 to 1024, 60 steps: 207.5 us and 205.7).
template <int MODE, int FORM>
__global__ void __launch_bounds__(kBatchBlock, 2) batch_kernel(BatchArgs a) {
    using A = typename Tr<MODE>::A;
    extern __shared__ __align__(16) unsigned char smem[];
    A *arena = (A *)smem;                                  // ring arena
    int *lists = (int *)(smem + a.ring_smem);              // spiker lists
    __shared__ int s_item, s_cnt, s_own[2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long my_spikes = 0, my_events = 0;
    bool overflow = false;

    // Some blocks, the last ones, take warps' networks from the start: a warp needs
    // as long for one of 128 neurons as a block for one of 1024, and begun after
    // the blocks' queue was empty they were the last 250 us of 480.
    constexpr bool OWN = FORM != 0;
    const int early = OWN && a.n_cta ? min((a.n_warp + kWarps - 1) / kWarps, (int)gridDim.x / 8) : 0;
    const bool warps_first = (int)(gridDim.x - blockIdx.x) <= early;
    // ---- networks run by the whole block
    while (!warps_first) {
        // thread 0 decides for the whole block (a latched status ends the work)
        if (threadIdx.x == 0)
            s_item = ld_status(a.ctl) != 0 ? a.n_cta : (int)atomicAdd(&a.ctl->queue[0], 1u);
        __syncthreads();
        const int item = s_item;
        __syncthreads();
        if (item >= a.n_cta) break;
        const BatchNet<MODE> nb = load_net<MODE>(a, a.cta_order[item]);
        A *gring = (A *)a.ring + a.ring_off[nb.b];
        const size_t ring_elems = (size_t)a.D1 * nb.n;
        const bool in_smem = ring_elems * sizeof(A) <= (size_t)a.ring_smem;
        A *ring = in_smem ? arena : gring;
        if (in_smem)
            for (size_t q = threadIdx.x; q < ring_elems; q += blockDim.x) arena[q] = __ldcg(gring + q);
        if (OWN && threadIdx.x < 2) s_own[threadIdx.x] = 0;
        __syncthreads();
        if constexpr (OWN)
        {
            int2 *list = (int2 *)lists, *rows = list + kOwn * kBatchBlock;
            if (FORM == 2 && nb.n <= kBatchBlock)
                run_own<MODE, kBatchBlock, 1>(a, nb, ring, !in_smem, threadIdx.x, list, rows, s_own, my_spikes,
                                              my_events, overflow);
            else
                run_own<MODE, kBatchBlock, kOwn>(a, nb, ring, !in_smem, threadIdx.x, list, rows, s_own, my_spikes,
                                                 my_events, overflow);
        }
        for (int s = OWN ? a.steps : 0; s < a.steps; ++s) {
            const int t = a.t0 + s;
            const int cur = t % a.D1;
            A *slot = ring + (size_t)cur * nb.n;
            unsigned *rrow = a.raster + (size_t)(t % a.cap) * a.total_words + nb.woff;
            if (threadIdx.x == 0) s_cnt = 0;
            __syncthreads();
            for (int jb0 = 0; jb0 < nb.n; jb0 += kUpdAhead * blockDim.x) {
                NeuronIn<MODE> in[kUpdAhead];
#pragma unroll
                for (int u = 0; u < kUpdAhead; ++u) {
                    const int j = jb0 + u * blockDim.x + threadIdx.x;
                    if (j < nb.n) batch_load<MODE>(a, nb, j, slot, !in_smem, in[u]);
                }
#pragma unroll
                for (int u = 0; u < kUpdAhead; ++u) {
                    const int jb = jb0 + u * blockDim.x;
                    if (jb >= nb.n) break;
                    const int j = jb + threadIdx.x;
                    const bool fire = j < nb.n && batch_finish<MODE>(a, nb, t, j, slot, in[u], overflow);
                    const unsigned ball = __ballot_sync(0xffffffffu, fire);
                    const int wb = jb + warp * 32;
                    if (lane == 0 && wb < nb.n) rrow[wb >> 5] = ball;
                    if (ball) {
                        int base = 0;
                        if (lane == 0) base = atomicAdd(&s_cnt, __popc(ball));
                        base = __shfl_sync(0xffffffffu, base, 0);
                        if (fire) lists[base + __popc(ball & ((1u << lane) - 1u))] = j;
                    }
                }
            }
            __syncthreads();
            const int k = s_cnt;
            if (threadIdx.x == 0) my_spikes += (unsigned long long)k;
            for (int q = warp; q < k; q += kWarps) {
                const long long len = batch_push<MODE>(a, nb, lists[q], cur, ring, lane);
                if (lane == 0) my_events += (unsigned long long)len;
            }
            __syncthreads();
        }
        if (in_smem)
            for (size_t q = threadIdx.x; q < ring_elems; q += blockDim.x) gring[q] = arena[q];
        __syncthreads();
    }

    const int warp_ring_bytes = (a.ring_smem / kWarps) & ~15;
    A *wring_smem = (A *)(smem + (size_t)warp * warp_ring_bytes);
    int *wlist = lists + warp * (kListInts / kWarps);
    // ---- networks run by single warps
    for (;;) {
        int item = 0;
        if (lane == 0) item = ld_status(a.ctl) != 0 ? a.n_warp : (int)atomicAdd(&a.ctl->queue[1], 1u);
        item = __shfl_sync(0xffffffffu, item, 0);
        if (item >= a.n_warp) break;
        const BatchNet<MODE> nb = load_net<MODE>(a, a.warp_order[item]);
        A *gring = (A *)a.ring + a.ring_off[nb.b];
        const size_t ring_elems = (size_t)a.D1 * nb.n;
        const bool in_smem = ring_elems * sizeof(A) <= (size_t)warp_ring_bytes;
        A *ring = in_smem ? wring_smem : gring;
        if (in_smem)
            for (size_t q = lane; q < ring_elems; q += 32) wring_smem[q] = __ldcg(gring + q);
        __syncwarp();
        if constexpr (OWN)
            run_own<MODE, 32, kOwn>(a, nb, ring, !in_smem, lane, (int2 *)wlist, (int2 *)wlist + kOwn * 32, nullptr,
                              my_spikes, my_events, overflow);
        for (int s = OWN ? a.steps : 0; s < a.steps; ++s) {
            const int t = a.t0 + s;
            const int cur = t % a.D1;
            A *slot = ring + (size_t)cur * nb.n;
            unsigned *rrow = a.raster + (size_t)(t % a.cap) * a.total_words + nb.woff;
            int cnt = 0;
            for (int jb0 = 0; jb0 < nb.n; jb0 += kUpdAhead * 32) {
                NeuronIn<MODE> in[kUpdAhead];
#pragma unroll
                for (int u = 0; u < kUpdAhead; ++u) {
                    const int j = jb0 + u * 32 + lane;
                    if (j < nb.n) batch_load<MODE>(a, nb, j, slot, !in_smem, in[u]);
                }
#pragma unroll
                for (int u = 0; u < kUpdAhead; ++u) {
                    const int jb = jb0 + u * 32;
                    if (jb >= nb.n) break;
                    const int j = jb + lane;
                    const bool fire = j < nb.n && batch_finish<MODE>(a, nb, t, j, slot, in[u], overflow);
                    const unsigned ball = __ballot_sync(0xffffffffu, fire);
                    if (lane == 0) rrow[jb >> 5] = ball;
                    if (fire) wlist[cnt + __popc(ball & ((1u << lane) - 1u))] = j;
                    cnt += __popc(ball);
                }
            }
            __syncwarp();
            if (lane == 0) my_spikes += (unsigned long long)cnt;
            for (int q = 0; q < cnt; ++q) {
                const long long len = batch_push<MODE>(a, nb, wlist[q], cur, ring, lane);
                if (lane == 0) my_events += (unsigned long long)len;
            }
            __syncwarp();
        }
        if (in_smem)
            for (size_t q = lane; q < ring_elems; q += 32) gring[q] = wring_smem[q];
        __syncwarp();
    }
    if (MODE == SN_I32 && overflow) atomicCAS(&a.ctl->status, 0, (int)SN_EOVERFLOW);
    if (my_spikes) atomicAdd(&a.ctl->spikes, my_spikes);
    if (my_events) atomicAdd(&a.ctl->events, my_events);
}

size_t batch_smem(int ring_smem) { return (size_t)ring_smem + (size_t)kListInts * sizeof(int); }

static const void *batch_fn(int dtype, int form) {
    const bool f = dtype == SN_F32;
    if (form == 2) return f ? (const void *)batch_kernel<SN_F32, 2> : (const void *)batch_kernel<SN_I32, 2>;
    if (form == 1) return f ? (const void *)batch_kernel<SN_F32, 1> : (const void *)batch_kernel<SN_I32, 1>;
    return f ? (const void *)batch_kernel<SN_F32, 0> : (const void *)batch_kernel<SN_I32, 0>;
}

// run_own where the largest networks of the blocks and of the warps fit kOwn neurons a
// thread (sizes of the blocks' networks: 0, 0 when there are none).
// Measured (100 steps, us, general form first): 512 networks of 64 to 1024, 492 and
// 275; 2000 of 32 to 128, 350 and 222; 32 of 64 to 300, 270 and 190; 2000 of 130, 885
// and 523; 1000 of 1000 with 304 of 20, 1913 and 1125.
int batch_form(int min_block_n, int max_block_n, int max_warp_n) {
    if (max_block_n > kOwn * kBatchBlock || max_warp_n > kOwn * 32) return 0;
    return min_block_n > 0 && min_block_n <= kBatchBlock ? 2 : 1;
}

cudaError_t batch_kernel_node(int dtype, int form, void **fn) {
    *fn = (void *)batch_fn(dtype, form);
    return cudaSuccess;
}

cudaError_t max_grid_batch(int dtype, int form, int ring_smem, int *grid) {
    int dev = 0, sms = 0, per = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const size_t smem = batch_smem(ring_smem);
    if ((e = allow_all_smem(batch_fn(dtype, form))) != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, batch_fn(dtype, form), kBatchBlock, smem);
    if (e != cudaSuccess) return e;
    *grid = per * sms;
    return cudaSuccess;
}

}  // namespace sn
