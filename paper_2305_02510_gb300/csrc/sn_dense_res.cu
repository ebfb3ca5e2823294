// Dense network whose weights fit the chip's shared memory: every block keeps
// its column slab for the whole launch.
//
// The streaming form (sn_kernels.cu) fetches the spikers' rows from L2 at every
// step.  For a network of one to two thousand neurons that is a chain of L2
// round trips, not bandwidth: 1001 neurons at 0.9 of them firing took 8.4 us a
// step, of which the 0.1 MB a block reads would be well under one.  Here block
// c loads W[:, slab] once per launch (n * 128 bytes at 32 columns), and a step is
//   update(t):  own neurons; the spike word goes to its slot of a two-row
//               buffer with the step's number in the high half, so the word
//               says itself that it has arrived (no grid barrier: the words
//               are the only thing blocks pass to one another);
//   row(t):     two warps read the row's words until each carries the step's
//               number, while the owners prepare the external input of t + 1;
//   gather(t):  the spikers' ranks, then the same partial sums, in the same
//               order, as the streaming form: bit-identical results;
//   STDP:       the slab's columns of every row belong to this block, so the
//               updates are shared-memory ones; each block keeps all the
//               traces (they follow from the spikes), and the slab goes back
//               to memory at the end of the launch.
// The words of a row lie a cache line apart: 32 blocks polling two lines full
// of words queue at one L2 slice (1001 neurons: 2.18 us a step against 1.82).
// What bounds it now (1001 neurons, nearly all firing: 2.5 us a step, of 8.4): the
// exchange of the words, about 1.2 us (store, line to the reader, one poll too
// early), and the slab's rows at one 128-byte row a cycle, 0.6 us.  200 steps
// take 501 us (1686 streaming); 1000 neurons at 0.2 with STDP 4.2 us a step (8.2),
// 128 neurons in one block 0.9 (2.2) and with STDP 4.3 (8.7).
// A row slot is reused two steps later: a block stores its word of t + 2 only
// after it has seen every word of t + 1, which every block stores after its
// last read of row t.

#include <cuda_runtime.h>

#include "sn_device.cuh"
#include "sn_internal.h"

namespace sn {

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kPollers = 64;               // the last threads of a block read the row, a word each
constexpr int kMaxWords = kPollers;

__host__ __device__ constexpr int chain_len(int n) { return ((n + kWarps - 1) / kWarps + 15) & ~15; }
// Columns from one row of the slab to the next: with STDP one more than the
// slab has, so that the rows of one column lie in different banks.
__host__ __device__ constexpr int slab_ld(int cw, bool stdp) { return stdp ? cw + 1 : cw; }

// Bytes of shared memory: slab with a row of zeros after it, the chains' row
// offsets, partial sums (as many as 8 warps * 4 * 32), two spike rows, traces.
size_t res_smem(int n, int cw, bool stdp) {
    return (((size_t)(n + 1) * slab_ld(cw, stdp) + 3) / 4 * 4 + (size_t)kWarps * chain_len(n) + kWarps * 128 + 2 * kMaxWords + (stdp ? n + 1 : 0)) * 4;
}

__device__ __forceinline__ void copy_async16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void copy_async4(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" :: "r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void copy_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ unsigned long long ld_word(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// One word of the row once it carries `tag`; bounded like the grid barrier.
__device__ __forceinline__ bool poll_word(const unsigned long long *p, unsigned tag, unsigned &bits, Control *ctl) {
    unsigned long long v = ld_word(p), began = 0;
    for (unsigned spins = 1; (unsigned)(v >> 32) != tag; ++spins) {
        if ((spins & 63u) == 0) {
            const unsigned long long now = global_timer_ns();
            if (began == 0) began = now;
            if (ld_status(ctl) != 0) return false;
            if (now - began > kBarrierTimeoutNs) {
                atomicCAS(&ctl->status, 0, (int)SN_ETIMEOUT);
                return false;
            }
        }
        v = ld_word(p);
    }
    bits = (unsigned)v;
    return true;
}

// CPL columns per lane; RPI chains per warp: the streaming form's vector gather
// sums 32 / (8 * CPL) rows side by side, its scalar gather one.
template <int CPL, int RPI, bool STDP>
__global__ void __launch_bounds__(kThreads, 1) dense_res_kernel(NetArgs a) {
    extern __shared__ float smem_f[];
    constexpr int cw = 32 * CPL, ld = slab_ld(cw, STDP);
    const int n = a.n, W = a.words;
    const int L8 = chain_len(n);
    float *slab = smem_f;                                    // [n + 1][ld], the last row zero
    int *chain = (int *)(slab + ((n + 1) * ld + 3) / 4 * 4); // [kWarps][L8] slab offsets of the spikers' rows
    float *wpart = (float *)(chain + kWarps * L8);           // [kWarps][RPI][cw]
    unsigned *s_bits = (unsigned *)(wpart + kWarps * 128);   // [2][kMaxWords]
    float *s_x = (float *)(s_bits + 2 * kMaxWords);          // [n + 1] traces x(t - 1)
    __shared__ int s_stop;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int c0 = blockIdx.x * cw;
    const int j = c0 + tid;
    const bool mine = tid < cw && j < n;
    float *ring = (float *)a.ring, *out = ring;

    if (tid == 0) s_stop = ld_status(a.ctl);
    __syncthreads();
    if (s_stop) return;
    if (!STDP && n % 4 == 0 && ((size_t)a.W & 15u) == 0) {
        constexpr int G = cw / 4;
        for (int i = tid; i < n * G; i += kThreads) {
            const int row = i / G, g = 4 * (i % G);
            if (c0 + g < n) copy_async16(slab + row * ld + g, a.W + (size_t)row * n + c0 + g);
        }
    } else {
        for (int i = tid; i < n * cw; i += kThreads) {
            const int row = i / cw, g = i % cw;
            if (c0 + g < n) copy_async4(slab + row * ld + g, a.W + (size_t)row * n + c0 + g);
        }
    }
    if (tid < cw) slab[n * ld + tid] = 0.0f;
    if constexpr (STDP)
        for (int i = tid; i < n; i += kThreads) s_x[i] = a.trace[(size_t)((a.t0 + 2) % 3) * n + i];

    float v = 0, th = 0, lk = 0, rs = 0, amp = 0, acc_in = 0, ext = 0;
    int rr = 0, R = 0;
    unsigned thr = 0;
    unsigned long long my_spikes = 0;
    // the external input of step t and, unless it is the last fold itself
    // (delay 1 after the first step), the pending synaptic input
    int at = a.t0 % a.cap;                                   // the step's raster row
    auto input = [&](int t, bool from_ring) {
        ext = 0.0f;
        if (t < a.ev_nsteps) {
            int lo = a.ev_off[t], hi = a.ev_off[t + 1];
            const int end = hi;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (a.ev_neuron[mid] < j) lo = mid + 1; else hi = mid;
            }
            if (lo < end && a.ev_neuron[lo] == j) ext = ((const float *)a.ev_val)[lo];
        }
        if (thr && poisson_fires(a.pkey, (unsigned)t, (unsigned)j, thr)) ext = __fadd_rn(ext, amp);
        if (from_ring) acc_in = ring[(size_t)(t % a.D1) * n + j];
    };
    if (mine) {
        v = ((const float *)a.V)[j];
        rr = a.r[j];
        th = ((const float *)a.th)[j];
        lk = ((const float *)a.lk)[j];
        rs = ((const float *)a.rs)[j];
        R = a.R[j];
        thr = a.prate[j];
        amp = ((const float *)a.pamp)[j];
        input(a.t0, true);
    }
    copy_async_wait();
    __syncthreads();

    for (int s = 0; s < a.steps; ++s) {
        const int t = a.t0 + s;
        const unsigned tag = (unsigned)s + 1u;
        unsigned *bits = s_bits + (s & 1) * kMaxWords;
        unsigned long long *row = a.ptag + (size_t)(s & 1) * W * kDenseTagStride;
        // ---- update(t)
        if (tid < cw) {
            const bool fire = mine && lif_update_f32(v, rr, acc_in, ext, th, lk, rs, R);
            const unsigned ball = __ballot_sync(0xffffffffu, fire);
            if (lane == 0 && c0 + warp * 32 < n) {
                const int word = (c0 >> 5) + warp;
                if (gridDim.x > 1) st_tagged(row + kDenseTagStride * word, tag, ball); else bits[word] = ball;
                a.spk[(size_t)(t & 1) * W + word] = ball;
                a.raster[(size_t)at * W + word] = ball;
                my_spikes += (unsigned long long)__popc(ball);
            }
            at = at + 1 < a.cap ? at + 1 : 0;
            out = ring + (size_t)((t + a.dense_delay) % a.D1) * n + j;
            // the next step's external input, while the other words arrive
            if (mine && s + 1 < a.steps) input(t + 1, a.dense_delay > 1);
        } else if (tid >= kThreads - kPollers && gridDim.x > 1) {
            const int w = tid - (kThreads - kPollers);
            if (w < W && !poll_word(row + kDenseTagStride * w, tag, bits[w], a.ctl)) s_stop = 1;
        }
        __syncthreads();
        if (s_stop) break;

        // ---- the spikers in ascending order: rank r is entry r / 8 of chain r % 8
        // (a lane holds the bits and the rank before them of words lane, lane + 32)
        const unsigned b0 = lane < W ? bits[lane] : 0u, b1 = lane + 32 < W ? bits[lane + 32] : 0u;
        int base0 = __popc(b0), base1 = __popc(b1);
        {
            const int p0 = base0, p1 = base1;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y0 = __shfl_up_sync(0xffffffffu, base0, o);
                const int y1 = __shfl_up_sync(0xffffffffu, base1, o);
                base0 += lane >= o ? y0 : 0;
                base1 += lane >= o ? y1 : 0;
            }
            const int low = __shfl_sync(0xffffffffu, base0, 31);
            base0 -= p0;
            base1 += low - p1;
        }
        const int k = __shfl_sync(0xffffffffu, base1 + __popc(b1), 31);
        const int rows = k > warp ? (k - warp + kWarps - 1) / kWarps : 0, rows_up = (rows + 15) & ~15;
        int *ch = chain + warp * L8;
        if (rows + lane < rows_up) ch[rows + lane] = n * ld;
        auto emit = [&](unsigned bl, int basel, int w) {
            const unsigned b = __shfl_sync(0xffffffffu, bl, w & 31);
            const int r = __shfl_sync(0xffffffffu, basel, w & 31) + __popc(b & ((1u << lane) - 1u));
            if ((b >> lane) & 1u) chain[(r & (kWarps - 1)) * L8 + r / kWarps] = (w * 32 + lane) * ld;
        };
#pragma unroll
        for (int w = 0; w < 32; w += kWarps) emit(b0, base0, w + warp);
        if (W > 32)
#pragma unroll
            for (int w = 32; w < kMaxWords; w += kWarps) emit(b1, base1, w + warp);
        __syncthreads();

        // ---- gather(t), and STDP of step t
        float acc[RPI][CPL];
#pragma unroll
        for (int q = 0; q < RPI; ++q)
#pragma unroll
            for (int c = 0; c < CPL; ++c) acc[q][c] = 0.0f;
        bool sc[CPL];
        float xc[CPL];
        if constexpr (STDP) {
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
                const int col = c0 + lane + 32 * c;
                sc[c] = col < n && spiked(bits, col);
                xc[c] = col < n ? s_x[col] : 0.0f;
            }
        }
        // U rows are loaded while the U before them are added.  An entry past the
        // chain's end is the row of zeros: a sum that began at +0 never becomes
        // -0, so adding +0 leaves its bits alone, and no branch parts a load
        // from the loads around it (a guard here made the compiler wait for each
        // row by itself: 52 cycles a row instead of 8)
        constexpr int U = 16 / CPL;
        int off[U];
        float wv[U][CPL];
        auto load = [&](int k0) {
#pragma unroll
            for (int u = 0; u < U; u += 4) {
                const int4 x = *(const int4 *)(ch + k0 + u);
                off[u] = x.x; off[u + 1] = x.y; off[u + 2] = x.z; off[u + 3] = x.w;
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int c = 0; c < CPL; ++c) wv[u][c] = slab[off[u] + lane + 32 * c];
        };
        if (rows > 0) load(0);
        for (int k0 = 0; k0 < rows; k0 += U) {
            float w[U][CPL];
            int o[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                o[u] = off[u];
#pragma unroll
                for (int c = 0; c < CPL; ++c) w[u][c] = wv[u][c];
            }
            load(min(k0 + U, rows_up - U));
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if constexpr (STDP) {
                    const int i = o[u] / ld;
                    const float up = __fmul_rn(a.a_plus, s_x[i]);
#pragma unroll
                    for (int c = 0; c < CPL; ++c) {
                        const float dw = __fsub_rn(sc[c] ? up : 0.0f, __fmul_rn(a.a_minus, xc[c]));
                        const float nw = clampf(__fadd_rn(w[u][c], dw), a.wmin, a.wmax);
                        const bool change = c0 + lane + 32 * c != i && i < n;
                        if (change) slab[o[u] + lane + 32 * c] = nw;
                        w[u][c] = change ? nw : w[u][c];
                    }
                }
#pragma unroll
                for (int c = 0; c < CPL; ++c) acc[u % RPI][c] = __fadd_rn(acc[u % RPI][c], w[u][c]);
            }
        }
        if constexpr (STDP) {
            // LTP in the slab's spiking columns, rows that did not spike: a lane a
            // row; where there are fewer words of rows than warps, the warps of
            // one word share out its columns
            const int share = W < kWarps ? kWarps / W : 1, step = W < kWarps ? W : kWarps;
            unsigned m[CPL];
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
                const unsigned b = (c0 >> 5) + c < W ? bits[(c0 >> 5) + c] : 0u;
                const int r = __popc(b & ((1u << lane) - 1u));
                m[c] = share == 1 ? b : __ballot_sync(0xffffffffu, ((b >> lane) & 1u) && r % share == warp / step);
            }
            if (warp < share * step) {
                for (int w = warp % step; w < W; w += step) {
                    const int i = w * 32 + lane;
                    const bool quiet = i < n && !((bits[w] >> lane) & 1u);
                    const float up = quiet ? __fmul_rn(a.a_plus, s_x[i]) : 0.0f;
                    float *p = slab + i * ld;
#pragma unroll
                    for (int c = 0; c < CPL; ++c) {
                        for (unsigned rest = m[c]; rest;) {
                            int col[4];
                            float val[4];
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                col[u] = rest ? 32 * c + __ffs(rest) - 1 : -1;
                                rest &= rest - 1u;
                                val[u] = (quiet && col[u] >= 0) ? p[col[u]] : 0.0f;
                            }
#pragma unroll
                            for (int u = 0; u < 4; ++u)
                                if (quiet && col[u] >= 0) p[col[u]] = clampf(__fadd_rn(val[u], up), a.wmin, a.wmax);
                        }
                    }
                }
            }
        }
#pragma unroll
        for (int q = 0; q < RPI; ++q)
#pragma unroll
            for (int c = 0; c < CPL; ++c) wpart[(warp * RPI + q) * cw + lane + 32 * c] = acc[q][c];
        __syncthreads();
        // fold in the streaming form's order; the input of t + delay
        if (mine) {
            float sum = 0.0f;
#pragma unroll
            for (int w = 0; w < kWarps * RPI; ++w) sum = __fadd_rn(sum, wpart[w * cw + tid]);
            *out = sum;
            if (a.dense_delay == 1) acc_in = sum;
        }
        if constexpr (STDP) {
            for (int i = tid; i < n; i += kThreads) {
                const float x = __fadd_rn(__fmul_rn(a.decay, s_x[i]), spiked(bits, i) ? 1.0f : 0.0f);
                s_x[i] = x;
                if (i >= c0 && i < c0 + cw) a.trace[(size_t)(t % 3) * n + i] = x;
            }
        }
    }
    if (mine) {
        ((float *)a.V)[j] = v;
        a.r[j] = rr;
    }
    if (my_spikes) {
        atomicAdd(&a.ctl->spikes, my_spikes);
        atomicAdd(&a.ctl->events, my_spikes * (unsigned long long)n);
    }
    if constexpr (STDP) {
        __syncthreads();
        for (int i = tid; i < n * cw; i += kThreads) {
            const int row = i / cw, g = i % cw;
            if (c0 + g < n) a.W[(size_t)row * n + c0 + g] = slab[row * ld + g];
        }
    }
}

__global__ void dense_tag_init_kernel(unsigned long long *tag, int words) {
    for (int i = threadIdx.x; i < words; i += blockDim.x) tag[i] = 0;
}

const void *res_fn(int cpl, bool stdp, bool vec) {
    if (stdp)
        return cpl == 1   ? (const void *)dense_res_kernel<1, 1, true>
               : cpl == 2 ? (const void *)dense_res_kernel<2, 1, true>
                          : (const void *)dense_res_kernel<4, 1, true>;
    if (vec)
        return cpl == 1   ? (const void *)dense_res_kernel<1, 4, false>
               : cpl == 2 ? (const void *)dense_res_kernel<2, 2, false>
                          : (const void *)dense_res_kernel<4, 1, false>;
    return cpl == 1   ? (const void *)dense_res_kernel<1, 1, false>
           : cpl == 2 ? (const void *)dense_res_kernel<2, 1, false>
                      : (const void *)dense_res_kernel<4, 1, false>;
}

}  // namespace

// Whether a run of `steps` steps takes the resident slabs: they fit (1715
// neurons at 32 columns a block, 1617 with STDP), every block has an SM of its
// own, and the launch is long enough to pay for loading them and, with STDP, for
// writing them back.  Measured at the line (launch included), resident against
// streaming: 1600 neurons, 4 steps, 20.4 us against 22.9; with STDP 4 steps 37
// against 32, 8 steps 54.5 against 52.4, 50 steps 318 against 513.
bool dense_res_fits(int n, int chunk, int grid, bool stdp, int steps) {
    int dev = 0, sms = 0, lim = 0;
    if (steps < (stdp ? kDenseResStepsStdp : kDenseResSteps) || chunk > 128 || (n + 31) / 32 > kMaxWords) return false;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&lim, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        return false;
    return grid <= sms && res_smem(n, chunk, stdp) + 1024 <= (size_t)lim;
}

size_t dense_tag_bytes(int n) {
    const int words = (n + 31) / 32;
    return words > kMaxWords ? 0 : (size_t)2 * words * kDenseTagStride * 8;
}

cudaError_t plan_dense_res(int chunk) {
    if (chunk > 128) return cudaSuccess;
    for (const void *fn : {res_fn(chunk / 32, false, false), res_fn(chunk / 32, false, true), res_fn(chunk / 32, true, false)})
        if (cudaError_t e = allow_all_smem(fn)) return e;
    return cudaSuccess;
}

cudaError_t launch_dense_res(const NetArgs &a, int grid, cudaStream_t s) {
    const bool vec = a.n % 4 == 0 && ((uintptr_t)a.W & 15u) == 0;
    const void *fn = res_fn(a.chunk / 32, a.stdp != 0, vec);
    if (grid > 1) {
        dense_tag_init_kernel<<<1, 256, 0, s>>>(a.ptag, 2 * a.words * kDenseTagStride);
        if (cudaError_t e = cudaGetLastError()) return e;
    }
    void *args[] = {(void *)&a};
    return cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(kThreads), args, res_smem(a.n, a.chunk, a.stdp != 0), s);
}

}  // namespace sn
