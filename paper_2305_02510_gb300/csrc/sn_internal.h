// Internal declarations shared by the host API (sn_api.cu) and the kernel
// translation units.  Not part of the public ABI.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "../../include/sn.h"

namespace sn {

// The limit on a kernel's dynamic shared memory is the function's, shared by every
// context and thread of the process.  It is set to all that a block may have, never
// to one network's bytes: a smaller network planned or launched by another thread
// between a set and its launch would lower it under that launch.
inline cudaError_t allow_all_smem(const void *fn) {
    int dev = 0, lim = 0;
    cudaFuncAttributes at;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&lim, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&at, fn);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, lim - (int)at.sharedSizeBytes);
}

enum Kind { KIND_SPARSE = 0, KIND_DENSE = 1, KIND_BATCH = 2, KIND_SHARED_I8 = 3, KIND_FF = 4 };

// Grid barrier state (one per context): the arrival count of the running
// launch, zeroed before every launch that uses it.
struct GridBarrier {
    unsigned int count;
    unsigned int pad;
};

// Device-side control block: latched status word and run counters.
struct Control {
    int status;                       // 0 or an sn_status latched by a kernel
    int pad;
    unsigned long long spikes;        // total spikes
    unsigned long long events;        // total synaptic events
    GridBarrier bar;
    unsigned queue[2];                // batched work queues: next block item, next warp item
};

// Wall-clock limit of one grid-barrier wait before the kernel gives up and
// latches SN_ETIMEOUT (nanoseconds of %globaltimer).
constexpr unsigned long long kBarrierTimeoutNs = 2000000000ull;

// Packed synapse of the CSR (pre-major) store: x = post | (delay-1) << 26,
// y = weight bits (float in SN_F32 mode, int32 in SN_I32 mode).
constexpr int kPostBits = 26;
constexpr unsigned kPostMask = (1u << kPostBits) - 1u;

// Arguments of the single-network kernels (sparse push and dense gather).
struct NetArgs {
    int n, D1, words, cap;            // neurons, ring slots (D+1), raster words/row, raster rows
    int t0, steps;                    // first absolute step, steps to run
    int chunk;                        // neurons owned per block (multiple of 32)
    // neuron state and parameters (float or int32 according to the mode)
    void *V;
    int *r;
    const void *th, *lk, *rs;
    const int *R;
    const unsigned *prate;            // Poisson threshold per neuron (0: no source)
    const void *pamp;                 // Poisson amplitude per neuron
    unsigned long long pkey;          // Poisson stream key of the network
    // explicit events, deduplicated per (step, neuron), sorted by neuron per step
    const int *ev_off;                // [ev_nsteps + 1] offsets by absolute step
    int ev_nsteps;
    const int *ev_neuron;
    const void *ev_val;
    // sparse store (CSR by pre)
    const long long *rowptr;
    uint2 *syn;                       // weights are rewritten in place by STDP
    const long long *colptr;          // CSC by post (STDP only)
    const uint2 *csc;                 // {pre, CSR position}
    void *ring;                       // [D1][n] pending input (int64 fixed point / int32 / float)
    // sparse store for pull propagation (sn_pull.cu): incoming synapses of
    // 32-neuron slices, plain ({bit offset, weight bits} pairs) or coded
    // (groups of 8 weights and 16-bit offset steps)
    const uint4 *pin;
    const long long *pin_off;         // [slices] first uint4 of each slice
    const int *pin_len;               // [regions][n] entries of each region of each position's list
                                      // (sn_pull.cu: delay >= 2, delay 1; sn_pull_block.cu: five)
    const unsigned *pin_y0;           // coded store: [2][n] window bit offset of each region's first entry
    const int *pin_perm;              // [n] the neuron whose lists thread position p sums (the store,
                                      // pin_len and pin_y0 are indexed by position)
    unsigned long long *ptag;         // blocked pull, resident dense: spike words of the last steps with
                                      // the step's number in the high half
    int wp, wt, rows_at, acc_at;     // blocked pull: words rounded up to 4 and to 2, bytes of shared
                                      // memory before the two rows and before the sums
    unsigned *hist;                   // [hD][words] spike bits of step tau in row tau % hD
    int hD;                           // history depth (the maximum delay D)
    int hL;                           // rows of the pull kernel's shared-memory window
    int ring_until;                   // the ring may hold pending input for steps < ring_until
    int j_first, j_end;               // pull: the neurons [j_first, j_end) this launch simulates
                                      // (a shard of the network; 0 and n otherwise)
    // dense store
    float *W;                         // [n][n]
    float *partial;                   // [S][n] gather partial sums
    int S, dense_delay;
    // spikes
    unsigned *raster;                 // [cap][words]
    unsigned *spk;                    // [2][words] spike bits of the last two steps (dense)
    // STDP
    int stdp;
    float decay, a_plus, a_minus, wmin, wmax;
    float *trace;                     // [3][n]: sparse kernels use buffer t & 1, dense t % 3
    Control *ctl;
};

// Arguments of the batched kernel: many independent networks, each run for
// all steps by one block or one warp.
struct BatchArgs {
    int nets, t0, steps, cap, total_words, D1;
    const int *net_off;               // [nets + 1] first neuron of each network
    const int *word_off;              // [nets + 1] first raster word of each network
    const long long *ring_off;        // [nets] first ring element of each network (D1 * n_b)
    const unsigned long long *pkey;   // [nets] Poisson stream key
    const int *cta_order;             // networks run by whole blocks, largest first
    int n_cta;
    const int *warp_order;            // networks run by single warps
    int n_warp;
    void *V;
    int *r;
    const void *th, *lk, *rs;
    const int *R;
    const unsigned *prate;
    const void *pamp;
    const int *ev_off;
    int ev_nsteps;
    const int *ev_neuron;
    const void *ev_val;
    const long long *rowptr;          // [sum n + 1] over global neuron index
    const unsigned short *sidx;       // post (12 bits) | (delay-1) << 12
    const unsigned *sw;               // weight bits
    void *ring;                       // all networks' pending-input rings
    unsigned *raster;                 // [cap][total_words]
    int ring_smem;                    // bytes of shared ring arena per block
    Control *ctl;
};

constexpr int kBatchBlock = 256;
constexpr int kBatchMaxN = 4096;      // largest network of a batched context
constexpr int kBatchMaxDelay = 16;

int batch_form(int min_block_n, int max_block_n, int max_warp_n);
cudaError_t batch_kernel_node(int dtype, int form, void **fn);
cudaError_t max_grid_batch(int dtype, int form, int ring_smem, int *grid);
size_t batch_smem(int ring_smem);

// Shared dense network on tensor cores: sn_shared.cu, and sn_shared_res.cu when
// every block holds one tile (spikes as tagged bit words instead of A0, A1)
struct SharedHostArgs {
    int n, B, t0, steps, cap;
    unsigned char *A0, *A1;
    int *V, *r;
    const int *th, *lk, *rs, *R;
    const unsigned *prate;
    const int *pamp;
    const unsigned long long *pkey;
    unsigned *raster;
    unsigned long long *bits;
    Control *ctl;
};
cudaError_t plan_shared_res(int n, int B, int *fits);
cudaError_t launch_shared_res(const void *tmap_w, const SharedHostArgs &h, cudaStream_t s);
int wt_res_pos(int i);
cudaError_t launch_shared(const void *tmaps, const SharedHostArgs &h, int grid, cudaStream_t s);
cudaError_t max_grid_shared(int *grid);
size_t shared_smem_bytes();
cudaError_t launch_shared_transpose(const int *src, int *dst, int n, int B, cudaStream_t s);

// Feedforward (BPTT) kernels, sn_ff.cu
// sbf (may be null): the spikes also as BF16 rows of ldbf elements
cudaError_t ff_pack(const uint8_t *in, int rows, int n, int words, unsigned *out, void *sbf, int ldbf,
                    cudaStream_t s);
cudaError_t ff_delay_fwd(const unsigned *sprev, int words_in, const float *W, const void *dm, int n_in,
                         int n_out, int B, int row0, int rows, float *I, cudaStream_t s);
cudaError_t ff_scan_fwd(const float *I, int n, int B, int T, int k, float theta, float leak, float reset,
                        int refractory, unsigned *S, float *vck, int *rck, float *counts, void *sbf, int ldbf,
                        cudaStream_t s);
// gI as floats [T*B][n], or (gbf given) as its two BF16 parts [2][T*B][ldg], with pad
// also zeros in columns n .. ldg - 1
cudaError_t ff_scan_bwd(const float *I, int n, int B, int T, int k, float theta, float leak, float reset,
                        int refractory, float slope, const float *vck, const int *rck, const float *gs,
                        const float *gc, float *gI, void *gbf, int ldg, bool pad, cudaStream_t s);
cudaError_t ff_bwd_data(const float *gI, const float *W, const uint8_t *D, int n_in, int n_out, int B, int T,
                        float *gsp, cudaStream_t s);
cudaError_t ff_dw(const float *gI, const unsigned *sprev, int words_in, const uint8_t *D, int n_in, int n_out,
                  int B, int T, int splits, float *part, float *dW, cudaStream_t s);

// Tensor-core contractions of the feedforward network (sn_ff_tc.cu).
// ff_tc_rows: C[r][n] over the delays d = 1..4, K blocks of 64 and part products.
// Maps: m[0], m[1] the A parts (rows, boxes of 128 x 64; the forward has m[0] only),
// m[2] the B parts (boxes of bn x 64), part p of delay d from row ((d - 1) * parts +
// p) * part_rows.  A's rows are shifted by shift * d.  bn: columns of a tile (128, or
// the whole of a narrower C rounded up to 16).
constexpr int kFfTcMaxMaps = 3;
struct FfTcMaps {
    CUtensorMap m[kFfTcMaxMaps];
};
struct FfTcArgs {
    int M, N, tiles_m, tiles_n, kblocks, shift, part_rows, bn;
    float *C;
    long long ldc;
    Control *ctl;
};
cudaError_t ff_tc_rows(const FfTcMaps &maps, const FfTcArgs &args, bool spike_grad, cudaStream_t s);
cudaError_t ff_tc_weights(const float *W, const uint8_t *D, int n_in, int n_out, int nout_p, int rows_in,
                          void *Wb, int nin_p, int rows_out, void *Wf, cudaStream_t s);
cudaError_t ff_tc_spikes(const unsigned *bits, int rows, int n_in, int words, int nin_p, void *S, cudaStream_t s);
// Weight gradient (ff_tc_dw_kernel): maps m[0] the spikes, m[1] and m[2] the
// gradient's parts, boxes of 64 rows x 64 columns; C [ksplit][M][N].
struct FfTcDwArgs {
    int M, N, tiles_m, tiles_n, ksplit, kblocks, B;
    float *C;
    long long cstride;
    const uint8_t *D;
    Control *ctl;
};
cudaError_t ff_tc_dw(const FfTcMaps &maps, const FfTcDwArgs &args, cudaStream_t s);
cudaError_t ff_dw_reduce(const float *part, int splits, long long count, float *dW, cudaStream_t s);

// Launchers (kernels live in sn_kernels.cu).  Return a CUDA error code.
cudaError_t launch_sparse(const NetArgs &a, int dtype, int grid, int block, cudaStream_t s);
cudaError_t launch_dense(const NetArgs &a, int grid, int block, cudaStream_t s);
cudaError_t max_grid_sparse(int dtype, int stdp, int block, int *grid);
cudaError_t max_grid_sparse_reg(int *grid);
cudaError_t launch_sparse_reg(const NetArgs &a, int dtype, int grid, cudaStream_t s);
constexpr int kSparseRegBlock = 512;
// sn_dense_res.cu: the form that keeps W in shared memory, and its rule
constexpr int kDenseResSteps = 4, kDenseResStepsStdp = 12;   // shortest runs that take it
constexpr int kDenseTagStride = 16;        // 64-bit words from one spike word of a tagged row to the next
size_t dense_tag_bytes(int n);             // 0: n never takes it
bool dense_res_fits(int n, int chunk, int grid, bool stdp, int steps);
cudaError_t plan_dense_res(int chunk);     // before the first launch
cudaError_t launch_dense_res(const NetArgs &a, int grid, cudaStream_t s);
cudaError_t plan_dense(int n, int *grid, int *chunk, int force_cpl = 0);
// Pull propagation (sn_pull.cu).  plan_pull sets *grid = 0 when the network
// does not fit the executor (a window of max_delay spike rows above a block's
// shared memory, or more than one neuron per thread).  Synapse words of the
// pull store: x = ((D - d) * Wp + pre / 32) << 7 | (pre & 31),
// Wp = roundup(ceil(n/32), 4).
cudaError_t plan_pull(int n, int D, long long m, int *grid, int *chunk, int *rows, size_t *smem,
                      int own_slices = -1);
cudaError_t launch_shard_put(unsigned *hist, unsigned *raster, int D, int cap, int words, int w0, int w1,
                             long long t0, int rows, const unsigned *src, cudaStream_t s);
cudaError_t launch_sparse_pull(const NetArgs &a, int dtype, bool coded, int grid, size_t smem, cudaStream_t s);
// Pull in blocks of three steps (sn_pull_block.cu).  Blocks of up to kPullNarrow threads
// have 80 registers a thread, wider ones 64.
constexpr int kPullNarrow = 672;
cudaError_t plan_pull_block(int n, int D, int dtype, int grid, int chunk, int *hb, size_t *smem);
size_t pull_tag_bytes(int words);
unsigned pull_hist_byte(unsigned pre, int hb);
cudaError_t launch_pull_block(NetArgs a, int dtype, int hb, int grid, size_t smem, bool rows_live, cudaStream_t s);
cudaError_t launch_pull_flush(const NetArgs &a, int dtype, int t0, cudaStream_t s);
cudaError_t launch_gather_weights(const uint2 *syn, const long long *perm_inv, long long m,
                                  float *out, cudaStream_t s);
cudaError_t launch_scatter_weights(uint2 *syn, const long long *perm_inv, long long m, const float *w,
                                   cudaStream_t s);
cudaError_t launch_barrier_selftest(Control *ctl, int blocks, cudaStream_t s);

}  // namespace sn
