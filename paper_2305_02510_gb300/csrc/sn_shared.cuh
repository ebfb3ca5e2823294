// What the two kernels of the shared dense network (sn_shared.cu,
// sn_shared_res.cu) have in common: the tile and the kernel arguments.
#pragma once

#include <stdint.h>

#include "sn_internal.h"

namespace sn {

constexpr int kTM = 128;                       // trains per tile (MMA M)
constexpr int kTN = 128;                       // post-neurons per tile (MMA N)
constexpr int kTK = 128;                       // bytes of K per stage (one 128B swizzle row)

struct SharedArgs {
    int n, B, t0, steps, cap, words;
    int tiles_m, tiles;
    unsigned char *A0, *A1;        // spike operands [B][n] bytes, A_(t & 1) holds step t
    int *V, *r;                    // [n][B] (neuron-major)
    const int *th, *lk, *rs, *R;   // [n]
    const unsigned *prate;         // [n]
    const int *pamp;               // [n]
    const unsigned long long *pkey;// [B]
    unsigned *raster;              // [cap][B][words]
    unsigned long long *bits;      // shared_res_kernel: spike words [2][words / 4][B][4], those of step
                                   // t in part t & 1, the step's number in the launch in the high half
    Control *ctl;
};

inline SharedArgs shared_args(const SharedHostArgs &h) {
    SharedArgs a;
    a.n = h.n; a.B = h.B; a.t0 = h.t0; a.steps = h.steps; a.cap = h.cap; a.words = h.n / 32;
    a.tiles_m = h.B / kTM;
    a.tiles = a.tiles_m * (h.n / kTN);
    a.A0 = h.A0; a.A1 = h.A1; a.V = h.V; a.r = h.r;
    a.th = h.th; a.lk = h.lk; a.rs = h.rs; a.R = h.R;
    a.prate = h.prate; a.pamp = h.pamp; a.pkey = h.pkey; a.raster = h.raster; a.bits = h.bits; a.ctl = h.ctl;
    return a;
}

}  // namespace sn
