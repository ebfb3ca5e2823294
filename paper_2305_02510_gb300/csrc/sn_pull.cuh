// What the two pull kernels (sn_pull.cu, sn_pull_block.cu) share: the
// accumulator of a neuron's synaptic input and the block size.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "sn_device.cuh"

namespace sn {

constexpr int kPullMaxBlock = 1024;

template <int MODE> struct PullAcc;
template <> struct PullAcc<SN_F32> {
    using T = float;
    static __device__ __forceinline__ T add(T acc, unsigned wbits) { return __fadd_rn(acc, __uint_as_float(wbits)); }
};
template <> struct PullAcc<SN_I32> {
    using T = long long;            // exact: int32 weights, at most 2^32 synapses
    static __device__ __forceinline__ T add(T acc, unsigned wbits) { return acc + (long long)(int)wbits; }
};

}  // namespace sn
