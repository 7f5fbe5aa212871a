// dd_kernels.h -- the compiled forward kernels (one-shot and persistent) by
// input type. dd_kernels.cu is compiled once per input type; the host code
// picks kernels through these functions.
#pragma once
#include <cuda_runtime.h>

#include <cstddef>

#include "dd_fwd_tile.cuh"

namespace dd {

constexpr int kMaxBatchPlans = 16;

// Arguments of the persistent batched launch.
struct BatchArgs {
    const FwdArgs *args;  // [n], device
    int n, stages;
    long long item_start[kMaxBatchPlans + 1];
    unsigned long long *counter;
};

using FwdLaunchFn = cudaError_t (*)(const FwdArgs &, dim3, dim3, size_t, cudaStream_t);

// A one-shot kernel and its launcher (null: not compiled).
struct FwdKernel {
    const void *fn = nullptr;
    FwdLaunchFn launch = nullptr;
};
// A persistent kernel and its occupancy query (resident CTAs per SM).
struct PersistentFn {
    const void *fn = nullptr;
    int (*occupancy)(int block, size_t smem) = nullptr;
};

#define DD_DECLARE_PICK(NAME_)                                  \
    FwdKernel pick_fwd_##NAME_(int kind, int dpt, int spt);     \
    PersistentFn pick_persistent_##NAME_(int kind, int dpt, int spt);
DD_DECLARE_PICK(f32)
DD_DECLARE_PICK(f16)
DD_DECLARE_PICK(bf16)
DD_DECLARE_PICK(u8)
#undef DD_DECLARE_PICK
FwdKernel pick_fwd_f32_live(int kind, int dpt, int spt);

}  // namespace dd
