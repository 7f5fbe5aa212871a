// dd_kernels.cu -- the forward kernels of one input type, one-shot and
// persistent. Compiled once per type, so that the types build in parallel:
// DD_INST 0 = FP32, 1 = FP32 with live-chunk ranges, 2 = FP16, 3 = BF16, 4 =
// 8-bit.
#include <atomic>

#include "dd_kernels.h"

namespace dd {

// LIVE: the plan has a live-chunk table (the adjoint's transposed gather,
// FP32 only); tiles sum only their live chunks.
template <int KIND, typename T, int DPT, int SPT, bool LIVE>
__global__ void __launch_bounds__(fwd_max_threads(KIND, DPT, SPT), fwd_min_blocks(KIND, DPT, SPT))
    dd_fwd_kernel(const FwdArgs a) {
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem);
    fwd_init_barriers<KIND>(bars, a.stages);
    uint32_t kbase = 0;
    const int x = int(blockIdx.x);
    const int dt = a.time_major ? x / a.grid_tt : x % a.grid_dt;
    const int tt = a.time_major ? x % a.grid_tt : x / a.grid_dt;
    fwd_tile_any<KIND, T, DPT, SPT, LIVE>(a, a.dtile0 + dt, a.ttile0 + tt, blockIdx.y, bars,
                                          smem + 128, kbase);
}

#if DD_INST != 1
template <int KIND, typename T, int DPT, int SPT>
__global__ void __launch_bounds__(fwd_max_threads(KIND, DPT, SPT), fwd_min_blocks(KIND, DPT, SPT))
    dd_fwd_persistent_kernel(const BatchArgs ba) {
    extern __shared__ __align__(128) unsigned char smem[];
    // The item number alternates between two words: thread 0 writes the
    // next one while a warp that is still leaving the previous tile may not
    // yet have read the current one (a tile with no more chunks than stages
    // lets the staging warp run ahead of the others).
    __shared__ long long s_item[2];
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem);
    const volatile int *gave_up = reinterpret_cast<const volatile int *>(&bars[7]);
    fwd_init_barriers<KIND>(bars, ba.stages);
    uint32_t kbase = 0;
    const long long n_items = ba.item_start[ba.n];
    for (int it = 0;; it ^= 1) {
        // a CTA that gave up a wait takes no further items
        if (threadIdx.x == 0)
            s_item[it] = *gave_up ? n_items : (long long)atomicAdd(ba.counter, 1ull);
        __syncthreads();
        const long long item = s_item[it];
        if (item >= n_items) break;
        int i = 0;
        while (item >= ba.item_start[i + 1]) ++i;
        const FwdArgs a = ba.args[i];
        long long loc = item - ba.item_start[i];
        const int dtile = int(loc % a.n_dtiles);
        loc /= a.n_dtiles;
        const int ttile = int(loc % a.n_ttiles);
        const int b = int(loc / a.n_ttiles);
        fwd_tile_any<KIND, T, DPT, SPT>(a, dtile, ttile, b, bars, smem + 128, kbase);
    }
}

#endif

namespace {

constexpr int kMaxDevices = 64;

template <int KIND, typename T, int DPT, int SPT, bool LIVE>
cudaError_t launch_fwd_t(const FwdArgs &a, dim3 grid, dim3 block, size_t smem, cudaStream_t st) {
    // Make sure the kernel's dynamic shared-memory limit (set per device)
    // covers smem, checking once per size increase; the limit is only ever
    // raised, since other launches of the same kernel may need more.
    static std::atomic<size_t> smem_set[kMaxDevices];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const bool cached = dev >= 0 && dev < kMaxDevices;
    if (smem > 48 * 1024 && (!cached || smem > smem_set[dev].load())) {
        cudaFuncAttributes fa{};
        e = cudaFuncGetAttributes(&fa, dd_fwd_kernel<KIND, T, DPT, SPT, LIVE>);
        if (e != cudaSuccess) return e;
        if (size_t(fa.maxDynamicSharedSizeBytes) < smem) {
            e = cudaFuncSetAttribute(dd_fwd_kernel<KIND, T, DPT, SPT, LIVE>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
            if (e != cudaSuccess) return e;
        }
        if (cached) smem_set[dev].store(smem);
    }
    dd_fwd_kernel<KIND, T, DPT, SPT, LIVE><<<grid, block, smem, st>>>(a);
    return cudaGetLastError();
}

#if DD_INST != 1
// Raises the kernel's dynamic shared-memory limit to smem if it is lower (never
// lowers it: another batch's captured graph may launch the same kernel with
// more) and returns its resident CTAs per SM at (block, smem).
template <int KIND, typename T, int DPT, int SPT>
int occupancy_t(int block, size_t smem) {
    cudaFuncAttributes fa{};
    if (cudaFuncGetAttributes(&fa, dd_fwd_persistent_kernel<KIND, T, DPT, SPT>) != cudaSuccess)
        return 0;
    if (size_t(fa.maxDynamicSharedSizeBytes) < smem &&
        cudaFuncSetAttribute(dd_fwd_persistent_kernel<KIND, T, DPT, SPT>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)) != cudaSuccess)
        return 0;
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &n, dd_fwd_persistent_kernel<KIND, T, DPT, SPT>, block, smem) != cudaSuccess)
        return 0;
    return n;
}
#endif

template <typename T, bool LIVE>
FwdKernel pick(int kind, int dpt, int spt) {
#define DD_PICK(K_, D_, S_)                                                   \
    if constexpr (key_has_type<T>(K_, S_))                                    \
        if (kind == K_ && dpt == D_ && spt == S_)                             \
        return FwdKernel{(const void *)&dd_fwd_kernel<K_, T, D_, S_, LIVE>,   \
                         &launch_fwd_t<K_, T, D_, S_, LIVE>};
    DD_FWD_KEYS(DD_PICK)
#undef DD_PICK
    return FwdKernel{};
}

#if DD_INST != 1
template <typename T>
PersistentFn pick_persistent(int kind, int dpt, int spt) {
#define DD_PICK(K_, D_, S_)                                                         \
    if constexpr (key_has_type<T>(K_, S_))                                          \
        if (kind == K_ && dpt == D_ && spt == S_)                                   \
        return PersistentFn{(const void *)&dd_fwd_persistent_kernel<K_, T, D_, S_>, \
                            &occupancy_t<K_, T, D_, S_>};
    DD_FWD_KEYS(DD_PICK)
#undef DD_PICK
    return PersistentFn{};
}
#endif

}  // namespace

#define DD_DEFINE_PICK(NAME_, T_)                                          \
    FwdKernel pick_fwd_##NAME_(int kind, int dpt, int spt) {               \
        return pick<T_, false>(kind, dpt, spt);                            \
    }                                                                      \
    PersistentFn pick_persistent_##NAME_(int kind, int dpt, int spt) {     \
        return pick_persistent<T_>(kind, dpt, spt);                        \
    }
#if DD_INST == 0
DD_DEFINE_PICK(f32, float)
#elif DD_INST == 1
FwdKernel pick_fwd_f32_live(int kind, int dpt, int spt) {
    return pick<float, true>(kind, dpt, spt);
}
#elif DD_INST == 2
DD_DEFINE_PICK(f16, __half)
#elif DD_INST == 3
DD_DEFINE_PICK(bf16, __nv_bfloat16)
#else
DD_DEFINE_PICK(u8, uint8_t)
#endif

}  // namespace dd
