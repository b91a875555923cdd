// pd_persist.cu -- the persistent step kernels of one precision and one thread
// count per node, with or without bond tiles, for blocks of 128 and 256 threads.
// Compiled once per combination, with PD_PERSIST_FP32 (1: FP32 split, 0: FP64),
// PD_PERSIST_LANES and PD_PERSIST_TILES (1: bond tiles, one thread per node)
// defined, and with the compile flags of that precision's other kernels.
#include <algorithm>

#include "pd_step.cuh"

#if !defined(PD_PERSIST_FP32) || !defined(PD_PERSIST_LANES) || !defined(PD_PERSIST_TILES)
#error "PD_PERSIST_FP32, PD_PERSIST_LANES and PD_PERSIST_TILES must be defined"
#endif

namespace pd {

template <bool FP32, int LANES, bool TILES>
cudaError_t launch_persistent_lanes(const DevPtrs &d, const KParams &k, int vin, int nsteps, int block,
                                    cudaStream_t s) {
    if (block == 256) return launch_persistent_cfg<FP32, LANES, 256, TILES>(d, k, vin, nsteps, s);
    return launch_persistent_cfg<FP32, LANES, 128, TILES>(d, k, vin, nsteps, s);
}

template cudaError_t launch_persistent_lanes<PD_PERSIST_FP32 != 0, PD_PERSIST_LANES, PD_PERSIST_TILES != 0>(
    const DevPtrs &, const KParams &, int, int, int, cudaStream_t);

#if PD_PERSIST_TILES
template <>
cudaError_t init_persistent_tiles<PD_PERSIST_FP32 != 0>() {
    constexpr bool kFp32 = PD_PERSIST_FP32 != 0;
    const cudaError_t e = cudaFuncSetAttribute(k_persistent<kFp32, 1, 128, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               run_smem<kFp32, 128>());
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_persistent<kFp32, 1, 256, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                run_smem<kFp32, 256>());
}
#endif

}  // namespace pd
