// Launchers of the spawning kernels (k_sweep, k_heavy), defined in one translation unit per determinant
// width so that their instantiations (plain, permitted space, spin-coupled functions, both) compile in
// parallel with the rest of the library. mode: bit 0 permitted space, bit 1 spin-coupled functions.
#pragma once

#include <cuda_runtime.h>

namespace fq {

struct Params;

// Launches a kernel of an iteration. next: with a programmatic dependency on the launch before it on the stream, so
// that its blocks are placed while that one drains (the kernels call grid_wait() before they read anything). Captured
// into a graph, the dependency becomes a programmatic edge.
template <typename... K, typename... A>
cudaError_t launch_next(void (*kernel)(K...), int grid, int block, size_t smem, cudaStream_t s, bool next, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = next ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<K>(args)...);
}

void launch_sweep_w1(int mode, int grid, cudaStream_t s, bool next, const Params &P);
void launch_heavy_w1(int mode, int grid, cudaStream_t s, bool next, const Params &P);
cudaError_t sweep_occupancy_w1(int n_elec, int *blocks_per_sm);  // also sets the kernels' shared-memory limits
void launch_sweep_w2(int mode, int grid, cudaStream_t s, bool next, const Params &P);
void launch_heavy_w2(int mode, int grid, cudaStream_t s, bool next, const Params &P);
cudaError_t sweep_occupancy_w2(int n_elec, int *blocks_per_sm);

}  // namespace fq
