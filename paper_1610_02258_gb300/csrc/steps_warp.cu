// The warp-tile step for models given at run time (meshes below the
// specialisation size, or without the run-time compiler) of up to
// kWarpGenericSpecies species: plain, flow and batched kernels. The loops over
// species are unrolled to 4 or 12, the reaction table is walked in loops.
#include <algorithm>
#include <string>

#include "steps_warp.cuh"

namespace steps {

namespace {

template <int SM>
__global__ void __launch_bounds__(512, 2)
    warp_kernel(const __grid_constant__ ModelDev m, const __grid_constant__ StepArgs a) {
    warp_step<0, 1, SM, RtWarp>(m, a, (int64_t)blockIdx.x);
}

template <int SM>
__global__ void __launch_bounds__(512, 2)
    warp_flow_kernel(const __grid_constant__ ModelDev m, const __grid_constant__ StepArgs a,
                     const __grid_constant__ FlowArgs f) {
    warp_step<0, 1, SM, RtWarp, 1>(m, a, 0, &f);
}

template <int SM>
__global__ void __launch_bounds__(512, 2)
    warp_batch_kernel(const BlockWork *__restrict__ work, const RepEntry *__restrict__ reps) {
    batch_member<0>(work, reps, 0, [](const ModelDev &m, const StepArgs &a, int64_t tile) {
        warp_step<0, 1, SM, RtWarp>(m, a, tile);
    });
}

// One warp, the tile of tets 32 to 63 (word 1), waits for window word 5 of the
// tiles of its tets' face neighbours.
__global__ void nbr_wait_test_kernel(const uint32_t *done, const int4 *nbr, long long limit, uint32_t *status) {
    const bool ok = flow_nbr_wait(done, 1u, 32, nbr[threadIdx.x], 5u, limit);
    if (threadIdx.x == 0) *status = ok ? 0u : 8u;
}

bool opt_in(const void *fn, size_t smem) {
    if (smem <= 44 * 1024) return true;  // with the static arrays below the 48 KB every launch may have
    const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) return true;
    set_error(std::string("warp-tile kernel shared memory: ") + cudaGetErrorString(e));
    return false;
}

int checked(cudaError_t e, const char *what) {
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess) return STEPS_OK;
    set_error(std::string(what) + ": " + cudaGetErrorString(e));
    return STEPS_ERR_CUDA;
}

template <int SM>
int launch_plain(const ModelDev &m, const StepArgs &a, int block, void *stream) {
    // A small mesh's windows are bound by the latency of a tile. Below a warp per
    // scheduler (4 on each of 152 SMs), warps take fewer tets, whose queues are
    // shorter: us per window, 32 tets -> this rule: 1,920 tets 7.4 -> 6.7, 8,670
    // tets 20.4 -> 19.8; but two warps per scheduler instead of one for 30,720
    // tets of 151 molecules 66 -> 73, and 2 tets a warp are no faster than 4.
    StepArgs b = a;
    while (b.lanes > 4 && ((int64_t)a.T + b.lanes - 1) / b.lanes < 4 * 152) b.lanes /= 2;
    const int64_t warps = ((int64_t)a.T + b.lanes - 1) / b.lanes;
    // warps of one block share an SM, so the blocks shrink until they cover the
    // SMs twice: 256 threads -> this rule, 30,720 tets 67.4 -> 65.8, 17,340 to
    // 52,020 tets of 14 molecules 22.2 -> 21.7, 24.4 -> 23.2, 24.7 -> 23.5 (up to
    // four times: 21.7, 23.7, 25.0)
    while (block > 32 && (warps * 32 + block - 1) / block < 2 * 152) block /= 2;
    const size_t smem = (size_t)(block / 32) * sizeof(WarpTile<SM>);
    if (!opt_in((const void *)warp_kernel<SM>, smem)) return STEPS_ERR_CUDA;
    // programmatic dependent launch, as the block-tile kernel
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((warps * 32 + block - 1) / block));
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = (cudaStream_t)stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return checked(cudaLaunchKernelEx(&cfg, warp_kernel<SM>, m, b), "warp-tile kernel launch");
}

template <int SM>
int launch_flow_sm(const ModelDev &m, const StepArgs &a, const FlowArgs &f, int block, void *stream) {
    const size_t smem = (size_t)(block / 32) * sizeof(WarpTile<SM>);
    if (!opt_in((const void *)warp_flow_kernel<SM>, smem)) return STEPS_ERR_CUDA;
    StepArgs b = a;
    b.window_base = nullptr;
    warp_flow_kernel<SM><<<f.nwin * f.ntiles, block, smem, (cudaStream_t)stream>>>(m, b, f);  // one item per block
    return checked(cudaSuccess, "warp-tile flow kernel launch");
}

template <int SM>
int launch_batch_sm(const BlockWork *work, int64_t nblocks, const RepEntry *reps, int block, void *stream) {
    const size_t smem = (size_t)(block / 32) * sizeof(WarpTile<SM>);
    if (!opt_in((const void *)warp_batch_kernel<SM>, smem)) return STEPS_ERR_CUDA;
    warp_batch_kernel<SM><<<(unsigned)nblocks, block, smem, (cudaStream_t)stream>>>(work, reps);
    return checked(cudaSuccess, "warp-tile batch kernel launch");
}

}  // namespace

int launch_nbr_wait_test(const uint32_t *d_done, const void *d_nbr, long long limit, uint32_t *d_status) {
    nbr_wait_test_kernel<<<1, 32>>>(d_done, (const int4 *)d_nbr, limit, d_status);
    return checked(cudaSuccess, "flow wait test launch");
}

int launch_warp(const ModelDev &m, const StepArgs &a, int block, void *stream) {
    return m.S <= 4 ? launch_plain<4>(m, a, block, stream) : launch_plain<kWarpGenericSpecies>(m, a, block, stream);
}

int launch_warp_flow(const ModelDev &m, const StepArgs &a, const FlowArgs &f, int block, void *stream) {
    return m.S <= 4 ? launch_flow_sm<4>(m, a, f, block, stream) : launch_flow_sm<kWarpGenericSpecies>(m, a, f, block, stream);
}

int launch_warp_batch(const BlockWork *work, int64_t nblocks, const RepEntry *reps, int max_S, int block, void *stream) {
    return max_S <= 4 ? launch_batch_sm<4>(work, nblocks, reps, block, stream)
                      : launch_batch_sm<kWarpGenericSpecies>(work, nblocks, reps, block, stream);
}

}  // namespace steps
