// FP32 instantiations of the batched stage kernel, and the per-step advance kernel.
#include "batch.cuh"

namespace hj {

cudaError_t launch_batch_stage_f32_eno2(const BatchTile* tiles, int ntiles, const BatchInst* insts, int stage,
                                        int ndim, int dynamics, int threads, size_t smem, cudaStream_t s);
cudaError_t launch_batch_stage_f32_eno13(const BatchTile* tiles, int ntiles, const BatchInst* insts, int stage,
                                         int ndim, int dynamics, int scheme, int threads, size_t smem, cudaStream_t s);

cudaError_t launch_batch_stage_f32(const BatchTile* tiles, int ntiles, const BatchInst* insts, int stage, int ndim,
                                   int dynamics, int scheme, int threads, size_t smem, cudaStream_t s) {
    if (scheme == HJ_ENO2) return launch_batch_stage_f32_eno2(tiles, ntiles, insts, stage, ndim, dynamics, threads, smem, s);
    if (scheme == HJ_ENO1 || scheme == HJ_ENO3)
        return launch_batch_stage_f32_eno13(tiles, ntiles, insts, stage, ndim, dynamics, scheme, threads, smem, s);
    HJ_BATCH_DISPATCH(launch_batch_weno5, float)
}

// After stage 3 of a step: count the step, and set up the next one. Every
// step uses dt_full except the one that completes a slice, which is clipped
// to land on the slice time (Listing 6) and also writes the slice output.
// One thread a tile: an instance's first tile advances it (other chains'
// descriptors may be advancing concurrently).
__global__ void batch_advance_kernel(const BatchTile* tiles, int ntiles, BatchInst* insts) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    grid_wait();
    if (i >= ntiles) return;
    const BatchTile t = tiles[i];
    if (t.tile != 0 || t.i2 != 0 || t.chunk != 0) return;
    BatchInst& I = insts[t.inst];
    if (I.k >= I.steps_total) return;
    const int k = ++I.k;
    I.slice_out = nullptr;
    if (k < I.steps_total) {
        double dt = I.dt_full;
        if (I.cursor < I.n_ends && I.ends[I.cursor] == (long long)k + 1) {
            dt = I.end_dt[I.cursor];
            I.slice_out = static_cast<char*>(I.out) + (size_t)I.end_slice[I.cursor] * (size_t)I.nodes * I.elem;
            I.cursor += 1;
        }
        I.dt = dt;
        I.dt_f = (float)dt;
    }
}

cudaError_t launch_batch_advance(const BatchTile* tiles, int ntiles, BatchInst* insts, cudaStream_t s) {
    return launch_dependent(batch_advance_kernel, dim3((ntiles + 127) / 128), dim3(128), 0, s, tiles, ntiles, insts);
}

}  // namespace hj
