// Host-side launchers of the AIR kernels (defined in kernels.cu).
#pragma once

#include <cuda_runtime.h>

#include "air_internal.cuh"

namespace air {

// Launches a kernel that begins with grid_wait(): its blocks take the places
// that the blocks of the kernel before it on the stream leave, and wait there
// for its results, instead of after a launch gap.  Two outer steps of five CG
// steps at 128^2 / 90 views take 464 us (688 without), at 512^2 / 800 views
// 2.38 ms (2.66).
template <typename... Params, typename... Args>
cudaError_t launch_overlapped(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, bool overlap,
                              cudaStream_t st, const Args &...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = overlap ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}

// One op over all tiles of one slice (overlap: see launch_overlapped).
cudaError_t launch_op(int op, const SliceDesc &s, int arg, cudaStream_t st, bool overlap = true);

// Blocks of a grouped backprojector (OP_BWD or OP_ORB_BWD) resident on the
// current device at once, for the given dynamic shared memory (0 on failure).
int group_bwd_capacity(int op, size_t smem);

// One op over the tiles of many slices in one launch (tasks all of that op).
cudaError_t launch_group(int op, const SliceDesc *d_slices, const Task *d_tasks, int ntasks, int total_tiles,
                         size_t smem, cudaStream_t st);

// Persistent batch solve: one cooperative launch runs every phase of every
// slice's program, with a bounded grid barrier between phases.
struct Phase {
    int op, arg;
};
struct BatchCtl {
    unsigned arrive;     // grid barrier: blocks arrived in this generation
    unsigned gen;        // grid barrier generation
    int error;           // AIR_ERR_TIMEOUT if a barrier wait gave up
    int pad;
    unsigned long long ticket;   // tiles handed out so far (see k_persistent)
};
// tile_base: [nphases][nslices + 1] prefix sums of the slices' tile counts in
// each phase; phase_base: [nphases] first ticket of each phase, the sum over
// earlier phases of their tiles plus one closing ticket per block.
cudaError_t launch_persistent(const SliceDesc *d_slices, int nslices, const Phase *d_prog,
                              int nphases, const int *d_tile_base, const unsigned long long *d_phase_base,
                              BatchCtl *d_ctl, int grid, size_t smem, bool orb, cudaStream_t st);
// Largest co-resident grid of the persistent kernel for the given smem (orb:
// the form that also runs the orbit ops).
int persistent_grid(size_t smem, bool orb);
// Poll budget of the persistent kernel's grid-barrier wait on the current
// device (negative: the default).  Synchronous.
cudaError_t set_barrier_budget(long long polls);

}  // namespace air
