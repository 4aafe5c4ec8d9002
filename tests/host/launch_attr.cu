// launch_attr.cu -- gbmd::launch (csrc/k_step.cu) against a stand-in for the two launch
// calls of the CUDA runtime, which records what each launch asks for.  No GPU is used.
#include <cstring>

#include "../../paper_1308_5587_gb300/csrc/launch.cuh"

namespace {
struct Seen { int plain, ex, cooperative; unsigned grid, block; size_t smem; } seen;
}

extern "C" cudaError_t cudaLaunchKernel(const void*, dim3 grid, dim3 block, void**, size_t smem,
                                        cudaStream_t) {
  seen = {1, 0, 0, grid.x, block.x, smem};
  return cudaSuccess;
}

extern "C" cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void*, void**) {
  seen = {0, 1, 0, c->gridDim.x, c->blockDim.x, c->dynamicSmemBytes};
  for (unsigned k = 0; k < c->numAttrs; ++k)
    if (c->attrs[k].id == cudaLaunchAttributeCooperative) seen.cooperative = c->attrs[k].val.cooperative;
  return cudaSuccess;
}

// out: plain calls, extended calls, cooperative attribute, grid, block, shared memory
extern "C" int launch_seen(int cooperative, int grid, int block, int smem, int* out) {
  gbmd::KernelCall k;
  memset(&k, 0, sizeof(k));
  k.func = (void*)launch_seen;
  k.grid = dim3(grid);
  k.block = dim3(block);
  k.smem = smem;
  k.cooperative = cooperative != 0;
  seen = {};
  const int rc = (int)gbmd::launch(k, nullptr);
  out[0] = seen.plain; out[1] = seen.ex; out[2] = seen.cooperative;
  out[3] = (int)seen.grid; out[4] = (int)seen.block; out[5] = (int)seen.smem;
  return rc;
}
