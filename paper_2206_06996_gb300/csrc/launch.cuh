// Programmatic dependent launch (option pdl): a kernel lets the next kernel
// of the stream start as soon as all of its CTAs are running
// (griddepcontrol.launch_dependents) and, before it reads anything an earlier
// kernel wrote, waits for that kernel to complete with its memory visible
// (griddepcontrol.wait).  Between the two it touches only stored matrices
// that no kernel in flight writes.  Every kernel launched this way waits
// itself, so a completed predecessor means that all earlier ones completed.
// Launched without the attribute, both instructions return at once.
//
// Nothing orders loads through the read-only path (__ldg, const __restrict__
// arguments) behind the wait.  As a precaution a kernel reads that way only
// what no kernel in flight may write (settled matrices), and vectors with
// ordinary loads behind the wait.
#pragma once
#include "common.cuh"

namespace scr {

__device__ __forceinline__ void pdl_allow_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait_prev() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

extern int g_pdl;

// Grids of at most half a CTA per SM, or of at least eight per SM, are launched
// early.  A chain of products of sizes between is slower that way: the next
// kernel's waiting CTAs take slots, and the last CTAs of this one and the first
// of the next fill the SMs unevenly.  Measured on 152 SMs (us per product in a
// chain, plain / early): FP64, 2 lanes, 6000 rows 5.0 / 8.2, 50,000 rows
// 18.0 / 18.2; FP32, 4 lanes 2.8 / 4.3 and 9.9 / 9.8; FP32, 300 rows 2.4 / 2.3;
// at the bench tube's size early launches take 1 % off an FP64 step.
inline bool early_grid(long long grid, int sms) { return 2 * grid <= sms || grid >= 8LL * sms; }

// kern<<<grid, blk, 0, s>>>(args...), with the programmatic-serialization
// attribute when early is set (and the option pdl); kern waits in
// griddepcontrol.wait
template <typename... KArgs, typename... Args>
inline void launch_early(bool early, void (*kern)(KArgs...), long long grid, int blk, cudaStream_t s, Args... args) {
  if (early && g_pdl) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)blk);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    SCR_CUDA(cudaLaunchKernelEx(&cfg, kern, args...));
  } else {
    kern<<<(unsigned)grid, blk, 0, s>>>(args...);
  }
}

}  // namespace scr
