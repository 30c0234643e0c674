// Chained kernel launches (programmatic dependent launch): a kernel launched with
// launch_after() may start while its predecessor on the stream finishes.  It calls grid_wait()
// before it reads anything the predecessor wrote or writes anything the predecessor reads (a no-op
// in kernels launched the ordinary way); what it does before that overlaps the predecessor's
// tail.  A kernel calls grid_release() to let its successor's launch begin as soon as every block
// of its own grid has started.  grid_wait() waits for the whole predecessor, which waited for its
// own, so everything before a chain is complete too.
//
// A kernel that calls grid_wait() is resident while its predecessor still writes, so what a kernel
// before it in the chain may write (psi, the advectors between the passes, bounds, factors,
// psi_bar) is read by ordinary loads: no __ldg, and no __restrict__ on the kernel's parameter,
// with which the compiler may take the array as constant for the whole kernel and read it through
// the read-only path or before the wait.  Neither is put on what the kernel writes itself.  Both
// stay for G, R and b, which no kernel of a forward call writes; the reverse sweep's kernels, whose
// first is a dependent of whatever the caller put on the stream before, have them nowhere.
#pragma once

#include <cuda_runtime.h>

namespace mpd {
namespace dev {

__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_release() { asm volatile("griddepcontrol.launch_dependents;" :::); }

}  // namespace dev

// The largest grid that releases its successor early: one block per SM.  The successor's blocks then
// start beside it, evenly.  The blocks of a larger one would take the slots the predecessor happens
// to leave and load the SMs unevenly (the compensated 1024^2 step, 288 blocks: 16.8 us released
// early, 13.3 not), so a larger grid releases its successor by ending; what remains saved is the
// 2 us step in which an ordinary launch waits for its predecessor.  Measured, ordinary -> chained
// launches: 59 x 61 (8 blocks) 6.1 -> 3.5 us per step, 512^2 8.5 -> 5.4, plain 1024^2 12.6 -> 10.5,
// compensated 15.0 -> 13.3, |psi| on 1021 x 1000 12.3 -> 10.8.
//
// FP64 blocks are bound by their SM's FP64 pipe, so that two on one SM while another has none cost
// twice the time: they are never released early.  Measured, released early up to 152 blocks -> not:
// band march 190 x 175 (96 blocks) 29.7 -> 19.4 us per step, 96^2 14.1 -> 9.8; tile kernel 256^2 with
// three passes and the limiter (128 blocks) 82 -> 61; ensemble of 16 fields of 128^2 in tiles of 12 rows
// (132 blocks) 137 -> 99; and with few blocks no difference (59 x 61 9.8, 9.8).
constexpr unsigned kChainBlocks = 152;
template <typename T>
__device__ __forceinline__ void grid_release_small(unsigned blocks) {
  if (sizeof(T) == 4 && blocks <= kChainBlocks) dev::grid_release();
}

// kern<<<grid, block, smem, st>>>(args...), as a dependent of the kernel before it where `chained`
template <typename... KArgs, typename... Args>
cudaError_t launch_chained(bool chained, void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                           Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = chained ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}

template <typename... KArgs, typename... Args>
cudaError_t launch_after(void (*kern)(KArgs...), dim3 grid, dim3 block, cudaStream_t st, Args... args) {
  return launch_chained(true, kern, grid, block, 0, st, args...);
}

}  // namespace mpd
