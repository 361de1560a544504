// Programmatic dependent launch for the stage kernels.
//
// Consecutive stage kernels of a time step run back to back on one stream.
// Each is launched with programmatic stream serialization, and every CTA
// signals griddepcontrol.launch_dependents as it starts: the next kernel may
// then be scheduled while this one drains, run its set-up (tensor memory,
// barriers, constant operators), and block in griddepcontrol.wait -- which
// returns once the previous grid has completed and its writes are visible --
// before it touches a field array.  The next grid starts only once every CTA of
// the previous one has signalled or left, so a waiting CTA never holds a slot that
// a CTA of the previous grid still has to start in (grids of many waves included).
// Tensor memory is what a CTA still has to take after it has started: see tc_smem().
#pragma once

#include <cuda_runtime.h>

#include "device.h"

namespace dgdev {

__device__ __forceinline__ void pdl_launch_dependents() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Shared memory of an SM, of which every resident CTA costs 1 KB beside its own.
constexpr int kSmSmem = 228 * 1024, kCtaSmem = 1024;

// Shared memory that a launch with `columns` tensor-memory columns a CTA asks for: one CTA
// of 512 columns an SM, two of 256, not three.  A CTA of 512 may share its SM with one of 256,
// so a CTA that had signalled its successor before it allocated could find its columns
// taken by a CTA of the next grid, which waits for this one.  Therefore a CTA signals once it
// has its columns (every CTA of a grid holds them before the next grid starts), or asks for
// so much shared memory that no CTA with tensor memory fits beside it (tc_sole) and signals
// as it starts.  Keeping all sizes apart by shared memory instead takes it from L1, which the
// neighbour gathers of large meshes need: order 2 in two CTAs of 110 KB, 279 936
// tetrahedra in random order, 224 us a stage (80 KB: 141), order 3 in one CTA of 148 KB, 384 000
// in random order, 413 us (124 KB: 400).
constexpr int tc_smem(int columns, int bytes) {
  const int least = (columns > 256 ? 120 : 80) * 1024;
  return bytes > least ? bytes : least;
}
constexpr bool tc_sole(int smem) { return smem + tc_smem(256, 0) + 2 * kCtaSmem > kSmSmem; }
static_assert(2 * (tc_smem(512, 0) + kCtaSmem) > kSmSmem, "one CTA of 512 columns an SM");
static_assert(2 * (tc_smem(256, 0) + kCtaSmem) <= kSmSmem &&
              3 * (tc_smem(256, 0) + kCtaSmem) > kSmSmem, "two of 256, not three");

inline cudaError_t launch_pdl(void (*kern)(const StageArgs), int grid, int threads, int smem,
                              cudaStream_t s, const StageArgs& a) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, a);
}

}  // namespace dgdev
