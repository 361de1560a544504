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
// What a CTA takes after its signal is tensor memory; tc_smem() below keeps two
// CTAs whose columns do not fit together off one SM, so that allocation finds its
// columns free unless their holder is a CTA that has left the SM.
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

// Shared memory a launch asks for so that tensor memory (512 columns an SM) is never
// contended: a CTA signals its successor before it allocates, so a CTA of the next grid
// beside it could take the columns and then wait for the grid whose CTA waits for them.
// A CTA of all 512 columns shares its SM with no other CTA of this size, one of 256 with
// one more of 256 at most.  The smaller floor is the low one because shared memory is taken
// from L1, which the neighbour gathers of two CTAs need (order 2 at a floor of 110 KB: 279 936
// tetrahedra in random order 224 us a stage instead of 141).
constexpr int tc_smem(int columns, int bytes) {
  const int least = (columns > 256 ? 148 : 80) * 1024;
  return bytes > least ? bytes : least;
}
static_assert(2 * (tc_smem(256, 0) + kCtaSmem) <= kSmSmem, "two CTAs of 256 columns fit");
static_assert(3 * (tc_smem(256, 0) + kCtaSmem) > kSmSmem, "three do not");
static_assert(tc_smem(512, 0) + tc_smem(256, 0) + 2 * kCtaSmem > kSmSmem, "nor 512 and 256");

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
