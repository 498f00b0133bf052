// Launches that overlap the end of the kernel before them in the stream
// (programmatic dependent launch).
//
// A plain launch starts after the last block of the kernel before it has ended
// and its writes are flushed, 3-4 us in which a request's next kernel does
// nothing; launched this way its blocks are already in place.  Measured (one
// request at a time, host's wait included, both sides in one session; J.2 and
// Gaborish / colour kernels launched this way): 48x40 u8 73 -> 64 us, 1920x1088
// u8 125 -> 119, 4096x4096 f32 530 -> 527, 8192x8192 the same; without
// let_next_start in the transform kernel 4096x4096 is 2-4 us slower.  The DC
// kernels (F.2, H) and the transform kernel behind them: 3001x2003 photograph
// 400 -> 393 us.  With several requests in flight a kernel lets the next one in
// only after its main work (k_dc_cell).  The JPEG1 output kernel behind its
// chroma planes gained nothing (4096x4096 113 us either way): a plain launch.
#ifndef JXLR_LAUNCH_H_
#define JXLR_LAUNCH_H_

#include <cuda_runtime.h>

namespace jxlr {

// Waits until the kernels before this one in the stream are done and their
// results visible.  Every thread of a kernel started by launch_after calls it
// before it reads what they wrote or writes anything (so that a kernel after
// this one, too, may rely on all of them).  Returns 0, to be added to the
// addresses of those loads: none of them can be moved before the wait then, not
// even one that the compiler takes for a load of constant memory (__ldg, or a
// __restrict__ pointer that the kernel only reads).  Copies by the TMA unit are
// issued after the wait and need nothing more.
__device__ __forceinline__ unsigned wait_for_stream() {
  unsigned zero;
  asm volatile("griddepcontrol.wait;\n\tmov.u32 %0, 0;" : "=r"(zero) :: "memory");
  return zero;
}

// Blocks of the kernel after this one (if launch_after starts it) may be set up
// once every block of this one has come here or ended.
__device__ __forceinline__ void let_next_start() {
  asm volatile("griddepcontrol.launch_dependents;");
}

// Launches kernel k so that it can start while the kernel before it in the
// stream ends; after anything but a kernel a plain launch.
template <class... P, class... A>
void launch_after(void (*k)(P...), dim3 grid, dim3 block, size_t shared, cudaStream_t s,
                  A&&... args) {
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = shared;
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k, static_cast<P>(args)...);
}

}  // namespace jxlr

#endif  // JXLR_LAUNCH_H_
