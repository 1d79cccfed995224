// sr_extend_n0.cu -- instantiations of the int16 extension kernel for readout mode 0
// (best cell anywhere) and score sets with mismatch > go + ge.
#include "sr_extend.cuh"

namespace sr {

int dispatch_neg0(uint32_t lanes, uint32_t rows, const ExtArgs& a, cudaStream_t st, uint64_t tasks) {
  return launch_shape<0, false>(lanes, rows, a, st, tasks);
}

int preload_neg0() { return touch_shapes<0, false>(); }

}  // namespace sr
