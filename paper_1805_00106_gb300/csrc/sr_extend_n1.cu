// sr_extend_n1.cu -- instantiations of the int16 extension kernel for readout mode 1
// (best cell of the final row) and score sets with mismatch > go + ge.
#include "sr_extend.cuh"

namespace sr {

int dispatch_neg1(uint32_t lanes, uint32_t rows, const ExtArgs& a, cudaStream_t st, uint64_t tasks) {
  return launch_shape<1, false>(lanes, rows, a, st, tasks);
}

int preload_neg1() { return touch_shapes<1, false>(); }

}  // namespace sr
