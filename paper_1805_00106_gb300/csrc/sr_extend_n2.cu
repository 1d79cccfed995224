// sr_extend_n2.cu -- instantiations of the int16 extension kernel for readout mode 2
// (end-row search of winning windows) and score sets with mismatch > go + ge.
#include "sr_extend.cuh"

namespace sr {

int dispatch_neg2(uint32_t lanes, uint32_t rows, const ExtArgs& a, cudaStream_t st) {
  return launch_shape<2, false>(lanes, rows, a, st, 0);
}

int preload_neg2() { return touch_shapes<2, false>(); }

}  // namespace sr
