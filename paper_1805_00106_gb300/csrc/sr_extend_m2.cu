// sr_extend_m2.cu -- instantiations of the int16 extension kernel for readout mode 2
// (end-row search of winning windows).
#include "sr_extend.cuh"

namespace sr {

int dispatch_mode2(uint32_t lanes, uint32_t rows, const ExtArgs& a, cudaStream_t st) {
  return ext_nonneg(a) ? launch_shape<2, true>(lanes, rows, a, st, 0) : dispatch_neg2(lanes, rows, a, st);
}

int preload_mode2() { return touch_shapes<2, true>(); }

}  // namespace sr
