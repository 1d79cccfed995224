// sr_extend_m0.cu -- instantiations of the int16 extension kernel for readout mode 0
// (best cell anywhere).
#include "sr_extend.cuh"

namespace sr {

int dispatch_mode0(bool persist, uint32_t lanes, uint32_t rows, const ExtArgs& a, cudaStream_t st,
                   uint64_t tasks) {
  const bool nn = ext_nonneg(a);
  if (persist) return nn ? launch_shape<0, true>(lanes, rows, a, st, tasks) : dispatch_neg0(lanes, rows, a, st, tasks);
#define SR_CASE(g, r)          \
  if (lanes == g && rows == r) \
    return nn ? launch16<g, r, 0, false, true>(a, st, tasks) : launch16<g, r, 0, false, false>(a, st, tasks);
  SR_PLAIN_SHAPES(SR_CASE)
#undef SR_CASE
  return -1;
}

int dispatch_all0(const ExtArgs& a, const uint32_t* upper, uint64_t pairs, cudaStream_t st) {
  return ext_nonneg(a) ? launch_all<0, true>(a, upper, pairs, st) : launch_all<0, false>(a, upper, pairs, st);
}

int preload_mode0() {
  int n_ = touch_shapes<0, true>();
  SR_TOUCH((k_extend_all<0, true>));
  SR_TOUCH((k_extend_all<0, false>));
#define SR_CASE(g, r)                              \
  SR_TOUCH((k_extend16<g, r, 0, false, true>)); \
  SR_TOUCH((k_extend16<g, r, 0, false, false>));
  SR_PLAIN_SHAPES(SR_CASE)
#undef SR_CASE
  return n_;
}

}  // namespace sr
