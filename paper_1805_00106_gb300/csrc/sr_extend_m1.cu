// sr_extend_m1.cu -- instantiations of the int16 extension kernel for readout mode 1
// (best cell of the final row).
#include "sr_extend.cuh"

namespace sr {

int dispatch_mode1(bool persist, uint32_t lanes, uint32_t rows, const ExtArgs& a, cudaStream_t st,
                   uint64_t tasks) {
  const bool nn = ext_nonneg(a);
  if (persist) return nn ? launch_shape<1, true>(lanes, rows, a, st, tasks) : dispatch_neg1(lanes, rows, a, st, tasks);
#define SR_CASE(g, r)          \
  if (lanes == g && rows == r) \
    return nn ? launch16<g, r, 1, false, true>(a, st, tasks) : launch16<g, r, 1, false, false>(a, st, tasks);
  SR_PLAIN_SHAPES(SR_CASE)
#undef SR_CASE
  return -1;
}

int dispatch_all1(const ExtArgs& a, const uint32_t* upper, uint64_t pairs, cudaStream_t st) {
  return ext_nonneg(a) ? launch_all<1, true>(a, upper, pairs, st) : launch_all<1, false>(a, upper, pairs, st);
}

int preload_mode1() {
  int n_ = touch_shapes<1, true>();
  SR_TOUCH((k_extend_all<1, true>));
  SR_TOUCH((k_extend_all<1, false>));
#define SR_CASE(g, r)                              \
  SR_TOUCH((k_extend16<g, r, 1, false, true>)); \
  SR_TOUCH((k_extend16<g, r, 1, false, false>));
  SR_PLAIN_SHAPES(SR_CASE)
#undef SR_CASE
  return n_;
}

}  // namespace sr
