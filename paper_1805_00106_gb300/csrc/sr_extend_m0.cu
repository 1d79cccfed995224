// sr_extend_m0.cu -- instantiations of the int16 extension kernel for readout mode 0
// (best cell anywhere).
#include "sr_extend.cuh"

namespace sr {

int dispatch_mode0(bool persist, uint32_t lanes, uint32_t rows, const ExtArgs& a, cudaStream_t st,
                   uint64_t tasks) {
  if (!persist) {
    if (!ext_nonneg(a)) return launch16<16, 16, 0, false, false>(a, st, tasks);
#define SR_CASE(g, r) \
  if (lanes == g && rows == r) return launch16<g, r, 0, false>(a, st, tasks);
    SR_PLAIN_SHAPES(SR_CASE)
#undef SR_CASE
    return -1;
  }
#define SR_CASE(g, r) \
  if (lanes == g && rows == r) return launch16<g, r, 0, true>(a, st, tasks);
  SR_SHAPES(SR_CASE)
#undef SR_CASE
  return -1;
}

int dispatch_all0(const ExtArgs& a, const uint32_t* upper, uint64_t pairs, cudaStream_t st) {
  return ext_nonneg(a) ? launch_all<32, 0, true>(a, upper, pairs, st) : launch_all<16, 0, false>(a, upper, pairs, st);
}

int preload_mode0() {
  int n_ = 0;
  SR_TOUCH((k_extend_all<32, 0, true>));
  SR_TOUCH((k_extend_all<16, 0, false>));
  SR_TOUCH((k_extend16<16, 16, 0, false, false>));
#define SR_CASE(g, r) SR_TOUCH((k_extend16<g, r, 0, true>));
  SR_SHAPES(SR_CASE)
#undef SR_CASE
#define SR_CASE(g, r) SR_TOUCH((k_extend16<g, r, 0, false>));
  SR_PLAIN_SHAPES(SR_CASE)
#undef SR_CASE
  return n_;
}

}  // namespace sr
