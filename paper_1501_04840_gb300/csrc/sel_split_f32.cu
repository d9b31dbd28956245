#define SEL_XT
#include "kernel_select.cuh"

namespace dynot {
template KRX<float> pick_krx<float, false>(int);
template KRX<float> pick_krx<float, true>(int);
}  // namespace dynot
