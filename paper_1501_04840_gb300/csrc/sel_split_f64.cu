#define SEL_XT
#include "kernel_select.cuh"

namespace dynot {
template KRX<double> pick_krx<double, false>(int);
template KRX<double> pick_krx<double, true>(int);
}  // namespace dynot
