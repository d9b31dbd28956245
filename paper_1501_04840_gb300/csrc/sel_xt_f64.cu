#define SEL_XT
#include "kernel_select.cuh"

namespace dynot {
template KA<double> pick_ka<double>(int, int);
template KC<double> pick_kc<double>(int, int);
template KCT<double> pick_kct<double>(int);
}  // namespace dynot
