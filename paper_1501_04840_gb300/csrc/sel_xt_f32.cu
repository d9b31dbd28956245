#define SEL_XT
#include "kernel_select.cuh"

namespace dynot {
template KA<float> pick_ka<float>(int, int);
template KC<float> pick_kc<float>(int, int);
template KCT<float> pick_kct<float>(int);
}  // namespace dynot
