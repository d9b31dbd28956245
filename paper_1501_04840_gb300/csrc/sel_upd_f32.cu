#define SEL_UPD
#define SEL_UPD_TMA
#include "kernel_select.cuh"

namespace dynot {
template KD<float> pick_kd<float>(int, bool, bool, bool);
}  // namespace dynot
