#define SEL_UPD
#include "kernel_select.cuh"

namespace dynot {
template KD<double> pick_kd<double>(int, bool, bool, bool);
}  // namespace dynot
