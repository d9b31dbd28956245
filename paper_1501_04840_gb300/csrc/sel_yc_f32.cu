#define SEL_YC
#include "kernel_select.cuh"

namespace dynot {
template KB<float> pick_kb<float>(int);
}  // namespace dynot
