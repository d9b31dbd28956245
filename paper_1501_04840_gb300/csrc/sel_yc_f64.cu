#define SEL_YC
#include "kernel_select.cuh"

namespace dynot {
template KB<double> pick_kb<double>(int);
}  // namespace dynot
