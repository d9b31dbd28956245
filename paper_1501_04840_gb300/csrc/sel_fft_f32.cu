#define SEL_FFT
#include "kernel_select.cuh"

namespace dynot {
template KFY<float> pick_kfy<float>(int, int);
}  // namespace dynot
