#define SEL_FFT_FWD
#include "kernel_select.cuh"
