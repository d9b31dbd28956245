#define SEL_FFT_INV
#include "kernel_select.cuh"
