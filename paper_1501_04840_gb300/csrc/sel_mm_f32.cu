#define SEL_MM
#include "kernel_select.cuh"

namespace dynot {
template KMF<float> pick_kmf<float>(int);
template KMI<float> pick_kmi<float>(int);
template KMY<float> pick_kmy<float>(int);
}  // namespace dynot
