#define SEL_MM
#include "kernel_select.cuh"

namespace dynot {
template KMF<double> pick_kmf<double>(int);
template KMI<double> pick_kmi<double>(int);
template KMY<double> pick_kmy<double>(int);
}  // namespace dynot
