// Definitions of the kernel selection (kernel_select.h).  A sel_*.cu file defines the part that it instantiates.
#pragma once
#include <type_traits>

#include "kernel_select.h"

namespace dynot {

#ifdef SEL_XT
template <typename T, int PM>
KA<T> pick_ka_p(int n) {
  if constexpr (std::is_same<T, float>::value) return k_rhs_fwd_xt<T, 0, 0, PM>;   // FFT lengths: pick_kff
  else switch (n) {
    case 64: return k_rhs_fwd_xt<T, 8, 8, PM>;
    case 96: return k_rhs_fwd_xt<T, 16, 6, PM>;
    case 128: return k_rhs_fwd_xt<T, 8, 16, PM>;
    case 192: return k_rhs_fwd_xt<T, 16, 12, PM>;
    case 256: return k_rhs_fwd_xt<T, 16, 16, PM>;
    case 512: return k_rhs_fwd_xt<T, 16, 32, PM>;
    default: return k_rhs_fwd_xt<T, 0, 0, PM>;
  }
}
template <typename T>
KA<T> pick_ka(int n, int pm) {
  return pm == 16 ? pick_ka_p<T, 16>(n) : (pm == 32 ? pick_ka_p<T, 32>(n) : pick_ka_p<T, 64>(n));
}
template <typename T, int PM>
KC<T> pick_kc_p(int n) {
  if constexpr (std::is_same<T, float>::value) return k_inv_xt<T, 0, 0, PM>;       // FFT lengths: pick_kfi
  else switch (n) {
    case 64: return k_inv_xt<T, 8, 8, PM>;
    case 96: return k_inv_xt<T, 16, 6, PM>;
    case 128: return k_inv_xt<T, 8, 16, PM>;
    case 192: return k_inv_xt<T, 16, 12, PM>;
    case 256: return k_inv_xt<T, 16, 16, PM>;
    case 512: return k_inv_xt<T, 16, 32, PM>;
    default: return k_inv_xt<T, 0, 0, PM>;
  }
}
template <typename T>
KC<T> pick_kc(int n, int pm) {
  return pm == 16 ? pick_kc_p<T, 16>(n) : (pm == 32 ? pick_kc_p<T, 32>(n) : pick_kc_p<T, 64>(n));
}
template <typename T, bool INV>
KRX<T> pick_krx(int n) {
  switch (n) {
    case 64: return k_rows_x<T, 8, 8, INV>;
    case 96: return k_rows_x<T, 16, 6, INV>;
    case 128: return k_rows_x<T, 8, 16, INV>;
    case 192: return k_rows_x<T, 16, 12, INV>;
    case 256: return k_rows_x<T, 16, 16, INV>;
    case 512: return k_rows_x<T, 16, 32, INV>;
    default: return k_rows_x<T, 0, 0, INV>;
  }
}
template <typename T>
KCT<T> pick_kct(int pm) {
  return pm == 16 ? k_cols_t<T, 16> : (pm == 32 ? k_cols_t<T, 32> : k_cols_t<T, 64>);
}
#endif

#ifdef SEL_YC
template <typename T>
KB<T> pick_kb(int n) {
  if constexpr (std::is_same<T, float>::value) return k_solve_yc<T, 0, 0, kW, 256>;   // FFT lengths: pick_kfy
  else switch (n) {
    case 64: return k_solve_yc<T, 8, 8, kW, yc_nt(8)>;
    case 96: return k_solve_yc<T, 16, 6, kW, yc_nt(16)>;
    case 128: return k_solve_yc<T, 8, 16, kW, yc_nt(8)>;
    case 192: return k_solve_yc<T, 16, 12, kW, yc_nt(16)>;
    case 256: return k_solve_yc<T, 16, 16, kW, yc_nt(16)>;
    case 512: return k_solve_yc<T, 16, 32, kW, yc_nt(16)>;
    default: return k_solve_yc<T, 0, 0, kW, 256>;
  }
}
#endif

#ifdef SEL_FFT
template <typename T, int C>
KFY<T> pick_kfy_c(int n) {
  switch (n) {
    case 64: return k_fft_yc<T, 8, 8, C>;
    case 96: return k_fft_yc<T, 16, 6, C>;
    case 128: return k_fft_yc<T, 8, 16, C>;
    case 192: return k_fft_yc<T, 16, 12, C>;
    case 256: return k_fft_yc<T, 16, 16, C>;
    case 512: return k_fft_yc<T, 16, 32, C>;
    default: return nullptr;
  }
}
template <typename T>
KFY<T> pick_kfy(int n, int C) {
  switch (C) {
    case 1: return pick_kfy_c<T, 1>(n);
    case 2: return pick_kfy_c<T, 2>(n);
    case 3: return pick_kfy_c<T, 3>(n);
    default: return pick_kfy_c<T, 4>(n);
  }
}
#endif

#ifdef SEL_FFT_FWD
template <int PM>
KFF pick_kff_p(int n) {
  switch (n) {
    case 64: return k_fft_fwd_xt<8, 8, PM>;
    case 96: return k_fft_fwd_xt<16, 6, PM>;
    case 128: return k_fft_fwd_xt<8, 16, PM>;
    case 192: return k_fft_fwd_xt<16, 12, PM>;
    case 256: return k_fft_fwd_xt<16, 16, PM>;
    case 512: return k_fft_fwd_xt<16, 32, PM>;
    default: return nullptr;
  }
}
KFF pick_kff(int n, int pm) { return pm == 16 ? pick_kff_p<16>(n) : (pm == 32 ? pick_kff_p<32>(n) : pick_kff_p<64>(n)); }
#endif

#ifdef SEL_FFT_INV
template <int PM>
KFI pick_kfi_p(int n) {
  switch (n) {
    case 64: return k_fft_inv_xt<8, 8, PM>;
    case 96: return k_fft_inv_xt<16, 6, PM>;
    case 128: return k_fft_inv_xt<8, 16, PM>;
    case 192: return k_fft_inv_xt<16, 12, PM>;
    case 256: return k_fft_inv_xt<16, 16, PM>;
    case 512: return k_fft_inv_xt<16, 32, PM>;
    default: return nullptr;
  }
}
KFI pick_kfi(int n, int pm) { return pm == 16 ? pick_kfi_p<16>(n) : (pm == 32 ? pick_kfi_p<32>(n) : pick_kfi_p<64>(n)); }
#endif

#ifdef SEL_MM
template <typename T>
KMF<T> pick_kmf(int pm) {
  switch (pm) {
    case 16: return k_mm_fwd_xt<T, 16>;
    case 24: return k_mm_fwd_xt<T, 24>;
    case 32: return k_mm_fwd_xt<T, 32>;
    case 48: return k_mm_fwd_xt<T, 48>;
    default: return k_mm_fwd_xt<T, 64>;
  }
}
template <typename T>
KMI<T> pick_kmi(int pm) {
  switch (pm) {
    case 16: return k_mm_inv_xt<T, 16>;
    case 24: return k_mm_inv_xt<T, 24>;
    case 32: return k_mm_inv_xt<T, 32>;
    case 48: return k_mm_inv_xt<T, 48>;
    default: return k_mm_inv_xt<T, 64>;
  }
}
template <typename T>
KMY<T> pick_kmy(int C) {
  switch (C) {
    case 1: return k_mm_yc<T, 1>;
    case 2: return k_mm_yc<T, 2>;
    case 3: return k_mm_yc<T, 3>;
    default: return k_mm_yc<T, 4>;
  }
}
#endif

#ifdef SEL_UPD
template <typename T, int C, bool PXY>
KD<T> pick_kd_c(bool check, bool wx) {
  if (check) return wx ? k_update_tiled<T, C, true, true, PXY> : k_update_tiled<T, C, true, false, PXY>;
  return wx ? k_update_tiled<T, C, false, true, PXY> : k_update_tiled<T, C, false, false, PXY>;
}
template <typename T, bool PXY>
KD<T> pick_kd_p(int C, bool check, bool wx) {
  switch (C) {
    case 1: return pick_kd_c<T, 1, PXY>(check, wx);
    case 2: return pick_kd_c<T, 2, PXY>(check, wx);
    case 3: return pick_kd_c<T, 3, PXY>(check, wx);
    default: return pick_kd_c<T, 4, PXY>(check, wx);
  }
}
template <typename T>
KD<T> pick_kd(int C, bool check, bool wx, bool per_xy) {
  return per_xy ? pick_kd_p<T, true>(C, check, wx) : pick_kd_p<T, false>(C, check, wx);
}
#endif

#ifdef SEL_UPD_TMA
// the update kernel with tensor-memory-accelerator staging (FP32, Neumann x and y)
template <int C>
KDT pick_kdt_c(bool check, bool wx) {
  if (check) return wx ? k_update_tma<C, true, true> : k_update_tma<C, true, false>;
  return wx ? k_update_tma<C, false, true> : k_update_tma<C, false, false>;
}
KDT pick_kdt(int C, bool check, bool wx) {
  switch (C) {
    case 1: return pick_kdt_c<1>(check, wx);
    case 2: return pick_kdt_c<2>(check, wx);
    case 3: return pick_kdt_c<3>(check, wx);
    default: return pick_kdt_c<4>(check, wx);
  }
}
#endif

}  // namespace dynot
