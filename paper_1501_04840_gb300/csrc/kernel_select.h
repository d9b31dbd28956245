// Kernel selection: which instance of each kernel of an iteration a plan launches.  The functions are defined in
// kernel_select.cuh and instantiated in the sel_*.cu files, so that the kernels compile as separate units.
#pragma once
#include <cuda.h>

#include "fft_kernels.cuh"
#include "hue_kernels.cuh"
#include "misc_kernels.cuh"
#include "mm_kernels.cuh"
#include "rgb_kernels.cuh"
#include "rgb_update_tma.cuh"

namespace dynot {

constexpr int kThreadsXt = 256;
constexpr int kThreadsUpd = 128;
constexpr int kW = 8;   // x-strip width of the row-based y/colour pass (k_solve_yc)

inline int pmax_for(int P) { return P <= 16 ? 16 : (P <= 32 ? 32 : 64); }
// lengths with an FFT path: 2^k (64-512) and 3 * 2^k (96 = 16 * 6, 192 = 16 * 12); N1 = fft_n1(n)
inline bool fft_len(int n) { return n == 64 || n == 96 || n == 128 || n == 192 || n == 256 || n == 512; }
inline int fft_n1(int n) { return n == 64 ? 8 : (n == 128 ? 8 : 16); }
// threads of k_solve_yc: 12 row pairs of length n2 per FFT chunk, 256 on the dense path
constexpr int yc_nt(int m1) { return 12 * m1; }
inline int yc_threads(int n2) { return fft_len(n2) ? yc_nt(fft_n1(n2)) : 256; }

// the folded-product transforms (mm_kernels.cuh): time lengths in register arrays of 16, 24, 32, 48 or 64
inline int mm_pm(int P) { return P <= 16 ? 16 : (P <= 24 ? 24 : (P <= 32 ? 32 : (P <= 48 ? 48 : 64))); }

template <typename T> using KA = void (*)(Geo<T>, const v4<T>*, const T*, const T*, T*, XtTables, int);
template <typename T> using KC = void (*)(Geo<T>, const T*, T*, XtTables, int);
template <typename T> using KB = void (*)(Geo<T>, T*, YcTables, int);
template <typename T> using KH = void (*)(Geo<T>, T*, HueTables);
template <typename T> using KRX = void (*)(Geo<T>, const T*, T*, XtTables, int);
template <typename T> using KCT = void (*)(Geo<T>, T*, const T*);
template <typename T> using KFY = void (*)(Geo<T>, T*, YcTables);
using KFF = void (*)(Geo<float>, const float4*, const float*, const float*, float*, FftXtTables);
using KFI = void (*)(Geo<float>, const float*, float*, FftXtTables);
template <typename T> using KMF = void (*)(Geo<T>, const v4<T>*, const T*, const T*, T*, MmAxis<T>, const T*);
template <typename T> using KMI = void (*)(Geo<T>, const T*, T*, MmAxis<T>, const T*);
template <typename T> using KMY = void (*)(Geo<T>, T*, YcTables, MmAxis<T>, int);
template <typename T> using KD = void (*)(Geo<T>, Arrays<T>, int, TileLayout, double*);
using KDT = void (*)(Geo<float>, Arrays<float>, int, double*, int*, const CUtensorMap, const CUtensorMap,
                     const CUtensorMap);

template <typename T> KA<T> pick_ka(int n, int pm);
template <typename T> KC<T> pick_kc(int n, int pm);
template <typename T, bool INV> KRX<T> pick_krx(int n);
template <typename T> KCT<T> pick_kct(int pm);
template <typename T> KB<T> pick_kb(int n);
template <typename T> KFY<T> pick_kfy(int n, int C);   // nullptr unless n is an FFT length
KFF pick_kff(int n, int pm);   // FFT lengths; pm = 16, 32 or 64
KFI pick_kfi(int n, int pm);
template <typename T> KMF<T> pick_kmf(int pm);
template <typename T> KMI<T> pick_kmi(int pm);
template <typename T> KMY<T> pick_kmy(int C);
template <typename T> KD<T> pick_kd(int C, bool check, bool wx, bool per_xy);
KDT pick_kdt(int C, bool check, bool wx);   // FP32, staged by bulk tensor copies

}  // namespace dynot
