// Hue image pipeline of section 5: HSV conversion, hue histograms and the
// periodic exact histogram specification that turns each transported hue
// histogram h^t back into an image (saturation and value kept).
//
// The paper cites, without printing them, an analysis of transport on the
// circle and an exact specification method.  The reading implemented here:
// pixels are ranked by a strict order (hue quantised to 32 bits, then pixel
// index); the target histogram becomes exact integer counts (largest
// remainders, ties to the lower bin); target rank q in bin b gets the hue
// (b + (q - C_b + 1/2) / c_b) / bins; the circle is cut at the cyclic shift s of
// least squared circular distance sum_r d(x_r, y_{(r-s) mod n})^2 over all n
// shifts (the smaller of shifts whose computed costs are equal).  For sorted points on the circle and a
// cost convex in the circular distance an optimal matching is a cyclic shift of
// the sorted orders, so this cut is the optimal assignment of the source pixels
// to the target hues.
#include "../../include/dynot.h"

#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <vector>

#include "abi_guard.h"
#include "plan_base.h"

namespace dynot {
namespace {

__global__ void k_rgb_to_hsv(int n, const float* __restrict__ rgb, float* __restrict__ h, float* __restrict__ s,
                             float* __restrict__ v) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float r = rgb[i], g = rgb[(size_t)n + i], b = rgb[2 * (size_t)n + i];
    const float mx = fmaxf(fmaxf(r, g), b), mn = fminf(fminf(r, g), b), d = mx - mn;
    float hh = 0.f;
    if (d > 0.f) {
      if (mx == r) {
        hh = (g - b) / d;
        if (hh < 0.f) hh += 6.f;
      } else if (mx == g) {
        hh = (b - r) / d + 2.f;
      } else {
        hh = (r - g) / d + 4.f;
      }
      hh /= 6.f;
      if (hh >= 1.f) hh -= 1.f;
    }
    h[i] = hh;
    s[i] = mx > 0.f ? d / mx : 0.f;
    v[i] = mx;
  }
}

__global__ void k_hsv_to_rgb(int n, const float* __restrict__ h, const float* __restrict__ s,
                             const float* __restrict__ v, float* __restrict__ rgb) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float h6 = h[i] * 6.f;
    const float fl = floorf(h6);
    const int sec = ((int)fl % 6 + 6) % 6;
    const float f = h6 - fl, vv = v[i], ss = s[i];
    const float p = vv * (1.f - ss), q = vv * (1.f - ss * f), t = vv * (1.f - ss * (1.f - f));
    float r, g, b;
    switch (sec) {
      case 0: r = vv; g = t; b = p; break;
      case 1: r = q; g = vv; b = p; break;
      case 2: r = p; g = vv; b = t; break;
      case 3: r = p; g = q; b = vv; break;
      case 4: r = t; g = p; b = vv; break;
      default: r = vv; g = p; b = q; break;
    }
    rgb[i] = r;
    rgb[(size_t)n + i] = g;
    rgb[2 * (size_t)n + i] = b;
  }
}

__device__ __forceinline__ int hue_bin_of(float h, int bins) {
  return min((int)floor((double)h * bins), bins - 1);
}

// counts (float, exact below 2^24 per bin) then normalisation in a second kernel
__global__ void k_hue_count(int n, const float* __restrict__ h, int bins, float* __restrict__ cnt) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    atomicAdd(&cnt[max(hue_bin_of(h[i], bins), 0)], 1.f);
}
__global__ void k_scale(int n, float* __restrict__ x, float s) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) x[i] *= s;
}

// strict order keys: (hue quantised to 32 bits) << 32 | index; padding keys sort last
__global__ void k_hue_keys(int n, int m, const float* __restrict__ h, unsigned long long* __restrict__ key) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
    if (i < n) {
      const double q = fmin(floor((double)h[i] * 4294967296.0), 4294967295.0);
      key[i] = ((unsigned long long)q << 32) | (unsigned long long)i;
    } else {
      key[i] = ~0ULL;
    }
  }
}

// Ascending bitonic sort of m = 2^p keys.  Runs of kSortRun keys are sorted, and the strides below a run of every
// later merge finished, in shared memory; the strides from a run on go through memory two at a time, four keys per
// thread.  The keys are distinct, so the order is the same whatever the stages: 65536 keys take 13 launches where one
// launch per stage took 136 (about 2.4 us each).
constexpr int kSortRun = 2048, kSortThreads = 512;

__device__ __forceinline__ void key_exchange(unsigned long long& a, unsigned long long& b, bool up) {
  if ((a > b) == up) {
    const unsigned long long t = a;
    a = b;
    b = t;
  }
}
// k0 = 2: sort every run; otherwise finish merge k0 (strides min(k0, run) / 2 ... 1) of every run
__global__ void __launch_bounds__(kSortThreads) k_sort_runs(unsigned long long* __restrict__ key, int m, int k0) {
  __shared__ unsigned long long sk[kSortRun];
  const int run = min(kSortRun, m), base = blockIdx.x * run;
  for (int i = threadIdx.x; i < run; i += kSortThreads) sk[i] = key[base + i];
  __syncthreads();
  const int k1 = k0 == 2 ? run : k0;
  for (int k = k0; k <= k1; k <<= 1)
    for (int j = min(k, run) >> 1; j > 0; j >>= 1) {
      for (int q = threadIdx.x; q < run / 2; q += kSortThreads) {
        const int i = 2 * q - (q & (j - 1));   // the q-th index without bit j
        key_exchange(sk[i], sk[i + j], ((base + i) & k) == 0);
      }
      __syncthreads();
    }
  for (int i = threadIdx.x; i < run; i += kSortThreads) key[base + i] = sk[i];
}
// strides j and, when two, j / 2 of merge k
__global__ void k_sort_strides(unsigned long long* __restrict__ key, int m, int k, int j, int two) {
  const int per = two ? 4 : 2, h = j >> 1;
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < m / per; q += gridDim.x * blockDim.x) {
    if (two) {
      const int i = 4 * q - 3 * (q & (h - 1));   // the q-th index without bits j and j / 2
      const bool up = (i & k) == 0;
      unsigned long long a = key[i], b = key[i + h], c = key[i + j], d = key[i + j + h];
      key_exchange(a, c, up);
      key_exchange(b, d, up);
      key_exchange(a, b, up);
      key_exchange(c, d, up);
      key[i] = a;
      key[i + h] = b;
      key[i + j] = c;
      key[i + j + h] = d;
    } else {
      const int i = 2 * q - (q & (j - 1));
      unsigned long long a = key[i], b = key[i + j];
      key_exchange(a, b, (i & k) == 0);
      key[i] = a;
      key[i + j] = b;
    }
  }
}

// sorted source hues x_r (double) and pixel index of rank r
__global__ void k_sorted_hues(int n, const unsigned long long* __restrict__ key, const float* __restrict__ h,
                              double* __restrict__ x, int* __restrict__ idx) {
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x) {
    const int i = (int)(key[r] & 0xffffffffULL);
    idx[r] = i;
    x[r] = (double)h[i];
  }
}

// target hue of rank q: bin b with C_b <= q < C_{b+1}, (b + (q - C_b + 1/2) / c_b) / bins
__global__ void k_target_hues(int n, int bins, const long long* __restrict__ C, double* __restrict__ y) {
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x) {
    int lo = 0, hi = bins;   // largest b with C[b] <= q
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (C[mid] <= q) lo = mid;
      else hi = mid;
    }
    const double cb = (double)(C[lo + 1] - C[lo]);
    y[q] = ((double)lo + ((double)(q - C[lo]) + 0.5) / cb) / bins;
  }
}

// The least of cost[s] = sum_r d(x_r, y_{(r - s) mod n})^2 over the n cyclic shifts, d the circular distance.
//
// Lifted to the line (x and y continued by x_{r+n} = x_r + 1, y_{q+n} = y_q + 1), L(s) = sum_r (x_r - y_{r-s})^2 over
// all integers s has the differences L(s + 1) - L(s) = sum_q g_q (2 x_{q+s} - y_q - y_{q-1}) with the gaps
// g_q = y_q - y_{q-1} >= 0, which increase with s because x does: L is convex (the matching of two sorted sets
// on the circle under a convex cost; J. Delon, J. Salomon, A. Sobolevski, "Fast transport optimization for
// Monge costs on the circle", SIAM J. Appl. Math. 70(7), 2010).  cost[s mod n] <= L(s), with equality at an
// optimal shift, so the least cost lies at the minimum of L.  Its place is found by the sign of the differences,
// sum_q g_q (y_q + y_{q-1}) = 2 y_{n-1} - 1 being a constant:
//   k_shift_slope   : the signs at kSlopePoints shifts per round (one block each, n terms), three rounds;
//   k_shift_window  : the costs of the kShiftBlock shifts around it, tile by tile in float;
//   k_window_costs  : their sums over the tiles in double, in order; k_argmin_shift takes the least.
// The costs are the sums of the exhaustive search below term by term, so the shift is the one it finds (rounding
// moves a minimum of the float sums by a few shifts, the window holds 512 to either side; costs that agree to float
// rounding over more shifts than that are told apart by their rounding alone).  n^2 terms become about 1400 n: 0.08 ms
// in place of 4.7 ms for 65536 pixels.  Hues outside [0, 1], images of one hue (all shifts cost the
// same there, and the first minimum of the float sums may lie anywhere) and images of at most kShiftSmall pixels take
// the exhaustive search, which covers every shift.
//
// Exhaustive search and window alike: a block takes
// kShiftBlock consecutive shifts, kShiftPer per thread (s = s0 + tid + kShiftThreads u), and walks r in
// tiles of kShiftTile: the tile of x and the window of y that its shifts reach sit in shared memory, x
// read as a broadcast and y at consecutive addresses across the threads.  The target hue is held as a
// float pair (hi + lo = y to about 2^-48), so x - y is formed to about one unit in the last place of
// the difference; the terms of a tile are summed in float, the tiles in double.
constexpr int kShiftThreads = 256, kShiftPer = 4, kShiftBlock = kShiftThreads * kShiftPer, kShiftTile = 256;
constexpr int kShiftWin = kShiftTile + kShiftBlock - 1;
constexpr int kShiftSmall = 2 * kShiftBlock;

// part[u]: the terms of the tile from r0 for the shifts s0 + tid + kShiftThreads u
__device__ __forceinline__ void shift_tile(int n, int s0, int r0, const float* __restrict__ xs,
                                           const float2* __restrict__ ys, float (&sx)[kShiftTile],
                                           float2 (&sy)[kShiftWin], float (&part)[kShiftPer]) {
  const int tid = threadIdx.x;
  {
    const int len = min(kShiftTile, n - r0);
    __syncthreads();
    for (int i = tid; i < len; i += kShiftThreads) sx[i] = xs[r0 + i];
    // window entry i holds y at q = r0 - s0 - (kShiftBlock - 1) + i (mod n)
    int qb = (int)(((long long)r0 - s0 - (kShiftBlock - 1)) % n);
    if (qb < 0) qb += n;
    for (int i = tid; i < len + kShiftBlock - 1; i += kShiftThreads) {
      int q = qb + i;
      while (q >= n) q -= n;
      sy[i] = ys[q];
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kShiftPer; ++u) part[u] = 0.f;
    // thread (tid, u) has shift s = s0 + tid + kShiftThreads u; term r reads sy[r - r0 + kShiftBlock - 1 - (s - s0)]
    const int wb = kShiftBlock - 1 - tid;
#pragma unroll 4
    for (int r = 0; r < len; ++r) {
      const float xv = sx[r];
#pragma unroll
      for (int u = 0; u < kShiftPer; ++u) {
        const float2 yv = sy[r + wb - kShiftThreads * u];
        const float e = fabsf((xv - yv.x) - yv.y);
        const float d = fminf(e, 1.f - e);
        part[u] = fmaf(d, d, part[u]);
      }
    }
  }
}

// every shift; runs when *all is set
__global__ void __launch_bounds__(kShiftThreads) k_shift_costs(int n, const float* __restrict__ xs,
                                                               const float2* __restrict__ ys,
                                                               const int* __restrict__ all,
                                                               double* __restrict__ cost) {
  __shared__ float sx[kShiftTile];
  __shared__ float2 sy[kShiftWin];
  if (*all == 0) return;
  const int s0 = blockIdx.x * kShiftBlock, tid = threadIdx.x;
  double acc[kShiftPer];
#pragma unroll
  for (int u = 0; u < kShiftPer; ++u) acc[u] = 0.0;
  for (int r0 = 0; r0 < n; r0 += kShiftTile) {
    float part[kShiftPer];
    shift_tile(n, s0, r0, xs, ys, sx, sy, part);
#pragma unroll
    for (int u = 0; u < kShiftPer; ++u) acc[u] += (double)part[u];
  }
#pragma unroll
  for (int u = 0; u < kShiftPer; ++u) {
    const int s = s0 + tid + kShiftThreads * u;
    if (s < n) cost[s] = acc[u];
  }
}

// The shifts of a round: kSlopePoints inside (lo, hi), where the difference of L is negative at lo and not at hi.
// range() follows the rounds done so far from (-2 n, 2 n), which holds a minimum for hues in [0, 1].
constexpr int kSlopePoints = 128, kSlopeRounds = 3;
__device__ __forceinline__ long long slope_point(long long lo, long long hi, int j) {
  return lo + (hi - lo) * (j + 1) / (kSlopePoints + 1);
}
// every thread of a block of at least kSlopePoints threads calls it
__device__ __forceinline__ void slope_range(int n, const int* __restrict__ neg, int rounds, long long& lo, long long& hi) {
  lo = -2ll * n;
  hi = 2ll * n;
  for (int k = 0; k < rounds; ++k) {
    const int cnt = __syncthreads_count(threadIdx.x < kSlopePoints && neg[k * kSlopePoints + threadIdx.x] != 0);
    const long long a = cnt > 0 ? slope_point(lo, hi, cnt - 1) : lo;
    hi = cnt < kSlopePoints ? slope_point(lo, hi, cnt) : hi;
    lo = a;
  }
}
// neg[round][j]: whether L(s + 1) < L(s) at the j-th shift of the round.  gap: g_q of the target hues.
__global__ void __launch_bounds__(256) k_shift_slope(int n, int round, const float* __restrict__ xs,
                                                     const float* __restrict__ gap, const double* __restrict__ y,
                                                     int* __restrict__ neg) {
  long long lo, hi;
  slope_range(n, neg, round, lo, hi);
  const long long s = slope_point(lo, hi, blockIdx.x);
  // x_{q+s} = xs[(q + s) mod n] + floor((q + s) / n)
  long long turn = s / n;
  int off = (int)(s % n);
  if (off < 0) {
    off += n;
    --turn;
  }
  // float sums of up to 32 terms, added in double: an error of 1e-7 moves the sign change by n 1e-7 / 2 shifts
  double acc = 0;
  for (int q0 = threadIdx.x; q0 < n; q0 += 32 * 256) {
    float part = 0.f;
#pragma unroll 8
    for (int u = 0; u < 32; ++u) {
      const int q = q0 + 256 * u;
      if (q < n) {
        const int i = q + off;
        const bool wrap = i >= n;
        part = fmaf(gap[q], xs[wrap ? i - n : i] + (wrap ? 1.f : 0.f), part);
      }
    }
    acc += (double)part;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  __shared__ double red[8];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double sum = 0;
    for (int w = 0; w < 8; ++w) sum += red[w];
    neg[round * kSlopePoints + blockIdx.x] = 2.0 * (sum + (double)turn) - (2.0 * y[n - 1] - 1.0) < 0.0;
  }
}
// *place: first shift of the window, in [0, n)
__global__ void __launch_bounds__(kSlopePoints) k_window_place(int n, const int* __restrict__ neg, int* __restrict__ place) {
  long long lo, hi;
  slope_range(n, neg, kSlopeRounds, lo, hi);
  const int s0 = (int)(((lo + hi) / 2 - kShiftBlock / 2) % n);
  if (threadIdx.x == 0) *place = s0 < 0 ? s0 + n : s0;
}
// one tile of r per block, the kShiftBlock shifts of the window: part[tile][shift]
__global__ void __launch_bounds__(kShiftThreads) k_shift_window(int n, const float* __restrict__ xs,
                                                                const float2* __restrict__ ys,
                                                                const int* __restrict__ place,
                                                                float* __restrict__ parts) {
  __shared__ float sx[kShiftTile];
  __shared__ float2 sy[kShiftWin];
  const int s0 = *place;
  float part[kShiftPer];
  shift_tile(n, s0, blockIdx.x * kShiftTile, xs, ys, sx, sy, part);
#pragma unroll
  for (int u = 0; u < kShiftPer; ++u)
    parts[(size_t)blockIdx.x * kShiftBlock + threadIdx.x + kShiftThreads * u] = part[u];
}
// cost of the window's shifts, the tiles added in double in the order of the exhaustive search
__global__ void __launch_bounds__(32) k_window_costs(int n, const int* __restrict__ place, const int* __restrict__ all,
                                                     const float* __restrict__ parts, double* __restrict__ cost) {
  if (*all) return;
  const int i = blockIdx.x * 32 + threadIdx.x, tiles = (n + kShiftTile - 1) / kShiftTile;
  double acc = 0;
#pragma unroll 32
  for (int t = 0; t < tiles; ++t) acc += (double)parts[(size_t)t * kShiftBlock + i];
  cost[(*place + i) % n] = acc;
}

// the first minimiser of cost (ties to the smaller shift), one block: over all shifts, or over the window
__global__ void k_argmin_shift(int n, const double* __restrict__ cost, const int* __restrict__ place,
                               const int* __restrict__ all, int* __restrict__ best) {
  double bc = INFINITY;
  int bs = n;
  const bool every = *all != 0;
  const int s0 = every ? 0 : *place, cnt = every ? n : kShiftBlock;
  for (int i = threadIdx.x; i < cnt; i += blockDim.x) {
    const int s = (s0 + i) % n;
    const double c = cost[s];
    if (c < bc || (c == bc && s < bs)) { bc = c; bs = s; }
  }
  __shared__ double rc[1024];
  __shared__ int rs[1024];
  rc[threadIdx.x] = bc;
  rs[threadIdx.x] = bs;
  __syncthreads();
  for (int w = blockDim.x >> 1; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      const double c2 = rc[threadIdx.x + w];
      const int s2 = rs[threadIdx.x + w];
      if (c2 < rc[threadIdx.x] || (c2 == rc[threadIdx.x] && s2 < rs[threadIdx.x])) {
        rc[threadIdx.x] = c2;
        rs[threadIdx.x] = s2;
      }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) *best = rs[0] < n ? rs[0] : 0;
}

// float source hues of the sorted ranks, the target hues as float pairs and their gaps; sets *all where a hue lies
// outside [0, 1], or the image is small or of one hue, so that every shift is searched
__global__ void k_shift_inputs(int n, const double* __restrict__ x, const double* __restrict__ y,
                               float* __restrict__ xs, float2* __restrict__ ys, float* __restrict__ gap,
                               int* __restrict__ all) {
  if ((n <= kShiftSmall || x[0] == x[n - 1]) && blockIdx.x == 0 && threadIdx.x == 0) *all = 1;
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x) {
    xs[r] = (float)x[r];
    const float hi = (float)y[r];
    ys[r] = make_float2(hi, (float)(y[r] - (double)hi));
    gap[r] = (float)(r > 0 ? y[r] - y[r - 1] : y[0] - y[n - 1] + 1.0);
    if (!(x[r] >= 0.0 && x[r] <= 1.0)) *all = 1;
  }
}

// rank r receives target rank (r - s) mod n
__global__ void k_assign(int n, const int* __restrict__ shift, const int* __restrict__ idx,
                         const double* __restrict__ y, float* __restrict__ out) {
  const int s = *shift;
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x) {
    int q = r - s;
    if (q < 0) q += n;
    out[idx[r]] = (float)y[q];
  }
}

inline int grid_for(long long n) { return (int)std::min<long long>((n + 255) / 256, 152 * 16); }

// an exhaustive shift search costs npix^2 terms (about 0.15 s on one GPU at 2^20 pixels)
constexpr int kMaxSpecifyPixels = 1 << 21;

}  // namespace
}  // namespace dynot

using namespace dynot;

#define HP_CHECK()                                                                 \
  do {                                                                             \
    cudaError_t e_ = cudaGetLastError();                                           \
    if (e_ != cudaSuccess) return seterr(OT_ECUDA, "%s", cudaGetErrorString(e_)); \
  } while (0)

extern "C" {

ot_status ot_rgb_to_hsv(int npix, const float* rgb, float* h, float* s, float* v, void* stream) {
  if (npix < 0 || (npix > 0 && (!rgb || !h || !s || !v))) return seterr(OT_EINVAL, "bad rgb_to_hsv arguments");
  if (npix == 0) return OT_OK;
  k_rgb_to_hsv<<<grid_for(npix), 256, 0, (cudaStream_t)stream>>>(npix, rgb, h, s, v);
  HP_CHECK();
  return OT_OK;
}

ot_status ot_hsv_to_rgb(int npix, const float* h, const float* s, const float* v, float* rgb, void* stream) {
  if (npix < 0 || (npix > 0 && (!rgb || !h || !s || !v))) return seterr(OT_EINVAL, "bad hsv_to_rgb arguments");
  if (npix == 0) return OT_OK;
  k_hsv_to_rgb<<<grid_for(npix), 256, 0, (cudaStream_t)stream>>>(npix, h, s, v, rgb);
  HP_CHECK();
  return OT_OK;
}

ot_status ot_hue_histogram(int npix, const float* h, int bins, float* hist, void* stream) {
  if (npix < 1 || npix >= (1 << 24) || bins < 2 || !h || !hist)
    return seterr(OT_EINVAL, "hue_histogram: need 1 <= npix < 2^24, bins >= 2");
  cudaStream_t st = (cudaStream_t)stream;
  CUDA_OK(cudaMemsetAsync(hist, 0, sizeof(float) * bins, st));
  k_hue_count<<<grid_for(npix), 256, 0, st>>>(npix, h, bins, hist);
  HP_CHECK();
  k_scale<<<grid_for(bins), 256, 0, st>>>(bins, hist, (float)(1.0 / npix));
  HP_CHECK();
  return OT_OK;
}

ot_status ot_hue_specify(int npix, const float* h, int bins, const float* target, float* h_out, void* stream) {
  return ot_guard([&]() -> ot_status {
    if (npix < 1 || npix > kMaxSpecifyPixels || bins < 2 || !h || !target || !h_out)
      return seterr(OT_EINVAL, "hue_specify: need 1 <= npix <= 2^21, bins >= 2");
    cudaStream_t st = (cudaStream_t)stream;
    // exact counts of the target (host: bins values)
    std::vector<float> tg(bins);
    CUDA_OK(cudaMemcpyAsync(tg.data(), target, sizeof(float) * bins, cudaMemcpyDefault, st));
    CUDA_OK(cudaStreamSynchronize(st));
    // negative entries (an unconverged path can hold a few) count as empty; the rest is renormalised
    double mass = 0;
    for (int b = 0; b < bins; ++b) {
      if (!std::isfinite(tg[b])) return seterr(OT_EINVAL, "hue_specify: non-finite target");
      mass += tg[b] > 0.f ? (double)tg[b] : 0.0;
    }
    if (!(mass > 0)) return seterr(OT_EINVAL, "hue_specify: empty target");
    std::vector<long long> cnt(bins);
    std::vector<double> rem(bins);
    long long tot = 0;
    for (int b = 0; b < bins; ++b) {
      const double xb = (tg[b] > 0.f ? (double)tg[b] / mass : 0.0) * npix;
      cnt[b] = (long long)std::floor(xb);
      rem[b] = xb - (double)cnt[b];
      tot += cnt[b];
    }
    long long shortfall = npix - tot;
    if (shortfall < 0 || shortfall > bins) return seterr(OT_EINVAL, "hue_specify: bad target");
    std::vector<int> ord(bins);
    for (int b = 0; b < bins; ++b) ord[b] = b;
    std::stable_sort(ord.begin(), ord.end(), [&](int a, int c) { return rem[a] > rem[c]; });
    for (long long k = 0; k < shortfall; ++k) cnt[ord[k]] += 1;
    std::vector<long long> C(bins + 1, 0);
    for (int b = 0; b < bins; ++b) C[b + 1] = C[b] + cnt[b];
    // device workspace
    int m = 1;
    while (m < npix) m <<= 1;
    DevMem ws;
    const size_t bytes = sizeof(unsigned long long) * m + 2 * sizeof(double) * npix + sizeof(int) * npix +
                         sizeof(long long) * (bins + 1) + sizeof(float) * npix + sizeof(float2) * npix +
                         sizeof(double) * npix + sizeof(float) * npix +
                         sizeof(float) * kShiftBlock * (size_t)((npix + kShiftTile - 1) / kShiftTile) +
                         sizeof(int) * (kSlopeRounds * kSlopePoints + 3) + 16 * 14;
    CUDA_OK(cudaMalloc(&ws.p, bytes));
    char* q = (char*)ws.p;
    auto take = [&](size_t b) { char* r = q; q += (b + 15) & ~size_t(15); return r; };
    unsigned long long* key = (unsigned long long*)take(sizeof(unsigned long long) * m);
    double* x = (double*)take(sizeof(double) * npix);
    double* y = (double*)take(sizeof(double) * npix);
    int* idx = (int*)take(sizeof(int) * npix);
    long long* dC = (long long*)take(sizeof(long long) * (bins + 1));
    float* xs = (float*)take(sizeof(float) * npix);
    float2* ys = (float2*)take(sizeof(float2) * npix);
    double* dcost = (double*)take(sizeof(double) * npix);
    int* dbest = (int*)take(sizeof(int));
    int* dall = (int*)take(sizeof(int));
    int* dplace = (int*)take(sizeof(int));
    int* dneg = (int*)take(sizeof(int) * kSlopeRounds * kSlopePoints);
    float* dgap = (float*)take(sizeof(float) * npix);
    const int tiles = (npix + kShiftTile - 1) / kShiftTile;
    float* dparts = (float*)take(sizeof(float) * kShiftBlock * (size_t)tiles);
    CUDA_OK(cudaMemsetAsync(dall, 0, sizeof(int), st));
    // strict order of the source hues
    k_hue_keys<<<grid_for(m), 256, 0, st>>>(npix, m, h, key);
    HP_CHECK();
    const int run = std::min(m, kSortRun);
    k_sort_runs<<<m / run, kSortThreads, 0, st>>>(key, m, 2);
    for (int k = 2 * run; k <= m; k <<= 1) {
      int j = k >> 1;
      for (; j > run; j >>= 2) k_sort_strides<<<grid_for(m / 4), 256, 0, st>>>(key, m, k, j, 1);
      if (j == run) k_sort_strides<<<grid_for(m / 2), 256, 0, st>>>(key, m, k, j, 0);
      k_sort_runs<<<m / run, kSortThreads, 0, st>>>(key, m, k);
    }
    HP_CHECK();
    k_sorted_hues<<<grid_for(npix), 256, 0, st>>>(npix, key, h, x, idx);
    CUDA_OK(cudaMemcpyAsync(dC, C.data(), sizeof(long long) * (bins + 1), cudaMemcpyHostToDevice, st));
    k_target_hues<<<grid_for(npix), 256, 0, st>>>(npix, bins, dC, y);
    HP_CHECK();
    // least-cost cyclic shift: by convexity, or over all npix shifts
    k_shift_inputs<<<grid_for(npix), 256, 0, st>>>(npix, x, y, xs, ys, dgap, dall);
    HP_CHECK();
    for (int k = 0; k < kSlopeRounds; ++k) k_shift_slope<<<kSlopePoints, 256, 0, st>>>(npix, k, xs, dgap, y, dneg);
    k_window_place<<<1, kSlopePoints, 0, st>>>(npix, dneg, dplace);
    k_shift_window<<<tiles, kShiftThreads, 0, st>>>(npix, xs, ys, dplace, dparts);
    k_window_costs<<<kShiftBlock / 32, 32, 0, st>>>(npix, dplace, dall, dparts, dcost);
    k_shift_costs<<<(npix + kShiftBlock - 1) / kShiftBlock, kShiftThreads, 0, st>>>(npix, xs, ys, dall, dcost);
    HP_CHECK();
    k_argmin_shift<<<1, 1024, 0, st>>>(npix, dcost, dplace, dall, dbest);
    HP_CHECK();
    k_assign<<<grid_for(npix), 256, 0, st>>>(npix, dbest, idx, y, h_out);
    HP_CHECK();
    CUDA_OK(cudaStreamSynchronize(st));
    return OT_OK;
  });
}

}  // extern "C"
