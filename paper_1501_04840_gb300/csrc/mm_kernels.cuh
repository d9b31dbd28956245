// The Poisson solve's transforms for axis lengths without an FFT: matrix products over folded rows.
//
// A DCT-II (or a real Fourier transform) of length n is even or odd under the mirror of its axis, so
// with s_i = x_i + x_mirror(i) and d_i = x_i - x_mirror(i) the even part of the spectrum needs only s
// and the odd part only d: two products of half the length and half the outputs, n / 2 multiply-adds
// per output instead of n.  The inverse runs the same way backwards: E_i from the even part, O_i from
// the odd part, x_i = E_i + O_i and x_mirror(i) = E_i - O_i.  A Neumann axis mirrors i to n - 1 - i
// (even part: even frequencies), a periodic one to (n - i) mod n (even part: cosines, odd part: sines).
// The spectrum of an axis is kept in the order [even part][odd part]; the eigenvalue tables of such an
// axis are in the same order.
//
// A thread holds 8 (or 12) rows x 4 outputs (forward) or x 2 mirrored pairs (inverse) in registers, so one
// step of the sum costs 2-3 broadcast shared-memory vectors and 1-2 table vectors per 32-48 multiply-adds.
// The tables (n^2 / 2 values, L2-resident) stream through shared memory in chunks of eight steps, copied
// asynchronously two chunks ahead: read per step from L2 instead, their latency bound the sums.
//
//   k_mm_fwd_xt : r = A a - f_b^-, the time DCT of every column in registers, the x transform;
//   k_mm_yc     : the y transform, the colour eigen-solve and divide, the inverse y transform;
//   k_mm_inv_xt : the inverse time DCT of every column, the inverse x transform -> phi.
// At 180x135x3, P = 24 (events, one GB300): 35, 39 and 25 us against 138, 185 and 234 us of the dense sums; the
// iteration 111 against 575 us.  What bounds them there is latency at three blocks per SM (issue slots 39-58 % busy,
// 1.7 M cells leave 10 warps per SM with this register tile); the multiply-adds alone would take 5-8 us each.
// They replace the dense sums of k_rhs_fwd_xt, k_solve_yc and k_inv_xt (one output and n dependent steps per
// thread), which remain for planes that do not fit shared memory in this layout and for FP64 grids whose pipe they load
// less (plan.cuh, choose_mm).
#pragma once
#include "rgb_kernels.cuh"

namespace dynot {

// Tables of one axis (device).  ft: forward, row i holds the weights of folded input i for the even outputs (l0 values)
// and the odd ones (lf - l0); it: inverse, row q the weights of input q of the even part (li values) and of the odd
// part (li).  h0 rows each, absent entries zero, every row part a multiple of 4.
template <typename T>
struct MmAxis {
  const T *ft, *it;
  int n, h0, h1;   // even and odd part, h0 + h1 = n, h1 <= h0
  int o1;          // first mirrored index: 0 (Neumann) or 1 (periodic)
  int l0, lf, li;
  __device__ __forceinline__ int mirror(int i) const { return o1 ? (i == 0 ? 0 : n - i) : n - 1 - i; }
};

// Row blockIdx.y of the tables of an axis from turn[m] = cos(2 pi m / 4n) and turn2 = 2 / n times it (0 <= m < 4n; a sine
// is 3n further).  n^2 values: 242 us of a hue plan's creation at 360 bins when the host filled them.
template <typename T>
__global__ void __launch_bounds__(128) k_mm_tables(MmAxis<T> ax, const T* __restrict__ turn, const T* __restrict__ turn2,
                                                   T* __restrict__ ft, T* __restrict__ it) {
  const int r = blockIdx.y, c = blockIdx.x * blockDim.x + threadIdx.x;
  const unsigned n = ax.n, N4 = 4 * n;
  if (c < ax.lf) {
    const bool odd = c >= ax.l0;
    const int q = odd ? c - ax.l0 : c, h = odd ? ax.h1 : ax.h0;
    T v = T(0);
    if (q < h && r < h) {
      // periodic: cos(2 pi q r / n), sin(2 pi (q + 1) (r + 1) / n); Neumann: cos(pi k (2 r + 1) / 2n), k = 2 q or 2 q + 1
      const unsigned m = ax.o1 ? (odd ? 4u * (q + 1) * (r + 1) + 3 * n : 4u * q * r) : (2u * q + odd) * (2u * r + 1);
      v = turn[m % N4];
    }
    ft[(size_t)r * ax.lf + c] = v;
  }
  const int d = c - ax.lf;
  if (d >= 0 && d < 2 * ax.li) {
    const bool odd = d >= ax.li;
    const int i = odd ? d - ax.li : d;
    T v = T(0);
    if (i < ax.h0 && r < (odd ? ax.h1 : ax.h0)) {
      const unsigned m = ax.o1 ? (odd ? 4u * (r + 1) * i + 3 * n : 4u * r * i) : (2u * r + odd) * (2u * i + 1);
      v = turn2[m % N4];
      if (!odd && (r == 0 || (ax.o1 && 2u * r == n))) v *= T(0.5);   // weight 1 / n, all others 2 / n
    }
    it[(size_t)r * 2 * ax.li + d] = v;
  }
}

// N consecutive values (N even; aligned to 16 bytes, or to 8 for two floats) to registers and back
template <typename T, int N>
__device__ __forceinline__ void ldv(const T* p, T (&r)[N]) {
  constexpr int V = 16 / (int)sizeof(T);
  if constexpr (sizeof(T) == 4) {
#pragma unroll
    for (int i = 0; i < N / V; ++i) {
      const float4 v = reinterpret_cast<const float4*>(p)[i];
      r[4 * i] = v.x; r[4 * i + 1] = v.y; r[4 * i + 2] = v.z; r[4 * i + 3] = v.w;
    }
  } else {
#pragma unroll
    for (int i = 0; i < N / V; ++i) {
      const double2 v = reinterpret_cast<const double2*>(p)[i];
      r[2 * i] = v.x; r[2 * i + 1] = v.y;
    }
  }
  if constexpr (sizeof(T) == 4 && N % 4 == 2) {
    const float2 v = *reinterpret_cast<const float2*>(p + N / V * V);
    r[N - 2] = v.x; r[N - 1] = v.y;
  }
}
template <typename T, int N>
__device__ __forceinline__ void stv(T* p, const T (&r)[N]) {
  constexpr int V = 16 / (int)sizeof(T);
  static_assert(N % V == 0, "whole vectors");
  if constexpr (sizeof(T) == 4) {
#pragma unroll
    for (int i = 0; i < N / V; ++i)
      reinterpret_cast<float4*>(p)[i] = make_float4(r[4 * i], r[4 * i + 1], r[4 * i + 2], r[4 * i + 3]);
  } else {
#pragma unroll
    for (int i = 0; i < N / V; ++i) reinterpret_cast<double2*>(p)[i] = make_double2(r[2 * i], r[2 * i + 1]);
  }
}

template <typename T, int RT, int E>
__device__ __forceinline__ void mm_zero(T (&acc)[RT][E]) {
#pragma unroll
  for (int r = 0; r < RT; ++r)
#pragma unroll
    for (int e = 0; e < E; ++e) acc[r][e] = T(0);
}

// Tables on their way through shared memory: chunks of kMmK rows in kMmStages slots.  The slots come first in a block's
// shared memory, so that they start on lines of 128 bytes as the tables do in global memory: a warp's copy of 512 bytes
// falls apart into more pieces otherwise (224x97x1, P = 16: y pass 15.8 us, 20.0 with the tables 16 bytes further, 21.7 with
// the slots 48 bytes off; 180x135x3, P = 24 38.9, 42.5, 42.3, its L2 traffic 68 MB, 128 with the slots off).
constexpr int kMmK = 8, kMmStages = 3;
__host__ __device__ inline int mm_buf(int l0, int lf, int li) { return kMmStages * kMmK * (lf > 2 * li ? lf : 2 * li); }

// Start the copy of chunk c (rows 8 c .. 8 c + 7 below h) of a table; every thread of the block calls it, and it
// counts as one group of asynchronous copies even where nothing is left to copy.
template <typename T>
__device__ __forceinline__ void mm_issue(T* buf, const T* tab, int row, int h, int c) {
  constexpr int V = 16 / (int)sizeof(T);
  const int cnt = min(kMmK, h - c * kMmK) * row;
  T* dst = buf + (c % kMmStages) * kMmK * row;
  const T* src = tab + (size_t)c * kMmK * row;
  for (int i = V * threadIdx.x; i < cnt; i += V * blockDim.x) cp_async16(dst + i, src + i);
  asm volatile("cp.async.commit_group;\n" ::: "memory");
}
template <typename T>
__device__ __forceinline__ void mm_start(T* buf, const T* tab, int row, int h) {
  mm_issue<T>(buf, tab, row, h, 0);
  mm_issue<T>(buf, tab, row, h, 1);
}
// Run step(i, table row of step i) for i < h, all threads together; chunks 0 and 1 are on their way.  Threads that are
// not live only copy.
template <typename T, class F>
__device__ __forceinline__ void mm_run(T* buf, const T* tab, int row, int h, bool live, F&& step) {
#pragma unroll 1
  for (int c = 0; c * kMmK < h; ++c) {
    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    __syncthreads();   // chunk c is there for every thread, and every thread is done with chunk c - 1
    mm_issue<T>(buf, tab, row, h, c + 2);
    if (!live) continue;
    const T* t = buf + (c % kMmStages) * kMmK * row;
    const int i0 = c * kMmK;
    if (i0 + kMmK <= h) {
#pragma unroll
      for (int u = 0; u < kMmK; ++u) step(i0 + u, t + u * row);
    } else {
#pragma unroll 1
      for (int u = 0; i0 + u < h; ++u) step(i0 + u, t + u * row);
    }
  }
}
// forward: acc[r][e] += rows[i * stride + r] * table[i][col + e].  Both parities run h0 steps (a missing odd step has
// zero weights), so the lanes of a warp can hold items of either.
template <typename T, int RT>
__device__ __forceinline__ void mm_forward(T (&acc)[RT][4], const T* rows, int stride, int col, const MmAxis<T>& ax,
                                           T* buf, bool live) {
  mm_run<T>(buf, ax.ft, ax.lf, ax.h0, live, [&](int, const T* t) {
    T v[RT], m[4];
    ldv<T, RT>(rows, v);
    ldv<T, 4>(t + col, m);
    rows += stride;
#pragma unroll
    for (int r = 0; r < RT; ++r)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[r][e] = fma(v[r], m[e], acc[r][e]);
  });
}
// inverse: E and O of samples i0, i0 + 1 from the even rows (from `rows`) and the odd rows (h0 rows further)
template <typename T, int RT>
__device__ __forceinline__ void mm_inverse(T (&E)[RT][2], T (&O)[RT][2], const T* rows, int stride, int i0,
                                           const MmAxis<T>& ax, T* buf, bool live) {
  const T* odd = rows + ax.h0 * stride;
  mm_run<T>(buf, ax.it, 2 * ax.li, ax.h0, live, [&](int q, const T* t) {
    T v[RT], m[2];
    ldv<T, RT>(rows, v);
    ldv<T, 2>(t + i0, m);
#pragma unroll
    for (int r = 0; r < RT; ++r)
#pragma unroll
      for (int e = 0; e < 2; ++e) E[r][e] = fma(v[r], m[e], E[r][e]);
    if (q < ax.h1) {
      ldv<T, RT>(odd, v);
      ldv<T, 2>(t + ax.li + i0, m);
#pragma unroll
      for (int r = 0; r < RT; ++r)
#pragma unroll
        for (int e = 0; e < 2; ++e) O[r][e] = fma(v[r], m[e], O[r][e]);
    }
    rows += stride;
    odd += stride;
  });
}

// s and d of every mirrored pair of rows, in place: s at the first row, d at its mirror (row n - 1 - i for pair i)
template <typename T>
__device__ __forceinline__ void mm_fold(T* X, int ld, int len4, const MmAxis<T>& ax) {
  for (int it = threadIdx.x; it < ax.h1 * len4; it += blockDim.x) {
    const int i = it / len4, k = 4 * (it - i * len4);
    T* pa = X + (i + ax.o1) * ld + k;
    T* pb = X + (ax.n - 1 - i) * ld + k;
    T a[4], b[4];
    ldv<T, 4>(pa, a);
    ldv<T, 4>(pb, b);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const T s = a[e] + b[e];
      b[e] = a[e] - b[e];
      a[e] = s;
    }
    stv<T, 4>(pa, a);
    stv<T, 4>(pb, b);
  }
}

// Row stride of the (x, t) plane in shared memory: whole groups of 8 time indices, padded to 4 (mod 8) so that
// the column threads' vector accesses spread over the banks.
__host__ __device__ constexpr int mm_ldt(int P) { return (P + 7) / 8 * 8 + 4; }
constexpr int kMmXtThreads = 256;
template <typename T>
inline size_t mm_xt_smem(int n1, int P, int PM, int buf, bool forward) {
  return sizeof(T) * ((size_t)n1 * mm_ldt(P) + (size_t)((P + 3) / 4 * 4) * (forward ? PM / 2 : PM) + buf +
                      (forward ? (size_t)n1 * P : 0));
}

// Forward pass of one (y, c) row per block.  Mt: the time DCT [k][PM / 2] against the folded samples
// (even k: sums, odd k: differences), rows padded to a multiple of 4 with zeros.
template <typename T, int PM>
__global__ void __launch_bounds__(kMmXtThreads, sizeof(T) == 4 ? 2 : 1)
    k_mm_fwd_xt(Geo<T> g, const v4<T>* __restrict__ ap, const T* __restrict__ f0, const T* __restrict__ f1,
                T* __restrict__ hat, MmAxis<T> ax, const T* __restrict__ Mtg) {
  constexpr int PH = PM / 2;
  extern __shared__ __align__(16) char smraw[];
  const int c = blockIdx.x, y = blockIdx.y, b = blockIdx.z;
  if (retired(g, b)) return;
  const int n1 = g.n1, P = g.P, ld = mm_ldt(P), P4 = (P + 3) / 4 * 4, hP = (P + 1) / 2;
  T* buf = (T*)smraw;        // table chunks
  T* X = buf + mm_buf(ax.l0, ax.lf, ax.li);   // [x][t]
  T* Mt = X + n1 * ld;       // [k][PH]
  T* R = Mt + P4 * PH;       // [t][x]
  mm_start<T>(buf, ax.ft, ax.lf, ax.h0);
  for (int j = threadIdx.x; j < P4 * PH; j += blockDim.x) Mt[j] = Mtg[j];
  __syncthreads();
  pdl_wait();   // a (previous update) is read from here on
  const int ym = y > 0 ? y - 1 : (g.per2 ? g.n2 - 1 : -1);
  const int cm = c > 0 ? c - 1 : (g.perc ? g.C - 1 : -1);
  const size_t S = g.S;
  const size_t rowbase = (size_t)b * P * S + (size_t)n1 * (y + (size_t)g.n2 * c);
  const T* as0 = reinterpret_cast<const T*>(ap + rowbase);   // component k of the row's cell i at as0[4 i + k]
  const int dy = ym >= 0 ? n1 * (ym - y) : 0;
  const int dc = cm >= 0 ? n1 * g.n2 * (cm - c) : 0;
  // r = divergence of a and the time difference with the boundary densities, cell by cell into the tile [t][x]
  {
    const v4<T>* pc = ap + rowbase;
    const T* pf0 = f0 + (size_t)b * S + (rowbase - (size_t)b * P * S);
    const T* pf1 = f1 + (size_t)b * S + (rowbase - (size_t)b * P * S);
    // four cells of the row-major plane per thread and pass, all their loads in flight together (eight were slower)
    constexpr int U = 4;
    const int total = P * n1, dt = blockDim.x / n1, dxs = blockDim.x - dt * n1;
    int t = threadIdx.x / n1, x = threadIdx.x - t * n1;
    for (int base = threadIdx.x; base < total; base += U * blockDim.x) {
      v4<T> av[U];
      T lx[U], ly[U], lc[U], lf[U], uf[U];
      bool hl[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (base + u * (int)blockDim.x < total) {
          const int o = t * (int)S + x;   // a problem's a holds fewer than 2^31 values on this path (host rule)
          const int xm = x > 0 ? x - 1 : (g.per1 ? n1 - 1 : x);
          hl[u] = xm != x;
          av[u] = pc[o];
          lx[u] = as0[4 * (o + xm - x)];
          ly[u] = as0[4 * (o + dy) + 1];
          lc[u] = as0[4 * (o + dc) + 2];
          lf[u] = t > 0 ? as0[4 * (o - (int)S) + 3] : pf0[x];
          uf[u] = t < P - 1 ? T(0) : pf1[x];
          if (t < P - 1) uf[u] = av[u].w;
          t += dt;
          x += dxs;
          if (x >= n1) {
            x -= n1;
            ++t;
          }
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int i = base + u * (int)blockDim.x;
        if (i < total) {
          T r = g.s1 * (av[u].x - (hl[u] ? lx[u] : T(0)));
          r += g.s2 * (av[u].y - (ym >= 0 ? ly[u] : T(0)));
          r += g.sc * (av[u].z - (cm >= 0 ? lc[u] : T(0)));
          r += g.sp * (uf[u] - lf[u]);
          R[i] = r;
        }
      }
    }
  }
  __syncthreads();
  for (int x = threadIdx.x; x < n1; x += blockDim.x) {
    T vs[PH], vd[PH];
#pragma unroll
    for (int t = 0; t < PH; ++t) {
      const bool in = t < hP, mid = 2 * t == P - 1;
      const T lo = in ? R[t * n1 + x] : T(0), hi = in && !mid ? R[(P - 1 - t) * n1 + x] : T(0);
      vs[t] = lo + hi;
      vd[t] = mid ? T(0) : lo - hi;
    }
    for (int k = 0; k < P; k += 4) {
      T acc[4] = {T(0), T(0), T(0), T(0)};
#pragma unroll
      for (int j = 0; j < PH; j += 4) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          T m[4];
          ldv<T, 4>(Mt + (k + e) * PH + j, m);
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[e] = fma(m[q], e & 1 ? vd[j + q] : vs[j + q], acc[e]);
        }
      }
      stv<T, 4>(X + x * ld + k, acc);
    }
  }
  __syncthreads();
  mm_fold<T>(X, ld, (P + 3) / 4, ax);
  __syncthreads();
  // FP64 releases its successor only at its end (XtTables::late): measured per iteration with the trigger here and
  // without, 40x48x3x32 402 -> 313 us, 58x59x3x48 787 -> 533, 128x40x3x16 390 -> 299, 93x129x3x16 778 -> 718;
  // 143x160x3x40 and 110x66x3x64 are the same (3790, 1613 us).
  if constexpr (sizeof(T) == 4) pdl_trigger();
  const int G = (P + 7) / 8, Q0 = ax.l0 / 4, Q = ax.lf / 4;
  for (int r0 = 0; r0 < G * Q; r0 += blockDim.x) {
    if (r0) {
      __syncthreads();
      mm_start<T>(buf, ax.ft, ax.lf, ax.h0);
    }
    const int it = r0 + threadIdx.x;
    const bool live = it < G * Q;
    const int gr = live ? it / Q : 0, u = live ? it - gr * Q : 0;
    const bool odd = u >= Q0;
    const int q0 = 4 * (odd ? u - Q0 : u), h = odd ? ax.h1 : ax.h0;
    T acc[8][4];
    mm_zero<T>(acc);
    mm_forward<T, 8>(acc, X + (odd ? (n1 - 1) * ld : 0) + 8 * gr, odd ? -ld : ld, 4 * u, ax, buf, live);
    if (!live) continue;
    T* dst = hat + rowbase + (size_t)(8 * gr) * S + (odd ? ax.h0 : 0) + q0;
#pragma unroll
    for (int r = 0; r < 8; ++r)
      if (8 * gr + r < P) {
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (q0 + e < h) dst[(size_t)r * S + e] = acc[r][e];
      }
  }
}

// Inverse pass of one (y, c) row per block.  Mt: the inverse time DCT [t][2][PM / 2], the weights of the even and the
// odd frequencies, t < (P + 1) / 2 padded to a multiple of 4.
template <typename T, int PM>
__global__ void __launch_bounds__(kMmXtThreads, sizeof(T) == 4 ? 2 : 1)
    k_mm_inv_xt(Geo<T> g, const T* __restrict__ hat, T* __restrict__ phi, MmAxis<T> ax, const T* __restrict__ Mtg) {
  constexpr int PH = PM / 2;
  extern __shared__ __align__(16) char smraw[];
  const int y = blockIdx.x, c = blockIdx.y, b = blockIdx.z;
  if (retired(g, b)) return;
  const int n1 = g.n1, P = g.P, ld = mm_ldt(P), hP = (P + 1) / 2, hP4 = (hP + 3) / 4 * 4;
  T* buf = (T*)smraw;        // table chunks
  T* X = buf + mm_buf(ax.l0, ax.lf, ax.li);   // [spectral x][t]
  T* Mt = X + n1 * ld;
  mm_start<T>(buf, ax.it, 2 * ax.li, ax.h0);
  for (int j = threadIdx.x; j < hP4 * PM; j += blockDim.x) Mt[j] = Mtg[j];
  __syncthreads();
  pdl_wait();   // the spectral array (y/colour pass) is read from here on
  const size_t S = g.S;
  const size_t rowbase = (size_t)b * P * S + (size_t)n1 * (y + (size_t)g.n2 * c);
  for (int x = threadIdx.x; x < n1; x += blockDim.x) {
    const T* src = hat + rowbase + x;
    T ve[PH], vo[PH];
#pragma unroll
    for (int j = 0; j < PH; ++j) {
      const T e = src[(size_t)min(2 * j, P - 1) * S], o = src[(size_t)min(2 * j + 1, P - 1) * S];
      ve[j] = 2 * j < P ? e : T(0);
      vo[j] = 2 * j + 1 < P ? o : T(0);
    }
    T* col = X + x * ld;
    for (int t = 0; t < hP; t += 4) {
      T lo[4], hi[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const T* row = Mt + (t + e) * PM;
        T E = T(0), O = T(0);
#pragma unroll
        for (int j = 0; j < PH; j += 4) {
          T m[4], w[4];
          ldv<T, 4>(row + j, m);
          ldv<T, 4>(row + PH + j, w);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            E = fma(m[q], ve[j + q], E);
            O = fma(w[q], vo[j + q], O);
          }
        }
        lo[e] = E + O;
        hi[3 - e] = E - O;
      }
      // samples t .. t + 3 and their mirrors; where both halves of an odd or short P reach the same sample, both
      // forms hold it
      stv<T, 4>(col + t, lo);
      if ((P & 3) == 0) {
        stv<T, 4>(col + P - 4 - t, hi);
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (t + e < hP) col[P - 1 - t - e] = hi[3 - e];
      }
    }
  }
  __syncthreads();
  if constexpr (sizeof(T) == 4) pdl_trigger();
  const int G = (P + 7) / 8, I = (ax.h0 + 1) / 2;
  for (int r0 = 0; r0 < G * I; r0 += blockDim.x) {
    if (r0) {
      __syncthreads();
      mm_start<T>(buf, ax.it, 2 * ax.li, ax.h0);
    }
    const int it = r0 + threadIdx.x;
    const bool live = it < G * I;
    const int gr = live ? it / I : 0, i0 = live ? 2 * (it - gr * I) : 0;
    T E[8][2], O[8][2];
    mm_zero<T>(E);
    mm_zero<T>(O);
    mm_inverse<T, 8>(E, O, X + 8 * gr, ld, i0, ax, buf, live);
    if (!live) continue;
    T* dst = phi + rowbase + (size_t)(8 * gr) * S;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int i = i0 + e;
      if (i >= ax.h0) continue;
      const int mi = ax.mirror(i);
#pragma unroll
      for (int r = 0; r < 8; ++r)
        if (8 * gr + r < P) {
          dst[(size_t)r * S + i] = E[r][e] + O[r][e];
          if (mi != i) dst[(size_t)r * S + mi] = E[r][e] - O[r][e];
        }
    }
  }
}

// y transform, colour solve, inverse y transform of a strip of W columns, one t-frequency per block.  A thread's rows
// in the products are all C channels of WT neighbouring columns.
template <int C> struct MmColour { static constexpr int WT = C == 1 ? 8 : (C == 4 ? 2 : 4), RT = C * WT; };
inline int mm_yc_wt(int C) { return C == 1 ? 8 : (C == 4 ? 2 : 4); }
inline int mm_yc_ld(int C, int W) { return (C * W + 7) / 8 * 8 + 4; }
constexpr int kMmYcThreads = 256;
template <typename T>
inline size_t mm_yc_smem(int n2, int C, int W, int buf) {
  return sizeof(T) * ((size_t)n2 * mm_yc_ld(C, W) + buf + n2 + W) + 8 + sizeof(double) * (n2 + W);
}
inline int mm_yc_items(int lf, int C, int W) { return (W / mm_yc_wt(C)) * (lf / 4); }

template <typename T, int C>
__global__ void __launch_bounds__(kMmYcThreads, sizeof(T) == 4 ? 2 : 1) k_mm_yc(Geo<T> g, T* __restrict__ hat, YcTables tb, MmAxis<T> ay, int W) {
  constexpr int WT = MmColour<C>::WT, RT = MmColour<C>::RT;
  extern __shared__ __align__(16) char smraw[];
  const int x0 = blockIdx.x * W, kt = blockIdx.y, b = blockIdx.z;
  if (retired(g, b)) return;
  const int n1 = g.n1, n2 = g.n2, ld = (C * W + 7) / 8 * 8 + 4, NW = W / WT;
  const int w_act = min(W, n1 - x0);
  T* buf = (T*)smraw;        // table chunks
  T* X = buf + mm_buf(ay.l0, ay.lf, ay.li);   // [y][wg][c][wi]
  mm_start<T>(buf, ay.ft, ay.lf, ay.h0);
  T Q[C][C], lc[C];
#pragma unroll
  for (int c = 0; c < C; ++c) {
    lc[c] = ((const T*)tb.lamc)[c];
#pragma unroll
    for (int j = 0; j < C; ++j) Q[c][j] = ((const T*)tb.Qc)[c * C + j];
  }
  const T lt = ((const T*)tb.lamt)[kt];
  const double ltd = tb.lamtd[kt];
  T* l2 = X + n2 * ld;       // eigenvalues along y and x (the strip), also in double
  T* l1 = l2 + n2;
  double* l2d = (double*)(((uintptr_t)(l1 + W) + 7) & ~uintptr_t(7));
  double* l1d = l2d + n2;
  for (int j = threadIdx.x; j < n2; j += blockDim.x) {
    l2[j] = ((const T*)tb.lam2)[j];
    l2d[j] = tb.lam2d[j];
  }
  if ((int)threadIdx.x < W) {
    l1[threadIdx.x] = ((const T*)tb.lam1)[min(x0 + (int)threadIdx.x, n1 - 1)];
    l1d[threadIdx.x] = tb.lam1d[min(x0 + (int)threadIdx.x, n1 - 1)];
  }
  pdl_wait();   // the spectral array (forward x/t pass) is read from here on
  const size_t plane = ((size_t)b * g.P + kt) * g.S + x0;
  constexpr int V = sizeof(T) == 4 ? 4 : 2;
  const bool vec = WT % V == 0 && w_act == W && n1 % V == 0 && x0 % V == 0 && ((uintptr_t)hat & 15) == 0;
  if (vec) {
    const int per = W / V;
    for (int it = threadIdx.x; it < C * n2 * per; it += blockDim.x) {
      const int r = it / per, w = V * (it - r * per);   // r = c * n2 + y
      const int c = r / n2, yy = r - c * n2;
      cp_async16(X + yy * ld + (w / WT) * RT + c * WT + w % WT, hat + plane + (size_t)r * n1 + w);
    }
  } else {
    for (int it = threadIdx.x; it < C * n2 * W; it += blockDim.x) {
      const int r = it / W, w = it - r * W;
      const int c = r / n2, yy = r - c * n2;
      T* dst = X + yy * ld + (w / WT) * RT + c * WT + w % WT;
      if (w < w_act) cp_async_small<sizeof(T)>(dst, hat + plane + (size_t)r * n1 + w);
      else *dst = T(0);
    }
  }
  cp_async_wait_all();
  __syncthreads();
  mm_fold<T>(X, ld, NW * RT / 4, ay);
  __syncthreads();
  // forward: at most one item per thread (the launch has that many), kept over the barrier
  const int Q0 = ay.l0 / 4, Qn = ay.lf / 4;
  const bool live = (int)threadIdx.x < NW * Qn;
  const int wg = live ? threadIdx.x / Qn : 0, u = live ? threadIdx.x - wg * Qn : 0;
  const bool odd = u >= Q0;
  const int q0 = 4 * (odd ? u - Q0 : u), h = odd ? ay.h1 : ay.h0, pos = (odd ? ay.h0 : 0) + q0;
  T acc[RT][4];
  mm_zero<T>(acc);
  mm_forward<T, RT>(acc, X + (odd ? (n2 - 1) * ld : 0) + wg * RT, odd ? -ld : ld, 4 * u, ay, buf, live);
  __syncthreads();   // every thread is done with the folded rows: the spectrum takes their place
  mm_start<T>(buf, ay.it, 2 * ay.li, ay.h0);
  if (live) {
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (q0 + e < h) {
        T v[RT];
#pragma unroll
        for (int r = 0; r < RT; ++r) v[r] = acc[r][e];
        stv<T, RT>(X + (pos + e) * ld + wg * RT, v);
      }
  }
  __syncthreads();
  // colour eigen-solve: phi_c = sum_j Q[c][j] (sum_c' Q[c'][j] r_c') / lambda(kx, ky, j, kt)
  {
    const float thr = (float)tb.lam_fp64;
    for (int it = threadIdx.x; it < n2 * W; it += blockDim.x) {
      const int ky = it / W, w = it - ky * W;
      if (w >= w_act) continue;
      T* p = X + ky * ld + (w / WT) * RT + w % WT;
      T r[C], co[C];
#pragma unroll
      for (int cc = 0; cc < C; ++cc) r[cc] = p[cc * WT];
      const T lxyt = l1[w] + l2[ky] + lt;
#pragma unroll
      for (int j = 0; j < C; ++j) {
        T s = 0;
#pragma unroll
        for (int cc = 0; cc < C; ++cc) s = fma(Q[cc][j], r[cc], s);
        const T lam = lxyt + lc[j];
        if (!(lam > T(0))) {
          co[j] = T(0);     // the zero eigenvalue of the pseudo-inverse
        } else if ((float)lam < thr) {
          // low modes: eigenvalue and quotient in double precision
          const double ld_ = l1d[w] + l2d[ky] + ltd + tb.lamcd[j];
          co[j] = ld_ > 0.0 ? (T)quot_low((double)s, ld_) : T(0);
        } else {
          co[j] = fdiv_fast(s, lam);
        }
      }
#pragma unroll
      for (int cc = 0; cc < C; ++cc) {
        T s = 0;
#pragma unroll
        for (int j = 0; j < C; ++j) s = fma(Q[cc][j], co[j], s);
        p[cc * WT] = s;
      }
    }
  }
  __syncthreads();
  if constexpr (sizeof(T) == 4) pdl_trigger();
  const int I = (ay.h0 + 1) / 2;
  for (int r0 = 0; r0 < NW * I; r0 += blockDim.x) {
    if (r0) {
      __syncthreads();
      mm_start<T>(buf, ay.it, 2 * ay.li, ay.h0);
    }
    const int it = r0 + threadIdx.x;
    const bool work = it < NW * I;
    const int wv = work ? it / I : 0, i0 = work ? 2 * (it - wv * I) : 0;
    T E[RT][2], O[RT][2];
    mm_zero<T>(E);
    mm_zero<T>(O);
    mm_inverse<T, RT>(E, O, X + wv * RT, ld, i0, ay, buf, work);
    if (!work) continue;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int i = i0 + e;
      if (i >= ay.h0) continue;
      const int mi = ay.mirror(i);
#pragma unroll
      for (int c = 0; c < C; ++c) {
        T* p = hat + plane + ((size_t)c * n2 + i) * n1 + wv * WT;
        T* pm = hat + plane + ((size_t)c * n2 + mi) * n1 + wv * WT;
        T lo[WT], hi[WT];
#pragma unroll
        for (int w = 0; w < WT; ++w) {
          lo[w] = E[c * WT + w][e] + O[c * WT + w][e];
          hi[w] = E[c * WT + w][e] - O[c * WT + w][e];
        }
        bool done = false;
        if constexpr (WT % V == 0) {
          if (vec) {
            stv<T, WT>(p, lo);
            if (mi != i) stv<T, WT>(pm, hi);
            done = true;
          }
        }
        if (!done) {
#pragma unroll
          for (int w = 0; w < WT; ++w)
            if (wv * WT + w < w_act) {
              p[w] = lo[w];
              if (mi != i) pm[w] = hi[w];
            }
        }
      }
    }
  }
}

}  // namespace dynot
