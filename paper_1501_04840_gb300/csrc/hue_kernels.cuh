// Poisson solve of the hue variant (section 5): one periodic axis of n bins and
// P time intervals, A A^T = n^2 Delta_{n,per} (x) I + p^2 Delta_p (x) I
// (section 3, the derivation case of the paper).
//
// Along the periodic axis the DFT diagonalises Delta_{n,per} with eigenvalues
// 4 sin^2(pi j / n), equal for j and n - j.  The pseudo-inverse therefore only
// needs the real Fourier basis (cos and sin pairs), which keeps everything real:
//   slot 0 = sum r_i, slots 2j-1, 2j = sum r_i cos, sum r_i sin (2 pi i j / n),
//   slot n-1 = sum r_i (-1)^i for even n.
// The time axis uses the DCT-II as on the RGB path.
//
//   H_A  hue_fwd  : r = A a - f_b^- and the forward real DFT, per time row.
//   H_B  hue_t    : forward DCT along t, divide, inverse DCT, per slot column.
//   H_C  hue_inv  : inverse real DFT -> phi, per time row.
// The cell update is the shared kernel K_D with n2 = C = 1.
#pragma once
#include "common.cuh"
#include "mm_kernels.cuh"
#include "rgb_kernels.cuh"

namespace dynot {

struct HueTables {
  const void* cs;      // c2<T>[n]: (cos, sin)(2 pi m / n)
  const void* lam;     // T[n] eigenvalue of each slot
  const double* lamd;
  const void* lamt;    // T[P]
  const double* lamtd;
  const void* Mt_f;    // [P][PMAX]
  const void* Mt_i;
  double lam_fp64;
};

template <typename T>
__device__ __forceinline__ T hue_basis(const c2<T>* cs, int n, int slot, int i) {
  if (slot == 0) return T(1);
  if ((n & 1) == 0 && slot == n - 1) return (i & 1) ? T(-1) : T(1);
  const int j = (slot + 1) >> 1;
  const c2<T> w = cs[(int)(((long long)i * j) % n)];
  return (slot & 1) ? w.x : w.y;
}

template <typename T>
__global__ void __launch_bounds__(256) k_hue_fwd(Geo<T> g, const v4<T>* __restrict__ ap, const T* __restrict__ f0,
                                                 const T* __restrict__ f1, T* __restrict__ hat, HueTables tb) {
  extern __shared__ __align__(16) char smraw[];
  const int t = blockIdx.x, b = blockIdx.y;
  if (retired(g, b)) return;
  const int n = g.n1, P = g.P;
  T* row = (T*)smraw;
  c2<T>* cs = (c2<T>*)(smraw + ((sizeof(T) * n + 15) & ~size_t(15)));
  for (int m = threadIdx.x; m < n; m += blockDim.x) cs[m] = ((const c2<T>*)tb.cs)[m];
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const int im = i > 0 ? i - 1 : n - 1;  // periodic
    const size_t i0 = (size_t)(b * P + t) * n + i;
    const v4<T> av = ap[i0];
    T r = g.s1 * (av.x - comp<T>(ap, (size_t)(b * P + t) * n + im, 0));
    const T fnext = (t == P - 1) ? f1[(size_t)b * n + i] : av.w;
    const T fprev = (t == 0) ? f0[(size_t)b * n + i] : comp<T>(ap, i0 - n, 3);
    r += g.sp * (fnext - fprev);
    row[i] = r;
  }
  __syncthreads();
  for (int slot = threadIdx.x; slot < n; slot += blockDim.x) {
    // four interleaved partial sums: shorter rounding chains and independent FMAs.  The basis
    // index (i j) mod n of the cos / sin slots advances by 4 j per step instead of a modulo per term.
    T acc[4] = {0, 0, 0, 0};
    int i = 0;
    if (slot == 0 || ((n & 1) == 0 && slot == n - 1)) {
      // the constant slot and, for even n, the alternating Nyquist slot
      const bool alt = slot != 0;
      for (; i + 3 < n; i += 4) {
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] = fma(row[i + q], (alt && ((i + q) & 1)) ? T(-1) : T(1), acc[q]);
      }
    } else {
      const bool use_cos = slot & 1;
      const int j = (slot + 1) >> 1;
      int idx[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) idx[q] = (int)(((long long)q * j) % n);
      const int step = (int)((4LL * j) % n);
      for (; i + 3 < n; i += 4) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const c2<T> w = cs[idx[q]];
          acc[q] = fma(row[i + q], use_cos ? w.x : w.y, acc[q]);
          idx[q] += step;
          if (idx[q] >= n) idx[q] -= n;
        }
      }
    }
    for (; i < n; ++i) acc[0] = fma(row[i], hue_basis<T>(cs, n, slot, i), acc[0]);
    hat[(size_t)(b * P + t) * n + slot] = (acc[0] + acc[1]) + (acc[2] + acc[3]);
  }
}

// Shared memory of k_hue_t: the two DCT matrices with padded rows, and one column per slot of the
// input and of the divided spectrum.
template <typename T, int PMAX>
__host__ __device__ constexpr size_t hue_t_smem() {
  return sizeof(T) * (2 * (size_t)PMAX * (PMAX + 1) + 2 * (size_t)(256 / PMAX) * PMAX);
}
template <typename T>
__host__ __device__ inline size_t hue_t_smem_for(int pmax) {
  return pmax == 16 ? hue_t_smem<T, 16>() : (pmax == 32 ? hue_t_smem<T, 32>() : hue_t_smem<T, 64>());
}

// 256 threads = 256 / PMAX slot columns x PMAX time indices: thread (slot, k) forms the k-th DCT
// coefficient of its column and divides it, then (after a barrier) the k-th time sample of the inverse.
template <typename T, int PMAX>
__global__ void __launch_bounds__(256) k_hue_t(Geo<T> g, T* __restrict__ hat, HueTables tb) {
  extern __shared__ __align__(16) char smraw[];
  constexpr int SL = 256 / PMAX, LD = PMAX + 1;
  const int P = g.P, n = g.n1, b = blockIdx.y;
  if (retired(g, b)) return;
  T* Mf = (T*)smraw;            // [k][t], row stride LD
  T* Mi = Mf + PMAX * LD;       // [t][k]
  T* v = Mi + PMAX * LD;        // [SL][PMAX] input columns
  T* w = v + SL * PMAX;         // [SL][PMAX] divided spectra
  for (int j = threadIdx.x; j < P * PMAX; j += blockDim.x) {
    const int r = j / PMAX, c = j - r * PMAX;
    Mf[r * LD + c] = ((const T*)tb.Mt_f)[j];
    Mi[r * LD + c] = ((const T*)tb.Mt_i)[j];
  }
  const int sl = threadIdx.x / PMAX, k = threadIdx.x - sl * PMAX;
  const int slot = blockIdx.x * SL + sl;
  const bool act = slot < n && k < P;
  v[sl * PMAX + k] = act ? hat[(size_t)(b * P + k) * n + slot] : T(0);
  __syncthreads();
  T acc = 0;
  if (act) {
#pragma unroll 16
    for (int t = 0; t < PMAX; ++t) acc = fma(Mf[k * LD + t], v[sl * PMAX + t], acc);
    const T lam = ((const T*)tb.lam)[slot] + ((const T*)tb.lamt)[k];
    if (!(lam > T(0))) {
      acc = T(0);
    } else if ((double)lam < tb.lam_fp64) {
      acc = (T)((double)acc / (tb.lamd[slot] + tb.lamtd[k]));
    } else {
      acc = acc / lam;
    }
  }
  w[sl * PMAX + k] = act ? acc : T(0);
  __syncthreads();
  if (act) {
    T y = 0;
#pragma unroll 16
    for (int kk = 0; kk < PMAX; ++kk) y = fma(Mi[k * LD + kk], w[sl * PMAX + kk], y);
    hat[(size_t)(b * P + k) * n + slot] = y;
  }
}

template <typename T>
__global__ void __launch_bounds__(256) k_hue_inv(Geo<T> g, const T* __restrict__ hat, T* __restrict__ phi,
                                                 HueTables tb) {
  extern __shared__ __align__(16) char smraw[];
  const int t = blockIdx.x, b = blockIdx.y;
  if (retired(g, b)) return;
  const int n = g.n1, P = g.P;
  T* row = (T*)smraw;
  c2<T>* cs = (c2<T>*)(smraw + ((sizeof(T) * n + 15) & ~size_t(15)));
  for (int m = threadIdx.x; m < n; m += blockDim.x) cs[m] = ((const c2<T>*)tb.cs)[m];
  for (int i = threadIdx.x; i < n; i += blockDim.x) row[i] = hat[(size_t)(b * P + t) * n + i];
  __syncthreads();
  const T invn = T(1) / T(n);
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    // slots 1..n-1 carry weight 2 except the Nyquist slot of even n (weight 1)
    T acc[4] = {0, 0, 0, 0};
    const int last = (n & 1) ? n : n - 1;
    int slot = 1;
    // slots s, s+1 (cos, sin of frequency j) and s+2, s+3 (frequency j+1) for odd s: the basis
    // indices i j and i (j+1) mod n advance by 2 i per step of 4 slots
    int ia = i % n, ib = (int)((2LL * i) % n);
    const int step = (int)((2LL * i) % n);
    for (; slot + 3 < last; slot += 4) {
      const c2<T> wa = cs[ia], wb = cs[ib];
      acc[0] = fma(row[slot], wa.x, acc[0]);
      acc[1] = fma(row[slot + 1], wa.y, acc[1]);
      acc[2] = fma(row[slot + 2], wb.x, acc[2]);
      acc[3] = fma(row[slot + 3], wb.y, acc[3]);
      ia += step;
      if (ia >= n) ia -= n;
      ib += step;
      if (ib >= n) ib -= n;
    }
    for (; slot < last; ++slot) acc[0] = fma(row[slot], hue_basis<T>(cs, n, slot, i), acc[0]);
    T sum = T(2) * ((acc[0] + acc[1]) + (acc[2] + acc[3])) + row[0];
    if (!(n & 1)) sum += row[n - 1] * hue_basis<T>(cs, n, n - 1, i);
    phi[(size_t)(b * P + t) * n + i] = sum * invn;
  }
}

// ---------------------------------------------------------------------------
// The same solve by folded products (mm_kernels.cuh), for bins whose rows fit shared memory:
//   k_hue_x_fwd : r of a group of time rows and their folded bins in shared memory, then the real DFT, 8 rows x 4
//                 slots per thread;
//   k_hue_tt    : the time DCT of SC slot columns, the divide, the inverse DCT;
//   k_hue_x_inv : the inverse real DFT -> phi, 8 rows x 2 mirrored pairs per thread.
// SMALL (few rows, a single pair) is bound by latency: blocks of 8 rows x 64 outputs whose table columns are copied
// while the previous kernel runs, every sum in 16 slices of at most n / 32 steps.  Otherwise the FP32 pipe and the
// instructions around it bound: 16 or 8 rows x all outputs or some per block, tables in chunks of K = 8 or 16 steps, sums
// in runs of 16 terms (which keep the rounding error of 16 + n / 32 additions).  plan.cuh (choose_hue_mm) picks.
// ---------------------------------------------------------------------------
constexpr int kHueMmThreads = 256;
constexpr int kHueSlices = 16, kHueItems = 16;   // SMALL: slices of a sum, items (64 table columns) per block

// Rows of X before and after the bins, so that whole steps of 16 stay inside: their table weights are zero.
__host__ __device__ inline int hue_hpad(int h0) { return (h0 + 15) / 16 * 16; }
__host__ __device__ inline int hue_xpad(int n, int h0) { return hue_hpad(h0) > n ? hue_hpad(h0) - n : 0; }
inline size_t hue_mm_vals(int n, int h0, int rb, int items, bool small, int K = kMmK) {
  const size_t x = (size_t)(n + 2 * hue_xpad(n, h0)) * (rb + 4);
  const size_t tab = (size_t)hue_hpad(h0) * 4 * kHueItems, red = (size_t)kHueSlices * 32 * kHueItems;
  return x + (small ? (tab > red ? tab : red) : (size_t)kMmStages * K * 4 * items);
}

// Copies of `width` columns of a table (row stride ld) in chunks of K rows into slots of row stride ldb.  The place of a
// thread's first vector and the step between its vectors are found once (a division per vector and chunk took a
// quarter of the kernel's instructions).
template <typename T, int K>
struct HueChunks {
  const T* tab;
  T* buf;
  int ld, ldb, per, r, k, dr, dk, hpad;
  static constexpr int V = 16 / (int)sizeof(T);
  __device__ __forceinline__ HueChunks(T* buf_, const T* tab_, int ld_, int width, int ldb_, int hpad_)
      : tab(tab_), buf(buf_), ld(ld_), ldb(ldb_), per(width / V), hpad(hpad_) {
    r = threadIdx.x / per;
    k = threadIdx.x - r * per;
    dr = blockDim.x / per;
    dk = blockDim.x - dr * per;
  }
  __device__ __forceinline__ void issue(int c) const {
    if (c * K >= hpad) return;
    T* dst = buf + (c % kMmStages) * K * ldb;
    const T* src = tab + (size_t)c * K * ld;
    for (int i = r, j = k; i < K;) {
      cp_async16(dst + i * ldb + V * j, src + i * ld + V * j);
      i += dr;
      j += dk;
      if (j >= per) {
        j -= per;
        ++i;
      }
    }
  }
};
__device__ __forceinline__ void hue_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
// SMALL: `quads` (at most 16) groups of 4 columns of every row
template <typename T>
__device__ __forceinline__ void hue_columns(T* buf, const T* tab, int ld, int quads, int ldb, int hpad) {
  const int k = threadIdx.x % 16;
  if (k < quads)
    for (int r = threadIdx.x / 16; r < hpad; r += blockDim.x / 16)
#pragma unroll
      for (int v = 0; v < (int)sizeof(T) / 4; ++v)
        cp_async16(buf + r * ldb + 4 * k + v * 16 / (int)sizeof(T), tab + (size_t)r * ld + 4 * k + v * 16 / (int)sizeof(T));
}
template <typename T>
__device__ __forceinline__ void hue_zero_pads(T* X, int n, int pad, int ld) {
  for (int i = threadIdx.x; i < pad * ld; i += blockDim.x) {
    X[i - pad * ld] = T(0);
    X[n * ld + i] = T(0);
  }
}
// visit the cells (row r, bin x) of a rows x n plane, consecutive threads along x; f(index, r, x)
template <int U, class F>
__device__ __forceinline__ void hue_cells(int rows, int n, F&& f) {
  const int nt = blockDim.x, dr = nt / n, dx = nt - dr * n, tot = rows * n;
  int r = threadIdx.x / n, x = threadIdx.x - r * n;
  for (int i0 = threadIdx.x; i0 < tot; i0 += U * nt) {
    int rr[U], xx[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      rr[u] = r;
      xx[u] = x;
      r += dr;
      x += dx;
      if (x >= n) {
        x -= n;
        ++r;
      }
    }
    f(i0, rr, xx, tot);
  }
}

template <typename T, bool SMALL, int K>
__global__ void __launch_bounds__(kHueMmThreads, sizeof(T) == 4 ? 2 : 1)
    k_hue_x_fwd(Geo<T> g, const v4<T>* __restrict__ ap, const T* __restrict__ f0, const T* __restrict__ f1,
                T* __restrict__ hat, MmAxis<T> ax, int RB, int QC) {
  extern __shared__ __align__(16) char smraw[];
  const int b = blockIdx.z, t0 = blockIdx.x * RB, u0 = blockIdx.y * QC;
  if (retired(g, b)) return;
  const int n = g.n1, P = g.P, ld = RB + 4, Q = ax.lf / 4, qn = min(QC, Q - u0), rows = min(RB, P - t0);
  const int hpad = hue_hpad(ax.h0), pad = hue_xpad(n, ax.h0);
  T* X = (T*)smraw + pad * ld;
  T* buf = X + (n + pad) * ld;
  const T* tab = ax.ft + 4 * u0;
  const HueChunks<T, K> chunks(buf, tab, ax.lf, 4 * qn, 4 * QC, hpad);
  if (SMALL) {
    hue_columns<T>(buf, tab, ax.lf, qn, 4 * kHueItems, hpad);
  } else {
    chunks.issue(0);
    hue_commit();
    chunks.issue(1);
    hue_commit();
  }
  hue_zero_pads<T>(X, n, pad, ld);
  pdl_wait();   // a (previous update) is read from here on
  {
    constexpr int U = 4;
    const v4<T>* pc = ap + (size_t)(b * P + t0) * n;
    const T* as = reinterpret_cast<const T*>(pc);
    const T *pf0 = f0 + (size_t)b * n, *pf1 = f1 + (size_t)b * n;
    hue_cells<U>(rows, n, [&](int i0, const int (&rr)[U], const int (&xx)[U], int tot) {
      v4<T> av[U];
      T lx[U], lf[U], uf[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int i = i0 + u * (int)blockDim.x;
        if (i < tot) {
          const int t = t0 + rr[u];
          av[u] = pc[i];
          lx[u] = as[4 * (xx[u] > 0 ? i - 1 : i + n - 1)];
          lf[u] = t > 0 ? as[4 * (i - n) + 3] : pf0[xx[u]];
          uf[u] = t < P - 1 ? av[u].w : pf1[xx[u]];
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (i0 + u * (int)blockDim.x < tot)
          X[xx[u] * ld + rr[u]] = g.s1 * (av[u].x - lx[u]) + g.sp * (uf[u] - lf[u]);
    });
  }
  __syncthreads();
  mm_fold<T>(X, ld, (rows + 3) / 4, ax);
  T* dst = hat + (size_t)(b * P + t0) * n;
  if (SMALL) {
    cp_async_wait_all();
    __syncthreads();
    const int ks = threadIdx.x / kHueItems, u = threadIdx.x % kHueItems;
    const bool odd = 4 * (u0 + u) >= ax.l0;
    const T* row = X + (odd ? (n - 1 - ks) * ld : ks * ld);
    const int stride = (odd ? -ld : ld) * kHueSlices;
    const T* tc = buf + ks * 4 * kHueItems + 4 * u;
    T acc[32];
#pragma unroll
    for (int q = 0; q < 32; ++q) acc[q] = T(0);
#pragma unroll 4
    for (int i = 0; i < hpad; i += kHueSlices) {
      T v[8], m[4];
      ldv<T, 8>(row, v);
      ldv<T, 4>(tc, m);
      row += stride;
      tc += kHueSlices * 4 * kHueItems;
#pragma unroll
      for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[4 * r + e] = fma(v[r], m[e], acc[4 * r + e]);
    }
    __syncthreads();   // the table's place takes the slices
#pragma unroll
    for (int q = 0; q < 32; ++q) buf[(ks * 32 + q) * kHueItems + u] = acc[q];
    __syncthreads();
    pdl_trigger();
    for (int o = threadIdx.x; o < 8 * 4 * kHueItems; o += blockDim.x) {
      const int e = o & 3, uo = (o >> 2) % kHueItems, r = o / (4 * kHueItems);
      const bool od = 4 * (u0 + uo) >= ax.l0;
      const int q = 4 * (u0 + uo) - (od ? ax.l0 : 0) + e;
      if (uo >= qn || r >= rows || q >= (od ? ax.h1 : ax.h0)) continue;
      T sum = T(0);
#pragma unroll
      for (int k = 0; k < kHueSlices; ++k) sum += buf[(k * 32 + 4 * r + e) * kHueItems + uo];
      dst[(size_t)r * n + (od ? ax.h0 : 0) + q] = sum;
    }
    return;
  }
  const int rg = threadIdx.x / QC, u = threadIdx.x - rg * QC;
  const bool live = u < qn && 8 * rg < rows;
  const bool odd = 4 * (u0 + u) >= ax.l0;
  const int stride = odd ? -ld : ld;
  const T* row = X + (odd ? (n - 1) * ld : 0) + 8 * rg;
  T acc[8][4], part[8][4];
  mm_zero<T>(acc);
  mm_zero<T>(part);
#pragma unroll 1
  for (int c = 0; c * K < hpad; ++c) {
    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    __syncthreads();   // chunk c is there (and, at first, the folded rows), and every thread is done with chunk c - 1
    chunks.issue(c + 2);
    hue_commit();
    if (!live) continue;
    const T* tc = buf + (c % kMmStages) * K * 4 * QC + 4 * u;
#pragma unroll
    for (int j = 0; j < K; ++j) {
      T v[8], m[4];
      ldv<T, 8>(row, v);
      ldv<T, 4>(tc, m);
      row += stride;
      tc += 4 * QC;
#pragma unroll
      for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int e = 0; e < 4; ++e) part[r][e] = fma(v[r], m[e], part[r][e]);
    }
    if (K == 16 || (c & 1)) {   // 16 terms
#pragma unroll
      for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          acc[r][e] += part[r][e];
          part[r][e] = T(0);
        }
    }
  }
  pdl_trigger();
  if (!live) return;
  const int q0 = 4 * (u0 + u) - (odd ? ax.l0 : 0), h = odd ? ax.h1 : ax.h0;
  dst += (size_t)(8 * rg) * n + (odd ? ax.h0 : 0) + q0;
#pragma unroll
  for (int r = 0; r < 8; ++r)
    if (8 * rg + r < rows) {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (q0 + e < h) dst[(size_t)r * n + e] = acc[r][e];
    }
}

template <typename T, bool SMALL, int K>
__global__ void __launch_bounds__(kHueMmThreads, sizeof(T) == 4 ? 2 : 1)
    k_hue_x_inv(Geo<T> g, const T* __restrict__ hat, T* __restrict__ phi, MmAxis<T> ax, int RB, int IC) {
  extern __shared__ __align__(16) char smraw[];
  const int b = blockIdx.z, t0 = blockIdx.x * RB, i00 = 2 * blockIdx.y * IC;   // IC even: table columns in whole vectors
  if (retired(g, b)) return;
  const int n = g.n1, P = g.P, ld = RB + 4, rows = min(RB, P - t0), wid = min(2 * IC, ax.li - i00);
  const int hpad = hue_hpad(ax.h0), pad = hue_xpad(n, ax.h0);
  T* X = (T*)smraw + pad * ld;   // [slot][t]
  T* buf = X + (n + pad) * ld;
  const HueChunks<T, K> ce(buf, ax.it + i00, 2 * ax.li, wid, 4 * IC, hpad);
  const HueChunks<T, K> co(buf + 2 * IC, ax.it + ax.li + i00, 2 * ax.li, wid, 4 * IC, hpad);
  auto issue = [&](int c) {
    ce.issue(c);
    co.issue(c);
    hue_commit();
  };
  if (SMALL) {
    hue_columns<T>(buf, ax.it + i00, 2 * ax.li, wid / 4, 4 * kHueItems, hpad);
    hue_columns<T>(buf + 2 * kHueItems, ax.it + ax.li + i00, 2 * ax.li, wid / 4, 4 * kHueItems, hpad);
  } else {
    issue(0);
    issue(1);
  }
  hue_zero_pads<T>(X, n, pad, ld);
  pdl_wait();   // the spectral array (time transforms) is read from here on
  {
    constexpr int U = 8;
    const T* src = hat + (size_t)(b * P + t0) * n;
    hue_cells<U>(rows, n, [&](int i0, const int (&rr)[U], const int (&xx)[U], int tot) {
      T v[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (i0 + u * (int)blockDim.x < tot) v[u] = src[i0 + u * (int)blockDim.x];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (i0 + u * (int)blockDim.x < tot) X[xx[u] * ld + rr[u]] = v[u];
    });
  }
  T* dst = phi + (size_t)(b * P + t0) * n;
  // the steps past the odd part's rows read the pads or the even part's rows of other steps: zero weights
  const int oddlast = n + pad - 1;
  if (SMALL) {
    cp_async_wait_all();
    __syncthreads();
    const int ks = threadIdx.x / kHueItems, u = threadIdx.x % kHueItems;
    const T* tc = buf + ks * 4 * kHueItems + 2 * u;
    T acc[32];   // E and O of the pair's two samples: acc[4 r + 2 part + e]
#pragma unroll
    for (int q = 0; q < 32; ++q) acc[q] = T(0);
#pragma unroll 2
    for (int q = ks; q < hpad; q += kHueSlices) {
      T v[8], w[8], m[2], k[2];
      ldv<T, 8>(X + q * ld, v);
      ldv<T, 8>(X + min(ax.h0 + q, oddlast) * ld, w);
      ldv<T, 2>(tc, m);
      ldv<T, 2>(tc + 2 * kHueItems, k);
      tc += kHueSlices * 4 * kHueItems;
#pragma unroll
      for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          acc[4 * r + e] = fma(v[r], m[e], acc[4 * r + e]);
          acc[4 * r + 2 + e] = fma(w[r], k[e], acc[4 * r + 2 + e]);
        }
    }
    __syncthreads();   // the table's place takes the slices
#pragma unroll
    for (int q = 0; q < 32; ++q) buf[(ks * 32 + q) * kHueItems + u] = acc[q];
    __syncthreads();
    pdl_trigger();
    for (int o = threadIdx.x; o < 8 * 2 * kHueItems; o += blockDim.x) {
      const int e = o & 1, uo = (o >> 1) % kHueItems, r = o / (2 * kHueItems), i = i00 + 2 * uo + e;
      if (i >= ax.h0 || r >= rows) continue;
      T E = T(0), O = T(0);
#pragma unroll
      for (int k = 0; k < kHueSlices; ++k) {
        E += buf[(k * 32 + 4 * r + e) * kHueItems + uo];
        O += buf[(k * 32 + 4 * r + 2 + e) * kHueItems + uo];
      }
      const int mi = ax.mirror(i);
      dst[(size_t)r * n + i] = E + O;
      if (mi != i) dst[(size_t)r * n + mi] = E - O;
    }
    return;
  }
  const int rg = threadIdx.x / IC, u = threadIdx.x - rg * IC, i0 = i00 + 2 * u;
  const bool live = i0 < ax.h0 && 8 * rg < rows;
  const T* even = X + 8 * rg;
  T acc[8][4], part[8][4];   // E and O of the pair's two samples: [r][2 part + e]
  mm_zero<T>(acc);
  mm_zero<T>(part);
#pragma unroll 1
  for (int c = 0; c * K < hpad; ++c) {
    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    __syncthreads();
    issue(c + 2);
    if (!live) continue;
    const T* tc = buf + (c % kMmStages) * K * 4 * IC + 2 * u;
#pragma unroll
    for (int j = 0; j < K; ++j) {
      const int q = c * K + j;
      T v[8], m[2];
      ldv<T, 8>(even + q * ld, v);
      ldv<T, 2>(tc, m);
#pragma unroll
      for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int e = 0; e < 2; ++e) part[r][e] = fma(v[r], m[e], part[r][e]);
      ldv<T, 8>(even + min(ax.h0 + q, oddlast) * ld, v);
      ldv<T, 2>(tc + 2 * IC, m);
#pragma unroll
      for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int e = 0; e < 2; ++e) part[r][2 + e] = fma(v[r], m[e], part[r][2 + e]);
      tc += 4 * IC;
    }
    if (K == 16 || (c & 1)) {   // 16 terms
#pragma unroll
      for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          acc[r][e] += part[r][e];
          part[r][e] = T(0);
        }
    }
  }
  pdl_trigger();
  if (!live) return;
  dst += (size_t)(8 * rg) * n;
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int i = i0 + e;
    if (i >= ax.h0) continue;
    const int mi = ax.mirror(i);
#pragma unroll
    for (int r = 0; r < 8; ++r)
      if (8 * rg + r < rows) {
        dst[(size_t)r * n + i] = acc[r][e] + acc[r][2 + e];
        if (mi != i) dst[(size_t)r * n + mi] = acc[r][e] - acc[r][2 + e];
      }
  }
}

// Tables of k_hue_tt: tf [t < hP][P4] forward, te / to [j][h4] inverse weights of frequencies 2 j and 2 j + 1 at the
// samples t < hP; P4, h4 = P and hP = (P + 1) / 2 rounded up to whole vectors of 4, absent entries zero.
__host__ __device__ inline int hue_p4(int P) { return (P + 3) / 4 * 4; }
__host__ __device__ inline int hue_h4(int P) { return ((P + 1) / 2 + 3) / 4 * 4; }
inline size_t hue_tt_vals(int P, int SC) {
  const int hP = (P + 1) / 2;
  return (size_t)hP * hue_p4(P) + 2 * (size_t)hP * hue_h4(P) + 2 * (size_t)(hue_p4(P) + 2) * SC;
}
// SMALL: 8 slots per block, one slot and 2 frequencies (then 1 mirrored pair of samples) per thread; otherwise 32
// slots, 2 slots and 4 frequencies (2 pairs) per thread
template <bool SMALL> struct HueTt {
  static constexpr int SC = SMALL ? 8 : 32, ST = SMALL ? 1 : 2, KT = SMALL ? 2 : 4, TT = SMALL ? 1 : 2, LANES = SC / ST;
};
template <typename T, bool SMALL>
__global__ void __launch_bounds__(256) k_hue_tt(Geo<T> g, T* __restrict__ hat, HueTables tb, const T* __restrict__ tabs) {
  using L = HueTt<SMALL>;
  constexpr int SC = L::SC, ST = L::ST, KT = L::KT, TT = L::TT;
  extern __shared__ __align__(16) char smraw[];
  const int b = blockIdx.y, x0 = blockIdx.x * SC;
  if (retired(g, b)) return;
  const int n = g.n1, P = g.P, hP = (P + 1) / 2, P4 = hue_p4(P), h4 = hue_h4(P), act = min(SC, n - x0);
  T* tf = (T*)smraw;
  T* te = tf + hP * P4;
  T* to = te + hP * h4;
  T* V = to + hP * h4;       // [t][slot]: samples, then sums (t < hP) and differences (mirrored rows)
  T* Y = V + (P4 + 2) * SC;  // [k][slot], two rows more
  {
    constexpr int W = 16 / (int)sizeof(T);
    const int cnt = hP * P4 + 2 * hP * h4;
    for (int i = W * threadIdx.x; i < cnt; i += W * blockDim.x) cp_async16(tf + i, tabs + i);
  }
  for (int i = threadIdx.x; i < 2 * SC; i += blockDim.x) Y[P * SC + i] = T(0);   // read with zero weights
  const int xs = threadIdx.x % L::LANES * ST, lane0 = threadIdx.x / L::LANES, lanes = blockDim.x / L::LANES;
  pdl_wait();   // the spectral array (bin transform) is read from here on
  T* base = hat + (size_t)b * P * n + x0;
  {
    // mirrored samples folded on the way in
    const int x = threadIdx.x % SC;
#pragma unroll 4
    for (int t = threadIdx.x / SC; t < hP; t += blockDim.x / SC) {
      const T lo = x < act ? base[(size_t)t * n + x] : T(0), hi = x < act ? base[(size_t)(P - 1 - t) * n + x] : T(0);
      const bool mid = 2 * t == P - 1;
      V[(P - 1 - t) * SC + x] = mid ? lo : lo - hi;
      if (!mid) V[t * SC + x] = lo + hi;
    }
  }
  cp_async_wait_all();
  __syncthreads();
  for (int k0 = KT * lane0; k0 < P; k0 += KT * lanes) {
    T acc[KT][ST];
    mm_zero<T, KT, ST>(acc);
    const T *ps = V + xs, *pd = V + (P - 1) * SC + xs, *pm = tf + k0;
#pragma unroll 8
    for (int t = 0; t < hP; ++t) {
      T m[KT];
      ldv<T, KT>(pm, m);
#pragma unroll
      for (int q = 0; q < ST; ++q) {
        const T s = ps[q], d = pd[q];   // the middle row of odd P meets zero weights of the odd frequencies
#pragma unroll
        for (int e = 0; e < KT; ++e) acc[e][q] = fma(m[e], e & 1 ? d : s, acc[e][q]);
      }
      ps += SC;
      pd -= SC;
      pm += P4;
    }
#pragma unroll
    for (int e = 0; e < KT; ++e) {
      const int k = k0 + e;
      if (k >= P) continue;
#pragma unroll
      for (int q = 0; q < ST; ++q) {
        const int slot = min(x0 + xs + q, n - 1);
        T v = acc[e][q];
        const T lam = ((const T*)tb.lam)[slot] + ((const T*)tb.lamt)[k];
        if (!(lam > T(0))) v = T(0);
        else if ((double)lam < tb.lam_fp64) v = (T)((double)v / (tb.lamd[slot] + tb.lamtd[k]));
        else v = v / lam;
        Y[k * SC + xs + q] = v;
      }
    }
  }
  __syncthreads();
  pdl_trigger();
  for (int t0 = TT * lane0; t0 < hP; t0 += TT * lanes) {
    T E[TT][ST], O[TT][ST];
    mm_zero<T, TT, ST>(E);
    mm_zero<T, TT, ST>(O);
    const T *py = Y + xs, *pe = te + t0, *po = to + t0;
#pragma unroll 8
    for (int j = 0; j < hP; ++j) {
#pragma unroll
      for (int q = 0; q < ST; ++q) {
        const T a = py[q], c = py[SC + q];
#pragma unroll
        for (int e = 0; e < TT; ++e) {
          E[e][q] = fma(pe[e], a, E[e][q]);
          O[e][q] = fma(po[e], c, O[e][q]);
        }
      }
      py += 2 * SC;
      pe += h4;
      po += h4;
    }
#pragma unroll
    for (int e = 0; e < TT; ++e) {
      const int t = t0 + e;
      if (t >= hP) continue;
#pragma unroll
      for (int q = 0; q < ST; ++q)
        if (xs + q < act) {
          base[(size_t)t * n + xs + q] = E[e][q] + O[e][q];
          if (t != P - 1 - t) base[(size_t)(P - 1 - t) * n + xs + q] = E[e][q] - O[e][q];
        }
    }
  }
}

}  // namespace dynot
