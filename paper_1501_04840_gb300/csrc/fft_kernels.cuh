// The Poisson solve's transforms on FFT lengths (FP32): the DCT engine of fft.cuh with its passes fused.
//
// Two real rows a, b travel as one complex sequence.  With Z its DFT (Makhoul order on a Neumann axis),
// V_a = (Z_k + conj Z_{N-k}) / 2 and V_b = (Z_k - conj Z_{N-k}) / (2i), the products q = exp(-i pi k / 2N) V hold two
// coefficients each, X_k = Re q and X_{N-k} = -Im q; backwards V = exp(+i pi k / 2N) (X_k - i X_{N-k}).  So whatever
// works on single coefficients (the colour solve and divide, the time transform) takes them from Z_k and Z_{N-k} and
// leaves the spectrum of the inverse in their place: the packed spectra are never unpacked to rows in memory.  A
// periodic axis keeps natural order and q = V (cosine and sine sums of one frequency).
//
// The DFT of length N = M1 M2 is Bailey's split with n = M2 n1 + n2, k = k1 + M1 k2: M1-point DFTs over n1 for every n2,
// twiddles, M2-point DFTs over n2 for every k1, in place (the M2 values of a k1 stay with its thread).  The inverse runs
// the same steps backwards: M2-point DFTs over k2, twiddles, M1-point DFTs over k1.
//
// Against the row-based passes of rgb_kernels.cuh (which unpacked every spectrum to rows and back), per launch from
// events on one GB300: 256x256x3, P = 32: y/colour 46.8 -> 28.1 us, inverse x/t 32.8 -> 20.5, forward x/t 58.8 -> 41.4;
// 512x512x3, P = 64 (whose time transform was a dense product): 432 -> 217, 587 -> 147, 886 -> 284 us; 128x128x3, P = 32:
// 21.4 -> 16.1, 14.3 -> 10.1, 21.7 -> 15.1 us.  Shared-memory accesses fall to about a third; the y/colour pass is left
// with issue and the barriers of its five passes, the forward x/t pass with the L2 traffic of forming r (a 16-byte
// cell and two neighbours' cells for 4 bytes of each).
#pragma once
#include <algorithm>
#include <type_traits>

#include "rgb_kernels.cuh"

namespace dynot {

// exp(-2 pi i j / R) for R dividing 32 or 12, folded at compile time
__host__ __device__ constexpr double cos32(int j) {   // cos(2 pi j / 32)
  j &= 31;
  if (j > 16) j = 32 - j;
  const double s = j > 8 ? -1.0 : 1.0;
  const int i = j > 8 ? 16 - j : j;
  switch (i) {
    case 0: return s;
    case 1: return s * 0.98078528040323044913;
    case 2: return s * 0.92387953251128675613;
    case 3: return s * 0.83146961230254523708;
    case 4: return s * 0.70710678118654752440;
    case 5: return s * 0.55557023301960222474;
    case 6: return s * 0.38268343236508977173;
    case 7: return s * 0.19509032201612826785;
    default: return 0.0;
  }
}
__host__ __device__ constexpr double cos12(int j) {   // cos(2 pi j / 12)
  j %= 12;
  if (j > 6) j = 12 - j;
  const double s = j > 3 ? -1.0 : 1.0;
  switch (j > 3 ? 6 - j : j) {
    case 0: return s;
    case 1: return s * 0.86602540378443864676;
    case 2: return s * 0.5;
    default: return 0.0;
  }
}
template <typename T, int R>
__device__ __forceinline__ c2<T> root(int j) {
  if constexpr (32 % R == 0) return mk2<T>((T)cos32(j * (32 / R)), (T)-cos32(j * (32 / R) + 24));
  else return mk2<T>((T)cos12(j * (12 / R)), (T)-cos12(j * (12 / R) + 9));
}

// DFT of length R = 2^k in registers, input in bit-reversed order, in place; INV: the conjugate.
template <typename T, int R, bool INV>
__device__ __forceinline__ void dftc_br(c2<T> (&a)[R]) {
  constexpr int L = Log2<R>::v;
#pragma unroll
  for (int stage = 0; stage < L; ++stage) {
    const int m = 2 << stage;
#pragma unroll
    for (int k = 0; k < R; k += m) {
#pragma unroll
      for (int j = 0; j < m / 2; ++j) {
        c2<T> t = a[k + j + m / 2];
        if (j != 0) {
          if (4 * j == m) {
            t = INV ? mk2<T>(-t.y, t.x) : mk2<T>(t.y, -t.x);
          } else {
            const c2<T> w = root<T, 32>(j * (32 / m));
            t = INV ? cmulc<T>(t, w) : cmul<T>(t, w);
          }
        }
        const c2<T> u = a[k + j];
        a[k + j] = cadd<T>(u, t);
        a[k + j + m / 2] = csub<T>(u, t);
      }
    }
  }
}
// DFT of length R = 2^k or 3 * 2^k (at most 32) in registers, natural order in and out (one radix-3 step, as dft_any).
template <typename T, int R, bool INV>
__device__ __forceinline__ void dftc(c2<T> (&z)[R]) {
  if constexpr (IsPow2<R>::v) {
    c2<T> a[R];
#pragma unroll
    for (int i = 0; i < R; ++i) a[bitrev_c(i, Log2<R>::v)] = z[i];
    dftc_br<T, R, INV>(a);
#pragma unroll
    for (int i = 0; i < R; ++i) z[i] = a[i];
  } else {
    constexpr int M = R / 3;
    c2<T> e[3][M];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
#pragma unroll
      for (int m = 0; m < M; ++m) e[r][m] = z[3 * m + r];
      if constexpr (M > 1) dftc<T, M, INV>(e[r]);
    }
    constexpr T wr = T(-0.5), wi = INV ? T(0.86602540378443864676) : T(-0.86602540378443864676);
#pragma unroll
    for (int k = 0; k < M; ++k) {
      c2<T> b = e[1][k], c = e[2][k];
      if (k != 0) {
        const c2<T> w1 = root<T, R>(k), w2 = root<T, R>(2 * k);
        b = INV ? cmulc<T>(b, w1) : cmul<T>(b, w1);
        c = INV ? cmulc<T>(c, w2) : cmul<T>(c, w2);
      }
      const c2<T> a = e[0][k];
      const c2<T> s = cadd<T>(b, c), d = csub<T>(b, c);
      const c2<T> base = mk2<T>(a.x + wr * s.x, a.y + wr * s.y);
      const c2<T> rot = mk2<T>(-wi * d.y, wi * d.x);
      z[k] = cadd<T>(a, s);
      z[k + M] = cadd<T>(base, rot);
      z[k + 2 * M] = csub<T>(base, rot);
    }
  }
}

// ---------------------------------------------------------------------------
// y transform, colour solve and divide, inverse y transform: strips of W = 24 / C columns (12 column pairs over the
// channels), one t-frequency per block.  The strip goes from global memory to registers (a pair of columns is one
// 8-byte load) and back from registers; shared memory holds the 12 packed spectra, [k1][j][pair] with a row stride
// of 12 (mod 16) so that every pass's half-warps touch distinct banks.
// ---------------------------------------------------------------------------
constexpr int kFftNP = 12;
template <int M2> __host__ __device__ constexpr int fft_yc_rs() { return M2 * kFftNP + (kFftNP + 16 - M2 * kFftNP % 16) % 16; }
inline int fft_yc_w(int C) { return 2 * kFftNP / C; }
template <typename T>
inline size_t fft_yc_smem(int m1, int m2, int C) {
  const int rs = m2 * kFftNP + (kFftNP + 16 - m2 * kFftNP % 16) % 16, n = m1 * m2;
  return sizeof(c2<T>) * ((size_t)m1 * rs + n + n / 2 + 1) + sizeof(T) * (n + fft_yc_w(C)) + 8 +
         sizeof(double) * (n + fft_yc_w(C));
}

template <typename T, int M1, int M2, int C>
__global__ void __launch_bounds__(kFftNP* M1, M2 >= 32 ? 2 : 768 / (kFftNP * M1))
    k_fft_yc(Geo<T> g, T* __restrict__ hat, YcTables tb) {
  constexpr int N = M1 * M2, NT = kFftNP * M1, W2 = kFftNP / C, W = 2 * W2, RS = fft_yc_rs<M2>();
  extern __shared__ __align__(16) char smraw[];
  c2<T>* S = (c2<T>*)smraw;
  c2<T>* tw = S + M1 * RS;
  c2<T>* hw = tw + N;
  T* l2 = (T*)(hw + N / 2 + 1);                    // eigenvalues along y, x (the strip) and colour
  T* l1 = l2 + N;
  double* l2d = (double*)(((uintptr_t)(l1 + W) + 7) & ~uintptr_t(7));   // the same in double, for the low modes
  double* l1d = l2d + N;
  const int x0 = blockIdx.x * W, kt = blockIdx.y, b = blockIdx.z;
  if (retired(g, b)) return;
  const int n1 = g.n1, tid = threadIdx.x;
  const bool per = g.per2;
  for (int j = tid; j < N; j += NT) {
    tw[j] = ((const c2<T>*)tb.tw)[j];
    l2[j] = ((const T*)tb.lam2)[j];
    l2d[j] = tb.lam2d[j];
    if (j <= N / 2) hw[j] = per ? mk2<T>(T(1), T(0)) : ((const c2<T>*)tb.hw)[j];
  }
  if (tid < W) {
    l1[tid] = ((const T*)tb.lam1)[min(x0 + tid, n1 - 1)];
    l1d[tid] = tb.lam1d[min(x0 + tid, n1 - 1)];
  }
  T Q[C][C], lc[C];
#pragma unroll
  for (int c = 0; c < C; ++c) {
    lc[c] = ((const T*)tb.lamc)[c];
#pragma unroll
    for (int j = 0; j < C; ++j) Q[c][j] = ((const T*)tb.Qc)[c * C + j];
  }
  const T lt = ((const T*)tb.lamt)[kt];
  const double ltd = tb.lamtd[kt];
  __syncthreads();
  pdl_wait();   // the spectral array (forward x/t pass) is read from here on
  // the pair of a thread in the first and last pass: lanes run along the pairs
  const bool wide = n1 % 2 == 0 && ((uintptr_t)hat & 7) == 0;
#pragma unroll
  for (int q = 0; q < (kFftNP * M2 + NT - 1) / NT; ++q) {
    const int it = tid + q * NT, p = it % kFftNP, n2 = it / kFftNP;
    if (kFftNP * M2 % NT != 0 && it >= kFftNP * M2) break;
    const int c = p / W2, x = x0 + 2 * (p - c * W2);
    const T* src = hat + ((size_t)b * g.P + kt) * g.S + (size_t)c * n1 * N + x;
    c2<T> z[M1];
#pragma unroll
    for (int i = 0; i < M1; ++i) {
      const int n = M2 * i + n2;
      const int y = per ? n : (i < M1 / 2 ? 2 * n : 2 * N - 1 - 2 * n);   // Makhoul order
      const T* s = src + (size_t)y * n1;
      if (wide) {
        z[i] = x < n1 ? *reinterpret_cast<const c2<T>*>(s) : mk2<T>(T(0), T(0));
      } else {
        z[i] = mk2<T>(x < n1 ? s[0] : T(0), x + 1 < n1 ? s[1] : T(0));
      }
    }
    dftc<T, M1, false>(z);
#pragma unroll
    for (int k1 = 0; k1 < M1; ++k1)
      S[k1 * RS + n2 * kFftNP + p] = k1 ? cmul<T>(z[k1], tw[n2 * k1]) : z[k1];
  }
  __syncthreads();
  const int p = tid % kFftNP, k1 = tid / kFftNP;
  {
    c2<T> y[M2];
#pragma unroll
    for (int j = 0; j < M2; ++j) y[j] = S[k1 * RS + j * kFftNP + p];
    dftc<T, M2, false>(y);
#pragma unroll
    for (int j = 0; j < M2; ++j) S[k1 * RS + j * kFftNP + p] = y[j];
  }
  __syncthreads();
  // colour eigen-solve of frequencies k and N - k of both columns of a pair, all channels:
  // phi_c = sum_j Q[c][j] (sum_c' Q[c'][j] r_c') / lambda(kx, ky, j, kt), over N for the inverse
  {
    const float thr = (float)tb.lam_fp64;
    const T invN = T(1) / T(N);
    for (int it = tid; it < W2 * (N / 2 + 1); it += NT) {
      const int w = it % W2, k = it / W2, m = k ? N - k : 0;
      const int ik = (k % M1) * RS + (k / M1) * kFftNP + w, im = (m % M1) * RS + (m / M1) * kFftNP + w;
      const c2<T> h = hw[k];
      c2<T> qa[C], qb[C];
#pragma unroll
      for (int c = 0; c < C; ++c) {
        const c2<T> zk = S[ik + c * W2], zm = S[im + c * W2];
        const c2<T> va = mk2<T>(T(0.5) * (zk.x + zm.x), T(0.5) * (zk.y - zm.y));
        const c2<T> vb = mk2<T>(T(0.5) * (zk.y + zm.y), T(0.5) * (zm.x - zk.x));
        qa[c] = cmul<T>(va, h);
        qb[c] = cmul<T>(vb, h);
      }
      // frequency index of the real and the imaginary parts (a periodic axis: slot of frequency k for both)
      const int kr = per ? (k ? 2 * k - 1 : 0) : k, ki = per ? kr : (k ? m : 0);
      auto solve = [&](T (&r)[C], int wx, int ky) {
        T co[C];
        const T lxyt = l1[wx] + l2[ky] + lt;
#pragma unroll
        for (int j = 0; j < C; ++j) {
          T s = 0;
#pragma unroll
          for (int c = 0; c < C; ++c) s = fma(Q[c][j], r[c], s);
          const T lam = lxyt + lc[j];
          if (!(lam > T(0))) {
            co[j] = T(0);     // the zero eigenvalue of the pseudo-inverse
          } else if ((float)lam < thr) {
            // low modes: eigenvalue and quotient in double precision
            const double ld = l1d[wx] + l2d[ky] + ltd + tb.lamcd[j];
            co[j] = ld > 0.0 ? (T)quot_low((double)s, ld) * invN : T(0);
          } else {
            co[j] = fdiv_fast(s, lam) * invN;
          }
        }
#pragma unroll
        for (int c = 0; c < C; ++c) {
          T s = 0;
#pragma unroll
          for (int j = 0; j < C; ++j) s = fma(Q[c][j], co[j], s);
          r[c] = s;
        }
      };
      T r[C];
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        auto part = [&](c2<T>& v) -> T& { return half ? v.y : v.x; };
#pragma unroll
        for (int c = 0; c < C; ++c) r[c] = part(qa[c]);
        solve(r, 2 * w, half ? ki : kr);
#pragma unroll
        for (int c = 0; c < C; ++c) part(qa[c]) = r[c];
#pragma unroll
        for (int c = 0; c < C; ++c) r[c] = part(qb[c]);
        solve(r, 2 * w + 1, half ? ki : kr);
#pragma unroll
        for (int c = 0; c < C; ++c) part(qb[c]) = r[c];
      }
#pragma unroll
      for (int c = 0; c < C; ++c) {
        if (k == 0) qa[c].y = qb[c].y = T(0);   // frequency 0 has no partner
        const c2<T> va = cmulc<T>(qa[c], h), vb = cmulc<T>(qb[c], h);
        S[ik + c * W2] = mk2<T>(va.x - vb.y, va.y + vb.x);
        if (k) S[im + c * W2] = mk2<T>(va.x + vb.y, vb.x - va.y);
      }
    }
  }
  __syncthreads();
  {
    c2<T> y[M2];
#pragma unroll
    for (int j = 0; j < M2; ++j) y[j] = S[k1 * RS + j * kFftNP + p];
    dftc<T, M2, true>(y);
#pragma unroll
    for (int j = 0; j < M2; ++j)
      S[k1 * RS + j * kFftNP + p] = j ? cmulc<T>(y[j], tw[j * k1]) : y[j];
  }
  __syncthreads();
  pdl_trigger();
#pragma unroll
  for (int q = 0; q < (kFftNP * M2 + NT - 1) / NT; ++q) {
    const int it = tid + q * NT, pp = it % kFftNP, n2 = it / kFftNP;
    if (kFftNP * M2 % NT != 0 && it >= kFftNP * M2) break;
    const int c = pp / W2, x = x0 + 2 * (pp - c * W2);
    T* dst = hat + ((size_t)b * g.P + kt) * g.S + (size_t)c * n1 * N + x;
    c2<T> z[M1];
#pragma unroll
    for (int i = 0; i < M1; ++i) z[i] = S[i * RS + n2 * kFftNP + pp];
    dftc<T, M1, true>(z);
#pragma unroll
    for (int i = 0; i < M1; ++i) {
      const int n = M2 * i + n2;
      const int y = per ? n : (i < M1 / 2 ? 2 * n : 2 * N - 1 - 2 * n);
      T* d = dst + (size_t)y * n1;
      if (wide) {
        if (x < n1) *reinterpret_cast<c2<T>*>(d) = z[i];
      } else {
        if (x < n1) d[0] = z[i].x;
        if (x + 1 < n1) d[1] = z[i].y;
      }
    }
  }
}

// ---------------------------------------------------------------------------
// x and t transforms of one (y, c) row per block.  Rows t = 2p and 2p + 1 travel as one complex sequence; shared memory
// holds [chunk of PC pairs][element][pair], a row of PC + 1 values per element: the passes run their lanes along the
// pairs, the loads, stores and time transforms along the elements, and both touch distinct banks.
//   forward: r straight into pairs, the x transform, then a thread per x-frequency forms its P coefficients from Z_k and
//            Z_{N-k}, transforms them along t in registers and stores them;
//   inverse: a thread per x-frequency transforms along t and leaves pairs, the first inverse pass reads Z_k from the
//            coefficients k and N - k, and the samples go out by columns.
// The time transform is a register FFT (dct_cols_fft's) where P fills PM, the folded product of mm_kernels.cuh otherwise.
// ---------------------------------------------------------------------------
template <int PM> struct FftXt {
  static constexpr int PC = PM == 16 ? 8 : 16, NCH = PM / 2 / PC, ST = PC + 1;
};
template <int N, int PM> __host__ __device__ constexpr int fft_xt_nt() {
  const int nt = N * FftXt<PM>::PC / 16;
  return nt < 128 ? 128 : nt;
}
template <int N, int PM> __host__ __device__ constexpr int fft_xt_minb() {   // register budget: 80 (128 where P or N is long)
  return (PM == 64 || N == 512 ? 512 : 768) / fft_xt_nt<N, PM>();
}
inline int fft_xt_threads(int n, int pm) { return std::max(128, pm == 16 ? n / 2 : n); }
inline size_t fft_xt_smem(int n, int P, int pm) {
  const int pc = pm == 16 ? 8 : 16;
  const size_t tt = P == pm ? sizeof(float2) * 2 * P : sizeof(float) * (size_t)std::max((P + 3) / 4 * 4 * (pm / 2), ((P + 1) / 2 + 3) / 4 * 4 * pm);
  return sizeof(float2) * ((size_t)(pm / 2 / pc) * n * (pc + 1) + 2 * n) + tt;
}
struct FftXtTables {
  const float2 *tw, *hw;     // exp(-2 pi i j / N), exp(-i pi k / 2N)
  const float2 *twt, *hwt;   // the same along t (P == PM)
  const float *mtf, *mti;    // folded time products (P < PM), as for k_mm_fwd_xt / k_mm_inv_xt
};

// DCT-II along t of the P values x[] in registers (the steps of dct_cols_fft): out(k, value)
template <int P, class F>
__device__ __forceinline__ void dct_reg(const float (&x)[P], const float2* tw, const float2* hw, F&& out) {
  constexpr int M = P / 2;
  float2 z[M];
#pragma unroll
  for (int m = 0; m < M; ++m) {
    const int j0 = 2 * m, j1 = 2 * m + 1;   // v[j] = x[2j] (j < M), x[2(P-1-j)+1] (j >= M)
    z[bitrev_c(m, Log2<M>::v)] =
        make_float2(x[j0 < M ? 2 * j0 : 2 * (P - 1 - j0) + 1], x[j1 < M ? 2 * j1 : 2 * (P - 1 - j1) + 1]);
  }
  dftc_br<float, M, false>(z);
#pragma unroll
  for (int k = 0; k < M; ++k) {
    const float2 zk = z[k], zm = z[(M - k) % M];
    const float ex = 0.5f * (zk.x + zm.x), ey = 0.5f * (zk.y - zm.y);
    const float ox = 0.5f * (zk.y + zm.y), oy = 0.5f * (zm.x - zk.x);
    const float2 w = tw[k];
    const float tx = w.x * ox - w.y * oy, ty = w.x * oy + w.y * ox;
    const float2 h0 = hw[k], h1 = hw[k + M];
    out(k, h0.x * (ex + tx) - h0.y * (ey + ty));
    out(k + M, h1.x * (ex - tx) - h1.y * (ey - ty));
  }
}
// its inverse, in place
template <int P>
__device__ __forceinline__ void idct_reg(float (&x)[P], const float2* tw, const float2* hw) {
  constexpr int M = P / 2;
  float2 z[M];
#pragma unroll
  for (int k = 0; k < M; ++k) {
    const float a0 = x[k], b0 = k ? x[P - k] : 0.f, a1 = x[k + M], b1 = x[M - k];
    const float2 h0 = hw[k], h1 = hw[k + M];
    const float v0x = h0.x * a0 - h0.y * b0, v0y = -h0.x * b0 - h0.y * a0;
    const float v1x = h1.x * a1 - h1.y * b1, v1y = -h1.x * b1 - h1.y * a1;
    const float ex = 0.5f * (v0x + v1x), ey = 0.5f * (v0y + v1y);
    const float dx = 0.5f * (v0x - v1x), dy = 0.5f * (v0y - v1y);
    const float2 w = tw[k];
    const float ox = dx * w.x + dy * w.y, oy = dy * w.x - dx * w.y;
    z[bitrev_c(k, Log2<M>::v)] = make_float2(ex - oy, ey + ox);
  }
  dftc_br<float, M, true>(z);
  constexpr float invM = 1.f / M;
#pragma unroll
  for (int m = 0; m < M; ++m) {
    const int j0 = 2 * m, j1 = 2 * m + 1;
    x[j0 < M ? 2 * j0 : 2 * (P - 1 - j0) + 1] = z[m].x * invM;
    x[j1 < M ? 2 * j1 : 2 * (P - 1 - j1) + 1] = z[m].y * invM;
  }
}

template <int M1, int M2, int PM>
__global__ void __launch_bounds__((fft_xt_nt<M1 * M2, PM>()), (fft_xt_minb<M1 * M2, PM>()))
    k_fft_fwd_xt(Geo<float> g, const float4* __restrict__ ap, const float* __restrict__ f0,   // grid (C, n2, B)
                 const float* __restrict__ f1, float* __restrict__ hat, FftXtTables tb) {
  using L = FftXt<PM>;
  constexpr int N = M1 * M2, NT = fft_xt_nt<N, PM>(), PC = L::PC, ST = L::ST, NCH = L::NCH, PH = PM / 2;
  extern __shared__ __align__(16) char smraw[];
  // channels run fastest: the row of channel c - 1, whose faces this block reads, is then in L2 (with y fastest it had
  // left it at large grids: 368 against 284 us at 512x512x3, P = 64; 47.6 against 41.4 at 256x256x3, P = 32)
  const int c = blockIdx.x, y = blockIdx.y, b = blockIdx.z, tid = threadIdx.x;
  if (retired(g, b)) return;
  const int P = g.P;
  const bool per = g.per1, tfft = P == PM;
  float2* Z = (float2*)smraw;             // [chunk][element][pair]
  float2* tw = Z + NCH * N * ST;
  float2* hw = tw + N;
  float* tt = (float*)(hw + N);           // tables of the time transform
  for (int j = tid; j < N; j += NT) {
    tw[j] = tb.tw[j];
    hw[j] = tb.hw[j];
  }
  if (tfft) {
    for (int j = tid; j < P; j += NT) {
      ((float2*)tt)[j] = tb.twt[j];
      ((float2*)tt)[P + j] = tb.hwt[j];
    }
  } else {
    for (int j = tid; j < (P + 3) / 4 * 4 * PH; j += NT) tt[j] = tb.mtf[j];
  }
  pdl_wait();   // a (previous update) is read from here on
  const int S = g.S;
  const size_t rowbase = (size_t)b * P * S + (size_t)N * (y + (size_t)g.n2 * c);
  {
    const int ym = y > 0 ? y - 1 : (g.per2 ? g.n2 - 1 : -1), cm = c > 0 ? c - 1 : (g.perc ? g.C - 1 : -1);
    const int dy = ym >= 0 ? N * (ym - y) : 0, dc = cm >= 0 ? N * g.n2 * (cm - c) : 0;
    const size_t sb = (size_t)b * S + (size_t)N * (y + (size_t)g.n2 * c);
    for (int x = tid; x < N; x += NT) {
      const int xm = x > 0 ? x - 1 : (per ? N - 1 : x);
      const bool hx = xm != x, hy = ym >= 0, hz = cm >= 0;
      const float4* pc = ap + rowbase + x;
      const float* as = reinterpret_cast<const float*>(ap);
      const float* px = as + 4 * (rowbase + xm);
      const float* py = as + 4 * (rowbase + x + dy) + 1;   // dy, dc = 0 where the face is absent
      const float* pz = as + 4 * (rowbase + x + dc) + 2;
      float below = f0[sb + x];              // f face below the plane
      const float above = f1[sb + x];
#pragma unroll 4
      for (int p = 0; p < (P + 1) / 2; ++p) {
        const size_t o = (size_t)(2 * p) * S;
        const bool two = 2 * p + 1 < P;
        const size_t o2 = two ? o + S : o;
        const float4 a0 = pc[o], a1 = pc[o2];
        const float x0 = px[4 * o], x1 = px[4 * o2], y0 = py[4 * o], y1 = py[4 * o2], z0 = pz[4 * o], z1 = pz[4 * o2];
        const float t0 = two ? a0.w : above, t1 = 2 * p + 2 < P ? a1.w : above;
        float r0 = g.s1 * (a0.x - (hx ? x0 : 0.f)), r1 = g.s1 * (a1.x - (hx ? x1 : 0.f));
        r0 += g.s2 * (a0.y - (hy ? y0 : 0.f));
        r1 += g.s2 * (a1.y - (hy ? y1 : 0.f));
        r0 += g.sc * (a0.z - (hz ? z0 : 0.f));
        r1 += g.sc * (a1.z - (hz ? z1 : 0.f));
        r0 += g.sp * (t0 - below);
        r1 += g.sp * (t1 - t0);
        below = t1;
        Z[((p / PC) * N + x) * ST + p % PC] = make_float2(r0, two ? r1 : 0.f);
      }
    }
  }
  __syncthreads();
  // M1-point DFTs over n1 (Makhoul order on a Neumann axis), twiddles
  {
    constexpr int R1 = (PC * M2 + NT - 1) / NT;
#pragma unroll
    for (int ch = 0; ch < NCH; ++ch) {
      float2* Zc = Z + ch * N * ST;
      float2 z[R1][M1];
#pragma unroll
      for (int q = 0; q < R1; ++q) {
        const int it = tid + q * NT, pl = it % PC, n2 = it / PC;
        if (PC * M2 % NT == 0 || it < PC * M2)
#pragma unroll
          for (int i = 0; i < M1; ++i) {
            const int n = M2 * i + n2;
            z[q][i] = Zc[(per ? n : (i < M1 / 2 ? 2 * n : 2 * N - 1 - 2 * n)) * ST + pl];
          }
      }
      __syncthreads();
#pragma unroll
      for (int q = 0; q < R1; ++q) {
        const int it = tid + q * NT, pl = it % PC, n2 = it / PC;
        if (PC * M2 % NT == 0 || it < PC * M2) {
          dftc<float, M1, false>(z[q]);
#pragma unroll
          for (int k1 = 0; k1 < M1; ++k1)
            Zc[(n2 * M1 + k1) * ST + pl] = k1 ? cmul<float>(z[q][k1], tw[n2 * k1]) : z[q][k1];
        }
      }
    }
  }
  __syncthreads();
  // M2-point DFTs over n2: elements j M1 + k1, in place
  for (int it = tid; it < NCH * PC * M1; it += NT) {
    const int pl = it % PC, k1 = (it / PC) % M1, ch = it / (PC * M1);
    float2* Zc = Z + ch * N * ST + pl;
    float2 v[M2];
#pragma unroll
    for (int j = 0; j < M2; ++j) v[j] = Zc[(j * M1 + k1) * ST];
    dftc<float, M2, false>(v);
#pragma unroll
    for (int j = 0; j < M2; ++j) Zc[(j * M1 + k1) * ST] = v[j];
  }
  __syncthreads();
  pdl_trigger();
  // a thread per x-frequency: coefficient X = al va.x + be va.y of row a (va.y, vb.y with the signs of the packing)
  for (int q = tid; q < N; q += NT) {
    const int k = per ? (q + 1) / 2 : (q <= N / 2 ? q : N - q), m = k ? N - k : 0;
    float al, be;
    if (per) {
      const bool cs = q == 0 || (q & 1);
      al = cs ? 0.5f : 0.f;
      be = cs ? 0.f : -0.5f;
    } else {
      const float2 h = hw[k];
      al = 0.5f * (q <= N / 2 ? h.x : -h.y);
      be = 0.5f * (q <= N / 2 ? -h.y : -h.x);
    }
    const float2 *zk = Z + k * ST, *zm = Z + m * ST;
    auto pair = [&](int ch, int pl) {   // rows 2p and 2p + 1
      const float2 u = zk[ch * N * ST + pl], w = zm[ch * N * ST + pl];
      return make_float2(al * (u.x + w.x) + be * (u.y - w.y), al * (u.y + w.y) + be * (w.x - u.x));
    };
    float* dst = hat + rowbase + q;
    if (tfft) {
      float x[PM];
#pragma unroll
      for (int p = 0; p < PM / 2; ++p) {
        const float2 v = pair(p / PC, p % PC);
        x[2 * p] = v.x;
        x[2 * p + 1] = v.y;
      }
      dct_reg<PM>(x, (const float2*)tt, (const float2*)tt + P, [&](int kt, float v) { dst[(size_t)kt * S] = v; });
    } else {
      const int hP = (P + 1) / 2;
      float vs[PH], vd[PH];
#pragma unroll
      for (int t = 0; t < PH; ++t) {
        const int tl = min(t, hP - 1), th = P - 1 - tl;
        const float2 a = pair((tl / 2) / PC, (tl / 2) % PC), e = pair((th / 2) / PC, (th / 2) % PC);
        const float lo = tl & 1 ? a.y : a.x, hi = th & 1 ? e.y : e.x;
        const bool in = t < hP, mid = tl == th;
        vs[t] = in ? (mid ? lo : lo + hi) : 0.f;
        vd[t] = in && !mid ? lo - hi : 0.f;
      }
      for (int k4 = 0; k4 < P; k4 += 4) {
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int j = 0; j < PH; j += 4)
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float4 w = *reinterpret_cast<const float4*>(tt + (k4 + e) * PH + j);
            const float (&v)[PH] = e & 1 ? vd : vs;
            acc[e] = fmaf(w.x, v[j], acc[e]);
            acc[e] = fmaf(w.y, v[j + 1], acc[e]);
            acc[e] = fmaf(w.z, v[j + 2], acc[e]);
            acc[e] = fmaf(w.w, v[j + 3], acc[e]);
          }
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (k4 + e < P) dst[(size_t)(k4 + e) * S] = acc[e];
      }
    }
  }
}

template <int M1, int M2, int PM>
__global__ void __launch_bounds__((fft_xt_nt<M1 * M2, PM>()), (fft_xt_minb<M1 * M2, PM>()))
    k_fft_inv_xt(Geo<float> g, const float* __restrict__ hat, float* __restrict__ phi, FftXtTables tb) {
  using L = FftXt<PM>;
  constexpr int N = M1 * M2, NT = fft_xt_nt<N, PM>(), PC = L::PC, ST = L::ST, NCH = L::NCH, PH = PM / 2;
  extern __shared__ __align__(16) char smraw[];
  const int y = blockIdx.x, c = blockIdx.y, b = blockIdx.z, tid = threadIdx.x;
  if (retired(g, b)) return;
  const int P = g.P;
  const bool per = g.per1, tfft = P == PM;
  float2* Z = (float2*)smraw;
  float2* tw = Z + NCH * N * ST;
  float2* hw = tw + N;                    // over N: the inverse's normalisation
  float* tt = (float*)(hw + N);
  constexpr float invN = 1.f / N;
  for (int j = tid; j < N; j += NT) {
    tw[j] = tb.tw[j];
    const float2 h = tb.hw[j];
    hw[j] = make_float2(h.x * invN, h.y * invN);
  }
  if (tfft) {
    for (int j = tid; j < P; j += NT) {
      ((float2*)tt)[j] = tb.twt[j];
      ((float2*)tt)[P + j] = tb.hwt[j];
    }
  } else {
    for (int j = tid; j < ((P + 1) / 2 + 3) / 4 * 4 * PM; j += NT) tt[j] = tb.mti[j];
  }
  __syncthreads();
  pdl_wait();   // the spectral array (y/colour pass) is read from here on
  const int S = g.S;
  const size_t rowbase = (size_t)b * P * S + (size_t)N * (y + (size_t)g.n2 * c);
  // inverse time transform, a thread per x-frequency; pairs of samples to Z
  for (int q = tid; q < N; q += NT) {
    const float* src = hat + rowbase + q;
    if (tfft) {
      float x[PM];
#pragma unroll
      for (int t = 0; t < PM; ++t) x[t] = src[(size_t)t * S];
      idct_reg<PM>(x, (const float2*)tt, (const float2*)tt + P);
#pragma unroll
      for (int p = 0; p < PM / 2; ++p) Z[((p / PC) * N + q) * ST + p % PC] = make_float2(x[2 * p], x[2 * p + 1]);
    } else {
      float ve[PH], vo[PH];
#pragma unroll
      for (int j = 0; j < PH; ++j) {
        const float e = src[(size_t)min(2 * j, P - 1) * S], o = src[(size_t)min(2 * j + 1, P - 1) * S];
        ve[j] = 2 * j < P ? e : 0.f;
        vo[j] = 2 * j + 1 < P ? o : 0.f;
      }
      auto put = [&](int t, float v) {
        const int p = t / 2;
        reinterpret_cast<float*>(Z + ((p / PC) * N + q) * ST + p % PC)[t & 1] = v;
      };
      if (P & 1) put(P, 0.f);
      for (int t = 0; t < (P + 1) / 2; ++t) {
        float E = 0.f, O = 0.f;
#pragma unroll
        for (int j = 0; j < PH; j += 4) {
          const float4 w = *reinterpret_cast<const float4*>(tt + t * PM + j);
          const float4 u = *reinterpret_cast<const float4*>(tt + t * PM + PH + j);
          E = fmaf(w.x, ve[j], E);
          O = fmaf(u.x, vo[j], O);
          E = fmaf(w.y, ve[j + 1], E);
          O = fmaf(u.y, vo[j + 1], O);
          E = fmaf(w.z, ve[j + 2], E);
          O = fmaf(u.z, vo[j + 2], O);
          E = fmaf(w.w, ve[j + 3], E);
          O = fmaf(u.w, vo[j + 3], O);
        }
        put(P - 1 - t, E - O);
        put(t, E + O);
      }
    }
  }
  __syncthreads();
  // Z_k from the coefficients k and N - k, M2-point DFTs over k2, twiddles
  {
    constexpr int RA = (NCH * PC * M1 + NT - 1) / NT;
    float2 v[RA][M2];
#pragma unroll
    for (int r = 0; r < RA; ++r) {
      const int it = tid + r * NT, pl = it % PC, k1 = (it / PC) % M1, ch = it / (PC * M1);
      if (NCH * PC * M1 % NT == 0 || it < NCH * PC * M1) {
        const float2* Zc = Z + ch * N * ST + pl;
#pragma unroll
        for (int j = 0; j < M2; ++j) {
          const int k = k1 + M1 * j;
          if (per) {
            // V_k = X[2k-1] - i X[2k], V_{N-k} = conj V_k; slot 0 and the Nyquist slot are real
            const int f = k <= N / 2 ? k : N - k;
            const float2 re = Zc[(f ? 2 * f - 1 : 0) * ST];
            float2 im = (f == 0 || f == N / 2) ? make_float2(0.f, 0.f) : Zc[2 * f * ST];
            if (k <= N / 2) im = make_float2(-im.x, -im.y);
            v[r][j] = make_float2((re.x - im.y) * invN, (im.x + re.y) * invN);
          } else {
            const float2 x = Zc[k * ST], xm = k ? Zc[(N - k) * ST] : make_float2(0.f, 0.f), h = hw[k];
            const float ax = h.x * x.x - h.y * xm.x, ay = -h.x * xm.x - h.y * x.x;
            const float bx = h.x * x.y - h.y * xm.y, by = -h.x * xm.y - h.y * x.y;
            v[r][j] = make_float2(ax - by, ay + bx);
          }
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RA; ++r) {
      const int it = tid + r * NT, pl = it % PC, k1 = (it / PC) % M1, ch = it / (PC * M1);
      if (NCH * PC * M1 % NT == 0 || it < NCH * PC * M1) {
        float2* Zc = Z + ch * N * ST + pl;
        dftc<float, M2, true>(v[r]);
#pragma unroll
        for (int j = 0; j < M2; ++j) Zc[(j * M1 + k1) * ST] = j ? cmulc<float>(v[r][j], tw[j * k1]) : v[r][j];
      }
    }
  }
  __syncthreads();
  // M1-point DFTs over k1 -> samples in their places
  {
    constexpr int R1 = (PC * M2 + NT - 1) / NT;
#pragma unroll
    for (int ch = 0; ch < NCH; ++ch) {
      float2* Zc = Z + ch * N * ST;
      float2 z[R1][M1];
#pragma unroll
      for (int q = 0; q < R1; ++q) {
        const int it = tid + q * NT, pl = it % PC, n2 = it / PC;
        if (PC * M2 % NT == 0 || it < PC * M2)
#pragma unroll
          for (int i = 0; i < M1; ++i) z[q][i] = Zc[(n2 * M1 + i) * ST + pl];
      }
      __syncthreads();
#pragma unroll
      for (int q = 0; q < R1; ++q) {
        const int it = tid + q * NT, pl = it % PC, n2 = it / PC;
        if (PC * M2 % NT == 0 || it < PC * M2) {
          dftc<float, M1, true>(z[q]);
#pragma unroll
          for (int i = 0; i < M1; ++i) {
            const int n = M2 * i + n2;
            Zc[(per ? n : (i < M1 / 2 ? 2 * n : 2 * N - 1 - 2 * n)) * ST + pl] = z[q][i];
          }
        }
      }
    }
  }
  __syncthreads();
  pdl_trigger();
  for (int x = tid; x < N; x += NT) {
    float* dst = phi + rowbase + x;
#pragma unroll 8
    for (int p = 0; p < (P + 1) / 2; ++p) {
      const float2 v = Z[((p / PC) * N + x) * ST + p % PC];
      dst[(size_t)(2 * p) * S] = v.x;
      if (2 * p + 1 < P) dst[(size_t)(2 * p + 1) * S] = v.y;
    }
  }
}

}  // namespace dynot
