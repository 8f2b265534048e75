// The DCT-I pass of tensor generation (FP64): per line of n + 1 values
// O[0..n], X[p] = O[0] + (-1)^p O[n] + 2 sum_{j=1}^{n-1} O[j] cos(pi j p / n), the
// length-2n DFT of the even extension O[min(m, 2n - m)].  Two lines ride in
// one complex transform (their DFTs are real, so they come back as the real
// and imaginary parts).
//
// What bounds it: the FP64 pipe (about 2 lanes per SM and clock on GB300).  So
// the Stockham transform is pruned by the symmetry.  With R the first radix
// and NB = M / R, the first stage's butterfly NB - b reads butterfly b's
// inputs in reverse: its outputs are A_{NB-b}[q] = w_R^{-q} A_b[R - q], and only
// b <= NB / 2 is computed (the factor joins the next stage's twiddle: no
// further rounding).  The later stages keep an element's class q =
// index mod R, and X is even, so only the classes q <= R / 2 are carried: 33
// of 64, 40 of 64 and 40 of 64 butterflies at length 512.
// Measured (GB300, 256^3 plan): 0.86 -> 0.60 ms a pass.
//
// Src(a, b, m): element m of line (a, b); Dst(a, b, p, v) takes its result; a
// line's number is a * inner + b.
#pragma once
#include "passes.cuh"

namespace fsa {

// Butterflies a line runs in stage S, and the i-th one's index.
template <class P, int S> constexpr int dct_count() {
  constexpr int R0 = P::R[0];
  return S == 0 ? P::M / R0 / 2 + 1 : P::M / P::R[S] / R0 * (R0 / 2 + 1);
}
template <class P, int S> __device__ __forceinline__ int dct_index(int i) {
  constexpr int R0 = P::R[0], H = R0 / 2 + 1;
  return S == 0 ? i : (i / H) * R0 + i % H;
}

template <class P, int S, int W, int T, class Ld, class St>
__device__ __forceinline__ void dct_stages(int t, double2* sm, const Ld& ld, const St& st) {
  constexpr int R0 = P::R[0], R = P::R[S], NS = P::ns(S), NB = P::M / R, CNT = dct_count<P, S>();
  constexpr int PER = (CNT + T - 1) / T;
  constexpr bool LAST = S == P::NST - 1;
  double2 v[PER][R];
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int i = t + k * T;
    if (PER * T == CNT || i < CNT) {
      const int b = dct_index<P, S>(i);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if constexpr (S == 0) v[k][r] = ld(b + r * NB);
        else v[k][r] = sm[(b + r * NB) * W];
      }
      if constexpr (NS > 1) {
#pragma unroll
        for (int r = 1; r < R; ++r) {
          const int q = b % NS;
          int e = r * q;
          // first exchange: elements of a mirrored butterfly carry w_R0^{-q}
          if (S == 1 && 2 * ((b + r * NB) / R0) > P::M / R0) e = q == 0 ? 0 : e + NS * R - R * q;
          v[k][r] = cmul(v[k][r], twiddle<double2, NS * R>(e));
        }
      }
      dft<R, true>(v[k]);
    }
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int i = t + k * T;
    if (PER * T == CNT || i < CNT) {
      const int b = dct_index<P, S>(i);
      if constexpr (LAST) {
        // p = b + r NS (NB = NS): p and M - p are equal; the classes 0 and R0 / 2
        // hold both, the others only p
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int p = b + r * NS, q = b % R0;
          const bool lo = p <= P::M / 2;
          if (lo || (P::NST > 1 && q != 0 && q != R0 / 2)) st(lo ? p : P::M - p, v[k][r]);
        }
      } else if constexpr (S == 0) {
#pragma unroll
        for (int q = 0; q <= R0 / 2; ++q) sm[(b * R0 + q) * W] = v[k][q];
        if (b > 0 && 2 * b < NB) {
#pragma unroll
          for (int q = 0; q <= R0 / 2; ++q) sm[((NB - b) * R0 + q) * W] = v[k][(R0 - q) % R0];
        }
      } else {
        const int j = (b / NS) * NS * R + b % NS;
#pragma unroll
        for (int r = 0; r < R; ++r) sm[(j + r * NS) * W] = v[k][r];
      }
    }
  }
  if constexpr (!LAST) {
    __syncthreads();
    dct_stages<P, S + 1, W, T>(t, sm, ld, st);
  }
}

template <class P, int W, int T, class Src, class Dst>
__global__ void __launch_bounds__(W * T) k_dct1(const Src src, const Dst dst, long long nlines, int inner) {
  constexpr int M = P::M, n = M / 2;
  static_assert(P::R[0] == 8 || P::R[0] == 4, "first radix");
  extern __shared__ __align__(16) unsigned char smraw[];
  const int l = threadIdx.x % W, t = threadIdx.x / W;
  double2* sm = reinterpret_cast<double2*>(smraw) + l;
  const long long L0 = 2 * ((long long)blockIdx.x * W + l), L1 = L0 + 1;
  const bool ok0 = L0 < nlines, ok1 = L1 < nlines;
  const int a0 = ok0 ? (int)(L0 / inner) : 0, b0 = ok0 ? (int)(L0 % inner) : 0;
  const int a1 = ok1 ? (int)(L1 / inner) : 0, b1 = ok1 ? (int)(L1 % inner) : 0;
  dct_stages<P, 0, W, T>(
      t, sm,
      [&](int m) -> double2 {
        const int mm = m <= n ? m : M - m;
        return mk(ok0 ? src(a0, b0, mm) : 0.0, ok1 ? src(a1, b1, mm) : 0.0);
      },
      [&](int p, double2 v) {
        if (ok0) dst(a0, b0, p, v.x);
        if (ok1) dst(a1, b1, p, v.y);
      });
}

// Element m of line (a, b) at O[a os + b is + m es].
struct DctArray {
  double* O;
  long long os, is, es;
  __device__ __forceinline__ long long at(int a, int b, int m) const { return a * os + b * is + m * es; }
  __device__ __forceinline__ double operator()(int a, int b, int m) const { return O[at(a, b, m)]; }
  __device__ __forceinline__ void operator()(int a, int b, int p, double v) const { O[at(a, b, p)] = v; }
};
// A radial function from its table: entry ra a^2 + rb b^2 + re m^2.
struct DctRadial {
  const double* tab;
  int ra, rb, re;
  __device__ __forceinline__ double operator()(int a, int b, int m) const {
    return __ldg(tab + ra * a * a + rb * b * b + re * m * m);
  }
};
// The stored spectrum: (X + W) norm, W from its table (the sum rounded by
// itself, as where X is read back: the two forms agree bit for bit).
template <typename R> struct DctSpectrum {
  R* S;
  DctArray idx;
  DctRadial w;
  double norm;
  __device__ __forceinline__ void operator()(int a, int b, int p, double v) const {
    S[idx.at(a, b, p)] = (R)(__dadd_rn(v, w(a, b, p)) * norm);
  }
};

}  // namespace fsa
