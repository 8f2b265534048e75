// The apply passes in paired double-word arithmetic (dw2.cuh): the five
// passes of passes.cuh, the plane's middle pass and the DDI forms.
//
// What bounds them: the FP32 pipes (a 256^3 middle pass needs 29.4e9 FP32
// operations, 0.75 ms at the measured FMA rate, against 0.18 ms for its
// bytes).  The paired operations do that work in half the issue slots; the
// rest of the design keeps the pipes fed:
//   * a line runs the Stockham stages of PlanDw<M>, first and last radix
//     equal, so in the middle pass the last forward stage leaves a thread
//     exactly the elements its first inverse stage takes (b + r M/R): the
//     spectrum multiply happens in registers;
//   * the first stage's inputs are staged by per-thread asynchronous copies:
//     in the R2C and row passes the next tile's under the current tile's work,
//     in the middle pass from its last store on (until then the same slots
//     hold the spectrum values, copied under the forward transform); the C2R
//     pass and the plane's middle pass load directly.  The twiddles sit in a
//     shared table;
//   * the last stage writes HBM from registers (the row passes too: lanes run
//     along a row, so their accesses are contiguous), except in the R2C pass,
//     whose split of two real lines needs each line whole;
//   * the middle pass runs the inner stages of its forward and inverse
//     transforms through the same code (the inverse is the forward one with
//     real and imaginary parts swapped): unrolled twice it outgrew the
//     instruction cache (1.8 of 6.9 stall cycles per issue).
//   * tiles are handed out dynamically (mbar.cuh, TileQueue).
// Measured (GB300, FP64 solve of 256^3, us): R2C 217 -> 180, row forward 367 ->
// 254, middle 1187 -> 981 (0.76 of the measured FP32 rate, from 0.63), row
// inverse 348 -> 251, C2R 204 -> 173; the solve 2.30 -> 1.82 ms.  Before: the
// same stages in scalar double-word operations, five shared-memory trips per
// transform, a fixed share of the tiles per CTA.  Pairing two lines instead of
// the two parts of a value took 128 registers and 1.30 ms for the middle pass.
#pragma once
#include "ddi.cuh"
#include "dw2.cuh"
#include "mbar.cuh"
#include "passes2.cuh"

namespace fsa {

// Radix plan per length, first and last radix equal.
template <int M> struct PlanDw;
template <> struct PlanDw<8> { using type = Plan<8, 8>; };
template <> struct PlanDw<12> { using type = Plan<12, 2, 3, 2>; };
template <> struct PlanDw<16> { using type = Plan<16, 4, 4>; };
template <> struct PlanDw<24> { using type = Plan<24, 2, 6, 2>; };
template <> struct PlanDw<32> { using type = Plan<32, 4, 2, 4>; };
template <> struct PlanDw<48> { using type = Plan<48, 4, 3, 4>; };
template <> struct PlanDw<64> { using type = Plan<64, 8, 8>; };
template <> struct PlanDw<96> { using type = Plan<96, 4, 6, 4>; };
template <> struct PlanDw<128> { using type = Plan<128, 8, 2, 8>; };
template <> struct PlanDw<192> { using type = Plan<192, 8, 3, 8>; };
template <> struct PlanDw<256> { using type = Plan<256, 8, 4, 8>; };
template <> struct PlanDw<384> { using type = Plan<384, 8, 6, 8>; };
template <> struct PlanDw<512> { using type = Plan<512, 8, 8, 8>; };
template <> struct PlanDw<768> { using type = Plan<768, 8, 3, 4, 8>; };
template <> struct PlanDw<1024> { using type = Plan<1024, 8, 4, 4, 8>; };

// One Stockham stage: NB butterflies over T threads, PER each.
template <class P, int S, int T> struct PSt {
  static constexpr int R = P::R[S], NS = P::ns(S), NB = P::M / R, PER = (NB + T - 1) / T;
  static constexpr bool EXACT = PER * T == NB;
};

// Tile geometry: T threads per line (one butterfly of the end radix each;
// where the inner radix has more of them, their count or half of it: whole
// warps then sit out the ends), W lines per CTA: CTAs of 256 threads for the
// long lines, smaller ones for the short lines, whose grids are small (32^3
// would fill 16 SMs with 256-thread tiles).
template <int M_> struct GeoDw {
  using P = typename PlanDw<M_>::type;
  static constexpr int M = M_;
  static constexpr int T = M == 384 ? 64 : M == 192 ? 32 : M == 48 ? 16 : M / P::R[0];
  static constexpr int W = T > 96 ? 2 : T >= 64 ? 4 : T >= 8 ? 8 : T >= 4 ? 16 : 32;
  static constexpr int NT = T * W;
  // lines per CTA of the R2C and C2R passes: half as many lines in all, so
  // narrower tiles up to length 256 (96^3 R2C: 1.26 waves of 8-line tiles)
  static constexpr int WX = M >= 384 || W == 2 ? W : W / 2;
  // Resident threads per SM the kernels are compiled for: 1024 (64 registers)
  // where they fit without spills, else 768 (80 registers); the FP32 pipes
  // are as busy with 24 warps as with 32.
  static constexpr int RES = M == 96 || M == 192 || M == 384 ? 768 : 1024;
  static constexpr int RES_MID = M > 128 ? 768 : RES;
  static constexpr int XCH = M * 16;  // exchange tile, bytes per line
};

// Exchange tile of one line: element p at slot(p) * STRIDE, the low bits of p
// exchanged with the next three so that a first stage's stores, eight
// elements apart, hit different banks.
template <int STRIDE> struct PLine {
  cdwp* base;
  static __device__ __forceinline__ int slot(int p) { return (p ^ ((p >> 3) & 7)) * STRIDE; }
  __device__ __forceinline__ cdwp get(int p) const { return base[slot(p)]; }
  __device__ __forceinline__ void put(int p, cdwp v) const { base[slot(p)] = v; }
};

// Twiddle table of a plan: stage S >= 1 holds w^(r k), r = 1 .. R - 1, k < NS,
// at entry NS - NS(1) + (r - 1) NS + k: M - R(0) entries in all.
template <class P> constexpr int tw_entries() { return P::M - P::R[0]; }
template <class P, int S> __device__ __forceinline__ void tw_fill(float4* tw) {
  if constexpr (S < P::NST) {
    constexpr int R = P::R[S], NS = P::ns(S), OFF = NS - P::R[0];
    static_assert(kTwN % (NS * R) == 0, "length must divide the twiddle table");
    for (int i = threadIdx.x; i < (R - 1) * NS; i += blockDim.x)
      tw[OFF + i] = __ldg(reinterpret_cast<const float4*>(g_twdw + (i / NS + 1) * (i % NS) * (kTwN / (NS * R))));
    tw_fill<P, S + 1>(tw);
  }
}

// A stage in two halves: pstage_load reads, twiddles and transforms a
// thread's butterflies, pstage_store writes them out (the barrier between
// them is the caller's).  ZIN / ZOUT as fft_core.cuh's stage.
template <class P, int S, bool FWD, int T, bool ZIN, bool ZOUT>
__device__ __forceinline__ void pstage_dft(cdwp* v) {
  using G = PSt<P, S, T>;
  if constexpr (ZIN && S == 0 && G::R % 2 == 0) pdft_half_in<G::R, FWD>(v);
  else if constexpr (ZOUT && S == P::NST - 1 && G::R % 2 == 0) pdft_half_out<G::R, FWD>(v);
  else pdft<G::R, FWD>(v);
}
// ld(p, i): element p, the thread's i-th
template <class P, int S, bool FWD, int T, bool ZIN, bool ZOUT, class Ld>
__device__ __forceinline__ void pstage_load(int t, cdwp (*v)[PSt<P, S, T>::R], const float4* tw, const Ld& ld) {
  using G = PSt<P, S, T>;
  constexpr int RIN = ZIN && S == 0 && G::R % 2 == 0 ? G::R / 2 : G::R;
#pragma unroll
  for (int q = 0; q < G::PER; ++q) {
    const int b = t + q * T;
    if (G::EXACT || b < G::NB) {
#pragma unroll
      for (int r = 0; r < RIN; ++r) v[q][r] = ld(b + r * G::NB, q * RIN + r);
      if constexpr (G::PER > 1) asm volatile("" ::: "memory");  // one butterfly's loads at a time (registers)
      if constexpr (G::NS > 1) {
        const float4* w = tw + (G::NS - P::R[0]) + b % G::NS;
#pragma unroll
        for (int r = 1; r < RIN; ++r) v[q][r] = cmul_tw<FWD>(v[q][r], w[(r - 1) * G::NS]);
      }
      pstage_dft<P, S, FWD, T, ZIN, ZOUT>(v[q]);
    }
  }
}
template <class P, int S, int T, bool ZOUT, class St>
__device__ __forceinline__ void pstage_store(int t, cdwp (*v)[PSt<P, S, T>::R], const St& st) {
  using G = PSt<P, S, T>;
  constexpr int ROUT = ZOUT && S == P::NST - 1 && G::R % 2 == 0 ? G::R / 2 : G::R;
#pragma unroll
  for (int q = 0; q < G::PER; ++q) {
    const int b = t + q * T;
    if (G::EXACT || b < G::NB) {
      const int j = (b / G::NS) * G::NS * G::R + (b % G::NS);
#pragma unroll
      for (int r = 0; r < ROUT; ++r) st(j + r * G::NS, v[q][r]);
    }
  }
}
// stages S .. NST - 2 through shared memory (S >= 1)
template <class P, bool FWD, int T, int S, class SL>
__device__ __forceinline__ void pinner_stages(int t, const float4* tw, const SL& sl) {
  if constexpr (S < P::NST - 1) {
    {
      cdwp v[PSt<P, S, T>::PER][PSt<P, S, T>::R];
      pstage_load<P, S, FWD, T, false, false>(t, v, tw, [&](int p, int) { return sl.get(p); });
      __syncthreads();
      pstage_store<P, S, T, false>(t, v, [&](int p, cdwp x) { sl.put(p, x); });
    }
    __syncthreads();
    pinner_stages<P, FWD, T, S + 1>(t, tw, sl);
  }
}
// the last stage's butterflies into vl
template <class P, bool FWD, int T, bool ZOUT, class SL>
__device__ __forceinline__ void plast_stage(int t, cdwp (*vl)[PSt<P, P::NST - 1, T>::R], const float4* tw, const SL& sl) {
  pstage_load<P, P::NST - 1, FWD, T, false, ZOUT>(t, vl, tw, [&](int p, int) { return sl.get(p); });
}
// A whole transform from `first` into the last stage's registers; `taken` runs
// once a thread has read its inputs, `synced` after the barrier that follows.  The shared tile must be free on entry;
// its last reads end with the call (a barrier is due before anything writes
// it again).
template <class P, bool FWD, int T, bool ZIN, bool ZOUT, class F, class C, class B, class SL>
__device__ __forceinline__ void pfft(int t, cdwp (*vl)[PSt<P, P::NST - 1, T>::R], const float4* tw, const F& first,
                                     const C& taken, const B& synced, const SL& sl) {
  if constexpr (P::NST == 1) {
    pstage_load<P, 0, FWD, T, ZIN, ZOUT>(t, vl, tw, first);
    taken();
    __syncthreads();
    synced();
  } else {
    {
      cdwp v[PSt<P, 0, T>::PER][PSt<P, 0, T>::R];
      pstage_load<P, 0, FWD, T, ZIN, false>(t, v, tw, first);
      taken();
      pstage_store<P, 0, T, false>(t, v, [&](int p, cdwp x) { sl.put(p, x); });
    }
    __syncthreads();
    synced();
    pinner_stages<P, FWD, T, 1>(t, tw, sl);
    plast_stage<P, FWD, T, ZOUT>(t, vl, tw, sl);
  }
}

// Per-thread staging of a tile's inputs by asynchronous copies: slot i of a
// thread is 16 bytes at stg[i * NT] (stg offset by the thread), written and
// read by that thread alone, so its own wait orders the copies (no barrier).
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem, int src_bytes) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(s), "l"(gmem), "r"(src_bytes) : "memory");
}
// elements a thread takes in the first stage of plan P, and f(p, i) for each
template <class P, int T, bool ZIN> constexpr int first_elems() {
  using G = PSt<P, 0, T>;
  return G::PER * (ZIN && G::R % 2 == 0 ? G::R / 2 : G::R);
}
template <class P, int T, bool ZIN, class F> __device__ __forceinline__ void for_first(int t, const F& f) {
  using G = PSt<P, 0, T>;
  constexpr int RIN = ZIN && G::R % 2 == 0 ? G::R / 2 : G::R;
#pragma unroll
  for (int q = 0; q < G::PER; ++q) {
    const int b = t + q * T;
    if (G::EXACT || b < G::NB) {
#pragma unroll
      for (int r = 0; r < RIN; ++r) f(b + r * G::NB, q * RIN + r);
    }
  }
}
// elements a thread holds after the last stage, and f(p, q, r) for each
template <class P, int T> constexpr int last_elems() { return PSt<P, P::NST - 1, T>::PER * P::R[P::NST - 1]; }
template <class P, int T, class F> __device__ __forceinline__ void for_last(int t, const F& f) {
  using L = PSt<P, P::NST - 1, T>;
#pragma unroll
  for (int q = 0; q < L::PER; ++q) {
    const int b = t + q * T;
    if (L::EXACT || b < L::NB) {
#pragma unroll
      for (int r = 0; r < L::R; ++r) f(b + r * L::NB, q, r);
    }
  }
}
// CTAs per SM: `res` threads by registers, and the 228 KB of shared memory
// (1 KB of it reserved per CTA)
constexpr int fit_ctas(int bytes, int res, int nt) {
  const int fit = 233472 / (bytes + 1024), reg = res / nt > 16 ? 16 : res / nt;
  return fit < 1 || reg < 1 ? 1 : (fit < reg ? fit : reg);
}

// ---------------------------------------------------------------- pass 1 --
// Shared memory of each kernel: the exchange tile, the twiddle table, the
// staging slots.
template <int M, int W, bool PAD = true> struct SmR2cDw {
  using G = GeoDw<M>;
  static constexpr int TW = W * G::XCH;
  static constexpr int STG = TW + tw_entries<typename G::P>() * 16;
  static constexpr int Q = STG + first_elems<typename G::P, G::T, PAD>() * 16 * G::T * W;
  static constexpr int BYTES = Q + (int)sizeof(TileQueue);
  static constexpr int MINB = fit_ctas(BYTES, G::RES, G::T * W);
};
template <int M, int W, bool PAD = true>
__global__ void __launch_bounds__(GeoDw<M>::T* W, SmR2cDw<M, W, PAD>::MINB) kd_r2c_ax0(const Jobs jobs, long long C) {
  using G = GeoDw<M>;
  using P = typename G::P;
  using SM = SmR2cDw<M, W, PAD>;
  constexpr int T = G::T, NT = T * W, NV = PAD ? M / 2 : M, K = M / 2 + 1, LS = P::NST - 1;
  extern __shared__ __align__(16) unsigned char smraw[];
  float4* tw = reinterpret_cast<float4*>(smraw + SM::TW);
  double2* stg = reinterpret_cast<double2*>(smraw + SM::STG) + threadIdx.x;
  const int l = threadIdx.x % W, t = threadIdx.x / W;
  const PLine<W> sl{reinterpret_cast<cdwp*>(smraw) + l};
  const long long tpj = (C + 2 * W - 1) / (2 * W);
  auto issue = [&](long long tile) {  // columns c, c + 1 as one complex line
    const long long c = (tile % tpj) * (2 * W) + 2 * l;
    const double* rho = static_cast<const double*>(jobs.j[tile / tpj].in);
    for_first<P, T, PAD>(t, [&](int p, int i) {
      const bool ok = p < NV && c < C;
      cp_async16(&stg[i * NT], ok ? rho + (long long)p * C + c : rho, ok ? 16 : 0);
    });
  };
  TileQueue* tq = reinterpret_cast<TileQueue*>(smraw + SM::Q);
  if (threadIdx.x == 0) tile_queue_init(tq);
  issue(blockIdx.x);
  cp_async_commit();
  tw_fill<P, 1>(tw);
  __syncthreads();
  int next = 0;
  unsigned par = 0;
  for (long long tile = blockIdx.x; tile >= 0; tile = next, par ^= 1) {
    const long long c = (tile % tpj) * (2 * W) + 2 * l;
    cp_async_wait_all();
    cdwp v[PSt<P, LS, T>::PER][PSt<P, LS, T>::R];
    pfft<P, true, T, PAD, false>(
        t, v, tw,
        [&](int, int i) -> cdwp {
          const double2 a = stg[i * NT];
          return mkp(dw_from_double(a.x), dw_from_double(a.y));
        },
        [&] {
          if (threadIdx.x == 0) tile_answer(tq, par, jobs.fault);
        },
        [&] {
          next = tq->next;
          if (next >= 0) {
            issue(next);
            if (threadIdx.x == 0) tile_request(tq);
          }
          cp_async_commit();
        },
        sl);
    if (P::NST > 1) __syncthreads();
    pstage_store<P, LS, T, false>(t, v, [&](int p, cdwp x) { sl.put(p, x); });
    __syncthreads();
    // Z = DFT(a + i b): A[k] = (Z[k] + conj Z[M-k]) / 2, B[k] = (Z[k] - conj Z[M-k]) / 2i
    if (c < C) {
      cdwp* __restrict__ X = static_cast<cdwp*>(jobs.j[tile / tpj].out) + c;
      for (int k = t; k < K; k += T) {
        const cdwp zk = sl.get(k), zm = conjp(sl.get((M - k) % M));
        X[(long long)k * C] = canonp(halfp(cadd(zk, zm)));
        X[(long long)k * C + 1] = canonp(halfp(rotp<true>(csub(zk, zm))));
      }
    }
    __syncthreads();
  }
  cp_async_wait_all();
}

// ----------------------------------------------------------- passes 2, 4 --
// The row passes: forward (rows of n values padded to M) and inverse (rows of
// M values cropped to n).  PAD = false: M values in and out.
template <int M, int W, bool FWD, bool PAD> struct SmRowDw {
  using G = GeoDw<M>;
  using P = typename G::P;
  static constexpr int TW = W * G::XCH;
  static constexpr int STG = TW + tw_entries<P>() * 16;
  static constexpr int Q = STG + first_elems<P, G::T, FWD && PAD>() * 16 * G::T * W;
  static constexpr int BYTES = Q + (int)sizeof(TileQueue);
  static constexpr int MINB = fit_ctas(BYTES, G::RES, G::T * W);
};
template <int M, int W, bool FWD, bool PAD = true>
__global__ void __launch_bounds__(GeoDw<M>::T* W, SmRowDw<M, W, FWD, PAD>::MINB)
    kd_row(const Jobs jobs, long long rows) {
  using G = GeoDw<M>;
  using SM = SmRowDw<M, W, FWD, PAD>;
  using P = typename G::P;
  constexpr int T = G::T, NT = T * W, LS = P::NST - 1;
  constexpr int NI = FWD && PAD ? M / 2 : M, NO = !FWD && PAD ? M / 2 : M;  // values of a row in, out
  extern __shared__ __align__(16) unsigned char smraw[];
  float4* tw = reinterpret_cast<float4*>(smraw + SM::TW);
  cdwp* stg = reinterpret_cast<cdwp*>(smraw + SM::STG) + threadIdx.x;
  const int t = threadIdx.x % T, l = threadIdx.x / T;
  const PLine<1> sl{reinterpret_cast<cdwp*>(smraw) + l * M};
  const long long tpj = (rows + W - 1) / W;
  auto issue = [&](long long tile) {
    const long long row = (tile % tpj) * W + l;
    const cdwp* in = static_cast<const cdwp*>(jobs.j[tile / tpj].in);
    for_first<P, T, FWD && PAD>(t, [&](int p, int i) {
      const bool ok = p < NI && row < rows;
      cp_async16(&stg[i * NT], ok ? in + row * NI + p : in, ok ? 16 : 0);
    });
  };
  TileQueue* tq = reinterpret_cast<TileQueue*>(smraw + SM::Q);
  if (threadIdx.x == 0) tile_queue_init(tq);
  issue(blockIdx.x);
  cp_async_commit();
  tw_fill<P, 1>(tw);
  __syncthreads();
  int next = 0;
  unsigned par = 0;
  for (long long tile = blockIdx.x; tile >= 0; tile = next, par ^= 1) {
    const long long row = (tile % tpj) * W + l;
    const bool ok = row < rows;
    cdwp* __restrict__ y = static_cast<cdwp*>(jobs.j[tile / tpj].out) + row * NO;
    cp_async_wait_all();
    cdwp v[PSt<P, LS, T>::PER][PSt<P, LS, T>::R];
    pfft<P, FWD, T, FWD && PAD, !FWD && PAD>(
        t, v, tw, [&](int, int i) -> cdwp { return stg[i * NT]; },
        [&] {
          if (threadIdx.x == 0) tile_answer(tq, par, jobs.fault);
        },
        [&] {
          next = tq->next;
          if (next >= 0) {
            issue(next);
            if (threadIdx.x == 0) tile_request(tq);
          }
          cp_async_commit();
        },
        sl);
    pstage_store<P, LS, T, !FWD && PAD>(t, v, [&](int p, cdwp z) {
      if (p < NO && ok) y[p] = canonp(z);
    });
    __syncthreads();
  }
  cp_async_wait_all();
}

// ---------------------------------------------------- the middle transform --
// Forward, multiply, inverse of one line: `first`, `taken`, `synced` as pfft; mul(k1,
// q, r) returns the real factor of element k1; last(p, v) stores p < n.
// Both directions run the inner stages through one copy of the code: the
// inverse transform is the forward one of the values with their parts
// swapped.
template <class P, int T, bool PAD, class F, class C, class B, class Mu, class L, class SL>
__device__ __forceinline__ void pmiddle(int t, const float4* tw, const F& first, const C& taken, const B& synced,
                                        const Mu& mul, const L& last, const SL& sl) {
  constexpr int LS = P::NST - 1;
  cdwp v[PSt<P, LS, T>::PER][PSt<P, LS, T>::R];
  auto scale = [&] {
    for_last<P, T>(t, [&](int k1, int q, int r) { v[q][r] = swapp(cscale(v[q][r], mul(k1, q, r))); });
  };
  if constexpr (P::NST == 1) {
    static_assert(T == 1, "one butterfly");
    pstage_load<P, 0, true, T, PAD, false>(t, v, tw, first);
    taken();
    __syncthreads();
    synced();
    scale();
    pstage_dft<P, 0, true, T, false, PAD>(v[0]);
  } else {
    {
      cdwp w[PSt<P, 0, T>::PER][PSt<P, 0, T>::R];
      pstage_load<P, 0, true, T, PAD, false>(t, w, tw, first);
      taken();
      pstage_store<P, 0, T, false>(t, w, [&](int p, cdwp x) { sl.put(p, x); });
    }
#pragma unroll 1
    for (int dir = 0;; ++dir) {
      __syncthreads();
      if (dir == 0) synced();
      pinner_stages<P, true, T, 1>(t, tw, sl);
      if (dir == 1) break;
      plast_stage<P, true, T, false>(t, v, tw, sl);
      scale();
      using G = PSt<P, 0, T>;
#pragma unroll
      for (int q = 0; q < G::PER; ++q)
        if (G::EXACT || t + q * T < G::NB) pdft<G::R, true>(v[q]);
      __syncthreads();  // the tile is free (last-stage reads)
      pstage_store<P, 0, T, false>(t, v, [&](int p, cdwp x) { sl.put(p, x); });
    }
    plast_stage<P, true, T, PAD>(t, v, tw, sl);
  }
  pstage_store<P, LS, T, PAD>(t, v, [&](int p, cdwp x) { last(p, swapp(x)); });
}

// ---------------------------------------------------------------- pass 3 --
template <int M, int W, bool PAD> struct SmMidDw {
  using G = GeoDw<M>;
  using P = typename G::P;
  static constexpr int TW = W * G::XCH;
  static constexpr int STG = TW + tw_entries<P>() * 16;
  // a thread's input slots hold its spectrum values (8 bytes each) from the
  // first stage's reads to the next tile's copies
  static constexpr int IN = first_elems<P, G::T, PAD>() * 16, SP = (last_elems<P, G::T>() + 1) / 2 * 16;
  static constexpr int Q = STG + (IN > SP ? IN : SP) * G::T * W;
  static constexpr int BYTES = Q + (int)sizeof(TileQueue);
  static constexpr int MINB = fit_ctas(BYTES, G::RES_MID, G::T * W);
};

// A tile is W adjacent columns k2 of one plane k0.  MODE as k_col_mid.
template <int M, int W, int MODE = kMulSpectrum>
__global__ void __launch_bounds__(GeoDw<M>::T* W, SmMidDw<M, W, MODE != kMulDdiGrid>::MINB)
    kd_col_mid(const Jobs jobs, int M2, int planes) {
  using G = GeoDw<M>;
  using P = typename G::P;
  constexpr bool PAD = MODE != kMulDdiGrid;
  using SM = SmMidDw<M, W, PAD>;
  constexpr int T = G::T, NT = T * W, n = PAD ? M / 2 : M, RL = P::R[P::NST - 1];
  extern __shared__ __align__(16) unsigned char smraw[];
  float4* tw = reinterpret_cast<float4*>(smraw + SM::TW);
  cdwp* stg = reinterpret_cast<cdwp*>(smraw + SM::STG) + threadIdx.x;
  // spectrum value e of this thread: half a slot of its own
  auto sslot = [&](int e) { return reinterpret_cast<float2*>(stg + (e >> 1) * NT) + (e & 1); };
  const int l = threadIdx.x % W, t = threadIdx.x / W;
  const PLine<W> sl{reinterpret_cast<cdwp*>(smraw) + l};
  const int tpp = (M2 + W - 1) / W;
  const long long tpj = (long long)tpp * planes;
  const int n2 = M2 / 2;
  auto issue = [&](long long tile) {
    const int lt = (int)(tile % tpj);
    const int k0 = lt / tpp, k2 = (lt % tpp) * W + l;
    const cdwp* Y = static_cast<const cdwp*>(jobs.j[tile / tpj].out);
    const cdwp* col = Y + (long long)k0 * n * M2 + k2;
    for_first<P, T, PAD>(t, [&](int p, int i) {
      const bool ok = p < n && k2 < M2;
      cp_async16(&stg[i * NT], ok ? col + (long long)p * M2 : Y, ok ? 16 : 0);
    });
  };
  TileQueue* tq = reinterpret_cast<TileQueue*>(smraw + SM::Q);
  if (threadIdx.x == 0) tile_queue_init(tq);
  issue(blockIdx.x);
  cp_async_commit();
  tw_fill<P, 1>(tw);
  __syncthreads();
  int next = 0;
  unsigned par = 0;
  for (long long tile = blockIdx.x; tile >= 0; tile = next, par ^= 1) {
    const Job& jb = jobs.j[tile / tpj];
    const int lt = (int)(tile % tpj);
    const int k0 = lt / tpp, k2 = (lt % tpp) * W + l;
    const bool ok = k2 < M2;
    cdwp* __restrict__ col = static_cast<cdwp*>(jb.out) + (long long)k0 * n * M2 + k2;
    DdiLine<cdw> ddi;
    cp_async_wait_all();
    pmiddle<P, T, PAD>(
        t, tw, [&](int, int i) -> cdwp { return stg[i * NT]; },
        [&] {
          if constexpr (PAD) {
            const float2* S = static_cast<const float2*>(jb.S) + (long long)k0 * (n + 1) * (n2 + 1);
            const float2* s0 = S + (ok ? min(k2, M2 - k2) : 0);
            for_last<P, T>(t, [&](int k1, int q, int r) {
              cp_async8(sslot(q * RL + r), s0 + min(k1, M - k1) * (n2 + 1), 8);
            });
            cp_async_commit();
          }
          if (threadIdx.x == 0) tile_answer(tq, par, jobs.fault);
        },
        [&] {
          next = tq->next;
          if (next >= 0 && threadIdx.x == 0) tile_request(tq);
        },
        [&](int k1, int q, int r) -> dw {
          if (q == 0 && r == 0) {
            cp_async_wait_all();
            if constexpr (MODE != kMulSpectrum) ddi.init(jb.par, k0, ok ? k2 : 0, M2);
          }
          dw s(0);
          if constexpr (PAD) {
            const float2 f = *sslot(q * RL + r);
            s = dw(f.x, f.y);
          }
          if constexpr (MODE != kMulSpectrum) s = ddi.template value<MODE>(s, k1, M);
          return s;
        },
        [&](int p, cdwp z) {
          if (p < n && ok) col[(long long)p * M2] = canonp(z);
        },
        sl);
    if (next >= 0) issue(next);
    cp_async_commit();
    __syncthreads();
  }
  cp_async_wait_all();
}

// ------------------------------------------------- middle pass, d = 2 --
template <int M, int W> struct SmRowMidDw {
  using G = GeoDw<M>;
  static constexpr int TW = W * G::XCH;
  static constexpr int BYTES = TW + tw_entries<typename G::P>() * 16;
};
template <int M, int W>
__global__ void __launch_bounds__(GeoDw<M>::T* W) kd_row_mid(const Jobs jobs, long long rows) {
  using G = GeoDw<M>;
  using P = typename G::P;
  constexpr int T = G::T, n = M / 2, RL = P::R[P::NST - 1];
  extern __shared__ __align__(16) unsigned char smraw[];
  float4* tw = reinterpret_cast<float4*>(smraw + SmRowMidDw<M, W>::TW);
  const int t = threadIdx.x % T, l = threadIdx.x / T;
  const PLine<1> sl{reinterpret_cast<cdwp*>(smraw) + l * M};
  const long long tpj = (rows + W - 1) / W;
  tw_fill<P, 1>(tw);
  __syncthreads();
  for (long long tile = blockIdx.x; tile < tpj * jobs.count; tile += gridDim.x) {
    const Job& jb = jobs.j[tile / tpj];
    const long long row = (tile % tpj) * W + l;
    const bool ok = row < rows;
    cdwp* __restrict__ x = static_cast<cdwp*>(jb.out) + row * n;
    const float2* __restrict__ s0 = static_cast<const float2*>(jb.S) + (ok ? row : 0) * (n + 1);
    float2 sp[last_elems<P, T>()];  // the spectrum values, loaded ahead of the transform
    for_last<P, T>(t, [&](int k1, int q, int r) { sp[q * RL + r] = __ldg(s0 + min(k1, M - k1)); });
    pmiddle<P, T, true>(
        t, tw, [&](int p, int) -> cdwp { return p < n && ok ? x[p] : zerop(); }, [] {}, [] {},
        [&](int, int q, int r) -> dw { return dw(sp[q * RL + r].x, sp[q * RL + r].y); },
        [&](int p, cdwp z) {
          if (p < n && ok) x[p] = canonp(z);
        },
        sl);
    __syncthreads();
  }
}

// ---------------------------------------------------------------- pass 5 --
// EPI: the output is phi + beta * rho (rho = jb.aux); an element of rho is
// read by the thread that writes the same element of phi, just before (phi
// may be rho).
template <int M, int W> struct SmC2rDw {
  using G = GeoDw<M>;
  static constexpr int TW = W * G::XCH;
  static constexpr int Q = TW + tw_entries<typename G::P>() * 16;
  static constexpr int BYTES = Q + (int)sizeof(TileQueue);
  static constexpr int MINB = fit_ctas(BYTES, G::RES, G::T * W);
};
template <int M, int W, bool PAD = true, bool EPI = false>
__global__ void __launch_bounds__(GeoDw<M>::T* W, SmC2rDw<M, W>::MINB) kd_c2r_ax0(const Jobs jobs, long long C) {
  using G = GeoDw<M>;
  using P = typename G::P;
  constexpr int T = G::T, n = M / 2, NV = PAD ? M / 2 : M, LS = P::NST - 1;
  extern __shared__ __align__(16) unsigned char smraw[];
  float4* tw = reinterpret_cast<float4*>(smraw + SmC2rDw<M, W>::TW);
  TileQueue* tq = reinterpret_cast<TileQueue*>(smraw + SmC2rDw<M, W>::Q);
  const int l = threadIdx.x % W, t = threadIdx.x / W;
  const PLine<W> sl{reinterpret_cast<cdwp*>(smraw) + l};
  const long long tpj = (C + 2 * W - 1) / (2 * W);
  if (threadIdx.x == 0) tile_queue_init(tq);
  tw_fill<P, 1>(tw);
  __syncthreads();
  int next = 0;
  unsigned par = 0;
  for (long long tile = blockIdx.x; tile >= 0; tile = next, par ^= 1) {
    const Job& jb = jobs.j[tile / tpj];
    const long long c = (tile % tpj) * (2 * W) + 2 * l;
    const bool ok = c < C;
    const cdwp* __restrict__ X = static_cast<const cdwp*>(jb.in) + c;
    cdwp v[PSt<P, LS, T>::PER][PSt<P, LS, T>::R];
    // Z[k] = A[k] + i B[k] with A, B Hermitian: rebuild k > n from M - k.
    pfft<P, false, T, false, PAD>(
        t, v, tw,
        [&](int k, int) -> cdwp {
          if (!ok) return zerop();
          const bool lo = k <= n;
          const cdwp* q = X + (long long)(lo ? k : M - k) * C;
          const cdwp a = q[0], b = q[1];
          return lo ? cadd(a, rotp<false>(b)) : cadd(conjp(a), swapp(b));
        },
        [&] {
          if (threadIdx.x == 0) tile_answer(tq, par, jobs.fault);
        },
        [&] {
          next = tq->next;
          if (next >= 0 && threadIdx.x == 0) tile_request(tq);
        },
        sl);
    double* phi = static_cast<double*>(jb.out) + c;
    const double* rho = nullptr;
    double beta = 0.0;
    if constexpr (EPI) {
      rho = static_cast<const double*>(jb.aux) + c;
      beta = ddi_beta<double>(jb.par);
    }
    pstage_store<P, LS, T, PAD>(t, v, [&](int p, cdwp z) {
      if (p >= NV || !ok) return;
      const long long o = (long long)p * C;
      dw a, b;
      partsp(z, a, b);
      double2 f = make_double2(dw_to_double(a), dw_to_double(b));
      if constexpr (EPI) {
        const double2 r0 = *reinterpret_cast<const double2*>(rho + o);
        f = make_double2(f.x + beta * r0.x, f.y + beta * r0.y);
      }
      *reinterpret_cast<double2*>(phi + o) = f;
    });
    __syncthreads();
  }
}

}  // namespace fsa
