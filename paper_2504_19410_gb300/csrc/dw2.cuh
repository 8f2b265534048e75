// Paired double-word complex arithmetic: a complex double-word value as two
// register pairs h = (re.hi, im.hi), l = (re.lo, im.lo), so that every FP32
// operation of the double-word building blocks (dw.cuh) issues as ONE paired
// instruction of sm_100 and later (add / sub / mul / fma .rn.f32x2) for both
// parts.  Each half runs the operations of dw.cuh; signs are folded into the
// operands (x - y for x + (-y), a product with -b for a negated product),
// which rounds alike.
//
// Pairing the parts of one value (and not two lines) keeps eight values of a
// radix-8 butterfly in 32 registers, so 32 warps fit on an SM; the swaps that
// multiplications by -i need and the broadcasts of the complex products run
// on the ALU pipe, which the double-word arithmetic leaves idle.
#pragma once
#include "fft_core.cuh"

namespace fsa {

using f2p = unsigned long long;  // two packed floats, first one low

__device__ __forceinline__ f2p pk2(float a, float b) {
  f2p r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpk2(f2p v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ f2p add2(f2p a, f2p b) {
  f2p r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2p sub2(f2p a, f2p b) {
  f2p r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2p mul2(f2p a, f2p b) {
  f2p r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2p fma2(f2p a, f2p b, f2p c) {
  f2p r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f2p neg2(f2p a) { return a ^ 0x8000000080000000ull; }
__device__ __forceinline__ f2p conj2(f2p a) { return a ^ 0x8000000000000000ull; }  // second part negated
__device__ __forceinline__ f2p swap2(f2p a) {
  float x, y;
  unpk2(a, x, y);
  return pk2(y, x);
}
// (y, -x) forward, (-y, x) inverse
template <bool FWD> __device__ __forceinline__ f2p rot2(f2p a) {
  float x, y;
  unpk2(a, x, y);
  return FWD ? pk2(y, -x) : pk2(-y, x);
}

// 16 bytes in HBM and shared memory: (re.hi, im.hi, re.lo, im.lo)
struct __align__(16) cdwp {
  f2p h, l;
};
__device__ __forceinline__ cdwp mkp(f2p h, f2p l) {
  cdwp r;
  r.h = h;
  r.l = l;
  return r;
}
__device__ __forceinline__ cdwp mkp(dw x, dw y) { return mkp(pk2(x.hi, y.hi), pk2(x.lo, y.lo)); }
__device__ __forceinline__ cdwp zerop() { return mkp(0ull, 0ull); }
__device__ __forceinline__ void partsp(cdwp v, dw& x, dw& y) {
  unpk2(v.h, x.hi, y.hi);
  unpk2(v.l, x.lo, y.lo);
}

// TwoSum of a and b, and of a and -b
__device__ __forceinline__ cdwp two_sum2(f2p a, f2p b) {
  const f2p s = add2(a, b), bb = sub2(s, a);
  return mkp(s, add2(sub2(a, sub2(s, bb)), sub2(b, bb)));
}
__device__ __forceinline__ cdwp two_diff2(f2p a, f2p b) {
  const f2p s = sub2(a, b), bb = sub2(s, a);
  return mkp(s, sub2(sub2(a, sub2(s, bb)), add2(b, bb)));
}
// Canonical form of a value leaving a pass for HBM.  The double-word
// operations skip their closing renormalisation, so a low part can grow past
// half an ulp of its high part over many operations; one TwoSum per part at
// each pass boundary bounds that growth to the operations of one pass.
__device__ __forceinline__ cdwp canonp(cdwp v) { return two_sum2(v.h, v.l); }
__device__ __forceinline__ cdwp cadd(cdwp a, cdwp b) {
  const cdwp s = two_sum2(a.h, b.h);
  return mkp(s.h, add2(s.l, add2(a.l, b.l)));
}
__device__ __forceinline__ cdwp csub(cdwp a, cdwp b) {
  const cdwp s = two_diff2(a.h, b.h);
  return mkp(s.h, add2(s.l, sub2(a.l, b.l)));
}
template <bool FWD> __device__ __forceinline__ cdwp rotp(cdwp a) { return mkp(rot2<FWD>(a.h), rot2<FWD>(a.l)); }
__device__ __forceinline__ cdwp conjp(cdwp a) { return mkp(conj2(a.h), conj2(a.l)); }
__device__ __forceinline__ cdwp swapp(cdwp a) { return mkp(swap2(a.h), swap2(a.l)); }
// exact halving
__device__ __forceinline__ cdwp halfp(cdwp x) {
  const f2p h = 0x3f0000003f000000ull;
  return mkp(mul2(x.h, h), mul2(x.l, h));
}
// both parts times the double-word real s
__device__ __forceinline__ cdwp cscale(cdwp a, dw s) {
  const f2p sh = pk2(s.hi, s.hi), sl = pk2(s.lo, s.lo), nsh = pk2(-s.hi, -s.hi);
  const f2p ch = mul2(a.h, sh);
  const f2p e = fma2(a.h, nsh, ch);  // minus the product's error
  return mkp(ch, sub2(fma2(a.l, sh, fma2(a.h, sl, mul2(a.l, sl))), e));
}
// a w (FWD) or a conj(w), w = (x.hi, y.hi, x.lo, y.lo).  Each part is a fused
// two-term dot product a b + c d: the two leading products exact (2Prod by
// FMA), summed by TwoSum, with the products' errors and the cross terms
// a.hi b.lo, a.lo b.hi, c.hi d.lo, c.lo d.hi folded in by FMA (a.lo b.lo and
// c.lo d.lo, of order u^2 |a b| and u^2 |c d|, are dropped): 16 operations
// against 20 for two multiplications and an addition.  The low parts are
// summed negated, which saves negating the products.
template <bool FWD> __device__ __forceinline__ cdwp cmul_tw(cdwp a, float4 w) {
  const float yh = FWD ? w.y : -w.y, yl = FWD ? w.w : -w.w;
  const f2p W = pk2(w.x, yh), nW = pk2(-w.x, -yh), nWl = pk2(-w.z, -yl);  // (x, y)
  const f2p V = pk2(-yh, w.x), nV = pk2(yh, -w.x), nVl = pk2(yl, -w.z);   // (-y, x)
  float xh, yyh, xl, yyl;
  unpk2(a.h, xh, yyh);
  unpk2(a.l, xl, yyl);
  const f2p Xh = pk2(xh, xh), Yh = pk2(yyh, yyh), Xl = pk2(xl, xl), Yl = pk2(yyl, yyl);
  const f2p p = mul2(Xh, W), q = mul2(Yh, V);
  f2p t = add2(fma2(Xh, nW, p), fma2(Yh, nV, q));  // minus the products' errors
  const cdwp s = two_sum2(p, q);
  t = fma2(Xh, nWl, t);
  t = fma2(Xl, nW, t);
  t = fma2(Yh, nVl, t);
  t = fma2(Yl, nV, t);
  return mkp(s.h, sub2(s.l, t));
}

// ------------------------------------------------------------ codelets ----
// The codelets of fft_core.cuh over cdwp.
template <bool FWD> __device__ __forceinline__ void pdft3(cdwp* v) {
  const dw s(0.86602540378443864676372317075294);  // sin(2 pi / 3)
  const cdwp t1 = cadd(v[1], v[2]);
  const cdwp t2 = csub(v[0], halfp(t1));
  const cdwp d = rotp<FWD>(cscale(csub(v[1], v[2]), s));
  v[0] = cadd(v[0], t1);
  v[1] = cadd(t2, d);
  v[2] = csub(t2, d);
}
template <bool FWD> __device__ __forceinline__ void pdft4(cdwp* v) {
  const cdwp a = cadd(v[0], v[2]), b = csub(v[0], v[2]);
  const cdwp c = cadd(v[1], v[3]), d = rotp<FWD>(csub(v[1], v[3]));
  v[0] = cadd(a, c);
  v[2] = csub(a, c);
  v[1] = cadd(b, d);
  v[3] = csub(b, d);
}
// outputs 0 and 1 of pdft4
template <bool FWD> __device__ __forceinline__ void pdft4_lo2(const cdwp* v, cdwp& o0, cdwp& o1) {
  const cdwp a = cadd(v[0], v[2]), b = csub(v[0], v[2]);
  const cdwp c = cadd(v[1], v[3]), d = rotp<FWD>(csub(v[1], v[3]));
  o0 = cadd(a, c);
  o1 = cadd(b, d);
}
// b_k *= w8^k: (1 -+ i)/sqrt(2) = (b + rot b) / sqrt(2)
template <bool FWD> __device__ __forceinline__ void prot8(cdwp* b) {
  const dw h(0.70710678118654752440084436210485);  // 1/sqrt(2)
  b[1] = cscale(cadd(b[1], rotp<FWD>(b[1])), h);
  b[3] = rotp<FWD>(cscale(cadd(b[3], rotp<FWD>(b[3])), h));
  b[2] = rotp<FWD>(b[2]);
}
template <bool FWD> __device__ __forceinline__ void pdft8_tail(cdwp* a, cdwp* b, cdwp* v) {
  prot8<FWD>(b);
  pdft4<FWD>(a);
  pdft4<FWD>(b);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    v[2 * q] = a[q];
    v[2 * q + 1] = b[q];
  }
}
template <bool FWD> __device__ __forceinline__ void pdft8(cdwp* v) {
  cdwp a[4], b[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    a[k] = cadd(v[k], v[k + 4]);
    b[k] = csub(v[k], v[k + 4]);
  }
  pdft8_tail<FWD>(a, b, v);
}
// Good-Thomas 2 x 3: inputs (3 a + 2 b) mod 6, outputs (3 a' + 4 b') mod 6
template <bool FWD> __device__ __forceinline__ void pdft6(cdwp* v) {
  cdwp e[3] = {v[0], v[2], v[4]}, o[3] = {v[3], v[5], v[1]};
  pdft3<FWD>(e);
  pdft3<FWD>(o);
  v[0] = cadd(e[0], o[0]);
  v[3] = csub(e[0], o[0]);
  v[4] = cadd(e[1], o[1]);
  v[1] = csub(e[1], o[1]);
  v[2] = cadd(e[2], o[2]);
  v[5] = csub(e[2], o[2]);
}
template <int R, bool FWD> __device__ __forceinline__ void pdft(cdwp* v) {
  if constexpr (R == 2) {
    const cdwp a = v[0];
    v[0] = cadd(a, v[1]);
    v[1] = csub(a, v[1]);
  } else if constexpr (R == 3) {
    pdft3<FWD>(v);
  } else if constexpr (R == 4) {
    pdft4<FWD>(v);
  } else if constexpr (R == 6) {
    pdft6<FWD>(v);
  } else {
    static_assert(R == 8, "unsupported radix");
    pdft8<FWD>(v);
  }
}
// the upper half of the inputs is zero (fft_core.cuh's dft_half_in)
template <int R, bool FWD> __device__ __forceinline__ void pdft_half_in(cdwp* v) {
  if constexpr (R == 2) {
    v[1] = v[0];
  } else if constexpr (R == 4) {
    const cdwp a = v[0], c = v[1], d = rotp<FWD>(v[1]);
    v[0] = cadd(a, c);
    v[2] = csub(a, c);
    v[1] = cadd(a, d);
    v[3] = csub(a, d);
  } else {
    static_assert(R == 8, "pruned codelet radix");
    cdwp a[4], b[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) a[k] = b[k] = v[k];
    pdft8_tail<FWD>(a, b, v);
  }
}
// only the outputs v[0 .. R/2) are formed (fft_core.cuh's dft_half_out)
template <int R, bool FWD> __device__ __forceinline__ void pdft_half_out(cdwp* v) {
  if constexpr (R == 2) {
    v[0] = cadd(v[0], v[1]);
  } else if constexpr (R == 4) {
    pdft4_lo2<FWD>(v, v[0], v[1]);
  } else {
    static_assert(R == 8, "pruned codelet radix");
    cdwp a[4], b[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      a[k] = cadd(v[k], v[k + 4]);
      b[k] = csub(v[k], v[k + 4]);
    }
    prot8<FWD>(b);
    pdft4_lo2<FWD>(a, v[0], v[2]);
    pdft4_lo2<FWD>(b, v[1], v[3]);
  }
}

}  // namespace fsa
