// Device helpers for runtime-compiled segment kernels: the pair and quad
// updates of gates on local qubits (Sec. 2, Fig. 1a) written for a tile held
// in registers.
//
// A compiled segment is straight-line code: every register index, layout,
// control pattern and coefficient offset is a constant of its source, so the
// kernel carries none of the register-tile interpreter's per-op dispatch.
// The helpers here are the pair and quad updates it is written in; they use
// the same arithmetic policies (arith.cuh) as every other kernel of the
// library, so a compiled segment and the interpreter compute the same
// products and sums.
#pragma once
#include "arith.cuh"
#include "tile.cuh"

namespace lqs {
namespace jit {

// Amplitude updates of a compiled segment.  For double-float they return the
// accumulator pair (leading sum, collected errors) without renormalising it:
// that pair stands for the same value, and the next product, sum or float64
// conversion takes it as it is (3 fewer float32 instructions per real
// output).  The low parts then grow with every update, so the segment
// renormalises every register after a bounded number of updates (renorm).
// The other policies have no renormalisation to skip.
template <class A> struct Lz {
  using W = typename A::W;
  using C = typename A::C;
  using R = typename A::R;
  static __device__ __forceinline__ W cmul(const C& c, const W& a) { return A::cmul(c, a); }
  static __device__ __forceinline__ W cmac2(const C& c0, const W& a, const C& c1, const W& b) {
    return A::cmac2(c0, a, c1, b);
  }
  static __device__ __forceinline__ W cmac4(const C* c, const W* a) { return A::cmac4(c, a); }
  static __device__ __forceinline__ W rmac2(const R& c0, const W& a, const R& c1, const W& b) {
    return A::rmac2(c0, a, c1, b);
  }
  static __device__ __forceinline__ C kmul(const C& a, const C& b) { return A::kmul(a, b); }
  static __device__ __forceinline__ C kmuln(const C& a, const C& b) { return A::kmul(a, b); }  // normalised
  static __device__ __forceinline__ void renorm(W&) {}
  // SX x + k y for a real k
  template <int SX>
  static __device__ __forceinline__ W uma(const W& x, const R& k, const W& y) {
    W r;
    r.x = k * y.x + (SX > 0 ? x.x : -x.x);
    r.y = k * y.y + (SX > 0 ? x.y : -x.y);
    return r;
  }
  static __device__ __forceinline__ W rscale(const R& g, const W& x) {
    W r;
    r.x = g * x.x;
    r.y = g * x.y;
    return r;
  }
  // x + SY y
  template <int SY>
  static __device__ __forceinline__ W uadd(const W& x, const W& y) {
    W r;
    r.x = SY > 0 ? x.x + y.x : x.x - y.x;
    r.y = SY > 0 ? x.y + y.y : x.y - y.y;
    return r;
  }
};
}  // namespace jit

// 128-bit shared-memory and global accesses of working amplitudes.
__device__ __forceinline__ void st_w(P2* p, const P2& v) {
  *reinterpret_cast<ulonglong2*>(p) = make_ulonglong2(v.h, v.l);
}
__device__ __forceinline__ P2 ld_w(const P2* p) {
  const ulonglong2 f = *reinterpret_cast<const ulonglong2*>(p);
  return P2{f.x, f.y};
}

namespace jit {
// A real coefficient; nh = -h, so that a product's error term needs no
// negation of the product.
struct R2 { f2 h, nh, l; };

// The policy of compiled complex128 double-float segments: ArDF's storage and
// coefficients, packed working amplitudes.
struct ArDFP {
  using S = double2;
  using W = P2;
  using C = DFK;
  using R = R2;
  static __device__ __forceinline__ W load(const S& s) {
    const DF re = d2df(s.x), im = d2df(s.y);
    return W{f2_pack(re.h, im.h), f2_pack(re.l, im.l)};
  }
  static __device__ __forceinline__ S store(const W& w) {
    DF re, im;
    p2_lanes(w, re, im);
    return make_double2(df2d(re), df2d(im));
  }
  static __device__ __forceinline__ C kmul(const C& a, const C& b) { return ArDF::kmul(a, b); }
  static __device__ __forceinline__ C cconst1() { return ArDF::cconst1(); }
  static __device__ __forceinline__ W neg(const W& a) { return p2_neg(a); }
  static __device__ __forceinline__ W mul_i(const W& a) {
    return W{f2_swap(f2_conj(a.h)), f2_swap(f2_conj(a.l))};
  }
};
template <> struct Lz<ArDFP> {
  using W = P2;
  // c (re, im) = (re, im) * (cr, cr) + (im, re) * (-ci, ci)
  struct K2 { P2 c, s; };
  static __device__ __forceinline__ K2 k2(const DFK& c) {
    return K2{P2{f2_dup(c.re.h), f2_dup(c.re.l)}, P2{f2_pack(-c.im.h, c.im.h), f2_pack(-c.im.l, c.im.l)}};
  }
  static __device__ __forceinline__ PAcc cprod(const K2& c, const W& a) {
    PAcc A = p2_prod(a, c.c);
    p2_mac(A, p2_swap(a), c.s);
    return A;
  }
  static __device__ __forceinline__ W cmul(const DFK& c, const W& a) { return p2_raw(cprod(k2(c), a)); }
  // Dense complex rows, two packed products per coefficient: results are those
  // of the scalar rows bit for bit, in half the instructions.  24 qubits, scalar
  // against packed: reverse sweep of 4 layers RX + RZ 18.7 -> 14.7 ms, of 3 brick
  // layers of U4 12.7 -> 9.4, forward 4 layers RX + RZ 6.4 -> 5.1, U4 windows
  // 5.1 -> 4.5; a reverse segment of RX gates builds in 6 s instead of 13.
  static __device__ __forceinline__ void cmac(PAcc& A, const K2& c, const W& a) {
    p2_mac(A, a, c.c);
    p2_mac(A, p2_swap(a), c.s);
  }
  static __device__ __forceinline__ W cmac2(const DFK& c0, const W& a, const DFK& c1, const W& b) {
    PAcc A = cprod(k2(c0), a);
    cmac(A, k2(c1), b);
    return p2_raw(A);
  }
  static __device__ __forceinline__ W cmac4(const DFK* c, const W* a) {
    PAcc A = cprod(k2(c[0]), a[0]);
#pragma unroll
    for (int i = 1; i < 4; ++i) cmac(A, k2(c[i]), a[i]);
    return p2_raw(A);
  }
  static __device__ __forceinline__ DFK lanes(const P2& w) {
    DFK r;
    p2_lanes(w, r.re, r.im);
    return r;
  }
  static __device__ __forceinline__ P2 pair(const DFK& b) { return P2{f2_pack(b.re.h, b.im.h), f2_pack(b.re.l, b.im.l)}; }
  static __device__ __forceinline__ DFK kmul(const DFK& a, const DFK& b) { return lanes(p2_raw(cprod(k2(a), pair(b)))); }
  static __device__ __forceinline__ DFK kmuln(const DFK& a, const DFK& b) { return lanes(p2_norm(cprod(k2(a), pair(b)))); }
  static __device__ __forceinline__ W rmac2(const R2& c0, const W& a, const R2& c1, const W& b) {
    PAcc A = p2_prod(a, P2{c0.h, c0.l});
    p2_mac(A, b, P2{c1.h, c1.l});
    return p2_raw(A);
  }
  static __device__ __forceinline__ void renorm(W& w) { w = p2_norm(PAcc{w.h, w.l}); }
  // SX x + k y for a real k: one exact product, one TwoSum and the error
  // terms, 12 packed operations (13 for SX < 0).  q is minus the product p.
  template <int SX>
  static __device__ __forceinline__ W uma(const W& x, const R2& k, const W& y) {
    const f2 q = f2_mul(y.h, k.nh);
    f2 e = f2_fma(y.h, k.h, q);
    e = f2_fma(y.h, k.l, e);
    e = f2_fma(y.l, k.h, e);
    if (SX > 0) {
      const f2 s = f2_sub(x.h, q);                        // p + x
      const f2 bp = f2_add(s, q);                         // s - p
      const f2 w = f2_add(f2_sub(s, bp), q);              // -(p - (s - bp))
      const f2 err = f2_sub(f2_sub(x.h, bp), w);
      return W{s, f2_add(e, f2_add(err, x.l))};
    }
    const f2 p = f2_mul(y.h, k.h);
    const f2 s = f2_sub(p, x.h);
    const f2 bp = f2_add(s, q);
    const f2 err = f2_sub(f2_sub(p, f2_sub(s, bp)), f2_add(x.h, bp));
    return W{s, f2_add(e, f2_sub(err, x.l))};
  }
  static __device__ __forceinline__ W rscale(const R2& g, const W& x) { return p2_raw(p2_prod(x, P2{g.h, g.l})); }
  // x + SY y: one TwoSum of the leading parts, the low parts and the error added
  template <int SY>
  static __device__ __forceinline__ W uadd(const W& x, const W& y) {
    if (SY > 0) {
      const f2 s = f2_add(x.h, y.h);
      const f2 bp = f2_sub(s, x.h);
      const f2 err = f2_add(f2_sub(x.h, f2_sub(s, bp)), f2_sub(y.h, bp));
      return W{s, f2_add(f2_add(x.l, y.l), err)};
    }
    const f2 s = f2_sub(x.h, y.h);
    const f2 bp = f2_sub(s, x.h);
    const f2 err = f2_sub(f2_sub(x.h, f2_sub(s, bp)), f2_add(y.h, bp));
    return W{s, f2_add(f2_sub(x.l, y.l), err)};
  }
};
template <class A>
__device__ __forceinline__ void renorm(typename A::W& a) { Lz<A>::renorm(a); }

template <class A> struct Re;
template <> struct Re<ArF32> { static __device__ __forceinline__ float get(const float2& c) { return c.x; } };
template <> struct Re<ArF64> { static __device__ __forceinline__ double get(const double2& c) { return c.x; } };
template <> struct Re<ArDFP> {
  static __device__ __forceinline__ R2 get(const DFK& c) {
    return R2{f2_dup(c.re.h), f2_dup(-c.re.h), f2_dup(c.re.l)};
  }
};

// (a, b) <- (u00 a + u01 b, u10 a + u11 b)
template <class A>
__device__ __forceinline__ void d1(typename A::W& a, typename A::W& b, const typename A::C& u00,
                                   const typename A::C& u01, const typename A::C& u10, const typename A::C& u11) {
  const typename A::W x = a, y = b;
  a = Lz<A>::cmac2(u00, x, u01, y);
  b = Lz<A>::cmac2(u10, x, u11, y);
}

// the same with a real matrix (real parts of the coefficients)
template <class A>
__device__ __forceinline__ void d1r(typename A::W& a, typename A::W& b, const typename A::C& u00,
                                    const typename A::C& u01, const typename A::C& u10, const typename A::C& u11) {
  const typename A::W x = a, y = b;
  a = Lz<A>::rmac2(Re<A>::get(u00), x, Re<A>::get(u01), y);
  b = Lz<A>::rmac2(Re<A>::get(u10), x, Re<A>::get(u11), y);
}

// A real 2x2 that is g times an orthogonal matrix, m11 = SG m00 and
// m10 = -SG m01 with SG = +-1 (rotations such as RY, reflections such as H).
// Divided by m00 or m10, whichever has the larger modulus, each row keeps one
// entry of modulus 1, so each output costs one product and one sum:
//   form A (g = m00, |m00| >= |m01|): a' = a + k0 b,     b' = SG b + k1 a
//   form B (g = m10, |m01| >  |m00|): a' = -SG b + k0 a,  b' = a + k1 b
// with |k0|, |k1| <= 1 for orthogonal matrices.  The caller multiplies the
// amplitudes by the product of the g's afterwards (rscale).
template <class A, int SG>
__device__ __forceinline__ void u1a(typename A::W& a, typename A::W& b, const typename A::C& k0,
                                    const typename A::C& k1) {
  const typename A::W x = a, y = b;
  a = Lz<A>::template uma<1>(x, Re<A>::get(k0), y);
  b = Lz<A>::template uma<SG>(y, Re<A>::get(k1), x);
}
template <class A, int SG>
__device__ __forceinline__ void u1b(typename A::W& a, typename A::W& b, const typename A::C& k0,
                                    const typename A::C& k1) {
  const typename A::W x = a, y = b;
  a = Lz<A>::template uma<-SG>(y, Re<A>::get(k0), x);
  b = Lz<A>::template uma<1>(x, Re<A>::get(k1), y);
}

// The Hadamard pattern (m00 = m01 = m10 = -m11 = g): form A with k0 = k1 = 1,
// a' = a + b and b' = a - b, sums only; g joins the product of the g's.
template <class A>
__device__ __forceinline__ void u1h(typename A::W& a, typename A::W& b) {
  const typename A::W x = a, y = b;
  a = Lz<A>::template uadd<1>(x, y);
  b = Lz<A>::template uadd<-1>(x, y);
}

// (x0..x3) <- U x with U row-major at u[0..15]
template <class A>
__device__ __forceinline__ void d2(typename A::W& x0, typename A::W& x1, typename A::W& x2, typename A::W& x3,
                                   const typename A::C* u) {
  const typename A::W x[4] = {x0, x1, x2, x3};
  x0 = Lz<A>::cmac4(u, x);
  x1 = Lz<A>::cmac4(u + 4, x);
  x2 = Lz<A>::cmac4(u + 8, x);
  x3 = Lz<A>::cmac4(u + 12, x);
}

// (a, b) <- (f0 b, f1 a)
template <class A>
__device__ __forceinline__ void anti(typename A::W& a, typename A::W& b, const typename A::C& f0,
                                     const typename A::C& f1) {
  const typename A::W x = a;
  a = Lz<A>::cmul(f0, b);
  b = Lz<A>::cmul(f1, x);
}

// exchange a and b where p holds (a per-thread predicate)
template <class W>
__device__ __forceinline__ void swap_if(bool p, W& a, W& b) {
  const W x = a, y = b;
  a = p ? y : x;
  b = p ? x : y;
}

// Exchange-buffer position of a local amplitude index (same fold as the
// interpreter's buffer, so bank spread is unchanged).  It is linear over XOR,
// so for a thread part jt and a register part c with disjoint bits,
// swz(jt | c) = swz(jt) ^ swz(c): the thread part is folded once per layout
// and the register parts are constants.
template <int SZ>
__device__ __forceinline__ uint32_t swz(uint32_t j) {
  if (SZ == 16) return j ^ (((j >> 3) ^ (j >> 6) ^ (j >> 9)) & 7u);
  return j ^ (((j >> 4) ^ (j >> 8)) & 15u);
}

// Bit q of a tile's base index (an outside qubit's value on that tile), as
// the 0 / 1 that selects a folded permutation's outside-controlled flips.
__device__ __forceinline__ uint32_t obit(uint64_t base, int q) { return (uint32_t)(base >> q) & 1u; }

// Bank bits an exchange's swizzle changes relative to swz: bit b is the
// parity of the position bits in m_b (the masks are literal constants, so
// unused ones vanish at compile time).
__device__ __forceinline__ uint32_t pfold(uint32_t j, uint32_t m0, uint32_t m1, uint32_t m2, uint32_t m3) {
  uint32_t f = 0;
  if (m0) f |= (uint32_t)__popc(j & m0) & 1u;
  if (m1) f |= ((uint32_t)__popc(j & m1) & 1u) << 1;
  if (m2) f |= ((uint32_t)__popc(j & m2) & 1u) << 2;
  if (m3) f |= ((uint32_t)__popc(j & m3) & 1u) << 3;
  return f;
}

// Issues the bulk copies of one tile into `buf`, one row per thread (rows
// beyond the block size wrap): the work is spread over the block instead of
// one warp, so no warp falls behind the others before the next barrier.
// `my_roff` is row_offset(G, tid), formed once per launch.  The phase's
// expected byte count (its only arrival) must already be posted by thread 0
// (seg_expect) before any thread issues a copy of that phase.
template <class S>
__device__ __forceinline__ void seg_copy(const TileGeom& G, S* buf, const S* psi, uint64_t base, uint64_t* bar,
                                         uint64_t my_roff) {
  const uint32_t tid = threadIdx.x;
  const uint32_t nrows = 1u << G.r;
  const uint32_t per_row = 1u << G.b;
  for (uint32_t row = tid; row < nrows; row += blockDim.x)
    bulk_g2s(buf + (size_t)row * per_row, psi + base + (row == tid ? my_roff : row_offset(G, row)), G.row_bytes, bar);
}
__device__ __forceinline__ void seg_expect(const TileGeom& G, uint64_t* bar, uint32_t ntiles = 1) {
  mbar_expect_tx(bar, ntiles * (1u << G.r) * G.row_bytes);
}

// ---------------------------------------------------------------------------
// compiled adjoint: gradient partials Im <lambda|G|psi>
// ---------------------------------------------------------------------------
template <class A> struct Dfc;
template <> struct Dfc<ArF64> {
  static __device__ __forceinline__ DFC get(const double2& w) { return DFC{d2df(w.x), d2df(w.y)}; }
};

// Per-tile partial sums: double-float for complex128 (the products must keep
// about 2^-46 relative accuracy), float32 for complex64 states.  Either is
// added in float64 across tiles.  T accumulates products of amplitudes (in
// packed kernels one sum per component, added at the warp sum), B signed sums
// of terms V.
template <class A> struct GAcc {
  using T = DAcc;  // running sum (leading part, accumulated errors)
  using B = DAcc;
  using V = DF;    // one term
  static __device__ __forceinline__ T zero() { return DAcc{0.f, 0.f}; }
  static __device__ __forceinline__ B bzero() { return DAcc{0.f, 0.f}; }
};
template <> struct GAcc<ArDFP> {
  using T = PAcc;
  using B = DAcc;
  using V = DF;
  static __device__ __forceinline__ T zero() { return PAcc{0ull, 0ull}; }
  static __device__ __forceinline__ B bzero() { return DAcc{0.f, 0.f}; }
};
template <> struct GAcc<ArF32> {
  using T = float;
  using B = float;
  using V = float;
  static __device__ __forceinline__ T zero() { return 0.f; }
  static __device__ __forceinline__ B bzero() { return 0.f; }
};

// acc += sign * Im(conj(l) p) = sign * (l.re p.im - l.im p.re)
__device__ __forceinline__ void gim_t(DAcc& acc, const DFC& l, const DFC& p, bool neg) {
  df_mac(acc, neg ? df_neg(l.re) : l.re, p.im);
  df_mac(acc, neg ? l.im : df_neg(l.im), p.re);
}
__device__ __forceinline__ void gim_t(float& acc, const float2& l, const float2& p, bool neg) {
  const float s = neg ? -1.f : 1.f;
  acc = __fmaf_rn(s * l.x, p.y, acc);
  acc = __fmaf_rn(-s * l.y, p.x, acc);
}
__device__ __forceinline__ void gim_t(DAcc& acc, const double2& l, const double2& p, bool neg) {
  gim_t(acc, Dfc<ArF64>::get(l), Dfc<ArF64>::get(p), neg);
}
__device__ __forceinline__ P2 p2_xor(const P2& a, f2 m) { return P2{a.h ^ m, a.l ^ m}; }
__device__ __forceinline__ void gim_t(PAcc& acc, const P2& l, const P2& p, bool neg) {
  p2_mac(acc, l, p2_xor(p2_swap(p), neg ? 0x0000000080000000ull : 0x8000000000000000ull));
}
// acc += sign * Re(conj(l) p) = sign * (l.re p.re + l.im p.im)
__device__ __forceinline__ void gre_t(DAcc& acc, const DFC& l, const DFC& p, bool neg) {
  df_mac(acc, neg ? df_neg(l.re) : l.re, p.re);
  df_mac(acc, neg ? df_neg(l.im) : l.im, p.im);
}
__device__ __forceinline__ void gre_t(float& acc, const float2& l, const float2& p, bool neg) {
  const float s = neg ? -1.f : 1.f;
  acc = __fmaf_rn(s * l.x, p.x, acc);
  acc = __fmaf_rn(s * l.y, p.y, acc);
}
__device__ __forceinline__ void gre_t(DAcc& acc, const double2& l, const double2& p, bool neg) {
  gre_t(acc, Dfc<ArF64>::get(l), Dfc<ArF64>::get(p), neg);
}
__device__ __forceinline__ void gre_t(PAcc& acc, const P2& l, const P2& p, bool neg) {
  p2_mac(acc, l, p2_xor(p, neg ? 0x8000000080000000ull : 0ull));
}
template <class A>
__device__ __forceinline__ void gim(typename GAcc<A>::T& acc, const typename A::W& l, const typename A::W& p, bool neg) {
  gim_t(acc, l, p, neg);
}
template <class A>
__device__ __forceinline__ void gre(typename GAcc<A>::T& acc, const typename A::W& l, const typename A::W& p, bool neg) {
  gre_t(acc, l, p, neg);
}
// the scalar value of an accumulator
__device__ __forceinline__ float gval(float a) { return a; }
__device__ __forceinline__ DAcc gval(const DAcc& a) { return a; }
__device__ __forceinline__ DAcc gval(const PAcc& a) {
  DF x, y;
  p2_lanes(P2{a.s, a.e}, x, y);
  DAcc A{x.h, x.l};
  df_acc(A, y);
  return A;
}

// One term w = Im(conj(l) p), shared by every Z / P1 partial of a merged
// diagonal run (those partials are signed sums of the same w_j).
__device__ __forceinline__ float gterm(float a) { return a; }
__device__ __forceinline__ DF gterm(const DAcc& a) { return df_norm(a); }
template <class A>
__device__ __forceinline__ typename GAcc<A>::V wim(const typename A::W& l, const typename A::W& p) {
  typename GAcc<A>::T a = GAcc<A>::zero();
  gim<A>(a, l, p, false);
  return gterm(gval(a));
}
template <>
__device__ __forceinline__ DF wim<ArDFP>(const P2& l, const P2& p) {
  return df_norm(gval(p2_prod(l, p2_xor(p2_swap(p), 0x8000000000000000ull))));
}
__device__ __forceinline__ void wadd(DAcc& acc, const DF& w, bool neg) { df_acc(acc, neg ? df_neg(w) : w); }
__device__ __forceinline__ void wadd(float& acc, float w, bool neg) { acc = neg ? acc - w : acc + w; }
__device__ __forceinline__ DAcc gneg(const DAcc& a, bool neg) { return neg ? DAcc{-a.s, -a.e} : a; }
__device__ __forceinline__ float gneg(float a, bool neg) { return neg ? -a : a; }

// Per-warp partial-sum slots.  Double-float kernels keep each 8-byte slot as
// a double-float pair and add to it with float32 operations (float64 adds run
// on a far narrower pipe); the slot is read as a float64 once, after the tile
// loop.  Float32 kernels add in float64.
__device__ __forceinline__ void slot_add(double* slot, const DF& v) {
  DF* d = reinterpret_cast<DF*>(slot);
  *d = df_add(*d, v);
}
template <class A>
__device__ __forceinline__ double slot_get(const double* slot) {
  if constexpr (sizeof(typename GAcc<A>::T) == sizeof(float)) return *slot;
  else return df2d(*reinterpret_cast<const DF*>(slot));
}

// Warp sum of a partial, added by lane 0 to the warp's slot.  All 32 lanes
// must call it.
__device__ __forceinline__ void gflush(DAcc a, double* slot) {
  DF v = df_norm(a);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1)
    v = df_add(v, DF{__shfl_xor_sync(0xffffffffu, v.h, off), __shfl_xor_sync(0xffffffffu, v.l, off)});
  if ((threadIdx.x & 31u) == 0) slot_add(slot, v);
}
__device__ __forceinline__ void gflush(float a, double* slot) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
  if ((threadIdx.x & 31u) == 0) *slot += (double)a;
}

// Four per-lane partials summed over the warp at once (a reduce-scatter):
// two halving exchanges leave each lane with one of the four (lanes with bit
// 4 take slots 2-3, with bit 3 the odd one), three butterfly steps complete
// the sums, and lanes 0, 8, 16, 24 add them to slots s0..s3 (null: unused).
// All 32 lanes must call it.
__device__ __forceinline__ DF shfl_df(const DF& v, int off) {
  return DF{__shfl_xor_sync(0xffffffffu, v.h, off), __shfl_xor_sync(0xffffffffu, v.l, off)};
}
__device__ __forceinline__ void gflush4(const DAcc& a0, const DAcc& a1, const DAcc& a2, const DAcc& a3, double* s0,
                                        double* s1, double* s2, double* s3) {
  const uint32_t lane = threadIdx.x & 31u;
  const bool u16 = lane & 16u, u8 = lane & 8u;
  const DF v0 = df_norm(a0), v1 = df_norm(a1), v2 = df_norm(a2), v3 = df_norm(a3);
  DF k0 = u16 ? v2 : v0, k1 = u16 ? v3 : v1;
  const DF t0 = u16 ? v0 : v2, t1 = u16 ? v1 : v3;
  k0 = df_add(k0, shfl_df(t0, 16));
  k1 = df_add(k1, shfl_df(t1, 16));
  DF k = u8 ? k1 : k0;
  k = df_add(k, shfl_df(u8 ? k0 : k1, 8));
  k = df_add(k, shfl_df(k, 4));
  k = df_add(k, shfl_df(k, 2));
  k = df_add(k, shfl_df(k, 1));
  double* s = u16 ? (u8 ? s3 : s2) : (u8 ? s1 : s0);
  if ((lane & 7u) == 0 && s) slot_add(s, k);
}
__device__ __forceinline__ void gflush4(const PAcc& a0, const PAcc& a1, const PAcc& a2, const PAcc& a3, double* s0,
                                        double* s1, double* s2, double* s3) {
  gflush4(gval(a0), gval(a1), gval(a2), gval(a3), s0, s1, s2, s3);
}
__device__ __forceinline__ void gflush4(float a0, float a1, float a2, float a3, double* s0, double* s1, double* s2,
                                        double* s3) {
  const uint32_t lane = threadIdx.x & 31u;
  const bool u16 = lane & 16u, u8 = lane & 8u;
  float k0 = u16 ? a2 : a0, k1 = u16 ? a3 : a1;
  const float t0 = u16 ? a0 : a2, t1 = u16 ? a1 : a3;
  k0 += __shfl_xor_sync(0xffffffffu, t0, 16);
  k1 += __shfl_xor_sync(0xffffffffu, t1, 16);
  float k = u8 ? k1 : k0;
  k += __shfl_xor_sync(0xffffffffu, u8 ? k0 : k1, 8);
  k += __shfl_xor_sync(0xffffffffu, k, 4);
  k += __shfl_xor_sync(0xffffffffu, k, 2);
  k += __shfl_xor_sync(0xffffffffu, k, 1);
  double* s = u16 ? (u8 ? s3 : s2) : (u8 ? s1 : s0);
  if ((lane & 7u) == 0 && s) *s += (double)k;
}

// A running sum held by one lane across the tile loop and stored in its
// slot once: double-float for complex128 kernels, float64 for complex64.
template <class A> struct LaneAcc {
  DF s;
  __device__ __forceinline__ void zero() { s = DF{0.f, 0.f}; }
  __device__ __forceinline__ void add(const DF& x, bool neg) { s = df_add(s, neg ? df_neg(x) : x); }
  __device__ __forceinline__ void put(double* slot) const { *reinterpret_cast<DF*>(slot) = s; }
};
template <> struct LaneAcc<ArF32> {
  double s;
  __device__ __forceinline__ void zero() { s = 0.0; }
  __device__ __forceinline__ void add(float x, bool neg) { s += neg ? -(double)x : (double)x; }
  __device__ __forceinline__ void put(double* slot) const { *slot = s; }
};
__device__ __forceinline__ DF shfl_idx(const DF& v, uint32_t src) {
  return DF{__shfl_sync(0xffffffffu, v.h, src), __shfl_sync(0xffffffffu, v.l, src)};
}
__device__ __forceinline__ float shfl_idx(float v, uint32_t src) { return __shfl_sync(0xffffffffu, v, src); }

// Walsh butterfly over the warp: lane l ends with sum_i (-1)^popc(i & l) v_i,
// so lane 0 holds the plain sum and lane 2^m the sum signed by lane bit m.
// All 32 lanes must call it.
__device__ __forceinline__ DF wht(DAcc a) {
  DF v = df_norm(a);
  const uint32_t lane = threadIdx.x & 31u;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const DF o{__shfl_xor_sync(0xffffffffu, v.h, off), __shfl_xor_sync(0xffffffffu, v.l, off)};
    v = (lane & (uint32_t)off) ? df_sub(o, v) : df_add(v, o);
  }
  return v;
}
__device__ __forceinline__ float wht(float v) {
  const uint32_t lane = threadIdx.x & 31u;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const float o = __shfl_xor_sync(0xffffffffu, v, off);
    v = (lane & (uint32_t)off) ? o - v : v + o;
  }
  return v;
}
// slot += (neg ? -w : w) where `cond` holds (one lane per slot).
__device__ __forceinline__ void gput(const DF& w, bool cond, bool neg, double* slot) {
  if (cond) slot_add(slot, neg ? df_neg(w) : w);
}
__device__ __forceinline__ void gput(float w, bool cond, bool neg, double* slot) {
  if (cond) *slot += neg ? -(double)w : (double)w;
}

// ---------------------------------------------------------------------------
// compiled Pauli passes: |psi_j|^2, lambda accumulators
// ---------------------------------------------------------------------------
__device__ __forceinline__ DF pnorm2(const DFC& v) {
  DAcc a = df_prod(v.re, v.re);
  df_mac(a, v.im, v.im);
  return df_norm(a);
}
__device__ __forceinline__ DF pnorm2(const double2& v) { return pnorm2(Dfc<ArF64>::get(v)); }
__device__ __forceinline__ DF pnorm2(const P2& v) { return df_norm(gval(p2_prod(v, v))); }
__device__ __forceinline__ float pnorm2(const float2& v) { return __fmaf_rn(v.x, v.x, __fmul_rn(v.y, v.y)); }
template <class A>
__device__ __forceinline__ typename GAcc<A>::V pn2(const typename A::W& w) { return pnorm2(w); }

// lambda_j accumulated per component: double-float for complex128 states,
// float32 for complex64.
template <class A> struct LAcc;
template <> struct LAcc<ArF64> {
  DAcc re, im;
  __device__ __forceinline__ void init(const double2& w) {
    const DFC v = Dfc<ArF64>::get(w);
    re = DAcc{v.re.h, v.re.l};
    im = DAcc{v.im.h, v.im.l};
  }
  __device__ __forceinline__ void zero() { re = im = DAcc{0.f, 0.f}; }
  // += c * sign * i^PH * w
  template <int PH>
  __device__ __forceinline__ void add(const double2& w, const DF& c, bool neg) {
    const DFC v = Dfc<ArF64>::get(w);
    DF vr = v.re, vi = v.im;
    if (PH & 1) { const DF t = vr; vr = df_neg(vi); vi = t; }
    if (PH & 2) { vr = df_neg(vr); vi = df_neg(vi); }
    if (neg) { vr = df_neg(vr); vi = df_neg(vi); }
    df_mac(re, vr, c);
    df_mac(im, vi, c);
  }
  __device__ __forceinline__ double2 out() const {
    return make_double2(df2d(df_norm(re)), df2d(df_norm(im)));
  }
};
template <> struct LAcc<ArDFP> {
  PAcc a;
  __device__ __forceinline__ void init(const P2& w) { a = PAcc{w.h, w.l}; }
  __device__ __forceinline__ void zero() { a = PAcc{0ull, 0ull}; }
  template <int PH>
  __device__ __forceinline__ void add(const P2& w, const DF& c, bool neg) {
    const bool n = neg != ((PH & 2) != 0);  // the sign goes to the coefficient
    const float ch = n ? -c.h : c.h, cl = n ? -c.l : c.l;
    p2_mac(a, (PH & 1) ? ArDFP::mul_i(w) : w, P2{f2_dup(ch), f2_dup(cl)});
  }
  __device__ __forceinline__ P2 out() const { return p2_norm(a); }
};
template <> struct LAcc<ArF32> {
  float re, im;
  __device__ __forceinline__ void init(const float2& w) { re = w.x; im = w.y; }
  __device__ __forceinline__ void zero() { re = im = 0.f; }
  template <int PH>
  __device__ __forceinline__ void add(const float2& w, float c, bool neg) {
    float vr = w.x, vi = w.y;
    if (PH & 1) { const float t = vr; vr = -vi; vi = t; }
    if (PH & 2) { vr = -vr; vi = -vi; }
    if (neg) { vr = -vr; vi = -vi; }
    re = __fmaf_rn(vr, c, re);
    im = __fmaf_rn(vi, c, im);
  }
  __device__ __forceinline__ float2 out() const { return make_float2(re, im); }
};
// Real coefficient of a Pauli word in the parameter block, per policy.
template <class A> struct PCoef { using T = DF; };
template <> struct PCoef<ArF32> { using T = float; };
// sum of signed coefficients (diagonal words of lambda)
__device__ __forceinline__ void cadd(DAcc& a, const DF& c, bool neg) { df_acc(a, neg ? df_neg(c) : c); }
__device__ __forceinline__ void cadd(float& a, float c, bool neg) { a = neg ? a - c : a + c; }
__device__ __forceinline__ DF cfin(const DAcc& a) { return df_norm(a); }
__device__ __forceinline__ float cfin(float a) { return a; }

// Barrier over a group of warps: named barrier `id` (1..15; 0 is the
// block-wide barrier) for `nthreads` threads, a multiple of 32.
__device__ __forceinline__ void bar_group(uint32_t id, uint32_t nthreads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

}  // namespace jit
}  // namespace lqs
