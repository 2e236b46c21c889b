// Batched Stockham (self-sorting) FFT of one line per group of L/8 threads.
//
// Each thread owns 8 complex values of its line.  A length-L transform is a
// sequence of radix passes (radix 8, then one radix-2 or radix-4 pass when
// log2 L is not a multiple of 3); the inverse plan runs the radices in reverse
// order so that the forward transform's last-pass register layout is exactly
// the inverse transform's first-pass layout.  That is what lets the z pass
// fuse forward FFT -> k-space multiply -> inverse FFT without touching shared
// memory at the turn.  Between passes values go through shared memory; the
// first-pass inputs and last-pass outputs stay in registers, so prologue and
// epilogue code reads and writes global memory directly in natural order.
//
// Pass p (radix r, Ns = product of earlier radices), butterfly j, element q:
//   input position  j + q L/r
//   twiddle         W_{Ns r}^{q (j mod Ns)}   (table entry q (j mod Ns) L/(Ns r))
//   output position (j div Ns) Ns r + (j mod Ns) + q Ns
// Thread t of a line owns butterflies j = t + b L/8 (b < 8/r).
//
// Lengths 48, 80 and 96 (8 times 6, 10 and 12) use the same register interface
// with a radix-8 pass, one pass of radix L/8 and natural entry/exit layouts; see
// fft_mixed.
#pragma once
#include <type_traits>

#include "common.cuh"

namespace egpe {

template <int L> struct IsPow2 {
  static constexpr bool v = L > 0 && (L & (L - 1)) == 0;
};

// The other lengths are 8 times 6, 10 or 12: a radix-8 pass and one pass of radix
// L/8, which is as many values as the line has threads.
template <int L> struct MixedPlan {
  static constexpr int TPL = L / 8;
  static_assert(TPL == 6 || TPL == 10 || TPL == 12, "unsupported FFT length");
  // natural layout on entry and exit, in both directions
  __device__ static __forceinline__ int entry_pos(bool, int t, int e) { return t + e * TPL; }
  __device__ static __forceinline__ int exit_pos(bool, int t, int e) { return t + e * TPL; }
};

template <int L, bool POW2 = IsPow2<L>::v> struct Plan;
template <int L> struct Plan<L, false> : MixedPlan<L> {};

template <int L> struct Plan<L, true> {
  static constexpr int TPL = L / 8;
  static constexpr int LOG2 = (L == 8) ? 3 : (L == 16) ? 4 : (L == 32) ? 5 : (L == 64) ? 6
                            : (L == 128) ? 7 : (L == 256) ? 8 : -1;
  static_assert(LOG2 > 0, "unsupported FFT length");
  static constexpr int P = (LOG2 + 2) / 3;
  static constexpr int LAST = L >> (3 * (P - 1));  // radix of the forward plan's last pass
  __host__ __device__ static constexpr int rad(bool inv, int p) {
    return inv ? (p == 0 ? LAST : 8) : (p == P - 1 ? LAST : 8);
  }
  __host__ __device__ static constexpr int ns(bool inv, int p) {
    return p == 0 ? 1 : ns(inv, p - 1) * rad(inv, p - 1);
  }
  // position of register e of thread t on entry to / exit from the transform
  __device__ static __forceinline__ int entry_pos(bool inv, int t, int e) {
    const int r = rad(inv, 0);
    return t + (e / r) * TPL + (e % r) * (L / r);
  }
  __device__ static __forceinline__ int exit_pos(bool inv, int t, int e) {
    const int r = rad(inv, P - 1);
    return t + (e / r) * TPL + (e % r) * (L / r);
  }
};

template <int MC> struct ColIdxT;
template <class SI> struct IsColIdx {
  static constexpr bool v = false;
};
template <int MC> struct IsColIdx<ColIdxT<MC>> {
  static constexpr bool v = true;
};
// Synchronisation of one transform's exchange buffer.  A row line's L/8
// threads are consecutive and, for the power-of-two lengths (L/8 <= 32
// dividing 32), inside one warp with a buffer of their own: a warp barrier
// suffices.  Column lines spread over the block and need the block barrier.
template <class SI> __device__ __forceinline__ void line_sync() {
  if constexpr (IsColIdx<SI>::v) __syncthreads();
  else __syncwarp();
}
// Column lines (power-of-two lengths) exchange through two buffers in turn,
// so one block barrier per exchange suffices: a buffer is written again only
// after the barrier of the exchange that used the other one, which every
// thread reaches after its reads of the first.  Row lines reuse one buffer
// with two warp barriers per exchange.
template <class SI> struct PingPong {
  static constexpr bool v = IsColIdx<SI>::v;
};

template <class C> __device__ __forceinline__ C mul_i(C a) { return cmk<C>(-a.y, a.x); }
template <class C> __device__ __forceinline__ C mul_mi(C a) { return cmk<C>(a.y, -a.x); }

template <bool INV, class C> __device__ __forceinline__ void dft2(C* v) {
  C a = v[0], b = v[1];
  v[0] = cadd(a, b);
  v[1] = csub(a, b);
}

template <bool INV, class C> __device__ __forceinline__ void dft4v(C& a0, C& a1, C& a2, C& a3) {
  C t0 = cadd(a0, a2), t1 = csub(a0, a2), t2 = cadd(a1, a3), t3 = csub(a1, a3);
  t3 = INV ? mul_i(t3) : mul_mi(t3);
  a0 = cadd(t0, t2);
  a2 = csub(t0, t2);
  a1 = cadd(t1, t3);
  a3 = csub(t1, t3);
}

template <bool INV, class C> __device__ __forceinline__ void dft4(C* v) { dft4v<INV>(v[0], v[1], v[2], v[3]); }

template <bool INV, class C> __device__ __forceinline__ void dft8(C* v) {
  using R = decltype(C::x);
  const R h = R(0.70710678118654752440084436210485);
  C e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
  C o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
  dft4v<INV>(e0, e1, e2, e3);
  dft4v<INV>(o0, o1, o2, o3);
  // odd outputs times W8^k (forward W8 = exp(-i pi/4); inverse its conjugate)
  if (INV) {
    o1 = cmk<C>((o1.x - o1.y) * h, (o1.x + o1.y) * h);
    o2 = mul_i(o2);
    o3 = cmk<C>((-o3.x - o3.y) * h, (o3.x - o3.y) * h);
  } else {
    o1 = cmk<C>((o1.x + o1.y) * h, (o1.y - o1.x) * h);
    o2 = mul_mi(o2);
    o3 = cmk<C>((o3.y - o3.x) * h, -(o3.x + o3.y) * h);
  }
  v[0] = cadd(e0, o0);
  v[4] = csub(e0, o0);
  v[1] = cadd(e1, o1);
  v[5] = csub(e1, o1);
  v[2] = cadd(e2, o2);
  v[6] = csub(e2, o2);
  v[3] = cadd(e3, o3);
  v[7] = csub(e3, o3);
}

// y_k = sum_q a_q W_3^{qk}: with c = cos(2 pi/3) = -1/2 and s = sin(2 pi/3),
// y_{1,2} = a0 + c (a1 + a2) -/+ i s (a1 - a2) (signs swapped for the inverse).
template <bool INV, class C> __device__ __forceinline__ void dft3(C* v) {
  using R = decltype(C::x);
  const R s = R(0.86602540378443864676372317075294);
  const C a0 = v[0], t1 = cadd(v[1], v[2]), t2 = csub(v[1], v[2]);
  const C b = cmk<C>(a0.x - R(0.5) * t1.x, a0.y - R(0.5) * t1.y);
  const C d = cscale(INV ? mul_i(t2) : mul_mi(t2), s);
  v[0] = cadd(a0, t1);
  v[1] = cadd(b, d);
  v[2] = csub(b, d);
}

// Five-point DFT from the real and imaginary parts of W_5^k:
// c1 = cos(2 pi/5), c2 = cos(4 pi/5), s1 = sin(2 pi/5), s2 = sin(4 pi/5).
template <bool INV, class C> __device__ __forceinline__ void dft5(C* v) {
  using R = decltype(C::x);
  const R c1 = R(0.30901699437494742410229341718282), c2 = R(-0.80901699437494742410229341718282);
  const R s1 = R(0.95105651629515357211643933337938), s2 = R(0.58778525229247312916870595463907);
  const C a0 = v[0];
  const C t1 = cadd(v[1], v[4]), t2 = cadd(v[2], v[3]), t3 = csub(v[1], v[4]), t4 = csub(v[2], v[3]);
  const C b1 = cmk<C>(a0.x + c1 * t1.x + c2 * t2.x, a0.y + c1 * t1.y + c2 * t2.y);
  const C b2 = cmk<C>(a0.x + c2 * t1.x + c1 * t2.x, a0.y + c2 * t1.y + c1 * t2.y);
  const C e1 = cmk<C>(s1 * t3.x + s2 * t4.x, s1 * t3.y + s2 * t4.y);
  const C e2 = cmk<C>(s2 * t3.x - s1 * t4.x, s2 * t3.y - s1 * t4.y);
  const C d1 = INV ? mul_i(e1) : mul_mi(e1), d2 = INV ? mul_i(e2) : mul_mi(e2);
  v[0] = cadd(a0, cadd(t1, t2));
  v[1] = cadd(b1, d1);
  v[4] = csub(b1, d1);
  v[2] = cadd(b2, d2);
  v[3] = csub(b2, d2);
}

// ----------------------------------------------------------------------------
// FP64 lines in 64-bit fixed point.
//
// GB300 issues two FP64 lanes per SM and clock, one 32-lane instruction in 16
// clocks, while the integer pipes take the two 32-bit halves of a 64-bit sum in
// one or two.  So a line of an FP64 transform is converted to 64-bit integers
// under one scale of its own, transformed in integers, and converted back:
//
// * Scale.  B >= sum_j (|Re x_j| + |Im x_j|) over the line bounds every
//   intermediate value and output of the transform.  With q = x 2^s, s the largest
//   with 2^s B <= 2^62, nothing overflows, sums are exact, and an input is rounded
//   towards minus infinity by at most one unit, 2^-62 to 2^-61 B.  For a line whose
//   values are comparable that is 2^-62 L to 2^-61 L of a typical |Re| + |Im| (at most
//   2^-54 at L = 128), against 2^-53 of each value in FP64.
// * Products.  Twiddles and constants carry 62 fractional bits as two signed
//   32-bit limbs; a product is three 32 x 32 + 64 multiply-adds, right to two
//   units.
//
// Measured: a y pass of three 128^3 fields 256 -> 77 us, of three 96^3 fields
// 115 -> 52 us; relative 2-norm error of a 3D transform of random data against
// extended precision 2.3e-16 -> 0.9e-16 (32^3), 2.7e-16 -> 1.0e-16 (64^3),
// 2.8e-16 -> 1.5e-16 (256 x 16 x 128), 2.9e-16 -> 1.2e-16 (80^3).  Lines with a
// value of at least 2^1013 (or not finite) give NaN; lines with no value above
// 2^-960 give 0.  Squares of such values are out of range anyway in the pipelines; the
// plain transforms of the caller's own fields are WIDE and take values up to the
// largest (in every pass that cost the FP64 attempt 0.5% at 128^3 and 1.8% at 96^3).
// ----------------------------------------------------------------------------
struct __align__(16) Q2 {
  long long x, y;
};
// (cos, -sin) of a twiddle angle: value = (h 2^32 + l) 2^-62, both limbs signed.
struct __align__(16) TwQ {
  int xh, xl, yh, yl;
};
static_assert(sizeof(Q2) == sizeof(double2) && sizeof(TwQ) == sizeof(double2), "fixed-point lines share FP64 buffers");

// Scale of one line: an input with biased exponent e is its 53-bit significand
// shifted left by 10 and then right by X - e; an output whose
// leading zeros are lz gets the biased exponent X + 1 - lz.
struct LineScale {
  int X;
  int keep;  // 0 for a line that is taken as 0: clears the signs of its values too
  int bad;  // bits or-ed into the outputs' high words: a NaN pattern for a line that is not finite
};
constexpr int kLineBad = 0x7ff80000;
constexpr int kLineBig = 0x7ffc0000;  // WIDE: finite, but exponents may overflow on the way (NaN to the others)

__device__ __forceinline__ long long to_fixed(double d, const LineScale& ls) {
  const int hi = __double2hiint(d);
  const unsigned lo = (unsigned)__double2loint(d);
  const int e = (hi >> 20) & 0x7ff;
  const int r = min(ls.X - e, 63);  // zeros (e = 0) leave by the clamp
  const unsigned mh = ((unsigned)hi & 0xfffffu) | 0x100000u;
  const unsigned long long m = (((unsigned long long)mh << 32) | lo) << 10;
  const long long s = (long long)((hi >> 31) & ls.keep);
  return (long long)(m >> r) ^ s;  // floor: ones' complement of a negative value's magnitude
}
__device__ __forceinline__ double from_fixed(long long q, const LineScale& ls) {
  const int sg = (int)(q >> 32) >> 31;
  const unsigned long long u = (unsigned long long)(q ^ (long long)sg);
  const int lz = __clzll((long long)u);
  const unsigned long long m = u << (lz & 63);
  const unsigned long long r = (m >> 11) + ((m >> 10) & 1ull);  // carries into the exponent
  int hi = (int)(r >> 32) + ((ls.X - lz) << 20);
  int lo = (int)r;
  hi = u == 0ull ? 0 : hi;  // r is 0 then
  return __hiloint2double(hi | (sg & (int)0x80000000) | ls.bad, lo);
}

// One thread's share of B: the largest biased exponent of its 16 values and the
// sum of their significands (top 21 bits, rounded up) in units of that exponent.
__device__ __forceinline__ uint2 thread_bound(const double2 (&v)[8]) {
  int mx = 0;
#pragma unroll
  for (int e = 0; e < 8; ++e)
    mx = max(mx, max(__double2hiint(v[e].x) & 0x7fffffff, __double2hiint(v[e].y) & 0x7fffffff));
  const int E = mx >> 20;
  unsigned S = 16;
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const unsigned hx = (unsigned)__double2hiint(v[e].x) & 0x7fffffffu, hy = (unsigned)__double2hiint(v[e].y) & 0x7fffffffu;
    S += ((hx & 0xfffffu) | 0x100000u) >> min(E - (int)(hx >> 20), 31);
    S += ((hy & 0xfffffu) | 0x100000u) >> min(E - (int)(hy >> 20), 31);
  }
  return make_uint2((unsigned)E, S);
}
// Sum of two shares (commutative: every thread of a line gets the same bits).
__device__ __forceinline__ uint2 add_bounds(uint2 a, uint2 b) {
  const int E = max((int)a.x, (int)b.x);
  return make_uint2((unsigned)E, (a.y >> min(E - (int)a.x, 31)) + (b.y >> min(E - (int)b.x, 31)) + 1u);
}
template <bool WIDE> __device__ __forceinline__ LineScale make_scale(uint2 b) {
  const int E = (int)b.x;
  LineScale s;
  s.X = E < 64 ? 4096 : E + (32 - __clz((int)b.y)) - 20;
  s.keep = E < 64 ? 0 : -1;
  s.bad = E >= 2036 ? (WIDE && E < 2047 ? kLineBig : kLineBad) : 0;
  return s;
}

// Scales of a thread's NF lines.  Row lines of power-of-two length sit in one
// warp; the other row lines exchange their shares through the line's (idle)
// exchange buffer, column lines through the slots `sc`, which are free again
// after the transform's first exchange barrier.
template <int L, int NF, bool WIDE, class SI>
__device__ __forceinline__ void line_scales(const double2 (&v)[NF][8], double2* sm, int fstride, int t, const SI& si,
                                            LineScale (&ls)[NF]) {
  constexpr int TPL = L / 8;
  uint2 b[NF];
#pragma unroll
  for (int f = 0; f < NF; ++f) b[f] = thread_bound(v[f]);
  if constexpr (IsColIdx<SI>::v) {
    static_assert(NF == 1, "column lines come one field at a time");
    si.sc[t * si.width()] = b[0];
    __syncthreads();
    uint2 a = si.sc[0];
#pragma unroll 8
    for (int k = 1; k < TPL; ++k) a = add_bounds(a, si.sc[k * si.width()]);
    ls[0] = make_scale<WIDE>(a);
  } else if constexpr (IsPow2<L>::v) {
#pragma unroll
    for (int f = 0; f < NF; ++f) {
#pragma unroll
      for (int off = TPL / 2; off > 0; off >>= 1)
        b[f] = add_bounds(b[f], make_uint2(__shfl_xor_sync(0xffffffffu, b[f].x, off),
                                           __shfl_xor_sync(0xffffffffu, b[f].y, off)));
      ls[f] = make_scale<WIDE>(b[f]);
    }
  } else {
#pragma unroll
    for (int f = 0; f < NF; ++f) reinterpret_cast<uint2*>(sm + f * fstride)[t] = b[f];
    __syncthreads();
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      const uint2* p = reinterpret_cast<const uint2*>(sm + f * fstride);
      uint2 a = p[0];
#pragma unroll
      for (int k = 1; k < TPL; ++k) a = add_bounds(a, p[k]);
      ls[f] = make_scale<WIDE>(a);
    }
    __syncthreads();
  }
}

__device__ __forceinline__ long long imad(int a, int b, long long c) { return (long long)a * b + c; }
// Signed limbs of a (|a| < 2^62): a = h 2^32 + l.
struct LimbQ {
  int h, h2, l;  // h2 = 2 h
};
__device__ __forceinline__ LimbQ limbs(long long a) {
  LimbQ r;
  r.l = (int)a;
  r.h = (int)(a >> 32) - (r.l >> 31);
  r.h2 = 2 * r.h;
  return r;
}
// a w for a real constant w = (wh 2^32 + wl) 2^-62: half the product from the limbs' upper parts.
__device__ __forceinline__ long long mulq(long long a, int wh, int wl) {
  const LimbQ x = limbs(a);
  return 2 * imad(x.h2, wh, imad(x.l, wh, imad(x.h, wl, 0)) >> 31);
}
__device__ __forceinline__ Q2 cmul_limbs(Q2 a, int wh, int wl, int vh, int vl) {  // w + i v
  const LimbQ x = limbs(a.x), y = limbs(a.y);
  const int nh = -vh, nl = -vl;
  const long long tr = imad(y.l, nh, imad(y.h, nl, imad(x.l, wh, imad(x.h, wl, 0))));
  const long long ti = imad(y.l, wh, imad(y.h, wl, imad(x.l, vh, imad(x.h, vl, 0))));
  return Q2{2 * imad(y.h2, nh, imad(x.h2, wh, tr >> 31)), 2 * imad(y.h2, wh, imad(x.h2, vh, ti >> 31))};
}
__device__ __forceinline__ Q2 cmul(Q2 a, TwQ w) { return cmul_limbs(a, w.xh, w.xl, w.yh, w.yl); }
__device__ __forceinline__ Q2 cmulc(Q2 a, TwQ w) { return cmul_limbs(a, w.xh, w.xl, -w.yh, -w.yl); }

template <bool INV> __device__ __forceinline__ void dft8(Q2* v) {
  constexpr int hh = 759250125, hl = -25716447;  // 2^62 / sqrt 2
  Q2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
  Q2 o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
  dft4v<INV>(e0, e1, e2, e3);
  dft4v<INV>(o0, o1, o2, o3);
  o1 = Q2{mulq(o1.x, hh, hl), mulq(o1.y, hh, hl)};
  o3 = Q2{mulq(o3.x, hh, hl), mulq(o3.y, hh, hl)};
  if (INV) {
    o1 = Q2{o1.x - o1.y, o1.x + o1.y};
    o2 = mul_i(o2);
    o3 = Q2{-o3.x - o3.y, o3.x - o3.y};
  } else {
    o1 = Q2{o1.x + o1.y, o1.y - o1.x};
    o2 = mul_mi(o2);
    o3 = Q2{o3.y - o3.x, -o3.x - o3.y};
  }
  v[0] = cadd(e0, o0);
  v[4] = csub(e0, o0);
  v[1] = cadd(e1, o1);
  v[5] = csub(e1, o1);
  v[2] = cadd(e2, o2);
  v[6] = csub(e2, o2);
  v[3] = cadd(e3, o3);
  v[7] = csub(e3, o3);
}
template <bool INV> __device__ __forceinline__ void dft3(Q2* v) {
  const Q2 a0 = v[0], t1 = cadd(v[1], v[2]), t2 = csub(v[1], v[2]);
  const Q2 b = Q2{a0.x - (t1.x >> 1), a0.y - (t1.y >> 1)};
  const Q2 m = Q2{mulq(t2.x, 929887697, -1332128537), mulq(t2.y, 929887697, -1332128537)};
  const Q2 d = INV ? mul_i(m) : mul_mi(m);
  v[0] = cadd(a0, t1);
  v[1] = cadd(b, d);
  v[2] = csub(b, d);
}
template <bool INV> __device__ __forceinline__ void dft5(Q2* v) {
  auto sc = [](Q2 a, int h, int l) { return Q2{mulq(a.x, h, l), mulq(a.y, h, l)}; };
  constexpr int c1h = 331804471, c1l = 803819395, c2h = -868675383, c2l = -803819395, s1h = 1021189159, s1l = -2002125123, s2h = 631129609, s2l = -357254181;
  const Q2 a0 = v[0];
  const Q2 t1 = cadd(v[1], v[4]), t2 = cadd(v[2], v[3]), t3 = csub(v[1], v[4]), t4 = csub(v[2], v[3]);
  const Q2 b1 = cadd(a0, cadd(sc(t1, c1h, c1l), sc(t2, c2h, c2l)));
  const Q2 b2 = cadd(a0, cadd(sc(t1, c2h, c2l), sc(t2, c1h, c1l)));
  const Q2 e1 = cadd(sc(t3, s1h, s1l), sc(t4, s2h, s2l));
  const Q2 e2 = csub(sc(t3, s2h, s2l), sc(t4, s1h, s1l));
  const Q2 d1 = INV ? mul_i(e1) : mul_mi(e1), d2 = INV ? mul_i(e2) : mul_mi(e2);
  v[0] = cadd(a0, cadd(t1, t2));
  v[1] = cadd(b1, d1);
  v[4] = csub(b1, d1);
  v[2] = cadd(b2, d2);
  v[3] = csub(b2, d2);
}

template <int R_, bool INV, class C> __device__ __forceinline__ void dft_r(C* v) {
  if constexpr (R_ == 8) dft8<INV>(v);  // Q2 lines: the fixed-point overloads
  else if constexpr (R_ == 5) dft5<INV>(v);
  else if constexpr (R_ == 4) dft4<INV>(v);
  else if constexpr (R_ == 3) dft3<INV>(v);
  else dft2<INV>(v);
}

// Runs passes p..P-1 of the (forward or inverse) plan on NF lines at once.
// v[f][8]: this thread's registers for field f; sm + f*fstride: the shared
// line buffer of field f for this thread's line; si(pos): offset of line
// position pos inside that buffer; tw: shared table W_L^m, m < L.
template <class C, int L, bool INV, int NF, int p, class SI, class TW>
__device__ __forceinline__ void fft_passes(C (&v)[NF][8], C* sm, int fstride, const TW* __restrict__ tw,
                                           int t, const SI& si) {
  using PL = Plan<L>;
  constexpr int r = PL::rad(INV, p);
  constexpr int Ns = PL::ns(INV, p);
  constexpr int NB = 8 / r;
  constexpr int TPL = PL::TPL;
  constexpr int STW = L / (Ns * r);
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    const int j = t + b * TPL;
    if constexpr (Ns > 1) {
      const int k = j % Ns;
#pragma unroll
      for (int q = 1; q < r; ++q) {
        const TW w = tw[q * k * STW];
#pragma unroll
        for (int f = 0; f < NF; ++f) v[f][b * r + q] = INV ? cmulc(v[f][b * r + q], w) : cmul(v[f][b * r + q], w);
      }
    }
#pragma unroll
    for (int f = 0; f < NF; ++f) dft_r<r, INV>(&v[f][b * r]);
  }
  if constexpr (p + 1 < PL::P) {
    // exchange p goes through the second buffer when p is even (column lines)
    C* xb = sm;
    if constexpr (PingPong<SI>::v) {
      if constexpr ((p & 1) == 0) xb = sm + si.alt;
    }
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const int j = t + b * TPL;
      const int base = (j / Ns) * Ns * r + (j % Ns);
#pragma unroll
      for (int q = 0; q < r; ++q) {
        const int o = si(base + q * Ns);
#pragma unroll
        for (int f = 0; f < NF; ++f) xb[f * fstride + o] = v[f][b * r + q];
      }
    }
    line_sync<SI>();
    constexpr int r2 = PL::rad(INV, p + 1);
    constexpr int NB2 = 8 / r2;
#pragma unroll
    for (int b = 0; b < NB2; ++b) {
      const int j = t + b * TPL;
#pragma unroll
      for (int q = 0; q < r2; ++q) {
        const int o = si(j + q * (L / r2));
#pragma unroll
        for (int f = 0; f < NF; ++f) v[f][b * r2 + q] = xb[f * fstride + o];
      }
    }
    if constexpr (!PingPong<SI>::v) line_sync<SI>();
    fft_passes<C, L, INV, NF, p + 1, SI, TW>(v, sm, fstride, tw, t, si);
  }
}

// DFT of 6 = 2 x 3, 10 = 2 x 5 or 12 = 4 x 3 points by the prime-factor algorithm
// (Good, Thomas): with n = NB na + NA nb and k = ka mod NA, kb mod NB the transform
// is NB DFTs of NA points and NA DFTs of NB points without twiddles.
template <int N, bool INV, class C> __device__ __forceinline__ void dft_pfa(C (&x)[N]) {
  constexpr int NA = N == 12 ? 4 : 2, NB = N / NA;
  C u[NA][NB];
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    C a[NA];
#pragma unroll
    for (int q = 0; q < NA; ++q) a[q] = x[(NB * q + NA * b) % N];
    dft_r<NA, INV>(a);
#pragma unroll
    for (int q = 0; q < NA; ++q) u[q][b] = a[q];
  }
#pragma unroll
  for (int q = 0; q < NA; ++q) dft_r<NB, INV>(u[q]);
#pragma unroll
  for (int k = 0; k < N; ++k) x[k] = u[k % NA][k % NB];
}

// Mixed-radix line transform with natural entry and exit layouts (register e of
// thread t holds position t + e L/8).  Input n = t + (L/8) e and output
// k = k1 + 8 k2: thread t's radix-8 DFT over e, the twiddle W_L^{t k1}, and for each
// k1 a DFT over t, taken in place at slots 8 t + k1, which become the outputs
// 8 k2 + k1 in natural order.  Two trips through shared memory and three barriers;
// plans of radix 8 and two more passes took three trips and six (FP32, 96^3: see
// kernels.cuh for the passes).  The eight DFTs go to the line's first eight threads
// (a second round for six); column lines keep whole warps busy or idle.
template <class C, int L, bool INV, int NF, class SI, class TW>
__device__ __forceinline__ void fft_mixed(C (&v)[NF][8], C* sm, int fstride, const TW* __restrict__ tw, int t,
                                          const SI& si) {
  constexpr int N2 = MixedPlan<L>::TPL;
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    dft8<INV>(v[f]);
#pragma unroll
    for (int q = 0; q < 8; ++q) sm[f * fstride + si(8 * t + q)] = v[f][q];
  }
  __syncthreads();
#pragma unroll
  for (int f = 0; f < NF; ++f) {
#pragma unroll
    for (int r = 0; r < (8 + N2 - 1) / N2; ++r) {
      const int k1 = t + r * N2;
      if (k1 < 8) {
        C w[N2];
#pragma unroll
        for (int n = 0; n < N2; ++n) w[n] = sm[f * fstride + si(8 * n + k1)];
#pragma unroll
        for (int n = 1; n < N2; ++n) {
          const TW q = tw[n * k1];
          w[n] = INV ? cmulc(w[n], q) : cmul(w[n], q);
        }
        dft_pfa<N2, INV>(w);
#pragma unroll
        for (int n = 0; n < N2; ++n) sm[f * fstride + si(8 * n + k1)] = w[n];
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int f = 0; f < NF; ++f)
#pragma unroll
    for (int e = 0; e < 8; ++e) v[f][e] = sm[f * fstride + si(t + e * N2)];
  __syncthreads();  // callers may reuse the buffer
}

template <class C, int L, bool INV, int NF, bool WIDE = false, class SI>
__device__ __forceinline__ void fft_line(C (&v)[NF][8], C* sm, int fstride, const C* __restrict__ tw, int t,
                                         const SI& si) {
  if constexpr (std::is_same<C, double2>::value) {
    Q2* qs = reinterpret_cast<Q2*>(sm);
    const TwQ* qt = reinterpret_cast<const TwQ*>(tw);
    Q2 q[NF][8];
    LineScale ls[NF];
    line_scales<L, NF, WIDE>(v, sm, fstride, t, si, ls);
#pragma unroll
    for (int f = 0; f < NF; ++f)
#pragma unroll
      for (int e = 0; e < 8; ++e) q[f][e] = Q2{to_fixed(v[f][e].x, ls[f]), to_fixed(v[f][e].y, ls[f])};
    if constexpr (IsPow2<L>::v) fft_passes<Q2, L, INV, NF, 0, SI, TwQ>(q, qs, fstride, qt, t, si);
    else fft_mixed<Q2, L, INV, NF, SI, TwQ>(q, qs, fstride, qt, t, si);
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      const bool big = WIDE && ls[f].bad == kLineBig;  // exponents 64 lower, then a product that may overflow
      if (big) ls[f] = LineScale{ls[f].X - 64, ls[f].keep, 0};
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        v[f][e] = make_double2(from_fixed(q[f][e].x, ls[f]), from_fixed(q[f][e].y, ls[f]));
        if (big) v[f][e] = make_double2(0x1p64 * v[f][e].x, 0x1p64 * v[f][e].y);
      }
    }
  } else {
    if constexpr (IsPow2<L>::v) fft_passes<C, L, INV, NF, 0, SI, C>(v, sm, fstride, tw, t, si);
    else fft_mixed<C, L, INV, NF, SI, C>(v, sm, fstride, tw, t, si);
  }
}

// Shared-memory index maps.  Row tiles (lines contiguous in global memory):
// one padded line per row, one pad element per 128 bytes to break the
// power-of-two strides of the Stockham writes.  Column tiles (lines strided
// in global memory, M adjacent lines per tile): position-major, so each
// quarter/half warp touches one 128-byte row of the tile.
template <int PADSHIFT> struct RowIdx {
  __device__ __forceinline__ int operator()(int pos) const { return pos + (pos >> PADSHIFT); }
};
// MC > 0: the tile width M is the compile-time constant MC (the default tile
// rows), so the exchange offsets fold into the shared-memory instructions;
// MC = 0: M at run time (the other tile widths).
template <int MC> struct ColIdxT {
  int M;
  int alt;    // offset (elements) of the second exchange buffer from the first
  uint2* sc;  // this column's slots of the FP64 line scales, one per thread of the line, M apart
  __device__ __forceinline__ int width() const { return MC > 0 ? MC : M; }
  __device__ __forceinline__ int operator()(int pos) const { return pos * width(); }
};
// Bytes of those slots in a column block of `threads` threads (FP64 only).
template <class R> __host__ __device__ constexpr size_t line_slots(int threads) {
  return sizeof(R) == sizeof(double) ? (size_t)threads * sizeof(uint2) : 0;
}
using ColIdx = ColIdxT<0>;
// A column transform of power-of-two length L makes P - 1 exchanges, the first
// through the second buffer.  When that count is odd the transform ends having
// written the second buffer last, so a following transform of the same line
// starts with the roles of the buffers swapped (its first exchange then writes
// the buffer whose last reads preceded the earlier barrier).
template <int L, class C, class SI> __device__ __forceinline__ void col_after(C*& sm, SI& si) {
  if constexpr (IsPow2<L>::v) {
    if constexpr (((Plan<L>::P - 1) & 1) != 0) {
      sm += si.alt;
      si.alt = -si.alt;
    }
  }
}
template <class R> struct PadShift;
template <> struct PadShift<double> { static constexpr int v = 3; };  // 8 x 16 B
template <> struct PadShift<float> { static constexpr int v = 4; };   // 16 x 8 B
template <class R, int L> __host__ __device__ constexpr int row_len_padded() {
  return L + (L >> PadShift<R>::v);
}

}  // namespace egpe
