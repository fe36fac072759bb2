// xfix.cuh -- 64-bit block-floating arithmetic on the integer pipes, and the Roe flux written in
// it for the FP64 path.
//
// Why.  This part issues one FP64 operation per 64 FP32 or integer ones: a warp's DADD or DMUL
// holds its sub-partition's FP64 lanes for 76 cycles, a DFMA for 64, while the integer pipes
// idle.  A 64-bit integer add takes 2 issue slots there, an arithmetic 64-bit shift 4, and the
// upper part of a 64 x 64 product about 12 (three 32 x 32 multiply-adds).  So the FP64 path's
// primitives, face fluxes and residuals are evaluated on 62-bit signed mantissas with an integer
// exponent each, in which a rounding is about 2^-57 of its class's largest value (FP64: 2^-53),
// and a result is rounded once to a double.
//
// A value is m 2^(E - 61), m a signed 64-bit integer, E an int.  Values that are added share E:
// before a sum the terms are shifted right to the sum's class, a bound on every |m| being known
// from the class (written beside each line as the number of bits), so nothing overflows for any
// finite input.  Sums then cost one 64-bit add.  Truncation is towards minus infinity.
//
// What shares a class: only terms that are added, and then a term that is far below its class (a difference, a
// product, a component that vanishes) is normalised before the class of the sum is taken, an exact zero having an exponent
// below all (XZERO): no term takes bits from another that is not there.  Sides of a face that are far apart go to
// FP64 (xfar), and so do edge values that are small in their stencil.  tests/test_xfix_classes.py holds each component's error to
// the FP64 form's; on smooth states the flux's is 4.5-6e-17 of its size (root mean square, the rounding to a double
// included) where that form's is 8-16e-17.
//
// The scheme is plain fixed-point arithmetic with scaling by exponents ("block floating point",
// J. H. Wilkinson, Rounding Errors in Algebraic Processes, 1963, ch. 1).
#pragma once

namespace gbcfd {

struct XVal {
  long long m;
  int e;
};

// (a b) >> 64, |a|, |b| < 2^63 - 2^31.  Each operand is split as h 2^32 + l with both halves signed (l
// the low word read as signed, its sign carried into h); of the four signed 32 x 32 products the
// upper one is kept whole, the middle ones by their upper words, l_a l_b not at all: the error is
// at most 2.25 units, and a zero factor gives zero (a velocity that is zero stays exactly zero).  So written it is three
// multiply-adds and a sign extension; the form that keeps the middle sum's 64 bits is 17
// instructions (opcode counts) for two more bits.
__host__ __device__ __forceinline__ int xmulhi(int a, int b) {
#ifdef __CUDA_ARCH__
  return __mulhi(a, b);
#else
  return (int)(((long long)a * b) >> 32);
#endif
}
__host__ __device__ __forceinline__ int xhi(long long a) {
  return (int)(a >> 32) + (int)((unsigned)(int)a >> 31);
}
__host__ __device__ __forceinline__ long long xmul(long long a, long long b) {
  const int al = (int)a, bl = (int)b, ah = xhi(a), bh = xhi(b);
  const int s = xmulhi(ah, bl) + xmulhi(al, bh);
  return (long long)ah * bh + s;
}
__host__ __device__ __forceinline__ long long xsq(long long a) {
  const int al = (int)a, ah = xhi(a);
  const int s = xmulhi(ah, al);
  return (long long)ah * ah + 2 * s;
}
// arithmetic shift right by s >= 0, any size (a shift of 64 or more leaves the sign)
__host__ __device__ __forceinline__ long long xshr(long long a, int s) {
#ifdef __CUDA_ARCH__
  long long r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(a), "r"(s));  // the hardware clamps the amount
  return r;
#else
  return a >> (s < 63 ? s : 63);
#endif
}
__host__ __device__ __forceinline__ int xmax(int a, int b) { return a > b ? a : b; }
__host__ __device__ __forceinline__ long long xabs(long long a) { return a < 0 ? -a : a; }

__host__ __device__ __forceinline__ unsigned long long xbits(double a) {
#ifdef __CUDA_ARCH__
  return (unsigned long long)__double_as_longlong(a);
#else
  unsigned long long b;
  __builtin_memcpy(&b, &a, 8);
  return b;
#endif
}
__host__ __device__ __forceinline__ double xdouble(unsigned long long b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double a;
  __builtin_memcpy(&a, &b, 8);
  return a;
#endif
}
__host__ __device__ __forceinline__ int xclz(unsigned long long a) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)a);
#else
  return a ? __builtin_clzll(a) : 64;
#endif
}

// a finite double as a value with 2^(B-1) <= |m| < 2^B, B = 61 or 62.  A zero or subnormal reads as
// +-2^-1022, far below everything it is added to (an exact zero is only needed of differences,
// and those of equal inputs are exact).
template <int B>
__host__ __device__ __forceinline__ XVal xdec(double a) {
  const unsigned long long b = xbits(a);
  const int hi = (int)(b >> 32);
  const unsigned long long mag = ((unsigned long long)(((unsigned)hi & 0xfffffu) | 0x100000u) << 32) | (unsigned)b;
  const long long s = hi >> 31;
  return {((long long)(mag << (B - 53)) ^ s) - s, (int)(((unsigned)hi >> 20) & 0x7ffu) - 1023 + (62 - B)};
}
template <int B>
__host__ __device__ __forceinline__ XVal xdec_pos(double a) {  // a > 0
  const unsigned long long b = xbits(a);
  const unsigned hi = (unsigned)(b >> 32);
  const unsigned long long mag = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | (unsigned)b;
  return {(long long)(mag << (B - 53)), (int)((hi >> 20) & 0x7ffu) - 1023 + (62 - B)};
}
// the exponent of an exact zero: below that of any product of doubles, so that a zero takes no part in the
// class of a sum
constexpr int XZERO = -8000;
// any finite double [62]: a zero as zero, a subnormal with its own (fewer) bits
__host__ __device__ __forceinline__ XVal xdec_zero(double a) {
  const unsigned long long b = xbits(a);
  const int hi = (int)(b >> 32), ex = (int)(((unsigned)hi >> 20) & 0x7ffu);
  const unsigned long long mag = ((unsigned long long)(((unsigned)hi & 0xfffffu) | (ex ? 0x100000u : 0u)) << 32) | (unsigned)b;
  const long long s = hi >> 31;
  return {((long long)(mag << 9) ^ s) - s, ex ? ex - 1023 : (mag ? -1022 : XZERO)};
}
// the double nearest to m 2^(e - 61), |m| < 2^63; below the normal range subnormal, above it infinity, and
// NaN for the exponents from XBAD up (a flux that has no value)
constexpr int XBAD = 8192;
__host__ __device__ __forceinline__ int xclz32(int a) {
#ifdef __CUDA_ARCH__
  return __clz(a);
#else
  return a ? __builtin_clz((unsigned)a) : 32;
#endif
}
__host__ __device__ inline double xenc_rare(long long m, int e) {
  const long long s = m >> 63;
  unsigned long long a = (unsigned long long)((m ^ s) - s);
  const int n = xclz(a);
  a <<= (n & 63);
  const int f = e + 2 - n + 1022;  // biased exponent - 1
  unsigned long long b = ((unsigned long long)(unsigned)f << 52) + (a >> 11) + ((a >> 10) & 1ull);
  if ((unsigned)f >= 2046u) b = 0x7ff0000000000000ull;
  if (f < 0) b = f < -53 ? 0ull : ((a >> (10 - f)) + 1ull) >> 1;
  if (a == 0ull) b = 0ull;
  if (e >= XBAD) b = 0x7ff8000000000000ull;
  return xdouble(b | ((unsigned long long)s & 0x8000000000000000ull));
}
__host__ __device__ __forceinline__ double xenc(long long m, int e) {
  const long long s = m >> 63;
  unsigned long long a = (unsigned long long)((m ^ s) - s);
  const int hi = (int)(a >> 32), n = xclz32(hi);
  const int f = e + 1024 - n;
  if (hi == 0 || (unsigned)f >= 2046u) return xenc_rare(m, e);  // small against its class, or out of range
  a <<= n;
  const unsigned long long b = ((unsigned long long)(unsigned)f << 52) + (a >> 11) + ((a >> 10) & 1ull);
  return xdouble(b | ((unsigned long long)s & 0x8000000000000000ull));
}

// the constants of the Roe flux as values (formed on the host)
struct XConsts {
  XVal ggm1, gm1, eps, gam;  // 62 bits
};
inline XConsts xconsts(double gamma, double eps) {
  return {xdec_pos<62>(gamma / (gamma - 1.0)), xdec_pos<62>(gamma - 1.0), xdec_pos<62>(eps), xdec_pos<62>(gamma)};
}

// shift m left until 2^61 <= |m| < 2^62, lowering its exponent; |m| < 2^62; 0 stays 0
__host__ __device__ __forceinline__ void xnorm(long long& m, int& e) {
  const int n = (xclz((unsigned long long)(m ^ (m >> 63))) - 2) & 63;
  m = (long long)((unsigned long long)m << n);
  e -= n;
}
__host__ __device__ __forceinline__ XVal xnormed(long long m, int e) {
  xnorm(m, e);
  return {m, e};
}
// the same from the upper word alone: at most 30 places, |m| < 2^63 in, [62] out.  For values whose
// later roundings should be relative to them (a value 2^30 times smaller than its class is left
// with 31 leading zeros, its roundings then at 2^-31 of it or 2^-61 of the class)
__host__ __device__ __forceinline__ XVal xquick(long long m, int e) {
  const int hi = (int)(m >> 32);
  const int n = xclz32(hi ^ (hi >> 31)) - 1;  // 0 .. 31
  return {(long long)((unsigned long long)m << n) >> 1, e + 1 - n};
}

// the same, an exact zero with its own exponent (a difference that vanishes)
__host__ __device__ __forceinline__ XVal xquick0(long long m, int e) {
  const XVal r = xquick(m, e);
  return {r.m, m ? r.e : XZERO};
}

// float seeds of the reciprocal (root) of x, 1 <= x < 4
__host__ __device__ __forceinline__ float xseed_rsqrt(float x) {
#ifdef __CUDA_ARCH__
  return rsqrtf(x);
#else
  return 1.0f / __builtin_sqrtf(x);
#endif
}
__host__ __device__ __forceinline__ float xseed_rcp(float x) {
#ifdef __CUDA_ARCH__
  return __fdividef(1.0f, x);
#else
  return 1.0f / x;
#endif
}
// y0 (1 + H 2^-60) as a 62-bit value, y0 = Y 2^-30 <= 1 (the root or reciprocal of a number in [1, 4))
__host__ __device__ __forceinline__ long long xcorrect(int Y, long long H) {
  const unsigned long long lo = (unsigned long long)(unsigned)Y * (unsigned)H;
  const long long hi = (long long)Y * (int)(H >> 32);
  const long long y = ((long long)Y << 32) + (long long)(lo >> 28) + (hi << 4);
  return y - (y >> 62);  // 1 itself becomes 1 - 2^-62
}
// 1 / sqrt(v), v > 0 normalised to [62]: the hardware's float estimate (relative error below 2^-21)
// and one step of the third-order iteration y (1 + e/2 + 3 e^2 / 8), e = 1 - v y^2 (Householder's
// method); the result's relative error is below 2^-57
__host__ __device__ __forceinline__ XVal xrsqrt(XVal v) {
  const int odd = v.e & 1;
  const long long M = v.m >> (1 - odd);  // f = M 2^-60 in [1, 4), v = f 2^(e - odd)
  const float x = (float)(int)(M >> 32) * (1.0f / 268435456.0f);
  const int Y = (int)(xseed_rsqrt(x) * 1073741824.0f);
  // f y^2 = M Y^2 2^-120: in units of 2^-58
  const long long e = (1ll << 58) - xmul(M, ((long long)Y * Y) << 2);
  const int es = (int)(e >> 16);  // units of 2^-42
  return {xcorrect(Y, 2 * e + ((3 * ((long long)es * es)) >> 27)), -((v.e - odd) >> 1) - 1};
}
// 1 / v, v > 0 normalised to [62]: the estimate and y (1 + e + e^2), e = 1 - v y
__host__ __device__ __forceinline__ XVal xrcp(XVal v) {
  const float x = (float)(int)(v.m >> 32) * (1.0f / 536870912.0f);
  const int Y = (int)(xseed_rcp(x) * 1073741824.0f);
  const unsigned long long t = (unsigned long long)(unsigned)v.m * (unsigned)Y;
  const long long r = (long long)(int)(v.m >> 32) * Y + (long long)(t >> 32);  // v.m Y >> 32
  const long long e = (1ll << 60) - ((r << 1) | (long long)((t >> 31) & 1ull));
  const int es = (int)(e >> 18);
  return {xcorrect(Y, e + (((long long)es * es) >> 24)), -v.e - 1};
}

// (x^2 + d^2) / (2 d) in the class of x and d, 0 <= x < d < 2^62: Harten's fix of |x| < d.  n =
// leading zeros that bring d to 62 bits, h 2^-62 = 1 / (d 2^n 2^-61)
struct XHid {
  long long h;
  int n;
};
__host__ __device__ __forceinline__ XHid xhid(long long d) {
  XHid r;
  r.n = (xclz((unsigned long long)d) - 2) & 63;  // d > 0 where it is used
  r.h = xrcp({d << r.n, 0}).m;
  return r;
}
__host__ __device__ __forceinline__ long long xharten(long long x, long long d, const XHid& r) {
  if (x >= d) return x;
  // squares of [62] are [60], class 3; their sum [61] times 1 / (2 d) (e = -1) is [59], class 4; up
  // to class 0, then back by n
  const long long q = xsq(x << r.n) + xsq(d << r.n);
  return xshr(xmul(q, r.h) << 4, r.n);
}

// the two sides of a face: one variable's left and right value in a common class, [62]
struct XPair {
  long long l, r;
  int e;
};
// a face's sides normalised together: the products of xroe are then rounded relative to the larger (edge
// values have up to four spare bits: their squares lost eight, three times the FP64 form's error in
// the energy residual)
__host__ __device__ __forceinline__ XPair xpair_norm(long long l, long long r, int e) {
  const int n = xclz32((int)((l ^ (l >> 63)) >> 32) | (int)((r ^ (r >> 63)) >> 32)) - 2;  // 0 .. 30
  return {l << n, r << n, e - n};
}
// a positive variable's sides: the pair, and either side by itself, normalised to [62]
struct XPos {
  XPair c;
  XVal l, r;
  __host__ __device__ __forceinline__ XPos(const XPair& p) : c(p), l(xquick(p.l, p.e)), r(xquick(p.r, p.e)) {}
};
// sides so far apart (more than 2^5) that the smaller one's bits in the pair's class, or its products in the
// classes of the larger one's, may be fewer than a double's: such a face is left to FP64
__host__ __device__ __forceinline__ bool xfar(const XPos& r, const XPos& p) {
  const int a = r.l.e - r.r.e, b = p.l.e - p.r.e;
  return a > 5 || a < -5 || b > 5 || b < -5;
}
// twice a face flux, each component in its own class, [62]; where a density or c^2 is not
// positive the exponents are XBAD or more (NaN)
struct XFlux {
  long long m[5];
  int e[5];
};

// Twice the Roe flux with Harten's fix in the face frame, as roe_frame (physics.cuh), from the
// sides' (rho, u_n, u_t1, u_t2, p).  [n] after a line: |m| < 2^n.  A product of [a] and [b] is
// [a + b - 64] with exponent e_a + e_b + 3; << 2 then brings [60] back to [62].  Classes: Eu, Ev, Ew of
// the velocities, EH of the enthalpies, Ek of q^2/2, El of the wave speeds, EM of the mass fluxes.
// Where a value may be much smaller than its class (jumps, products of several factors) it is
// normalised, so that later roundings are relative to it.
// CURVI: (u, v, w) are the x, y, z velocities, un the velocity along the face normal n, whose components have their
// own classes (a component that is zero or small on the face keeps the pressure's class out of that momentum);
// the shear jumps are du - dun n, so the momentum flux is a x, y, z vector and needs no
// tangents.
template <bool CURVI>
__host__ __device__ __forceinline__ void xroe(const XPos& r, const XPair& u, const XPair& v, const XPair& w,
                                              const XPos& p, const XConsts& K, XFlux& F, const XPair& un,
                                              const XVal* n) {
  const int Eu = u.e, Ev = v.e, Ew = w.e, Ep = p.c.e, En = CURVI ? un.e : Eu;
  const long long ul = u.l, ur = u.r, vl = v.l, vr = v.r, wl = w.l, wr = w.r;
  // densities and pressures by themselves; reciprocal roots; the Roe weights a_l = isr iw,
  // a_r = isl iw with iw = 1 / (isl + isr), class -1 (below 1, so [62])
  const XVal rl = r.l, rr = r.r, pl = p.l, pr = p.r;  // [62]
  const XVal isl = xrsqrt(rl), isr = xrsqrt(rr);
  const int Ei = xmax(isl.e, isr.e) + 1;
  const XVal iw = xrcp(xnormed(xshr(isl.m, Ei - isl.e) + xshr(isr.m, Ei - isr.e), Ei));
  const long long al = xshr(xmul(isr.m, iw.m) << 3, -1 - (isr.e + iw.e));
  const long long ar = xshr(xmul(isl.m, iw.m) << 3, -1 - (isl.e + iw.e));
  // sqrt(rho_l rho_r)
  const XVal rt = xquick(xmul(xmul(rl.m, isl.m) << 2, xmul(rr.m, isr.m) << 2), rl.e + isl.e + rr.e + isr.e + 5);  // [62]
  // mass fluxes
  const long long nl = CURVI ? un.l : ul, nr = CURVI ? un.r : ur;
  const XVal ml = xquick(xmul(rl.m, nl), rl.e + En + 3), mr = xquick(xmul(rr.m, nr), rr.e + En + 3);  // [62]
  // enthalpies gamma/(gamma-1) p / rho + |u|^2 / 2, each side in its own class
  const XVal gl = xquick(xmul(K.ggm1.m, xmul(pl.m, xsq(isl.m) << 2) << 2), K.ggm1.e + pl.e + 2 * isl.e + 5);  // [62]
  const XVal gr = xquick(xmul(K.ggm1.m, xmul(pr.m, xsq(isr.m) << 2) << 2), K.ggm1.e + pr.e + 2 * isr.e + 5);
  const int Ek = 2 * xmax(xmax(Eu, Ev), Ew) + 2;
  const int EHl = xmax(gl.e, Ek) + 1, EHr = xmax(gr.e, Ek) + 1, EH = xmax(EHl, EHr) + 2;
  const long long hl = xshr(gl.m, EHl - gl.e) + xshr(xsq(ul), EHl - 2 * Eu - 2) + xshr(xsq(vl), EHl - 2 * Ev - 2) +
                       xshr(xsq(wl), EHl - 2 * Ew - 2);  // [62]
  const long long hr = xshr(gr.m, EHr - gr.e) + xshr(xsq(ur), EHr - 2 * Eu - 2) + xshr(xsq(vr), EHr - 2 * Ev - 2) +
                       xshr(xsq(wr), EHr - 2 * Ew - 2);
  // Roe averages: velocities in the classes of the sides [62]; enthalpy in class EH [60], q^2 / 2 in
  // its own, Ek (in the enthalpies' the entropy wave's energy at a contact of 1 to 100 had 5e-15 of itself in error)
  const long long ut = (xmul(al, ul) + xmul(ar, ur)) << 2;
  const long long vt = (xmul(al, vl) + xmul(ar, vr)) << 2;
  const long long wt = (xmul(al, wl) + xmul(ar, wr)) << 2;
  const long long nt = CURVI ? (xmul(al, nl) + xmul(ar, nr)) << 2 : ut;
  const long long ht = xshr(xmul(al, hl), EH - EHl - 2) + xshr(xmul(ar, hr), EH - EHr - 2);
  const long long q2 = xshr(xsq(ut), Ek - 2 * Eu - 2) + xshr(xsq(vt), Ek - 2 * Ev - 2) + xshr(xsq(wt), Ek - 2 * Ew - 2);
  const long long c2m = xmul(K.gm1.m, ht - xshr(q2, EH - Ek));
  const bool bad = r.c.l <= 0 || r.c.r <= 0 || c2m <= 0;
  // c^2 normalised, its reciprocal root, c
  const XVal c2 = xnormed(c2m, K.gm1.e + EH + 3);
  const XVal ic = xrsqrt(c2);
  const long long ic2 = xsq(ic.m) << 2;       // [62], class 2 ic.e + 1
  const long long cc = xmul(c2.m, ic.m) << 2;  // [62]
  const int Ec = c2.e + ic.e + 1;
  // wave speeds, |u_n| in its own class unless Harten's fix replaces it; room for delta = eps (|u| + c) where eps >= 1
  const int hx = K.eps.e >= 0 ? K.eps.e + 1 : 0;
  const int El = xmax(En, Ec) + 1 + hx;
  const long long ue = xshr(nt, El - En), ce = xshr(cc, El - Ec);  // [61]
  long long l1 = xabs(ue - ce), l5 = xabs(ue + ce);  // [62]
  const long long ua = xabs(ue);
  XVal l2 = {xabs(nt), En};
  {
    long long d = xmul(K.eps.m, ua + ce);  // class El + eps.e + 3
    d = K.eps.e >= -3 ? d << (K.eps.e + 3) : xshr(d, -3 - K.eps.e);  // [62]
    if (l1 < d || ua < d || l5 < d) {
      const XHid hid = xhid(d);
      l1 = xharten(l1, d, hid);
      if (ua < d) l2 = {xharten(ua, d, hid), El};
      l5 = xharten(l5, d, hid);
    }
  }
  // jumps, normalised [62], and wave strengths: a1, a5 = (dp -+ rho c du) / (2 c^2), a2 = drho - dp / c^2
  const XVal jr = xquick0(r.c.r - r.c.l, r.c.e), ju = xquick(nr - nl, En), jv = xquick(vr - vl, Ev),
             jw = xquick(wr - wl, Ew), jp = xquick0(p.c.r - p.c.l, Ep);
  const XVal rcd = xquick(xmul(xmul(rt.m, cc) << 2, ju.m), rt.e + Ec + ju.e + 4);
  const int Eq = xmax(rcd.e, jp.e) + 1;
  const long long dp = xshr(jp.m, Eq - jp.e), rq = xshr(rcd.m, Eq - rcd.e);               // [61]
  const int Ea = Eq + 2 * ic.e + 3;                                                       // (the half included)
  const XVal a1 = xquick(xmul(dp - rq, ic2), Ea), a5 = xquick(xmul(dp + rq, ic2), Ea);
  const int Ew15 = El + 3 + xmax(a1.e, a5.e);
  const long long w1 = xshr(xmul(l1, a1.m), Ew15 - El - 3 - a1.e), w5 = xshr(xmul(l5, a5.m), Ew15 - El - 3 - a5.e);  // [60]
  const XVal s = xquick(w1 + w5, Ew15), dw = xquick(w5 - w1, Ew15);                       // [62]
  const int Ed = jp.e + 2 * ic.e + 4, EA = xmax(Ed, jr.e + 2);
  const XVal a2 = xquick(xshr(jr.m, EA - jr.e) - xshr(xmul(jp.m, ic2), EA - Ed), EA);
  const XVal w2 = xquick(xmul(l2.m, a2.m), l2.e + a2.e + 3);                              // [62]
  // in the class of the mass fluxes [60]
  const int EM = xmax(xmax(ml.e, mr.e), xmax(s.e, w2.e)) + 2;
  const long long fl = xshr(ml.m, EM - ml.e), fr = xshr(mr.m, EM - mr.e);
  const long long ws = xshr(s.m, EM - s.e) + xshr(w2.m, EM - w2.e);
  const long long dq = xmul(dw.m, cc);                                  // [60]
  const XVal lrt = xquick(xmul(l2.m, rt.m), l2.e + rt.e + 3);           // [62]
  const long long g1 = xmul(lrt.m, jv.m), g2 = xmul(lrt.m, jw.m);       // [60]
  const int Edq = dw.e + Ec + 3, Eg1 = lrt.e + jv.e + 3, Eg2 = lrt.e + jw.e + 3;
  const long long a1m = xmul(fl, ul) + xmul(fr, ur) - xmul(ws, ut);  // [60]
  const long long a2m = xmul(fl, vl) + xmul(fr, vr) - xmul(ws, vt);
  const long long a3m = xmul(fl, wl) + xmul(fr, wr) - xmul(ws, wt);
  const int f1 = EM + Eu + 3, f2 = EM + Ev + 3, f3 = EM + Ew + 3;
  const int el = ml.e + EHl + 3, er = mr.e + EHr + 3, e1 = s.e + EH + 3, e2 = Edq + En + 3, e3 = Eg1 + Ev + 3, e4 = Eg2 + Ew + 3,
            e5 = w2.e + Ek + 3;
  const int E4 = xmax(xmax(xmax(el, er), xmax(e1, e2)), xmax(xmax(e3, e4), e5));
  const long long a4 = xshr(xmul(ml.m, hl), E4 - el) + xshr(xmul(mr.m, hr), E4 - er);  // terms [60]
  const long long b4 = xshr(xmul(s.m, ht), E4 - e1) + xshr(xmul(w2.m, q2), E4 - e5);
  long long d4 = xshr(xmul(dq, nt), E4 - e2) + xshr(xmul(g1, vt), E4 - e3) + xshr(xmul(g2, wt), E4 - e4);
  F.m[0] = fl + fr - ws;
  F.e[0] = EM;
  if constexpr (!CURVI) {
    F.e[1] = xmax(xmax(f1, Edq), Ep + 2);
    F.e[2] = xmax(f2, Eg1);
    F.e[3] = xmax(f3, Eg2);
    F.m[1] = xshr(a1m, F.e[1] - f1) + xshr(p.c.l + p.c.r, F.e[1] - Ep) - xshr(dq, F.e[1] - Edq);
    F.m[2] = xshr(a2m, F.e[2] - f2) - xshr(g1, F.e[2] - Eg1);
    F.m[3] = xshr(a3m, F.e[3] - f3) - xshr(g2, F.e[3] - Eg2);
  } else {
    const XVal jx = xquick(ur - ul, Eu);
    const long long g0 = xmul(lrt.m, jx.m), gn = xmul(lrt.m, ju.m);  // [60]
    const int Eg0 = lrt.e + jx.e + 3, Egn = lrt.e + ju.e + 3;
    const int EP = xmax(xmax(Edq, Egn), Ep + 2);
    const XVal P = xquick(xshr(p.c.l + p.c.r, EP - Ep) - xshr(dq, EP - Edq) + xshr(gn, EP - Egn), EP);  // along n, [62]
    const int p0 = P.e + n[0].e + 3, p1 = P.e + n[1].e + 3, p2 = P.e + n[2].e + 3;                   // P n_x [60]
    F.e[1] = xmax(xmax(f1, p0), Eg0);
    F.e[2] = xmax(xmax(f2, p1), Eg1);
    F.e[3] = xmax(xmax(f3, p2), Eg2);
    F.m[1] = xshr(a1m, F.e[1] - f1) + xshr(xmul(P.m, n[0].m), F.e[1] - p0) - xshr(g0, F.e[1] - Eg0);
    F.m[2] = xshr(a2m, F.e[2] - f2) + xshr(xmul(P.m, n[1].m), F.e[2] - p1) - xshr(g1, F.e[2] - Eg1);
    F.m[3] = xshr(a3m, F.e[3] - f3) + xshr(xmul(P.m, n[2].m), F.e[3] - p2) - xshr(g2, F.e[3] - Eg2);
    // shear work ut . (du - dun n); class E4 may be below these terms' own: they are aligned both ways
    const int e0 = Eg0 + Eu + 3, en = Egn + En + 3, E5 = xmax(E4, xmax(e0, en));
    d4 = xshr(d4, E5 - E4) + xshr(xmul(g0, ut), E5 - e0) - xshr(xmul(gn, nt), E5 - en);
    F.e[4] = E5;
    F.m[4] = xshr(a4 - b4, E5 - E4) - d4;
  }
  if constexpr (!CURVI) {
    F.e[4] = E4;
    F.m[4] = a4 - b4 - d4;
  }
  if (bad) {
    F.e[0] = F.e[1] = F.e[2] = F.e[3] = F.e[4] = 2 * XBAD;
  }
}
__host__ __device__ __forceinline__ void xroe(const XPos& r, const XPair& u, const XPair& v, const XPair& w,
                                              const XPos& p, const XConsts& K, XFlux& F) {
  xroe<false>(r, u, v, w, p, K, F, u, nullptr);
}

// the unit normal, each component in its own class [62], and half the length of a face's area vector
struct XNormal {
  XVal n[3];
  XVal half;
};
__host__ __device__ __forceinline__ XNormal xnormal(double sx, double sy, double sz) {
  const XVal a = xdec_zero(sx), b = xdec_zero(sy), c = xdec_zero(sz);
  const int E = xmax(a.e, xmax(b.e, c.e));
  const XVal s2 = xnormed(xsq(xshr(a.m, E - a.e)) + xsq(xshr(b.m, E - b.e)) + xsq(xshr(c.m, E - c.e)), 2 * E + 3);
  const XVal ia = xrsqrt(s2);
  XNormal N;
  N.n[0] = {xmul(a.m, ia.m) << 2, a.e + ia.e + 1};
  N.n[1] = {xmul(b.m, ia.m) << 2, b.e + ia.e + 1};
  N.n[2] = {xmul(c.m, ia.m) << 2, c.e + ia.e + 1};
  N.half = {xmul(s2.m, ia.m) << 2, s2.e + ia.e};
  return N;
}

// twice the flux through a face of area vector (sx, sy, sz) from the sides' (rho, u, v, w, p), x, y, z
// momentum, times half the area: the face flux itself
__host__ __device__ __forceinline__ void xroe_area(const XPos& r, const XPair& u, const XPair& v, const XPair& w,
                                                   const XPos& p, double sx, double sy, double sz, const XConsts& K,
                                                   XFlux& F) {
  const XNormal N = xnormal(sx, sy, sz);
  // the velocities along n, in the class of the largest product ([60] each)
  const int e0 = u.e + N.n[0].e + 3, e1 = v.e + N.n[1].e + 3, e2 = w.e + N.n[2].e + 3, E = xmax(xmax(e0, e1), e2);
  auto dot = [&](long long a, long long b, long long c) {
    return xshr(xmul(a, N.n[0].m), E - e0) + xshr(xmul(b, N.n[1].m), E - e1) + xshr(xmul(c, N.n[2].m), E - e2);
  };
  const XPair un = xpair_norm(dot(u.l, v.l, w.l), dot(u.r, v.r, w.r), E);
  xroe<true>(r, u, v, w, p, K, F, un, N.n);
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int q = 0; q < 5; ++q) {
    const XVal f = xquick(F.m[q], F.e[q]);
    F.m[q] = xmul(f.m, N.half.m);
    F.e[q] = f.e + N.half.e + 3;
  }
}

// a flux given in doubles
__host__ __device__ __forceinline__ XFlux xflux_of(const double* f) {
  XFlux F;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int q = 0; q < 5; ++q) {
    const XVal v = xdec_zero(f[q]);
    F.m[q] = v.m;
    F.e[q] = v.e < 1024 ? v.e : 2 * XBAD;
  }
  return F;
}
// a flux component as a double, times 2^-h; below the normal range zero
__host__ __device__ __forceinline__ double xflux(const XFlux& F, int q, int h) {
  const double f = xenc(F.m[q], F.e[q] - h);
  return (xbits(f) & 0x7ff0000000000000ull) == 0ull ? 0.0 : f;
}
// ---- MUSCL ---------------------------------------------------------------------------------------
// half the minmod slope's double: 0 when a and b differ in sign, else the one of smaller magnitude
__host__ __device__ __forceinline__ long long xminmod(long long a, long long b) {
  const long long r = ((a < b) != (a < 0)) ? a : b;
  return (a ^ b) < 0 ? 0ll : r;
}
// the sides of the face between cells 1 and 2 of a stencil of four [61] (normalised but for zeros and the
// smallest doubles) and for the viscous flux the difference and the sum of these two, class ed
struct XSten {
  XPair s;
  long long d, sum;
  int ed;
};
// With minmod the states lie between cells 1 and 2 and keep their class: a cell 0 or 3 that is larger by
// more than 2^4 only has to give a slope larger than theirs, which it also does shifted into 2^4 times
// that class (|m| >= 2^59 against a difference below 2^58).  In the class of all four a state beside a jump
// had lost as many bits as the jump is high, less 8.  Doubled (class e - 1); with the central slope, where
// the larger cell is a term of the state, the class of all four, not doubled.
__host__ __device__ __forceinline__ XSten xmuscl(const long long (&m)[4], const int (&e)[4], int lim) {
  const int Ei = xmax(e[1], e[2]), Eo = xmax(e[0], e[3]), Ec = Ei + 4, E = xmax(Ei, lim || Eo < Ec ? Eo : Ec);
  const long long m0 = xshr(m[0], xmax(E - e[0], 0)), m1 = xshr(m[1], E - e[1]), m2 = xshr(m[2], E - e[2]),
                  m3 = xshr(m[3], xmax(E - e[3], 0));
  const long long d01 = m1 - m0, d12 = m2 - m1, d23 = m3 - m2;
  XSten S;
  S.d = d12;
  S.sum = m1 + m2;
  S.ed = E;
  if (lim) S.s = xpair_norm(m1 + ((d01 + d12) >> 2), m2 - ((d12 + d23) >> 2), E);
  else S.s = {(2 * m1 + xminmod(d01, d12)) << (E - Ei), (2 * m2 - xminmod(d12, d23)) << (E - Ei), Ei - 1};
  return S;
}

// both sides of one variable from doubles
__host__ __device__ __forceinline__ XPair xpair(double l, double r) {
  const XVal a = xdec<62>(l), b = xdec<62>(r);
  const int e = xmax(a.e, b.e);
  return {xshr(a.m, e - a.e), xshr(b.m, e - b.e), e};
}
// the primitives of a conserved state (rho, rho u, rho v, rho w, rho E): velocities [62] and pressure
// [62] each in its own class, 1 / rho; false where the density or the pressure is not positive or
// not finite
struct XPrim {
  XVal r, ir, u[3], p;
};
__host__ __device__ __forceinline__ bool xprim(const double* q, const XConsts& K, XPrim& W) {
  W.r = xdec_pos<62>(q[0]);
  W.ir = xrcp(W.r);
  const XVal E = xdec_zero(q[4]);
  long long k[3];
  int ek[3];
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int x = 0; x < 3; ++x) {
    const XVal m = xdec_zero(q[1 + x]);
    W.u[x].m = xmul(m.m, W.ir.m) << 2;
    W.u[x].e = m.e + W.ir.e + 1;
    k[x] = xmul(m.m, W.u[x].m);  // [60]; rho u^2 / 2 with the exponent lowered by 1
    ek[x] = m.e + W.u[x].e + 2;
  }
  const int Ek = xmax(xmax(ek[0], ek[1]), xmax(ek[2], E.e + 2));
  const long long d = xshr(E.m, Ek - E.e) - xshr(k[0], Ek - ek[0]) - xshr(k[1], Ek - ek[1]) - xshr(k[2], Ek - ek[2]);
  W.p = xnormed(xmul(K.gm1.m, d), K.gm1.e + Ek + 3);
  const long long br = (long long)xbits(q[0]);
  // a non-finite momentum or energy has the exponent 1024
  return br > 0 && br < 0x7ff0000000000000ll && W.p.m > 0 && E.e < 1024 && W.u[0].e - W.ir.e < 1025 &&
         W.u[1].e - W.ir.e < 1025 && W.u[2].e - W.ir.e < 1025;
}
// c = sqrt(gamma p / rho), [62]
__host__ __device__ __forceinline__ XVal xsound(const XPrim& W, const XVal& gam) {
  const XVal c2 = xnormed(xmul(gam.m, xmul(W.p.m, W.ir.m) << 2), gam.e + W.p.e + W.ir.e + 4);
  const XVal ic = xrsqrt(c2);
  return {xmul(c2.m, ic.m) << 2, c2.e + ic.e + 1};
}

// the spectral-radius rate of a cell, normalised: uniform grids, (|u| + c) / hx + (|v| + c) / hy +
// (|w| + c) / hz (+ vs / rho, viscous), from h2 = 1 / (2 h), hsum = the sum of 1 / h
template <bool VISC>
__host__ __device__ __forceinline__ XVal xrate(const XPrim& W, const XVal& c, const XVal* h2, const XVal& hsum,
                                               const XVal& vs) {
  long long t[5];
  int e[5];
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int a = 0; a < 3; ++a) {
    t[a] = xmul(xabs(W.u[a].m), h2[a].m);  // [60]
    e[a] = W.u[a].e + h2[a].e + 4;
  }
  t[3] = xmul(c.m, hsum.m);
  e[3] = c.e + hsum.e + 3;
  t[4] = VISC ? xmul(W.ir.m, vs.m) : 0;
  e[4] = VISC ? W.ir.e + vs.e + 3 : e[3];
  const int E = xmax(xmax(xmax(e[0], e[1]), xmax(e[2], e[3])), e[4]) + 1;
  return xnormed(xshr(t[0], E - e[0]) + xshr(t[1], E - e[1]) + xshr(t[2], E - e[2]) + xshr(t[3], E - e[3]) +
                     xshr(t[4], E - e[4]), E);
}
// curvilinear grids: one direction's part, |u . S| + c |S| (+ f |S|^2, viscous: f = 4 max(4/3, gamma/Pr)
// mu / (rho V)), S the mean of the cell's lower and upper face vectors; [61] or less
template <bool VISC>
__host__ __device__ __forceinline__ XVal xradius(const XPrim& W, const XVal& c, const double* lo, const double* up,
                                                 const XVal& f) {
  long long s[3];
  int es[3];
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int x = 0; x < 3; ++x) {
    const XPair p = xpair(lo[x], up[x]);
    s[x] = (p.l >> 1) + (p.r >> 1);  // [62], the mean in the class itself
    es[x] = p.e;
  }
  const int E = xmax(es[0], xmax(es[1], es[2]));
  long long dot[3], s2 = 0;
  int ec[3];
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int x = 0; x < 3; ++x) {
    s[x] = xshr(s[x], E - es[x]);
    s2 += xsq(s[x]);  // [60] each, class 2 E + 3
    dot[x] = xmul(s[x], W.u[x].m);
    ec[x] = E + W.u[x].e + 3;
  }
  const XVal n2 = xnormed(s2, 2 * E + 3);
  const XVal in = xrsqrt(n2);
  const long long cs = xmul(xmul(n2.m, in.m) << 2, c.m);  // c |S| [60]
  const int ecs = n2.e + in.e + 1 + c.e + 3;
  const long long fs = VISC ? xmul(f.m, n2.m) : 0;
  const int efs = VISC ? f.e + n2.e + 3 : ecs;
  const int e = xmax(xmax(xmax(ec[0], ec[1]), xmax(ec[2], ecs)), efs) + 2;
  return {xabs(xshr(dot[0], e - ec[0]) + xshr(dot[1], e - ec[1]) + xshr(dot[2], e - ec[2])) + xshr(cs, e - ecs) +
              xshr(fs, e - efs), e};
}
__host__ __device__ __forceinline__ XVal xsum3(const XVal& a, const XVal& b, const XVal& c) {  // [60] each
  const int E = xmax(a.e, xmax(b.e, c.e)) + 1;
  return xnormed(xshr(a.m, E - a.e) + xshr(b.m, E - b.e) + xshr(c.m, E - c.e), E);
}

// ---- the viscous flux on uniform grids -------------------------------------------------------------
// a block's coefficients: half the inverse cell sizes (of the doubled face fluxes); the viscous
// ones, 2 mu / h and the tangential 2 mu / (4 h) with the factors 4/3 and 2/3 of the normal
// stress, and 4 kappa / h; for the time step the sum of the inverse sizes and (viscous)
// 4 max(4/3, gamma/Pr) mu (sum of their squares)
struct XBlk {
  XVal h2[3], a[3], a43[3], b[3], b23[3], k[3], hsum, vs;
};
// the sum over a face's two cells of the central differences along a tangent, from the neighbours
// (+, -) of either; ring values [61] with biased exponents
__host__ __device__ __forceinline__ XVal xtang(const long long (&m)[4], const int (&e)[4], int bias) {
  const int E = xmax(xmax(e[0], e[1]), xmax(e[2], e[3])) + 1;  // [60] each
  return xquick0((xshr(m[0], E - e[0]) - xshr(m[1], E - e[1])) + (xshr(m[2], E - e[2]) - xshr(m[3], E - e[3])), E - bias);
}
// Twice the viscous flux of a face normal to direction d, taken from twice the inviscid one: dn the
// differences R - L of the velocities (n, t1, t2) and of theta, us (class eu) the sums of the two
// cells' velocities, gnn1 and gnn2 the tangential sums of u_n along t1 and t2, gt1, gt2 those of u_t1 along t1
// and of u_t2 along t2.  The differences come normalised, exact zeros with XZERO, so that every term of a stress has the
// class of its own size: in the velocities' class a stress of a component 10^6 times smaller than u_n, or
// next to a u_n that does not vary, had lost 20 bits.
__host__ __device__ __forceinline__ void xviscous(int d, int d1, int d2, const XBlk& X, const XVal (&dn)[4],
                                                  const long long (&us)[3], const int (&eu)[3], const XVal& gnn1,
                                                  const XVal& gnn2, const XVal& gt1, const XVal& gt2, XFlux& F) {
  // tau_nn = (4/3) 2 mu dun/dn - (2/3) 2 mu (dut1/dt1 + dut2/dt2), tau_nt = 2 mu (dut/dn + dun/dt); products [60]
  XVal tn, t1, t2;
  {
    const int f0 = X.a43[d].e + dn[0].e + 3, f1 = X.b23[d1].e + gt1.e + 3, f2 = X.b23[d2].e + gt2.e + 3;
    tn.e = xmax(f0, xmax(f1, f2));
    tn.m = xshr(xmul(X.a43[d].m, dn[0].m), tn.e - f0) - xshr(xmul(X.b23[d1].m, gt1.m), tn.e - f1) -
           xshr(xmul(X.b23[d2].m, gt2.m), tn.e - f2);
  }
  {
    const int f0 = X.a[d].e + dn[1].e + 3, f1 = X.b[d1].e + gnn1.e + 3;
    t1.e = xmax(f0, f1);
    t1.m = xshr(xmul(X.a[d].m, dn[1].m), t1.e - f0) + xshr(xmul(X.b[d1].m, gnn1.m), t1.e - f1);
  }
  {
    const int f0 = X.a[d].e + dn[2].e + 3, f2 = X.b[d2].e + gnn2.e + 3;
    t2.e = xmax(f0, f2);
    t2.m = xshr(xmul(X.a[d].m, dn[2].m), t2.e - f0) + xshr(xmul(X.b[d2].m, gnn2.m), t2.e - f2);
  }
  const XVal th = {xmul(X.k[d].m, dn[3].m), X.k[d].e + dn[3].e + 3};
  auto sub = [&](int q, const XVal& t) {
    const int E = xmax(F.e[q], t.e) + 1;
    F.m[q] = xshr(F.m[q], E - F.e[q]) - xshr(t.m, E - t.e);
    F.e[q] = E;
  };
  sub(1, tn);
  sub(2, t1);
  sub(3, t2);
  const int f0 = eu[0] + tn.e + 3, f1 = eu[1] + t1.e + 3, f2 = eu[2] + t2.e + 3;
  const int E = xmax(xmax(f0, f1), xmax(f2, th.e));
  const long long g = xshr(xmul(us[0], tn.m), E - f0) + xshr(xmul(us[1], t1.m), E - f1) +
                      xshr(xmul(us[2], t2.m), E - f2) + xshr(th.m, E - th.e);
  sub(4, {g, E - 1});
}

// ---- WCNS-E-5 lines ----------------------------------------------------------------------------
#ifdef __CUDACC__
#define XNOINLINE __noinline__  // called per variable: inlined five times it was half the kernel's code
#else
#define XNOINLINE
#endif
constexpr int XW_BIAS = 1018;       // staged value = m 2^(e - 1018 - 61), |m| < 2^57
constexpr int XW_BAD = 2 * XBAD;    // exponent of a staged value that is not finite

// a double as a staged value (subnormals with their own bits, a value that is not finite by its exponent)
__host__ __device__ __forceinline__ void xline_value(double v, long long* m, short* e) {
  const unsigned long long bits = xbits(v);
  const int hi = (int)(bits >> 32), ex = (int)(((unsigned)hi >> 20) & 0x7ffu);
  const unsigned long long mag = ((unsigned long long)(((unsigned)hi & 0xfffffu) | (ex ? 0x100000u : 0u)) << 32) | (unsigned)bits;
  const long long sg = hi >> 31;
  *m = ((long long)(mag << 4) ^ sg) - sg;
  *e = (short)(ex == 0x7ff ? XW_BAD : xmax(ex, 1));
}
// both edge values of a cell: u_{i+1/2} from the left, u_{i-1/2} from the right, class e, [62]; weak: both the cell's
// value and an edge value's distance from it are small beside the stencil's largest value, whose class leaves them
// fewer bits than a double has (a jump that the weights keep out of the value)
struct XEdge {
  long long up, um;
  int e;
  bool weak;
};
// the interpolation in doubles, as edges() in wcns.cu, for weak edges; staged values are doubles, so nothing is
// lost on the way in
inline __host__ __device__ XNOINLINE XEdge xedges_f64(double u0, double u1, double u2, double u3, double u4, bool linear) {
  const double gA = 0.5 * (u0 - 4.0 * u1 + 3.0 * u2), gB = 0.5 * (u3 - u1), gC = 0.5 * (4.0 * u3 - 3.0 * u2 - u4);
  const double sA = u0 - 2.0 * u1 + u2, sB = u1 - 2.0 * u2 + u3, sC = u2 - 2.0 * u3 + u4;
  double wA = 1.0, wB = 1.0, wC = 1.0;  // products of the other stencils' (1e-6 + g^2 + s^2)^2
  if (!linear) {
    const double a = 1e-6 + (gA * gA + sA * sA), b = 1e-6 + (gB * gB + sB * sB), c = 1e-6 + (gC * gC + sC * sC);
    wA = b * b * (c * c);
    wB = a * a * (c * c);
    wC = a * a * (b * b);
  }
  const double nB = 10.0 * wB, n = wA + nB + 5.0 * wC, k = 5.0 * wA + nB + wC;
  const double up = wA * (0.5 * gA + 0.125 * sA) + nB * (0.5 * gB + 0.125 * sB) + 5.0 * wC * (0.5 * gC + 0.125 * sC);
  const double um = 5.0 * wA * (0.125 * sA - 0.5 * gA) + nB * (0.125 * sB - 0.5 * gB) + wC * (0.125 * sC - 0.5 * gC);
  const XPair e = xpair(u2 + up / n, u2 + um / k);
  return {e.l, e.r, e.e, false};
}
// the weighted interpolation of WCNS-E-5 (edges() in wcns.cu) from the five staged values at wm, we.
// With d_j the first differences of u_{i-2} .. u_{i+2}: eight times the candidates' distances from u_i
// are small integer combinations of them, twice the first derivatives too.  Each stencil's
// smoothness is formed from its own normalised differences, and the weights are compared in the
// class of the largest: one 2^61 times smaller has no part in the value.
template <int STRIDE>
__host__ __device__ XNOINLINE XEdge xedges(const long long* __restrict__ wm, const short* __restrict__ we, bool linear,
                                             XVal eps) {
  long long u[5];
  int e[5];
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    u[c] = wm[c * STRIDE];
    e[c] = we[c * STRIDE];
  }
  int E = xmax(xmax(xmax(e[0], e[1]), xmax(e[2], e[3])), e[4]);
#pragma unroll
  for (int c = 0; c < 5; ++c) u[c] = xshr(u[c], E - e[c]);  // [57]
  E -= XW_BIAS;
  const long long d0 = u[1] - u[0], d1 = u[2] - u[1], d2 = u[3] - u[2], d3 = u[4] - u[3];  // [58]
  auto x3 = [](long long a) { return (a << 1) + a; };
  auto x5 = [](long long a) { return (a << 2) + a; };
  auto x7 = [](long long a) { return (a << 3) - a; };
  auto x10 = [](long long a) { return (a << 3) + (a << 1); };
  // 8 (candidate - u_i) at i + 1/2 and i - 1/2 [62]
  long long pA = x7(d1) - x3(d0), pB = x3(d2) + d1, pC = x5(d2) - d3;
  long long qA = d0 - x5(d1), qB = -(x3(d1) + d2), qC = x3(d3) - x7(d2);
  auto edge = [&](long long tp, long long tm) -> XEdge {  // u_i and the distances in class E - 3; |u| is 2^60 at most
    const long long uc = u[2] << 3;
    const int hu = (int)(uc >> 32), hp = (int)(tp >> 32), hm = (int)(tm >> 32), ap = hp ^ (hp >> 31), am = hm ^ (hm >> 31);
    return {uc + tp, uc + tm, E - 3, (hu ^ (hu >> 31)) + (ap < am ? ap : am) < (1 << 24)};  // 2^56
  };
  if (linear)
    return edge(((pA >> 2) + x10(pB >> 2) + x5(pC >> 2)) >> 2, (x5(qA >> 2) + x10(qB >> 2) + (qC >> 2)) >> 2);
  // 1e-6 + g^2 + s^2 of a stencil from 2 g and 2 s [60], normalised [62]
  auto smooth = [&](long long g, long long s) -> XVal {
    const int n = xclz32((int)((g ^ (g >> 63)) >> 32) | (int)((s ^ (s >> 63)) >> 32)) - 2;  // 2 .. 30
    const long long q = xsq(g << n) + xsq(s << n);                                          // 4 (g^2 + s^2) [61]
    const int eb = 2 * (E - n) + 1, ed = xmax(eb, eps.e + 1);
    return xquick(xshr(q, ed - eb) + xshr(eps.m, ed - eps.e), ed);
  };
  const XVal A = smooth(x3(d1) - d0, (d1 - d0) << 1), B = smooth(d1 + d2, (d2 - d1) << 1),
             C = smooth(x3(d2) - d3, (d3 - d2) << 1);
  // a stencil's weight: the square of the product of the others' smoothness, in [2^58, 2^60)
  auto weight = [](const XVal& x, const XVal& y) -> XVal {
    const long long m = xmul(x.m, y.m);  // [2^58, 2^60)
    const int n = 3 - (int)(m >> 59);
    return {xsq(m << n), 2 * (x.e + y.e + 3 - n) + 3};
  };
  const XVal wa = weight(B, C), wb = weight(A, C), wc = weight(A, B);
  const int Em = xmax(wa.e, xmax(wb.e, wc.e)) + 2;
  const long long a = xshr(wa.m, Em - wa.e), b = x10(xshr(wb.m, Em - wb.e)), c = xshr(wc.m, Em - wc.e);
  const XVal rp = xrcp(xquick(a + b + x5(c), Em)), rm = xrcp(xquick(x5(a) + b + c, Em));  // sums [62]
  // the weights' shares first (2^62 = 1, to 2^-59), then the distances of the candidates, normalised together: the error is
  // some 2^-60 of the largest distance.  (Products of weights and distances summed first and divided last left 2^-50 of
  // it beside a jump, where one weight outgrows the others.)
  const long long any = (pA ^ (pA >> 63)) | (pB ^ (pB >> 63)) | (pC ^ (pC >> 63)) | (qA ^ (qA >> 63)) | (qB ^ (qB >> 63)) |
                        (qC ^ (qC >> 63));
  const int n = xclz32((int)(any >> 32)) - 2;
  auto part = [&](long long m, int e, const XVal& r, long long p) {
    return xmul(xshr(xmul(m, r.m) << 2, 1 - (e + r.e)) << 3, p << n);
  };
  const long long tp = xshr((part(wa.m << 2, wa.e - 2, rp, pA) + part(x5(wb.m), wb.e + 1, rp, pB) + part(x5(wc.m), wc.e, rp, pC)) << 2, n);
  const long long tm = xshr((part(x5(wa.m), wa.e, rm, qA) + part(x5(wb.m), wb.e + 1, rm, qB) + part(wc.m << 2, wc.e - 2, rm, qC)) << 2, n);
  return edge(tp, tm);
}
// the edge values of a cell: on integers, weak ones in FP64
template <int STRIDE>
__host__ __device__ __forceinline__ XEdge xedge_values(const long long* __restrict__ wm, const short* __restrict__ we,
                                                       bool linear, XVal eps) {
  const XEdge g = xedges<STRIDE>(wm, we, linear, eps);
  if (g.weak && g.e < XBAD && (g.up | g.um) != 0) {
    double u[5];
#pragma unroll
    for (int c = 0; c < 5; ++c) u[c] = xenc(wm[c * STRIDE], we[c * STRIDE] - XW_BIAS);
    const XEdge h = xedges_f64(u[0], u[1], u[2], u[3], u[4], linear);
    if (h.e < 1024) return h;  // (fourth powers of values past 1e38 overflow)
  }
  return g;
}

}  // namespace gbcfd
