// xfix.cuh -- 64-bit block-floating arithmetic on the integer pipes, and the Roe flux written in
// it for the FP64 path.
//
// Why.  This part issues one FP64 operation per 64 FP32 or integer ones: a warp's DADD or DMUL
// holds its sub-partition's FP64 lanes for 76 cycles, a DFMA for 64, while the integer pipes
// idle.  A 64-bit integer add takes 2 issue slots there, an arithmetic 64-bit shift 4, and the
// upper part of a 64 x 64 product about 15 (three 32 x 32 + 64 multiply-adds).  So the face flux of
// the FP64 path is evaluated on 62-bit signed mantissas with an integer exponent each, in which
// every rounding is at 2^-57 or finer of its class's largest value (FP64: 2^-53), and the result
// is rounded once to a double.
//
// A value is m 2^(E - 61), m a signed 64-bit integer, E an int.  Values that are added share E:
// before a sum the terms are shifted right to the sum's class, a bound on every |m| being known
// from the class (written beside each line as the number of bits), so nothing overflows for any
// finite input.  Sums then cost one 64-bit add, and no result is normalised but where its
// reciprocal root is taken.  Truncation is towards minus infinity.
//
// Measured on random states against quadruple precision (tests/test_xfix.py holds a bound): the
// flux's root mean square error is 4-6e-17 of its size where the FP64 form's is 7-14e-17.
//
// The scheme is plain fixed-point arithmetic with scaling by exponents ("block floating point",
// J. H. Wilkinson, Rounding Errors in Algebraic Processes, 1963, ch. 1).
#pragma once

namespace gbcfd {

struct XVal {
  long long m;
  int e;
};

// (a b) >> (64 - K): the product of two 64-bit values, |a b| < 2^(126 - K).  Each operand is split as
// h 2^32 + l with both halves signed (l the low word read as signed, its sign carried into h), so
// the three products kept are signed 32 x 32 -> 64; l_a l_b (less than 2^30 units of the middle
// sum) is left out: the error is below 2^(K - 2) + 1 units of the result.
template <int K>
__host__ __device__ __forceinline__ long long xmul(long long a, long long b) {
  const int al = (int)a, bl = (int)b;
  const int ah = (int)(a >> 32) + (int)((unsigned)al >> 31), bh = (int)(b >> 32) + (int)((unsigned)bl >> 31);
  const long long t = (long long)ah * bl + (long long)al * bh;
  const long long r = (long long)ah * bh + (t >> 32);
  return (long long)(((unsigned long long)r << K) | ((unsigned)t >> (32 - K)));
}
template <int K>
__host__ __device__ __forceinline__ long long xsq(long long a) {
  const int al = (int)a;
  const int ah = (int)(a >> 32) + (int)((unsigned)al >> 31);
  const long long t = (long long)ah * al;  // half the middle sum
  const long long r = (long long)ah * ah + (t >> 31);
  return (long long)(((unsigned long long)r << K) | (((unsigned)t << 1) >> (32 - K)));
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
// the double nearest to m 2^(e - 61), |m| < 2^63; below the normal range 0, above it infinity
__host__ __device__ __forceinline__ double xenc(long long m, int e) {
  const long long s = m >> 63;
  unsigned long long a = (unsigned long long)((m ^ s) - s);
  const int n = xclz(a);
  a <<= (n & 63);
  const int f = e + 2 - n + 1022;  // biased exponent - 1
  const unsigned long long mant = (a >> 11) + ((a >> 10) & 1ull);
  unsigned long long b = ((unsigned long long)(unsigned)f << 52) + mant;
  if ((unsigned)f >= 2046u) b = f < 0 ? 0ull : 0x7ff0000000000000ull;
  if (a == 0ull) b = 0ull;
  return xdouble(b | ((unsigned long long)s & 0x8000000000000000ull));
}

// the constants of the Roe flux as values (formed on the host)
struct XConsts {
  XVal ggm1, gm1, eps;  // 62 bits
};
inline XConsts xconsts(double gamma, double eps) {
  return {xdec_pos<62>(gamma / (gamma - 1.0)), xdec_pos<62>(gamma - 1.0), xdec_pos<62>(eps)};
}

// shift m left until 2^61 <= |m| < 2^62 (m < 2^62), lowering its exponent; 0 stays 0 with a far
// smaller exponent
__host__ __device__ __forceinline__ void xnorm(long long& m, int& e) {
  const int n = (xclz((unsigned long long)(m ^ (m >> 63))) - 2) & 63;
  m = (long long)((unsigned long long)m << n);
  e -= n;
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
  const long long e = (1ll << 60) - xmul<4>(M, (long long)Y * Y);
  const int es = (int)(e >> 18);
  return {xcorrect(Y, (e >> 1) + ((3 * ((long long)es * es)) >> 27)), -((v.e - odd) >> 1) - 1};
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
__host__ __device__ __forceinline__ XVal xnormed(long long m, int e) {
  xnorm(m, e);
  return {m, e};
}

// (x^2 + d^2) / (2 d) in the class of x and d, 0 <= x < d < 2^62: Harten's fix of |x| < d.  n =
// leading zeros that bring d to 62 bits, h 2^(e - 61) = 1 / (d 2^n 2^-61)
struct XHid {
  long long h;
  int e, n;
};
__host__ __device__ __forceinline__ XHid xhid(long long d) {
  XHid r;
  r.n = (xclz((unsigned long long)d) - 2) & 63;  // d > 0 where it is used
  const XVal v = xrcp({d << r.n, 0});
  r.h = v.m;
  r.e = v.e;
  return r;
}
__host__ __device__ __forceinline__ long long xharten(long long x, long long d, const XHid& r) {
  if (x >= d) return x;
  // squares of 62-bit numbers, class 1; halved so that their sum keeps 62 bits: class 2; the
  // product with 1 / (2 d) has class 2 + (e - 1) + 1 = 1 for e = -1: one bit up, then back by n
  const long long q = (xsq<2>(x << r.n) >> 1) + (xsq<2>(d << r.n) >> 1);
  return xshr(xmul<2>(q, r.h) << 1, r.n);
}

// the two sides of a face: one variable's left and right value in a common class, |m| < 2^61
struct XPair {
  long long l, r;
  int e;
};
// twice a face flux, each component in its own class, |m| < 2^63; bad: a density or c^2 that is
// not positive (NaN fluxes)
struct XFlux {
  long long m[5];
  int e[5];
  bool bad;
};

// Twice the Roe flux with Harten's fix in the face frame, as roe_frame (physics.cuh), from the
// sides' (rho, u_n, u_t1, u_t2, p).  [n] after a line: |m| < 2^n.  Classes: Er, Eu, Ev, Ew, Ep of
// the five variables, EH of the enthalpies and q^2/2, El of the wave speeds, EA of the wave
// strengths, EM of the mass fluxes.  Where a value may be much smaller than its class (jumps,
// products of several factors) it is normalised, so that later roundings are relative to it.
__host__ __device__ __forceinline__ void xroe(const XPair& r, const XPair& u, const XPair& v, const XPair& w,
                                              const XPair& p, const XConsts& K, XFlux& F) {
  const int Eu = u.e, Ev = v.e, Ew = w.e, Ep = p.e;
  const long long ul = u.l, ur = u.r, vl = v.l, vr = v.r, wl = w.l, wr = w.r;
  // densities and pressures by themselves; reciprocal roots; the Roe weights a_l = isr iw,
  // a_r = isl iw with iw = 1 / (isl + isr), class -1 (below 1, so [62])
  const XVal rl = xnormed(r.l, r.e), rr = xnormed(r.r, r.e), pl = xnormed(p.l, p.e), pr = xnormed(p.r, p.e);  // [62]
  const XVal isl = xrsqrt(rl), isr = xrsqrt(rr);
  const int Ei = xmax(isl.e, isr.e) + 1;
  const XVal iw = xrcp(xnormed(xshr(isl.m, Ei - isl.e) + xshr(isr.m, Ei - isr.e), Ei));
  const long long al = xshr(xmul<3>(isr.m, iw.m), -1 - (isr.e + iw.e));
  const long long ar = xshr(xmul<3>(isl.m, iw.m), -1 - (isl.e + iw.e));
  // sqrt(rho_l rho_r)
  const XVal rt = xnormed(xmul<2>(xmul<2>(rl.m, isl.m), xmul<2>(rr.m, isr.m)), rl.e + isl.e + rr.e + isr.e + 3);  // [62]
  // mass fluxes
  const long long ml = xmul<3>(rl.m, ul), mr = xmul<3>(rr.m, ur);  // [62]
  const int Eml = rl.e + Eu, Emr = rr.e + Eu;
  // enthalpies gamma/(gamma-1) p / rho + |u|^2 / 2, each side in its own class
  const XVal gl = xnormed(xmul<2>(K.ggm1.m, xmul<2>(pl.m, xsq<2>(isl.m))), K.ggm1.e + pl.e + 2 * isl.e + 3);
  const XVal gr = xnormed(xmul<2>(K.ggm1.m, xmul<2>(pr.m, xsq<2>(isr.m))), K.ggm1.e + pr.e + 2 * isr.e + 3);
  const int Ek = 2 * xmax(xmax(Eu, Ev), Ew) - 2;
  const int EHl = xmax(gl.e, Ek) + 2, EHr = xmax(gr.e, Ek) + 2, EH = xmax(EHl, EHr);
  const long long hl = xshr(gl.m, EHl - gl.e) + xshr(xsq<4>(ul), EHl + 2 - 2 * Eu) + xshr(xsq<4>(vl), EHl + 2 - 2 * Ev) +
                       xshr(xsq<4>(wl), EHl + 2 - 2 * Ew);  // [62]
  const long long hr = xshr(gr.m, EHr - gr.e) + xshr(xsq<4>(ur), EHr + 2 - 2 * Eu) + xshr(xsq<4>(vr), EHr + 2 - 2 * Ev) +
                       xshr(xsq<4>(wr), EHr + 2 - 2 * Ew);
  // Roe averages, in the classes of the sides
  const long long ut = xmul<2>(al, ul) + xmul<2>(ar, ur);  // [61]
  const long long vt = xmul<2>(al, vl) + xmul<2>(ar, vr);  // [61]
  const long long wt = xmul<2>(al, wl) + xmul<2>(ar, wr);  // [61]
  const long long ht = xshr(xmul<2>(al, hl), EH - EHl) + xshr(xmul<2>(ar, hr), EH - EHr);  // [62]
  const long long q2 = xshr(xsq<4>(ut), EH + 2 - 2 * Eu) + xshr(xsq<4>(vt), EH + 2 - 2 * Ev) +
                       xshr(xsq<4>(wt), EH + 2 - 2 * Ew);  // q^2 / 2
  const long long c2m = xmul<2>(K.gm1.m, ht - q2);
  F.bad = r.l <= 0 || r.r <= 0 || c2m <= 0;
  // c^2 normalised, its reciprocal root, c
  const XVal c2 = xnormed(c2m, K.gm1.e + EH + 1);
  const XVal ic = xrsqrt(c2);
  const long long ic2 = xsq<2>(ic.m);  // [62], class 2 ic.e + 1
  const long long cc = xmul<2>(c2.m, ic.m);
  const int Ec = c2.e + ic.e + 1;
  // wave speeds; room for delta = eps (|u| + c) where eps >= 1
  const int hx = K.eps.e >= 0 ? K.eps.e + 1 : 0;
  const int El = xmax(Eu - 1, Ec) + 1 + hx;
  const long long ue = xshr(ut, El - Eu), ce = xshr(cc, El - Ec);  // [61]
  const long long au = xabs(ue);
  long long l1 = xabs(ue - ce), l5 = xabs(ue + ce), l2 = au;       // [62]
  {
    long long d = xmul<2>(K.eps.m, au + ce);
    d = K.eps.e >= 0 ? d << hx : xshr(d, -1 - K.eps.e);            // [62]
    if (l1 < d || l2 < d || l5 < d) {
      const XHid hid = xhid(d);
      l1 = xharten(l1, d, hid);
      l2 = xharten(l2, d, hid);
      l5 = xharten(l5, d, hid);
    }
  }
  // jumps, normalised [62], and wave strengths: a1, a5 = (dp -+ rho c du) / (2 c^2), a2 = drho - dp / c^2
  const XVal jr = xnormed(r.r - r.l, r.e), ju = xnormed(ur - ul, Eu), jv = xnormed(vr - vl, Ev), jw = xnormed(wr - wl, Ew),
             jp = xnormed(p.r - p.l, Ep);
  const long long rcd = xmul<2>(xmul<2>(rt.m, cc), ju.m);
  const int Ercd = rt.e + Ec + 1 + ju.e + 1;
  const int Eq = xmax(Ercd, jp.e) + 1;
  const long long dp = xshr(jp.m, Eq - jp.e), rq = xshr(rcd, Eq - Ercd);  // [61]
  const int Ea = Eq + 2 * ic.e + 1;                                       // of a1 and a5 (the half included)
  const long long w1 = xmul<1>(l1, xmul<2>(dp - rq, ic2)), w5 = xmul<1>(l5, xmul<2>(dp + rq, ic2));  // [61]
  const XVal s = xnormed(w1 + w5, El + Ea + 2), dw = xnormed(w5 - w1, El + Ea + 2);                  // [62]
  const int EA = xmax(Ea + 1, jr.e) + 1;
  const XVal w2 = xnormed(xmul<2>(l2, xshr(jr.m, EA - jr.e) - xshr(xmul<2>(dp, ic2), EA - Ea - 1)), El + EA + 1);
  // in the class of the mass fluxes [60]
  const int EM = xmax(xmax(Eml, Emr), xmax(s.e, w2.e) + 1) + 2;
  const long long fl = xshr(ml, EM - Eml), fr = xshr(mr, EM - Emr);
  const long long ws = xshr(s.m, EM - s.e) + xshr(w2.m, EM - w2.e);
  const XVal dq = {xmul<2>(dw.m, cc), dw.e + Ec + 1};                  // [62]
  const long long lrt = xmul<2>(l2, rt.m);                             // [62]
  const XVal g1 = xnormed(xmul<2>(lrt, jv.m), El + rt.e + jv.e + 2), g2 = xnormed(xmul<2>(lrt, jw.m), El + rt.e + jw.e + 2);
  F.m[0] = fl + fr - ws;
  F.e[0] = EM;
  {
    const int e2 = EM + Ev - 1, e3 = EM + Ew - 1;
    const long long a = xmul<4>(fl, vl) + xmul<4>(fr, vr) - xmul<4>(ws, vt);  // < 3 2^61
    const long long b = xmul<4>(fl, wl) + xmul<4>(fr, wr) - xmul<4>(ws, wt);
    F.e[2] = xmax(e2, g1.e) + 1;
    F.e[3] = xmax(e3, g2.e) + 1;
    F.m[2] = xshr(a, F.e[2] - e2) - xshr(g1.m, F.e[2] - g1.e);
    F.m[3] = xshr(b, F.e[3] - e3) - xshr(g2.m, F.e[3] - g2.e);
  }
  {
    const int e1 = EM + Eu - 1, E1 = xmax(xmax(e1, dq.e), Ep) + 2;
    const long long a = xmul<4>(fl, ul) + xmul<4>(fr, ur) - xmul<4>(ws, ut);
    F.e[1] = E1;
    F.m[1] = xshr(a, E1 - e1) + xshr(p.l + p.r, E1 - Ep) - xshr(dq.m, E1 - dq.e);
  }
  {
    const int el = Eml + EHl + 2, er = Emr + EHr + 2, e1 = s.e + EH + 1, e2 = dq.e + Eu + 1, e3 = g1.e + Ev + 1,
              e4 = g2.e + Ew + 1, e5 = w2.e + EH + 1;
    const int E4 = xmax(xmax(xmax(el, er), xmax(e1, e2)), xmax(xmax(e3, e4), e5)) + 2;
    const long long a = xshr(xmul<1>(ml, hl), E4 - el) + xshr(xmul<1>(mr, hr), E4 - er);
    const long long b = xshr(xmul<2>(s.m, ht), E4 - e1) + xshr(xmul<2>(w2.m, q2), E4 - e5);
    const long long d = xshr(xmul<2>(g1.m, vt), E4 - e3) + xshr(xmul<2>(g2.m, wt), E4 - e4);
    F.e[4] = E4;
    F.m[4] = a - b - xshr(xmul<2>(dq.m, ut), E4 - e2) - d;
  }
}

// a flux component as a double, times 2^-h
__host__ __device__ __forceinline__ double xflux(const XFlux& F, int q, int h) {
  return F.bad ? xdouble(0x7ff8000000000000ull) : xenc(F.m[q], F.e[q] - h);
}
// both sides of one variable from doubles
__host__ __device__ __forceinline__ XPair xpair(double l, double r) {
  const XVal a = xdec<61>(l), b = xdec<61>(r);
  const int e = xmax(a.e, b.e);
  return {xshr(a.m, e - a.e), xshr(b.m, e - b.e), e};
}
// roe_frame's interface: L, R = (rho, u_n, u_t1, u_t2, p), F twice the flux or (TWICE false) the flux
template <bool TWICE = true>
__host__ __device__ __forceinline__ void xroe(const double* L, const double* R, const XConsts& K, double* F) {
  XFlux f;
  xroe(xpair(L[0], R[0]), xpair(L[1], R[1]), xpair(L[2], R[2]), xpair(L[3], R[3]), xpair(L[4], R[4]), K, f);
  for (int q = 0; q < 5; ++q) F[q] = xflux(f, q, TWICE ? 0 : 1);
}

}  // namespace gbcfd
