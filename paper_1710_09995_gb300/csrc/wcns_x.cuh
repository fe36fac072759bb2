// wcns_x.cuh -- the direction passes and the viscous residual of the FP64 WCNS-E-5 path on the integer
// pipes (xfix.cuh).
// Included by wcns.cu, whose Args, Box and tile constants it uses.
//
// Same tiles, lines and passes as dir_kernel.  The FP64 form spent ~65 FP64 operations per
// variable and edge pair on the weighted interpolation alone (the pipe issues one per 64 integer
// operations).  Here a landed tile is converted once, in place, to 57-bit integers with an exponent
// each; the interpolation's differences and candidates are then exact integer sums, its weights
// and the Roe flux 62-bit products, and Eq. 2 is taken of the integer fluxes.  One primitive
// buffer (the next tile is requested when the fluxes are done, behind Eq. 2) and a separate flux
// buffer keep two CTAs per SM.  Measured: a 128^3 Navier-Stokes step
// 30.6 -> 9.75 ms (24.7 with only the Roe flux on integers), with the viscous pass and the primitives below 7.44, and 8.14 since
// edges beside jumps and small components keep the FP64 form's accuracy.  Residuals of smooth states are
// 2.6 to 2.8 times closer to long double than the FP64 form's, states after a step 1.01 to 1.8 times.
#pragma once

namespace gbcfd {
namespace wcns {

struct XSmem {
  static constexpr int NW_ = 5 * (LMAX + 10) * NLP, NF = 5 * (LMAX + 5) * NLP;
  static constexpr size_t wm = 0;                                             // staged doubles, then their integers
  static constexpr size_t fm = wm + sizeof(long long) * NW_;
  static constexpr size_t we = fm + sizeof(long long) * NF;
  static constexpr size_t fe = we + sizeof(short) * NW_;
  static constexpr size_t red = (fe + sizeof(short) * NF + 15) / 16 * 16;
  static constexpr size_t cst = red + sizeof(double) * (NTW / 32) * 5;        // Eq. 2's coefficients, the weights' 1e-6
  static constexpr size_t bytes = (cst + 4 * sizeof(XVal) + 127) / 128 * 128;
};
// an edge whose sides are far apart (xfar) in FP64: twice the flux.  Out of line: only edges at a jump of 2^5 or more in
// the density or the pressure call it
template <int D>
__device__ __noinline__ void xedge_f64(const double (&L)[5], const double (&R)[5], double gm1, double ggm1, double eps,
                                       long long* Fm, short* Fe, int o, bool bad) {
  Consts<double> K;
  K.gm1 = gm1;
  K.ggm1 = ggm1;
  K.eps = eps;
  constexpr int idx[5] = {0, Fr<D>::N, Fr<D>::T1, Fr<D>::T2, 4};
  double f[5];
  roe_frame<double, true>(L, R, K, f);
  const XFlux F = xflux_of(f);
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    Fm[idx[q] * (LMAX + 5) * NLP + o] = F.m[q];
    Fe[idx[q] * (LMAX + 5) * NLP + o] = (short)(bad ? XW_BAD : F.e[q]);
  }
}

template <int D, int MODE>
__global__ void __launch_bounds__(NTW, 2) xdir_kernel(Args a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* const Ws = reinterpret_cast<double*>(smem_raw + XSmem::wm);
  long long* const Wm = reinterpret_cast<long long*>(smem_raw + XSmem::wm);
  short* const We = reinterpret_cast<short*>(smem_raw + XSmem::we);
  long long* const Fm = reinterpret_cast<long long*>(smem_raw + XSmem::fm);
  short* const Fe = reinterpret_cast<short*>(smem_raw + XSmem::fe);
  double* red = reinterpret_cast<double*>(smem_raw + XSmem::red);
  XVal* cst = reinterpret_cast<XVal*>(smem_raw + XSmem::cst);
  __shared__ int last;
  const Box& b = a.b;
  const int nd = D == 0 ? b.nx : (D == 1 ? b.ny : b.nz);   // along the lines
  const int na = D == 0 ? b.ny : b.nx;                      // across the lines (16 per tile)
  const int nb = D == 2 ? b.ny : b.nz;                      // the third direction
  const int L = a.Lseg[D];
  const int nseg = (nd + L - 1) / L, ngrp = (na + NL - 1) / NL;
  const long long tiles = (long long)nseg * ngrp * nb;
  const double* W = static_cast<const double*>(a.W);
  double* R = static_cast<double*>(a.R);
  const bool linear = a.linear != 0;
  const double dt = (MODE == 2 && a.stage > 0) ? a.ctrl->dt : 0.0;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double sq[5] = {0, 0, 0, 0, 0};
  constexpr int idx[5] = {0, Fr<D>::N, Fr<D>::T1, Fr<D>::T2, 4};
  if (threadIdx.x == 0) {
    const double ih = a.cd.ih[D];  // the fluxes are doubled: Eq. 2's coefficients halved
    cst[0] = xdec_pos<62>(75.0 / 128.0 * ih);
    cst[1] = xdec_pos<62>(25.0 / 768.0 * ih);
    cst[2] = xdec_pos<62>(3.0 / 1280.0 * ih);
    cst[3] = xdec_pos<62>(1e-6);
  }
  struct TileInfo { int s0, Ls, a0, ob; };
  auto decode = [&](long long tile) {
    TileInfo t;
    const int seg = (int)(tile % nseg);
    const long long r = tile / nseg;
    t.s0 = seg * L;
    t.Ls = min(L, nd - t.s0);
    t.a0 = (int)(r % ngrp) * NL;
    t.ob = (int)(r / ngrp);
    return t;
  };
  // the primitives of cells s0 - 5 .. s0 + Ls + 4 of every line (staged cell s is cell s0 - 5 + s),
  // asynchronously, as one commit group
  auto issue_stage = [&](const TileInfo& t) {
    const int nst = t.Ls + 10;
    auto off = [&](int l, int s) {
      if (D == 0) return ((t.ob + H) * (b.ny + 2 * H) + t.a0 + l + H) * b.px + s + H;
      if (D == 1) return ((t.ob + H) * (b.ny + 2 * H) + s + H) * b.px + t.a0 + l + H;
      return ((s + H) * (b.ny + 2 * H) + t.ob + H) * b.px + t.a0 + l + H;
    };
    if (D == 0) {  // a warp per (variable, line), lanes along x
      for (int vl = warp; vl < 5 * NL; vl += NTW / 32) {
        const int v = vl / NL, l = vl % NL;
        double* drow = Ws + v * (LMAX + 10) * NLP + l;
        if (t.a0 + l < na) {
          const double* srow = W + (long long)v * b.field + off(l, t.s0 - H);
          for (int s = lane; s < nst; s += 32) cp_async(drow + s * NLP, srow + s);
        } else {
          for (int s = lane; s < nst; s += 32) drow[s * NLP] = (v == 0 || v == 4) ? 1.0 : 0.0;
        }
      }
    } else {       // 16 lines (x) per row s
      for (int v = 0; v < 5; ++v) {
        const double* src = W + (long long)v * b.field;
        double* dv = Ws + v * (LMAX + 10) * NLP;
        for (int e = threadIdx.x; e < nst * NL; e += NTW) {
          const int s = e / NL, l = e % NL;
          if (t.a0 + l < na) cp_async(dv + s * NLP + l, src + off(l, t.s0 - H + s));
          else dv[s * NLP + l] = (v == 0 || v == 4) ? 1.0 : 0.0;  // lines past the block
        }
      }
    }
    cp_async_commit();
  };
  if ((long long)blockIdx.x < tiles) issue_stage(decode(blockIdx.x));
  for (long long tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const TileInfo t = decode(tile);
    const int s0 = t.s0, Ls = t.Ls, a0 = t.a0, nfc = Ls + 5;
    cp_async_wait_all();
    __syncthreads();  // the tile has landed; the previous tile's cells are done with the fluxes
    // 1. in place to integers (zero and subnormals as zero, a value that is not finite by its exponent)
    for (int e = threadIdx.x; e < 5 * (Ls + 10) * NL; e += NTW) {
      const int r = e / NL, l = e % NL, v = r / (Ls + 10), s = r - v * (Ls + 10);
      const int o = (v * (LMAX + 10) + s) * NLP + l;
      xline_value(Ws[o], Wm + o, We + o);
    }
    __syncthreads();
    // 2. edge fluxes: edge f lies between staged cells f + 2 and f + 3, so cell c (staged c + 5)
    //    has edges c .. c + 5 around it.  Item (line, chunk): lane t takes staged cell
    //    m = 31 chunk + t + 2, evaluates its two edge states, and edge f = m - 2 pairs its
    //    left state with lane t + 1's right state.
#pragma unroll 1
    for (int it = 0; it < ITEMS; ++it) {
      const int item = warp * ITEMS + it, l = item >> 1, ch = item & 1;
      const int f = FCH * ch + lane;
      if (a0 + l >= na || FCH * ch >= nfc) continue;  // warp-uniform
      const int m = min(f + 2, nfc + 2);              // centres 2 .. nfc + 2 (stencil <= nst - 1)
      // one variable's value on either side of the lane's edge
      auto sides = [&](int q, XVal& left, XVal& right) {
        const int o = (idx[q] * (LMAX + 10) + m - 2) * NLP + l;
        const XEdge g = xedge_values<NLP>(Wm + o, We + o, linear, cst[3]);
        left = {g.up, g.e};
        right = {__shfl_down_sync(0xffffffffu, g.um, 1), __shfl_down_sync(0xffffffffu, g.e, 1)};
      };
      XPair S[5];
      int worst = 0;
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        XVal left, right;
        sides(q, left, right);
        const int E = xmax(left.e, right.e);
        S[q] = xpair_norm(xshr(left.m, E - left.e), xshr(right.m, E - right.e), E);
        worst = xmax(worst, E);
      }
      bool far = false;
      if (lane < FCH && f < nfc) {
        const XPos r = S[0], p = S[4];
        far = xfar(r, p);
        if (!far) {
          XFlux F;
          xroe(r, S[1], S[2], S[3], p, a.cd.x, F);
#pragma unroll
          for (int q = 0; q < 5; ++q) {
            const int o = (idx[q] * (LMAX + 5) + f) * NLP + l;
            Fm[o] = F.m[q];
            Fe[o] = (short)(worst >= XBAD ? XW_BAD : F.e[q]);
          }
        }
      }
      if (__any_sync(0xffffffffu, far)) {  // edges between densities or pressures far apart, in FP64
        double Ld[5], Rd[5];
#pragma unroll
        for (int q = 0; q < 5; ++q) {
          XVal left, right;
          sides(q, left, right);
          Ld[q] = xenc(left.m, left.e);
          Rd[q] = xenc(right.m, right.e);
        }
        if (far) xedge_f64<D>(Ld, Rd, a.cd.K.gm1, a.cd.K.ggm1, a.cd.K.eps, Fm, Fe, f * NLP + l, worst >= XBAD);
      }
    }
    __syncthreads();
    if (tile + gridDim.x < tiles) issue_stage(decode(tile + gridDim.x));
    // 3. Eq. 2 per cell (plus the viscous residual in the x pass), then the pass's output
    const int ncell = D == 0 ? NL * 64 : Ls * NL;  // D = 0: a warp per line, lanes along x
    for (int e = threadIdx.x; e < ncell; e += NTW) {
      int l, c;
      if (D == 0) {
        l = e >> 6;
        c = e & 63;
        if (c >= Ls) continue;
      } else {
        c = e / NL;
        l = e % NL;
      }
      if (a0 + l >= na) continue;
      int i, j, k;
      if (D == 0) { i = s0 + c; j = a0 + l; k = t.ob; }
      else if (D == 1) { i = a0 + l; j = s0 + c; k = t.ob; }
      else { i = a0 + l; j = t.ob; k = s0 + c; }
      const long long cc = ((long long)k * b.ny + j) * b.nx + i;
      // what the cell reads of global memory, before its first store (else each variable waits for its own:
      // 96^3 passes 284, 282, 304 -> 271, 269, 298 us)
      double rin[5], qs[5], qn[5];
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        rin[q] = 0.0;
        if (D == 0 && a.viscous && q >= 1) rin[q] = static_cast<const double*>(a.Rv)[(q - 1) * a.n + cc];
        if (MODE != 0) rin[q] = R[q * a.n + cc];
        if (MODE == 2 && a.stage >= 1) qs[q] = a.qs[q * a.n + cc];
        if (MODE == 2 && a.stage >= 2) qn[q] = a.qn[q * a.n + cc];
      }
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        const int o = (q * (LMAX + 5) + c) * NLP + l;
        long long d[3];
        int ed[3];
#pragma unroll
        for (int x = 0; x < 3; ++x) {  // edges 3 - 2, 4 - 1, 5 - 0 around the cell
          const int h = o + (3 + x) * NLP, w = o + (2 - x) * NLP, e1 = Fe[h], e0 = Fe[w], E = xmax(e1, e0) + 1;
          // normalised, so that the product's truncation is relative to the difference
          const XVal g = xquick0(xshr(Fm[h], E - e1) - xshr(Fm[w], E - e0), E);
          d[x] = xmul(g.m, cst[x].m);  // [60]
          ed[x] = g.e + cst[x].e + 3;
        }
        const int E = xmax(ed[0], xmax(ed[1], ed[2]));
        double add = xenc(xshr(d[0], E - ed[0]) - xshr(d[1], E - ed[1]) + xshr(d[2], E - ed[2]), E);
        if (D == 0 && a.viscous && q >= 1)  // the viscous residual, once (x pass)
          add = add + rin[q];
        const long long oc = q * a.n + cc;
        if (MODE == 0) {
          R[oc] = add;
        } else if (MODE == 1) {
          R[oc] = rin[q] + add;
        } else {  // Eqs. 4-6
          const double tot = rin[q] + add;
          if (a.stage == 0) {
            a.rout[oc] = tot;
            continue;
          }
          if (a.stage == 1) sq[q] = fma(tot, tot, sq[q]);
          const double adv = qs[q] - dt * tot;
          double out;
          if (a.stage == 1) out = adv;
          else if (a.stage == 2) out = fma(0.25, adv, 0.75 * qn[q]);  // rounded as the FP64 form was
          else {  // Q^n / 3 with one correction of the product (a division costs ~5 FMAs here)
            const double q3 = (1.0 / 3.0) * qn[q];
            out = fma(2.0 / 3.0, adv, fma(fma(-3.0, q3, qn[q]), 1.0 / 3.0, q3));
          }
          a.qout[oc] = out;
        }
      }
    }
  }
  if (MODE == 2 && a.stage == 1) norm_fold(a, sq, red, &last);
}

// ---- the viscous residual, FP64 ------------------------------------------------------------------
// Same tiles, planes and passes as viscres_kernel, on integers: that form's 204 FP64 operations a cell
// held the FP64 pipe 78% of the time.  A plane that has landed is converted once, in place: velocities to
// integers with an exponent each, theta (positive) to a word of mantissa and exponent.  A difference D4 is
// formed in the class of its four values with four bits of room, so that it is exact in them, and normalised; gradients,
// stresses and the energy flux are then 62-bit products, and sums in the class of their largest term.
// The fluxes are kept as integers with an exponent each, and differenced in the same way; the sum of
// the three directions is rounded once.  (With one exponent for a cell's velocities, one for a gradient cell's
// neighbours and one for its stresses, a component 10^6 times smaller than the others had 2^-38 of itself left.)
// 16 warps (the FP64 form had 8): a cell's four equations are
// shared by two threads.  Two barriers a plane: the conversion of the next plane runs beside the
// differences.  Measured (96^3): 434 -> 134 us a stage, 160 with the exponents of today; with the primitives' 117 -> 70 a
// 128^3 step 9.75 -> 7.85 ms (7.43 with the loads of the passes' ends brought forward and a warp per row of primitives).
// An exponent for each velocity, difference and stress cost the step 0.15 ms.
constexpr int XVT = 512, XWX = 42;  // threads; columns of the primitive box (41 are read; 16-byte rows)
struct XRSmem {
  static constexpr int WF = WY * XWX, WP = 4 * WF;
  static constexpr int FX = RY * GX, GY_ = GY * RX, HZ = RY * RX;  // cells of one flux buffer
  static constexpr int ERING = 5;                                  // exponents: of planes p - 2 .. p + 2
  static constexpr size_t w = 0;                                   // staged doubles, then their integers
  static constexpr size_t fx = w + 8 * WRING * WP;
  static constexpr size_t gy = fx + 8 * 4 * FX;
  static constexpr size_t hz = gy + 8 * 4 * GY_;
  static constexpr size_t we = hz + 8 * ZRING * 4 * HZ;            // exponents: u, v, w
  static constexpr size_t fxe = we + 2 * ERING * 3 * WF;           // of the fluxes: three stresses, energy
  static constexpr size_t gye = fxe + 2 * 4 * FX;
  static constexpr size_t hze = gye + 2 * 4 * GY_;
  static constexpr size_t bar = (hze + 2 * ZRING * 4 * HZ + 15) / 16 * 16;
  static constexpr size_t bytes = bar + 8 * WRING + 16;
  static_assert(bytes <= 232448 - 256, "227 KB of shared memory per CTA");
};
// a velocity: as xdec_zero, its exponent XBAD and more if it is not finite
__device__ __forceinline__ XVal xvalue(double d) {
  XVal v = xdec_zero(d);
  if (v.e >= 1024) v.e = 2 * XBAD;
  return v;
}
// theta > 0 as a word: its 53-bit mantissa above its biased exponent
__device__ __forceinline__ long long xword(long long bits) {
  const int ex = (int)(bits >> 52) & 0x7ff;
  const long long m = bits & 0xfffffffffffffll;
  return (ex ? (m | (1ll << 52)) << 11 | ex : m << 11 | 1);
}
__device__ __forceinline__ int xword_e(long long w) { return (int)w & 0x7ff; }
__device__ __forceinline__ long long xword_m(long long w) {  // [62]
  return (long long)(((unsigned long long)w & ~0x7ffull) >> 2);
}
// (a - d) + 8 (b - c) of four values brought to a class by right shifts s; [58] in, below 2^62.2
__device__ __forceinline__ long long xd4(long long a, int sa, long long b, int sb, long long c, int sc, long long d, int sd) {
  return (xshr(a, sa) - xshr(d, sd)) + ((xshr(b, sb) - xshr(c, sc)) << 3);
}

__global__ void __launch_bounds__(XVT, 1) xviscres_kernel(const __grid_constant__ Args a) {
  extern __shared__ __align__(128) unsigned char rsm[];
  using SM = XRSmem;
  long long* const wr = reinterpret_cast<long long*>(rsm + SM::w);
  short* const wer = reinterpret_cast<short*>(rsm + SM::we);
  long long* const fxr = reinterpret_cast<long long*>(rsm + SM::fx);
  long long* const gyr = reinterpret_cast<long long*>(rsm + SM::gy);
  long long* const hzr = reinterpret_cast<long long*>(rsm + SM::hz);
  short* const fxe = reinterpret_cast<short*>(rsm + SM::fxe);
  short* const gye = reinterpret_cast<short*>(rsm + SM::gye);
  short* const hze = reinterpret_cast<short*>(rsm + SM::hze);
  uint64_t* const bar = reinterpret_cast<uint64_t*>(rsm + SM::bar);
  __shared__ XVal cst[6];  // 1 / (12 h), mu, 2 mu / 3, kappa
  const Box& b = a.b;
  double* Rv = static_cast<double*>(a.Rv);
  const int ntx = (b.nx + RX - 1) / RX, nty = (b.ny + RY - 1) / RY;
  const long long units = (long long)ntx * nty * b.nz;
  const long long u0 = (long long)blockIdx.x * units / gridDim.x, u1 = (long long)(blockIdx.x + 1) * units / gridDim.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    for (int q = 0; q < WRING; ++q) mbar_init(&bar[q], 1);
    fence_barrier_init();
  }
  if (threadIdx.x < 3) cst[threadIdx.x] = xdec_pos<62>(a.cd.ih12[threadIdx.x]);
  if (threadIdx.x == 32) cst[3] = xdec_pos<62>(a.cd.mu);
  if (threadIdx.x == 64) cst[4] = xdec_pos<62>(2.0 / 3.0 * a.cd.mu);
  if (threadIdx.x == 96) cst[5] = xdec_pos<62>(a.cd.kappa);
  __syncthreads();
  unsigned parity = 0, pending = 0;  // per W slot (parity uniform; pending in thread 0)
  bool fail = false;                 // a copy did not arrive (uniform)
  auto ws = [](int kp) { return (kp + 4 * WRING) % WRING; };
  auto es = [](int kp) { return (kp + 4 * SM::ERING) % SM::ERING; };
  auto zs = [](int kp) { return (kp + 4 * ZRING) % ZRING; };
  for (long long u = u0; u < u1 && !fail;) {
    const long long tile = u / b.nz;
    const int k0 = (int)(u - tile * b.nz);
    const int k1 = (int)min((long long)b.nz, k0 + (u1 - u));
    u += k1 - k0;
    const int tx = (int)(tile % ntx), x0 = tx * RX, y0 = (int)(tile / ntx) * RY;
    auto issue = [&](int kp) {  // thread 0: u, v, w, theta of plane kp (fields 1, 2, 3, 5)
      const int q = ws(kp);
      long long* dst = wr + q * SM::WP;
      mbar_expect_tx(&bar[q], (unsigned)(8 * SM::WP));
      const int fld[4] = {1, 2, 3, 5};
      for (int f = 0; f < 4; ++f)  // storage column x0 is cell x0 - 5; storage row y0 + 1 is cell y0 - 4
        tma_load_4d(dst + f * SM::WF, &a.mwv, &bar[q], x0, y0 + 1, kp + H, fld[f]);
      pending |= 1u << q;
    };
    auto convert = [&](int kp) -> bool {  // all threads: wait for plane kp, make integers of it
      const int q = ws(kp);
      const bool ok = mbar_wait_bounded(&bar[q], (parity >> q) & 1u);
      long long* m = wr + q * SM::WP;
      short* e = wer + es(kp) * 3 * SM::WF;
      for (int c = threadIdx.x; c < SM::WF; c += XVT) {
        long long x[4];
#pragma unroll
        for (int f = 0; f < 4; ++f) x[f] = m[f * SM::WF + c];
#pragma unroll
        for (int f = 0; f < 3; ++f) {
          const XVal v = xvalue(__longlong_as_double(x[f]));
          m[f * SM::WF + c] = v.m;
          e[f * SM::WF + c] = (short)v.e;
        }
        m[3 * SM::WF + c] = xword(x[3]);
      }
      return ok;
    };
    auto converted = [&](int kp) {  // behind the barrier that follows
      parity ^= 1u << ws(kp);
      pending &= ~(1u << ws(kp));
    };
    // a thread owns tile cell (lane, warp % 8), equations 2 (warp / 8) and the next: its x- and y-parts of
    // Rv for planes p - 2, p - 1, p stay in registers until the z-part of plane p - 2 is known
    const int crow = warp & 7, q0 = (warp >> 3) * 2;
    XVal rv2[2] = {{0, XZERO}, {0, XZERO}}, rv1[2] = {{0, XZERO}, {0, XZERO}};
    if (threadIdx.x == 0) {
      fence_proxy_async();
      for (int kp = k0 - 4; kp <= k0 + 1; ++kp) issue(kp);
    }
    {
      bool ok = true;
      for (int kp = k0 - 4; kp <= k0; ++kp) ok = convert(kp) && ok;
      fail = __syncthreads_or(!ok);
      if (fail) break;
      for (int kp = k0 - 4; kp <= k0; ++kp) converted(kp);
    }
    for (int p = k0 - 2; p <= k1 + 1; ++p) {  // lead plane p, output plane p - 2
      // the union box: a warp per 32-cell row, and warps 12, 13 take the 4 extra columns of all 12 rows
      int gy = warp, gx = lane;
      if (warp >= GY) {
        const int sidx = (warp - GY) * 32 + lane;
        gy = sidx / (GX - RX);
        gx = RX + sidx % (GX - RX);
      }
      if (gy < GY) {
        const int c = (gy + 2) * XWX + gx + 3;  // the cell in the primitive box
        // neighbours along d at distances -2, -1, +1, +2: slots of the planes and offsets in them
        const int s0 = ws(p), nb[3][4] = {{s0, s0, s0, s0}, {s0, s0, s0, s0}, {ws(p - 2), ws(p - 1), ws(p + 1), ws(p + 2)}};
        const int t0 = es(p), ne[3][4] = {{t0, t0, t0, t0}, {t0, t0, t0, t0}, {es(p - 2), es(p - 1), es(p + 1), es(p + 2)}};
        const int of[3][4] = {{c - 2, c - 1, c + 1, c + 2}, {c - 2 * XWX, c - XWX, c + XWX, c + 2 * XWX}, {c, c, c, c}};
        XVal gr[4][3];  // [60]
#pragma unroll
        for (int d = 0; d < 3; ++d)
#pragma unroll
          for (int f = 0; f < 4; ++f) {
            long long v[4];
            int sv[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              v[i] = wr[nb[d][i] * SM::WP + f * SM::WF + of[d][i]];
              if (f < 3) {
                sv[i] = wer[(ne[d][i] * 3 + f) * SM::WF + of[d][i]];
              } else {
                sv[i] = xword_e(v[i]);
                v[i] = xword_m(v[i]);
              }
            }
            int E = xmax(xmax(sv[0], sv[1]), xmax(sv[2], sv[3]));
            const XVal D = xquick0(xd4(v[0], E + 4 - sv[0], v[2], E + 4 - sv[2], v[1], E + 4 - sv[1], v[3], E + 4 - sv[3]),
                                   f < 3 ? E + 4 : (E == 0x7ff ? 2 * XBAD : E - 1023 + 4));
            gr[f][d] = {xmul(D.m, cst[d].m), D.e + cst[d].e + 3};
          }
        const int Ed = xmax(gr[0][0].e, xmax(gr[1][1].e, gr[2][2].e));
        long long dg[3];  // the diagonal in one class
#pragma unroll
        for (int d = 0; d < 3; ++d) dg[d] = xshr(gr[d][d].m, Ed - gr[d][d].e);
        const long long div = dg[0] + dg[1] + dg[2];  // below 2^61.6
        XVal off[3];  // stresses xy, yz, zx
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const int q = (d + 1) % 3, E = xmax(gr[q][d].e, gr[d][q].e);
          off[d] = {xmul(xshr(gr[q][d].m, E - gr[q][d].e) + xshr(gr[d][q].m, E - gr[d][q].e), cst[3].m), E + cst[3].e + 3};  // [59]
        }
        const short* ve = wer + t0 * 3 * SM::WF + c;
        const long long* vel = wr + s0 * SM::WP + c;
        const bool rows = gy >= 2 && gy < RY + 2, cols = gx >= 2 && gx < RX + 2;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          if ((d == 0 && !rows) || (d == 1 && !cols) || (d == 2 && !(rows && cols))) continue;
          XVal tau[3];
          // 2 g - 2/3 div = 2/3 (3 g - div); 3 g - div is 2 of g less the others: below 2^62
          tau[d] = {xmul(3 * dg[d] - div, cst[4].m), Ed + cst[4].e + 3};
          tau[(d + 1) % 3] = off[d];
          tau[(d + 2) % 3] = off[(d + 2) % 3];
          long long w[4];  // u . tau + kappa dtheta, [58]
          int we[4], E = -32768;
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            w[q] = xmul(vel[q * SM::WF], tau[q].m);
            we[q] = ve[q * SM::WF] + tau[q].e + 3;
          }
          w[3] = xmul(gr[3][d].m, cst[5].m);
          we[3] = gr[3][d].e + cst[5].e + 3;
#pragma unroll
          for (int q = 0; q < 4; ++q) E = xmax(E, we[q]);
          const long long e = xshr(w[0], E - we[0]) + xshr(w[1], E - we[1]) + xshr(w[2], E - we[2]) + xshr(w[3], E - we[3]);
          long long* dst;
          short* de;
          int stride;
          if (d == 0) { dst = fxr; de = fxe; stride = SM::FX; dst += (gy - 2) * GX + gx; de += (gy - 2) * GX + gx; }
          else if (d == 1) { dst = gyr; de = gye; stride = SM::GY_; dst += gy * RX + gx - 2; de += gy * RX + gx - 2; }
          else {
            const int o = zs(p) * 4 * SM::HZ + (gy - 2) * RX + gx - 2;
            dst = hzr + o; de = hze + o; stride = SM::HZ;
          }
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            dst[q * stride] = tau[q].m;
            de[q * stride] = (short)min(tau[q].e, 3 * XBAD);
          }
          dst[3 * stride] = e;
          de[3 * stride] = (short)min(E, 3 * XBAD);
        }
      }
      __syncthreads();
      if (threadIdx.x == 0 && p <= k1 - 1) {  // plane p + 4 (the last needed is k1 + 3), into the slot of plane p - 2
        fence_proxy_async();
        issue(p + 4);
      }
      bool ok = true;
      if (p <= k1) ok = convert(p + 3);
      // D4 of a flux along one direction, [60]; flux values [60]
      auto diff = [&](const long long* f, const short* e, int st, int d) -> XVal {
        const int e0 = e[-2 * st], e1 = e[-st], e2 = e[st], e3 = e[2 * st];
        const int E = xmax(xmax(e0, e1), xmax(e2, e3)) + 2;
        const XVal D = xquick0(xd4(f[-2 * st], E - e0, f[st], E - e2, f[-st], E - e1, f[2 * st], E - e3), E);
        return {xmul(D.m, cst[d].m), D.e + cst[d].e + 3};
      };
      const int k = p - 2, i = x0 + lane, j = y0 + crow;
      const bool out = k >= k0 && i < b.nx && j < b.ny;
      const long long cc = ((long long)k * b.ny + j) * b.nx + i;
#pragma unroll
      for (int n = 0; n < 2; ++n) {
        const int q = q0 + n;
        const int ox = q * SM::FX + crow * GX + lane + 2, oy = q * SM::GY_ + (crow + 2) * RX + lane;
        const XVal dx = diff(fxr + ox, fxe + ox, 1, 0);
        const XVal dy = diff(gyr + oy, gye + oy, RX, 1);
        const int E = xmax(dx.e, dy.e);
        const XVal rv0 = {xshr(dx.m, E - dx.e) + xshr(dy.m, E - dy.e), E};  // [61]
        if (out) {
          const int o = q * SM::HZ + crow * RX + lane;
          auto zf = [&](int kp) { return hzr[zs(kp) * 4 * SM::HZ + o]; };
          auto ze = [&](int kp) { return (int)hze[zs(kp) * 4 * SM::HZ + o]; };
          const int e0 = ze(k - 2), e1 = ze(k - 1), e2 = ze(k + 1), e3 = ze(k + 2);
          const int Ez = xmax(xmax(e0, e1), xmax(e2, e3)) + 2;
          const XVal D = xquick0(xd4(zf(k - 2), Ez - e0, zf(k + 1), Ez - e2, zf(k - 1), Ez - e1, zf(k + 2), Ez - e3), Ez);
          const XVal dz = {xmul(D.m, cst[2].m), D.e + cst[2].e + 3};
          const int Es = xmax(rv2[n].e, dz.e);
          Rv[q * a.n + cc] = xenc(-(xshr(rv2[n].m, Es - rv2[n].e) + xshr(dz.m, Es - dz.e)), Es);
        }
        rv2[n] = rv1[n];
        rv1[n] = rv0;
      }
      fail = __syncthreads_or(!ok);  // the x-, y-flux buffers and the z-slot of plane p - 2 are reused
      if (fail) break;
      if (p <= k1) converted(p + 3);
    }
  }
  if (fail && threadIdx.x == 0) tma_abort(bar, pending, parity, WRING, a.ctrl);
}

}  // namespace wcns
}  // namespace gbcfd
