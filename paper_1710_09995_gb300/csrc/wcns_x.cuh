// wcns_x.cuh -- the direction passes of the FP64 WCNS-E-5 path on the integer pipes (xfix.cuh).
// Included by wcns.cu, whose Args, Box and tile constants it uses.
//
// Same tiles, lines and passes as dir_kernel.  The FP64 form spent ~65 FP64 operations per
// variable and edge pair on the weighted interpolation alone (the pipe issues one per 64 integer
// operations).  Here a landed tile is converted once, in place, to 57-bit integers with an exponent
// each; the interpolation's differences and candidates are then exact integer sums, its weights
// and the Roe flux 62-bit products, and Eq. 2 is taken of the integer fluxes.  One primitive
// buffer (the next tile is requested when the fluxes are done, behind Eq. 2) and a separate flux
// buffer keep two CTAs per SM.  Measured: a 128^3 Navier-Stokes step
// 30.5 -> 9.75 ms (24.7 with only the Roe flux on integers); residuals against long double 1.4 to 2.3
// times closer than the FP64 form's, 5 to 40 times on the finite-volume path.
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
      XPair S[5];
      int worst = 0;
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        const int o = (idx[q] * (LMAX + 10) + m - 2) * NLP + l;
        const XEdge g = xedges<NLP>(Wm + o, We + o, linear, cst[3]);
        const long long r = __shfl_down_sync(0xffffffffu, g.um, 1);
        const int er = __shfl_down_sync(0xffffffffu, g.e, 1), E = xmax(g.e, er);
        S[q] = xpair_norm(xshr(g.up, E - g.e), xshr(r, E - er), E);
        worst = xmax(worst, E);
      }
      if (lane < FCH && f < nfc) {
        XFlux F;
        xroe(S[0], S[1], S[2], S[3], S[4], a.cd.x, F);
#pragma unroll
        for (int q = 0; q < 5; ++q) {
          const int o = (idx[q] * (LMAX + 5) + f) * NLP + l;
          Fm[o] = F.m[q];
          Fe[o] = (short)(worst >= XBAD ? XW_BAD : F.e[q]);
        }
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
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        const int o = (q * (LMAX + 5) + c) * NLP + l;
        long long d[3];
        int ed[3];
#pragma unroll
        for (int x = 0; x < 3; ++x) {  // edges 3 - 2, 4 - 1, 5 - 0 around the cell
          const int h = o + (3 + x) * NLP, w = o + (2 - x) * NLP, e1 = Fe[h], e0 = Fe[w], E = xmax(e1, e0) + 1;
          // normalised, so that the product's truncation is relative to the difference
          const XVal g = xquick(xshr(Fm[h], E - e1) - xshr(Fm[w], E - e0), E);
          d[x] = xmul(g.m, cst[x].m);  // [60]
          ed[x] = g.e + cst[x].e + 3;
        }
        const int E = xmax(ed[0], xmax(ed[1], ed[2]));
        double add = xenc(xshr(d[0], E - ed[0]) - xshr(d[1], E - ed[1]) + xshr(d[2], E - ed[2]), E);
        if (D == 0 && a.viscous && q >= 1)  // the viscous residual, once (x pass)
          add = add + static_cast<const double*>(a.Rv)[(q - 1) * a.n + cc];
        const long long oc = q * a.n + cc;
        if (MODE == 0) {
          R[oc] = add;
        } else if (MODE == 1) {
          R[oc] = R[oc] + add;
        } else {  // Eqs. 4-6
          const double tot = R[oc] + add;
          if (a.stage == 0) {
            a.rout[oc] = tot;
            continue;
          }
          if (a.stage == 1) sq[q] = fma(tot, tot, sq[q]);
          const double adv = a.qs[oc] - dt * tot;
          double out;
          if (a.stage == 1) out = adv;
          else if (a.stage == 2) out = fma(0.75, a.qn[oc], 0.25 * adv);
          else {  // Q^n / 3 with one correction of the product (a division costs ~5 FMAs here)
            const double qn = a.qn[oc], q3 = (1.0 / 3.0) * qn;
            out = fma(2.0 / 3.0, adv, fma(fma(-3.0, q3, qn), 1.0 / 3.0, q3));
          }
          a.qout[oc] = out;
        }
      }
    }
  }
  if (MODE == 2 && a.stage == 1) norm_fold(a, sq, red, &last);
}

}  // namespace wcns
}  // namespace gbcfd
