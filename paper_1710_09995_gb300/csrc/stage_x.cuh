// stage_x.cuh -- the fused Runge-Kutta stage of the FP64 path (Cartesian blocks, and inviscid
// curvilinear ones), with the faces in 64-bit block-floating arithmetic (xfix.cuh).
//
// Same method, tiles, TMA staging, group table and reductions as stage_kernel (stage.cuh); what
// differs is where the work runs.  This part's FP64 pipe issues one operation per 64 integer ones,
// and the faces' reconstruction and fluxes were ~95% of the FP64 operations of a cell.  Here the
// staged planes are converted once per cell to primitives in the ring as a 61-bit signed integer
// and an exponent each; the faces (MUSCL, Roe, viscous flux), the residual and the time step's rate
// run on the integer pipes.  FP64 is left with the stage update itself and the norm (5 to 15
// operations a cell; with the conversion, the assembly and the rate in FP64 too its pipe was
// 26% busy, alone between two barriers: 25.7 ms a step on the 256^3 case against 21.2 then).
//
// Faces are work items of a warp: the tile's z-, y- and x-rows (32 faces each) and one item of the
// TY faces on the tile's upper x side, 3 TY + 2 items per plane dealt round-robin to the warps.  The
// three directions go through the same instructions (index offsets and the frame's permutation
// are data): a face is about 2000 instructions, and a copy per direction (six call sites in the
// first version) streamed the code through the instruction caches on every plane.  16 warps of 128
// registers: 26 items (TY 8) give the sub-partitions 7, 7, 6, 6; with 13 warps of one item each
// round one of them had 8.  On Cartesian blocks at TY 8 the flux buffers of two planes fit (PIPE): the warps
// that have one face item update the rows of the plane before in the same turn, where 8 warps updated
// between two barriers while 8 waited (36 uneven Euler blocks 19.6 -> 18.4 ms, 256^3 Navier-Stokes 20.4 -> 19.6).
// Bound by the integer pipes: ALU 60% busy, issue slots 57-61%, the rest multiply-add latency at 4 warps a
// scheduler.  Measured against the FP64-pipe form: 256^3 Navier-Stokes step 81.7 -> 20.9 ms, 36 uneven Euler
// blocks (14.4M cells) 69.0 -> 19.4 ms, two steps of the bump channel 14.2 -> 4.04 ms (19.6, 18.4 and 3.86 before every
// term had a class of its own size: components far below the others, and cells beside jumps, then had errors 10^2 to
// 10^9 times the FP64 form's).  Residuals of smooth states are 24 to 50 times closer to long double than
// that form's, states after a step the same to 2.6 times.
#pragma once
#include "stage.cuh"

namespace gbcfd {

// CURVI: one staging slot (a plane's work is far longer than its copy) leaves room for the metric ring
template <bool VISC, bool CURVI, int TYV, int NWV>
struct XPlan {
  static constexpr int TY = TYV, BY = box_rows(TYV), NW = NWV;
  static constexpr int NV = VISC ? 6 : 5;  // rho u v w p [theta]
  static constexpr int BOX = BY * BX;
  // PIPE: the update of a plane runs beside the faces of the next one (more flux buffers); where they fit
  static constexpr bool PIPE = !CURVI && TYV == TY_DEFAULT;
  static constexpr int NST = CURVI || (PIPE && VISC) ? 1 : NSTAGE, NMS = CURVI ? 2 : 0;  // staging slots, metric planes
  static constexpr size_t QSLOT = (sizeof(double) * 5 * BOX + 127) / 128 * 128;
  static constexpr size_t stq = 0;                                          // staged conserved planes
  static constexpr size_t ringm = stq + NST * QSLOT;                     // primitives: 61-bit integers
  static constexpr size_t ringe = ringm + sizeof(long long) * NRING * NV * BOX;  // and their exponents (biased)
  // face fluxes, 62-bit integers and exponents: one or two planes of x and y, two or three of z
  static constexpr int NFX = 5 * TY * (TX + 1), NFY = 5 * (TY + 1) * TX, NFZ = 5 * TY * TX;
  static constexpr int NBX = PIPE ? 2 : 1, NBZ = PIPE ? 3 : 2;
  static constexpr int FY0 = NBX * NFX, FZ0 = FY0 + NBX * NFY, NF = FZ0 + NBZ * NFZ;
  static constexpr size_t fm = (ringe + sizeof(short) * NRING * NV * BOX + 15) / 16 * 16;
  static constexpr size_t fe = fm + sizeof(long long) * NF;
  static constexpr size_t MSLOT = (sizeof(double) * 10 * BOX + 127) / 128 * 128;
  static constexpr size_t mring = (fe + sizeof(short) * NF + 127) / 128 * 128;
  static constexpr size_t red = mring + NMS * MSLOT;
  static constexpr size_t blk = red + sizeof(double) * NW * NPART;          // the block's coefficients (XBlk)
  static constexpr size_t bar = blk + 20 * sizeof(XVal);
  static constexpr size_t misc = bar + 8 * (NST + NMS);
  static constexpr size_t push = (misc + 16 + 15) / 16 * 16;
  static constexpr size_t bytes = (push + 27 * sizeof(PushDst) + 127) / 128 * 128;
  static_assert(bytes <= 232448, "227 KB of shared memory per CTA");
};

static_assert(sizeof(XBlk) == 20 * sizeof(XVal), "XPlan::blk");

// ring values are 61-bit integers with a biased exponent: value = m 2^(e - 1022 - 61)
constexpr int XRING_BIAS = 1022;

// one warp item's index data: cells c[0..3] along the normal (c[1] = L, c[2] = R) as indices into
// variable 0 of the ring; variable offsets of the normal and tangential velocities; tangential
// neighbours (added to c[1], c[2])
struct XItem {
  int c[4];
  int vn, v1, v2;
  int t1p, t1m, t2p, t2m;
};

// a face whose sides are far apart (xfar) in FP64, from the stencil's values rounded to doubles: twice the flux
// (CURVI: the flux).  Out of line: only faces with a jump of 2^5 or more in the density or the pressure call it.
template <bool CURVI, int MS>
__device__ __noinline__ XFlux xface_f64(const long long* rm, const short* re, int c0, int c1, int c2, int c3, int vn, int v1,
                                        int v2, const double* S, double gm1, double ggm1, double eps, int lim) {
  const int at[4] = {c0, c1, c2, c3}, var[5] = {0, vn, v1, v2, 4 * MS};
  Consts<double> K;
  K.gm1 = gm1;
  K.ggm1 = ggm1;
  K.eps = eps;
  double L[5], R[5], F[5];
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    double x[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) x[c] = xenc(rm[at[c] + var[q]], re[at[c] + var[q]] - XRING_BIAS);
    muscl(x[0], x[1], x[2], x[3], lim, L[q], R[q]);
  }
  if constexpr (CURVI) {
    const double a[3] = {S[0], S[MS], S[2 * MS]};
    roe_area<double>(L, R, a, K, F);
  } else {
    roe_frame<double, true>(L, R, K, F);
  }
  return xflux_of(F);
}

// twice the flux (F - Fv) through the lane's face; CURVI: the flux, S its area vector (strides MS)
template <bool VISC, bool CURVI, int MS>
__device__ __forceinline__ void xface(const long long* __restrict__ rm, const short* __restrict__ re, const XItem& I,
                                      int d, const XBlk* __restrict__ X, const double* __restrict__ S,
                                      const XConsts& K, const PathK<double>& PK, int lim, XFlux& F) {
  XVal dn[4];  // R - L of the velocities and theta (viscous)
  long long us[3];
  int eu[3];
  auto load = [&](const int (&ix)[4], int off, long long (&m)[4], int (&e)[4]) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      m[c] = rm[ix[c] + off];
      e[c] = re[ix[c] + off];
    }
  };
  auto states = [&](int off, int q) -> XPair {
    long long m[4];
    int e[4];
    load(I.c, off, m, e);
    XSten s = xmuscl(m, e, lim);
    if (VISC && q >= 0) {
      dn[q] = xquick0(s.d, s.ed - XRING_BIAS);
      us[q] = s.sum;
      eu[q] = s.ed - XRING_BIAS;
    }
    s.s.e -= XRING_BIAS;
    return s.s;
  };
  const XPos r = states(0, -1), p = states(4 * MS, -1);
  const XPair u = states(I.vn, 0), v = states(I.v1, 1), w = states(I.v2, 2);
  if (xfar(r, p)) {
    F = xface_f64<CURVI, MS>(rm, re, I.c[0], I.c[1], I.c[2], I.c[3], I.vn, I.v1, I.v2, S, PK.gm1, PK.ggm1, PK.eps, lim);
  } else if constexpr (CURVI) {
    xroe_area(r, u, v, w, p, S[0], S[MS], S[2 * MS], K, F);
  } else {
    xroe(r, u, v, w, p, K, F);
  }
  if constexpr (VISC) {
    auto tang = [&](int off, int tp, int tm) -> XVal {
      const int ix[4] = {I.c[1] + tp, I.c[1] + tm, I.c[2] + tp, I.c[2] + tm};
      long long m[4];
      int e[4];
      load(ix, off, m, e);
      return xtang(m, e, XRING_BIAS);
    };
    const int d1 = d == 2 ? 0 : d + 1, d2 = d == 0 ? 2 : d - 1;
    const int el = re[I.c[1] + 5 * MS], er = re[I.c[2] + 5 * MS], E = xmax(el, er);
    dn[3] = xquick0(xshr(rm[I.c[2] + 5 * MS], E - er) - xshr(rm[I.c[1] + 5 * MS], E - el), E - XRING_BIAS);
    xviscous(d, d1, d2, *X, dn, us, eu, tang(I.vn, I.t1p, I.t1m), tang(I.vn, I.t2p, I.t2m), tang(I.v1, I.t1p, I.t1m),
             tang(I.v2, I.t2p, I.t2m), F);
  }
}

// registers: NW warps in one CTA per SM (65536 / (32 NW) per thread)
template <bool VISC, int STAGE, bool CURVI, int TYV, int NWV, bool PUSH>
__global__ void __launch_bounds__(32 * NWV, 1) xstage_kernel(const GroupParams P) {
  using PL = XPlan<VISC, CURVI, TYV, NWV>;
  static_assert(TYV <= NWV && !(VISC && CURVI), "a warp owns at most one row; viscous curvilinear blocks: stage_kernel");
  constexpr int NST = PL::NST, NMS = PL::NMS;
  constexpr int TY = TYV, BY = PL::BY, NW = NWV, NT = 32 * NWV, NV = PL::NV, MS = BY * BX, SL = NV * MS;
  constexpr int NITEM = 3 * TY + 2;
  constexpr bool PIPE = PL::PIPE;
  constexpr int W1 = PIPE ? NITEM - NW : 0, WU = NW - W1;  // PIPE: warps W1 .. have one item, and update
  static_assert(!PIPE || (W1 > 0 && WU > 0), "two items a warp at most");

  extern __shared__ __align__(128) unsigned char smem[];
  long long* rm = reinterpret_cast<long long*>(smem + PL::ringm);
  short* re = reinterpret_cast<short*>(smem + PL::ringe);
  long long* fm = reinterpret_cast<long long*>(smem + PL::fm);
  short* fe = reinterpret_cast<short*>(smem + PL::fe);
  double* mring = reinterpret_cast<double*>(smem + PL::mring);
  double* red = reinterpret_cast<double*>(smem + PL::red);
  XBlk* xb = reinterpret_cast<XBlk*>(smem + PL::blk);
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + PL::bar);
  int* sabort = reinterpret_cast<int*>(smem + PL::misc);
  int* slast = sabort + 1;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const Physics& ph = P.ph;
  const XConsts& XK = P.pk.x;

  // the block of this CTA and the CTA's contiguous share of its tile-planes
  int bsel;
  {
    int lo = 0, hi = P.nblocks - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (P.table[mid].cta0 <= (int)blockIdx.x) lo = mid; else hi = mid - 1;
    }
    bsel = lo;
  }
  const BlockDesc* D = P.table + bsel;
  const double hx = D->ihx, hy = D->ihy, hz = D->ihz;
  PushDst* pushdst = reinterpret_cast<PushDst*>(smem + PL::push);
  if (tid == 0) {
    for (int s = 0; s < NST + NMS; ++s) mbar_init(&bar[s], 1);
    fence_barrier_init();
    *sabort = 0;
  }
  if (tid < 3) {
    const double h = tid == 0 ? hx : (tid == 1 ? hy : hz), m2 = P.pk.d.mu + P.pk.d.mu;
    xb->h2[tid] = xdec_pos<62>(0.5 * h);
    if (VISC) {
      xb->a[tid] = xdec_pos<62>(m2 * h);
      xb->a43[tid] = xdec_pos<62>((4.0 / 3.0) * m2 * h);
      xb->b[tid] = xdec_pos<62>(m2 * (0.25 * h));
      xb->b23[tid] = xdec_pos<62>((2.0 / 3.0) * m2 * (0.25 * h));
      xb->k[tid] = xdec_pos<62>(4.0 * P.pk.d.kappa * h);
    }
    if (tid == 0) {
      xb->hsum = xdec_pos<62>(hx + hy + hz);
      xb->vs = xdec_pos<62>(P.pk.d.vf * (hx * hx + hy * hy + hz * hz));
    }
  }
  if constexpr (PUSH && (STAGE == 1 || STAGE == 2)) {
    if (tid < 27) push_table<double, STAGE>(P.table, bsel, tid, pushdst);
  }
  __syncthreads();

  const double dt = (STAGE == 0) ? 0.0 : P.gctrl->dt;
  unsigned phase_bits = 0;  // parity of each staging slot (uniform across the CTA)
  unsigned pending = 0;     // slots with a copy in flight (meaningful in thread 0)
  unsigned mphase = 0, mpending = 0;  // the same of the metric slots
  bool bad = false;         // non-physical value met by this thread
  double nacc[5] = {0, 0, 0, 0, 0};
  double rate_max = 0.0;

  const int lcta = (int)blockIdx.x - D->cta0, nctas = D->ctas;
  const long long W = D->units;
  const long long u_begin = (long long)lcta * W / nctas;
  const long long u_end = (long long)(lcta + 1) * W / nctas;
  constexpr unsigned QBYTES = 5u * MS * sizeof(double);
  const Geometry g = D->g;
  // arrays of this stage
  constexpr int in = STAGE == 0 ? 0 : STAGE - 1;
  const CUtensorMap* tmq = &D->tq[in];
  const double *qs = D->q[in], *qn = D->q[0];
  double* qout = D->q[STAGE % 3];

  for (long long u = u_begin; u < u_end;) {
    const int nz = g.nz;
    const long long tile = u / nz;
    const int k0 = (int)(u - tile * nz);
    const int k1 = (int)min((long long)nz, (long long)k0 + (u_end - u));
    u += k1 - k0;
    const int tix = (int)(tile % D->ntx), tiy = (int)(tile / D->ntx);
    const int x0 = tix * TX, y0 = tiy * TY;  // storage coordinates of the box origin
    const int last_plane = k1 + 1;
    // the last plane's update reads the metric slots that this tile's first copy lands in, with no barrier behind it
    if constexpr (CURVI) __syncthreads();

    auto request = [&](int kp) {  // thread 0 only
      const int s = (kp + 2) & (NST - 1);
      fence_proxy_async();
      mbar_expect_tx(&bar[s], QBYTES);
      tma_load_4d(smem + PL::stq + s * PL::QSLOT, tmq, &bar[s], x0, y0, kp + HALO, 0);
      pending |= 1u << s;
    };
    // wait for plane kp, convert it into ring slot kp & 3, then refill the staging slot
    auto consume = [&](int kp) -> bool {
      const int s = (kp + 2) & (NST - 1);
      const bool ok = mbar_wait_bounded(&bar[s], (phase_bits >> s) & 1u);
      if (!ok) atomicOr(sabort, 1);
      phase_bits ^= 1u << s;
      const double* sq = reinterpret_cast<const double*>(smem + PL::stq + s * PL::QSLOT);
      long long* m = rm + (kp & 3) * SL;
      short* e = re + (kp & 3) * SL;
      for (int c = tid; c < MS; c += NT) {
        const int cy = c / BX, cx = c - cy * BX;
        double q[5];
#pragma unroll
        for (int v = 0; v < 5; ++v) q[v] = sq[v * MS + c];
        const bool valid = (x0 - HALO + cx < g.nx + HALO) && (y0 - HALO + cy < g.ny + HALO);
        XPrim W;
        const bool phys = xprim(q, XK, W);
        if (valid && !phys) bad = true;
        const bool fill = !valid || !phys;  // rho = p = 1, no velocity
        auto put = [&](int v, long long a, int ea, bool one) {
          m[v * MS + c] = fill ? (one ? 1ll << 60 : 0ll) : a;
          e[v * MS + c] = (short)(fill ? (one ? XRING_BIAS + 1 : XZERO) : XRING_BIAS + ea);
        };
        put(0, W.r.m >> 1, W.r.e + 1, true);
#pragma unroll
        for (int x = 0; x < 3; ++x) put(1 + x, W.u[x].m >> 1, W.u[x].e + 1, false);
        put(4, W.p.m >> 1, W.p.e + 1, true);
        if (VISC) put(5, xmul(W.p.m, W.ir.m), W.p.e + W.ir.e + 3, true);
      }
      __syncthreads();
      if (tid == 0) {
        pending &= ~(1u << s);
        if (kp + NST <= last_plane && *sabort == 0) request(kp + NST);
      }
      return *sabort == 0;
    };

    // metric planes (curvilinear): plane kp in slot kp & 1; iteration k reads k and k + 1
    int m_req = k0 - 1, m_wait = k0 - 1;
    auto mrequest_upto = [&](int upto) {  // thread 0 only
      if constexpr (CURVI) {
        upto = min(upto, k1);
        while (m_req < upto) {
          ++m_req;
          const int s = m_req & 1;
          fence_proxy_async();
          mbar_expect_tx(&bar[NST + s], 10u * MS * sizeof(double));
          tma_load_4d(smem + PL::mring + s * PL::MSLOT, &D->tm, &bar[NST + s], x0, y0, m_req + HALO, 0);
          mpending |= 1u << s;
        }
      }
    };
    auto mwait_upto = [&](int upto) {  // all threads
      if constexpr (CURVI) {
        while (m_wait < upto) {
          ++m_wait;
          const int s = m_wait & 1;
          if (!mbar_wait_bounded(&bar[NST + s], (mphase >> s) & 1u)) atomicOr(sabort, 1);
          mphase ^= 1u << s;
          if (tid == 0) mpending &= ~(1u << s);
        }
      }
    };

    if (tid == 0) {
      tensormap_acquire(tmq);
      if (CURVI) tensormap_acquire(&D->tm);
      for (int i = 0; i < NST; ++i) request(k0 - 2 + i);
      mrequest_upto(k0);
    }
    bool ok = true;
    for (int kp = k0 - 2; kp <= k0 && ok; ++kp) ok = consume(kp);
    if (!ok) break;

    auto zslot = [](int k) { return PL::FZ0 + (k + 1) % PL::NBZ * PL::NFZ; };  // of the upper z-faces of plane k >= -1
    auto xslot = [](int k) { return PL::NBX == 2 ? k & 1 : 0; };
    // the update of the tile's row `row` of plane k, a cell a lane
    auto update = [&](int k, int row) {
      const int ci = x0 + lane, cj = y0 + row;
      if (ci >= g.nx || cj >= g.ny) return;
      const long long o = gidx(g, ci, cj, k);
      double dtc = dt;
      if constexpr (STAGE >= 1 && !VISC)  // local time steps: inviscid blocks only
        if (ph.local_dt) dtc = __ldg(static_cast<const double*>(D->dtl) + o);
      double qs_[5], qn_[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        if constexpr (STAGE >= 1) qs_[v] = __ldg(qs + v * g.field + o);
        if constexpr (STAGE >= 2) qn_[v] = __ldg(qn + v * g.field + o);
      }
      const int mk = k & 1, mk1 = (k + 1) & 1;
      constexpr int MSD = PL::MSLOT / sizeof(double);
      const double* mc = mring + mk * MSD + (row + HALO) * BX + lane + HALO;  // the cell's metrics
      XVal iv = {0, 0};
      if constexpr (CURVI) iv = xrcp(xdec_pos<62>(mc[9 * MS]));
      double R[5], out[5];
      // R = sum over directions of (upper - lower face flux) / h (CURVI: / V)
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        const int x = xslot(k) * PL::NFX + q * TY * (TX + 1) + row * (TX + 1) + lane,
                  y = PL::FY0 + xslot(k) * PL::NFY + q * (TY + 1) * TX + row * TX + lane, z = q * TY * TX + row * TX + lane;
        const int up[3] = {x + 1, y + TX, z + zslot(k)}, lo[3] = {x, y, z + zslot(k - 1)};
        long long d[3];
        int ed[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          const int e1 = fe[up[a]], e0 = fe[lo[a]];
          ed[a] = xmax(e1, e0) + 1;
          d[a] = xshr(fm[up[a]], ed[a] - e1) - xshr(fm[lo[a]], ed[a] - e0);  // [62]
          // normalised first: the product's truncation is then relative to the difference (left to the
          // flux's own scale it doubled the 32^3 pulse's error against 64-bit references), and a direction in
          // which a component does not change does not take the others' bits
          const XVal f = xquick0(d[a], ed[a]);
          d[a] = CURVI ? f.m : xmul(f.m, xb->h2[a].m);  // [60]; CURVI [62]
          ed[a] = f.e + (CURVI ? 0 : xb->h2[a].e + 3);
        }
        const int E = xmax(ed[0], xmax(ed[1], ed[2])) + (CURVI ? 2 : 0);
        const long long t = xshr(d[0], E - ed[0]) + xshr(d[1], E - ed[1]) + xshr(d[2], E - ed[2]);
        if constexpr (CURVI) {
          const XVal r = xquick(t, E);
          R[q] = xenc(xmul(r.m, iv.m), r.e + iv.e + 3);
        } else {
          R[q] = xenc(t, E);
        }
      }
      if constexpr (STAGE == 0) {
        const long long oc = ((long long)k * g.ny + cj) * g.nx + ci;
        const long long n = (long long)g.nx * g.ny * g.nz;
#pragma unroll
        for (int m = 0; m < 5; ++m) P.rout[m * n + oc] = R[m];
      } else {
#pragma unroll
        for (int m = 0; m < 5; ++m) {
          const double adv = qs_[m] - dtc * R[m];
          if constexpr (STAGE == 1) out[m] = adv;
          else if constexpr (STAGE == 2) out[m] = fma(0.75, qn_[m], 0.25 * adv);
          else out[m] = fma(2.0 / 3.0, adv, (1.0 / 3.0) * qn_[m]);  // an FP64 division costs ~7 FMAs here
          qout[m * g.field + o] = out[m];
        }
        if constexpr (PUSH && (STAGE == 1 || STAGE == 2))
          if (ci < HALO || cj < HALO || k < HALO || ci >= g.nx - HALO || cj >= g.ny - HALO || k >= g.nz - HALO)
            push_halo<double>(pushdst, g.nx, g.ny, g.nz, ci, cj, k, out[0], out[1], out[2], out[3], out[4]);
        if constexpr (STAGE == 1) {
#pragma unroll
          for (int m = 0; m < 5; ++m) nacc[m] = fma(R[m], R[m], nacc[m]);
        }
        if constexpr (STAGE == 3) {
          XPrim W;
          const bool phys = xprim(out, XK, W);
          if (!phys) bad = true;
          const XVal c = xsound(W, XK.gam);
          XVal rate;
          if constexpr (!CURVI) {
            rate = xrate<VISC>(W, c, xb->h2, xb->hsum, xb->vs);
          } else {  // sum over directions of |u . S| + c |S|, over V
            const double* mu[3] = {mc + 1, mc + BX, mring + mk1 * MSD + (row + HALO) * BX + lane + HALO};
            XVal r[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
              const double lo[3] = {mc[3 * a * MS], mc[(3 * a + 1) * MS], mc[(3 * a + 2) * MS]};
              const double up[3] = {mu[a][3 * a * MS], mu[a][(3 * a + 1) * MS], mu[a][(3 * a + 2) * MS]};
              r[a] = xradius<false>(W, c, lo, up, iv);
            }
            const XVal v = xsum3(r[0], r[1], r[2]);
            rate = xnormed(xmul(v.m, iv.m), v.e + iv.e + 3);
          }
          // the largest rate, as the bits of a non-negative double
          const long long rb = __double_as_longlong(xenc(rate.m, rate.e));
          if (phys && rb > __double_as_longlong(rate_max)) rate_max = __longlong_as_double(rb);
          if constexpr (!VISC)
            if (ph.local_dt) {
              const XVal ir = xrcp(rate);
              static_cast<double*>(D->dtl)[o] = ph.cfl * xenc(ir.m, ir.e);
            }
        }
      }
    };

    // plane k0 - 1 only gives the lower z-faces of plane k0; PIPE: turn k1 is the last plane's update only
    for (int k = k0 - 1; k < k1 + (PIPE ? 1 : 0); ++k) {
      if (k < k1 && !consume(k + 2)) { ok = false; break; }
      if (tid == 0) mrequest_upto(k + 1);  // its slot held plane k - 1, last read before consume's barrier
      mwait_upto(k < k0 ? k0 : k + 1);
      const int sm = ((k - 1) & 3) * SL, sk = (k & 3) * SL, sp = ((k + 1) & 3) * SL, s2 = ((k + 2) & 3) * SL;
      const int nitem = k == k1 ? 0 : (k < k0 ? TY : NITEM);
      if constexpr (PIPE)
        if (k > k0 && (k == k1 || warp >= W1))
#pragma unroll 1
          for (int row = k == k1 ? warp : warp - W1; row < TY; row += k == k1 ? NW : WU) update(k - 1, row);
#pragma unroll 1
      for (int it = warp; it < nitem; it += NW) {
        const int d = it < TY ? 2 : (it < 2 * TY + 1 ? 1 : 0);
        int row = it < TY ? it : (it < 2 * TY + 1 ? it - TY : it - (2 * TY + 1));
        int col = lane;
        // rows of a ragged tile past the block's edge: y-rows up to the block's upper face
        if (y0 + row > g.ny - (d == 1 ? 0 : 1) && row < TY) continue;
        if (d == 1 && row == TY && y0 + TY > g.ny) continue;
        if (d == 0 && row == TY) {  // the upper x-faces of the tile
          if (x0 + TX > g.nx || lane >= TY || y0 + lane >= g.ny) continue;
          row = lane;
          col = TX;
        }
        const int b = sk + (row + HALO) * BX + col + HALO;
        XItem I;
        I.vn = (1 + d) * MS;
        I.v1 = (d == 2 ? 1 : 2 + d) * MS;
        I.v2 = (d == 0 ? 3 : d) * MS;
        if (d == 2) {
          I.c[0] = b - sk + sm; I.c[1] = b; I.c[2] = b - sk + sp; I.c[3] = b - sk + s2;
          I.t1p = 1; I.t1m = -1; I.t2p = BX; I.t2m = -BX;
        } else {
          const int st = d == 0 ? 1 : BX;
          I.c[0] = b - 2 * st; I.c[1] = b - st; I.c[2] = b; I.c[3] = b + st;
          const int zp = sp - sk, zm = sm - sk;
          I.t1p = d == 0 ? BX : zp; I.t1m = d == 0 ? -BX : zm;
          I.t2p = d == 0 ? zp : 1; I.t2m = d == 0 ? zm : -1;
        }
        const double* S = nullptr;
        if constexpr (CURVI) {  // x, y, z velocities as they are; the face's area vector: z-faces are plane k + 1's lower ones
          I.vn = MS; I.v1 = 2 * MS; I.v2 = 3 * MS;
          S = mring + ((d == 2 ? k + 1 : k) & 1) * (PL::MSLOT / sizeof(double)) + 3 * d * MS + (row + HALO) * BX + col + HALO;
        }
        XFlux F;
        xface<VISC, CURVI, MS>(rm, re, I, d, xb, S, XK, P.pk.d, ph.limiter, F);
        const int f = d == 2 ? zslot(k) + row * TX + col
                             : (d == 1 ? PL::FY0 + xslot(k) * PL::NFY + row * TX + col
                                       : xslot(k) * PL::NFX + row * (TX + 1) + col);
        const int fs = d == 2 ? TY * TX : (d == 1 ? (TY + 1) * TX : TY * (TX + 1));
        const int to[5] = {f, f + (CURVI ? 1 : 1 + d) * fs, f + (CURVI ? 2 : (d == 2 ? 1 : 2 + d)) * fs,
                           f + (CURVI ? 3 : (d == 0 ? 3 : d)) * fs, f + 4 * fs};
#pragma unroll
        for (int q = 0; q < 5; ++q) {
          fm[to[q]] = F.m[q];
          fe[to[q]] = (short)F.e[q];
        }
      }
      __syncthreads();
      if (!PIPE && k >= k0 && warp < TY) update(k, warp);  // warp `row` owns row `row` of the tile
    }
    if (!ok) break;
  }

  // abort path: drain copies still in flight (bounded), flag the timeout
  if (*sabort) {
    if (tid == 0) {
      for (int s = 0; s < NST; ++s)
        if (pending & (1u << s)) mbar_wait_bounded(&bar[s], (phase_bits >> s) & 1u);
      for (int s = 0; s < NMS; ++s)
        if (mpending & (1u << s)) mbar_wait_bounded(&bar[NST + s], (mphase >> s) & 1u);
      atomicOr(&D->ctrl->flag, FLAG_TIMEOUT);
    }
  }
  if (bad) atomicOr(&D->ctrl->flag, FLAG_NONPHYSICAL);

  if constexpr (STAGE == 1 || STAGE == 3) stage_reduce<STAGE, NW>(P, reinterpret_cast<double*>(smem + PL::ringm), red, slast, nacc, rate_max);
}

// ---- launch helpers --------------------------------------------------------------------------
// warps per tile height: 3 TY + 2 items a plane
constexpr int xwarps(int) { return 16; }

template <bool VISC, int STAGE, bool CURVI, int TYV, bool PUSH = false>
cudaError_t xstage_attr() {
  constexpr int NW = xwarps(TYV);
  static std::atomic<unsigned long long> done{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 64 && ((done.load(std::memory_order_acquire) >> dev) & 1ull)) return cudaSuccess;
  e = cudaFuncSetAttribute(xstage_kernel<VISC, STAGE, CURVI, TYV, NW, PUSH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)XPlan<VISC, CURVI, TYV, NW>::bytes);
  if (e == cudaSuccess && dev < 64) done.fetch_or(1ull << dev, std::memory_order_acq_rel);
  return e;
}
template <bool VISC, int STAGE, bool CURVI, int TYV, bool PUSH = false>
cudaError_t xstage_go(const GroupParams& P, int grid, cudaStream_t s) {
  constexpr int NW = xwarps(TYV);
  cudaError_t e = xstage_attr<VISC, STAGE, CURVI, TYV, PUSH>();
  if (e != cudaSuccess) return e;
  xstage_kernel<VISC, STAGE, CURVI, TYV, NW, PUSH><<<grid, 32 * NW, XPlan<VISC, CURVI, TYV, NW>::bytes, s>>>(P);
  return cudaGetLastError();
}
template <bool VISC, bool CURVI, int TYV>
cudaError_t xstage_prepare() {
  cudaError_t e = xstage_attr<VISC, 0, CURVI, TYV>();
  if (e == cudaSuccess) e = xstage_attr<VISC, 1, CURVI, TYV>();
  if (e == cudaSuccess) e = xstage_attr<VISC, 2, CURVI, TYV>();
  if (e == cudaSuccess) e = xstage_attr<VISC, 3, CURVI, TYV>();
  return e;
}
template <bool VISC, bool CURVI, int TYV>
cudaError_t xstage_dispatch(int stage, const GroupParams& P, int grid, cudaStream_t s) {
  switch (stage) {
    case 0: return xstage_go<VISC, 0, CURVI, TYV>(P, grid, s);
    case 1: return xstage_go<VISC, 1, CURVI, TYV>(P, grid, s);
    case 2: return xstage_go<VISC, 2, CURVI, TYV>(P, grid, s);
    case 3: return xstage_go<VISC, 3, CURVI, TYV>(P, grid, s);
  }
  return cudaErrorInvalidValue;
}
template <int TYV>
cudaError_t xstage_dispatch_push(int stage, const GroupParams& P, int grid, cudaStream_t s) {
  switch (stage) {
    case 1: return xstage_go<false, 1, false, TYV, true>(P, grid, s);
    case 2: return xstage_go<false, 2, false, TYV, true>(P, grid, s);
  }
  return cudaErrorInvalidValue;
}
template <int TYV>
cudaError_t xstage_prepare_push() {
  cudaError_t e = xstage_attr<false, 1, false, TYV, true>();
  if (e == cudaSuccess) e = xstage_attr<false, 2, false, TYV, true>();
  return e;
}

}  // namespace gbcfd
