// stage_c.cuh -- the fused Runge-Kutta stage on curvilinear blocks, mixed path (FP64: stage_x.cuh for
// inviscid blocks, stage.cuh for viscous ones).
//
// Same method, tiles, TMA staging and reductions as stage_kernel (stage.cuh), another schedule.  A
// curvilinear face takes about 600 instructions and its metric ring leaves room for one CTA per SM; with
// the faces spread over the directions (five copies of the code, nine warps, two barriers a plane)
// the instruction cache missed on 44% of its requests and the SMs issued half of the time.  Here the
// faces are work items of a warp (the tile's z-, y- and x-rows and one item of its upper x side,
// 3 TY + 2 a plane), all through one copy of face_flux_curvi with the direction in the index data,
// dealt to 16 warps.  The first 3 TY + 2 - 16 warps take two items; the others take one, and in the
// same phase the update of the plane before and the conversion of the plane after, so that a plane
// costs one barrier and every warp carries about 1,400 instructions between two of them.  For that the
// state ring has five planes, the metric ring four, the fluxes two or three, and all of a share's
// first four planes are requested at once (four staging slots).  In
// stage 3 the new time-step rates are taken by the two-face warps from the state that the update
// leaves in shared memory.  Measured (warped 128^3 Navier-Stokes block): stages 1 and 2 246 and 239 ->
// 195 and 191 us, issue slots 51 -> 71%, instruction-cache hits 56 -> 99.7%; a whole step 1.20x, of the
// 192 x 96 x 16 bump channel (7.6 planes a CTA) 1.08x.
#pragma once
#include <atomic>

#include "launch.h"
#include "stage.cuh"

namespace gbcfd {

template <bool VISC, int TYV>
struct CPlan {
  static constexpr int TY = TYV, BY = box_rows(TYV), NW = 16;
  static constexpr int NV = VISC ? 6 : 5;           // rho u v w p [theta]
  static constexpr int BOX = BY * BX;               // cells per staged plane
  static constexpr int NST = 4, NR = 5, NMS = 4;    // staging slots, state planes, metric planes
  static constexpr size_t SLOT = (sizeof(float) * 5 * BOX + 127) / 128 * 128;
  static constexpr size_t MSLOT = (sizeof(float) * 10 * BOX + 127) / 128 * 128;
  // floats of one buffer of x-, y- and z-fluxes
  static constexpr int FX = 5 * TY * (TX + 1), FY = 5 * (TY + 1) * TX, FZ = 5 * TY * TX;
  static constexpr size_t stq = 0;                        // state staging
  static constexpr size_t std_ = stq + NST * SLOT;        // increment staging
  static constexpr size_t mring = std_ + NST * SLOT;
  static constexpr size_t ring = mring + NMS * MSLOT;
  static constexpr size_t fx = ring + sizeof(float) * NR * NV * BOX;
  static constexpr size_t fy = fx + sizeof(float) * 2 * FX;
  static constexpr size_t fz = fy + sizeof(float) * 2 * FY;
  static constexpr size_t red = (fz + sizeof(float) * 3 * FZ + 15) / 16 * 16;
  static constexpr size_t bar = red + sizeof(double) * NW * NPART;
  static constexpr size_t misc = bar + 8 * (NST + NMS);
  static constexpr size_t bytes = (misc + 16 + 127) / 128 * 128;
  static_assert(bytes <= 232448, "227 KB of shared memory per CTA");
};

// Offsets of a face's stencil from the cell (of plane k) whose lower x- or y-face, or upper z-face, it
// is: the cells along the normal and the neighbours of L and R along tangents 1 and 2 (x, y, z
// cyclic) in the state ring, and in the metric ring the face's vector, the vectors averaged for the
// tangents and the volumes.  They depend on the direction and on the ring slot of plane k only, so they
// are tabulated: forming them at each face cost 8% more instructions (stage 1 of the block
// above: 204 us, with the table 195).
struct alignas(16) FaceOff {
  int sten[4], tg[8];
};
struct alignas(16) MetOff : MetIdx {
  int pad;
};
template <int NV, int BY>
struct FaceTab {
  static constexpr int NR = 5, NMS = 4, MS = BY * BX;
  FaceOff face[NR][3];
  MetOff met[NMS][3];
  constexpr FaceTab() : face{}, met{} {
    for (int s = 0; s < NR; ++s)
      for (int d = 0; d < 3; ++d) {
        const int Sk = s * NV * MS, Sm = (s + NR - 1) % NR * NV * MS, Sp = (s + 1) % NR * NV * MS,
                  S2 = (s + 2) % NR * NV * MS, zp = Sp - Sk, zm = Sm - Sk;
        const int st = d == 0 ? 1 : BX, L = d == 2 ? Sk : Sk - st, R = d == 2 ? Sp : Sk;
        const int t1p = d == 0 ? BX : (d == 1 ? zp : 1), t1m = d == 0 ? -BX : (d == 1 ? zm : -1);
        const int t2p = d == 0 ? zp : (d == 1 ? 1 : BX), t2m = d == 0 ? zm : (d == 1 ? -1 : -BX);
        const int sten[4] = {d == 2 ? Sm : Sk - 2 * st, L, R, d == 2 ? S2 : Sk + st};
        const int tg[8] = {L + t1p, L + t1m, R + t1p, R + t1m, L + t2p, L + t2m, R + t2p, R + t2m};
        for (int i = 0; i < 4; ++i) face[s][d].sten[i] = sten[i];
        for (int i = 0; i < 8; ++i) face[s][d].tg[i] = tg[i];
      }
    for (int s = 0; s < NMS; ++s)
      for (int d = 0; d < 3; ++d) {
        // fields 3 (d + 1) % 3 and 3 (d + 2) % 3 of L, L + tangent, R, R + tangent
        const int M0 = s * 10 * MS, M1 = (s + 1) % NMS * 10 * MS, mzp = M1 - M0, st = d == 0 ? 1 : BX;
        const int mL = d == 2 ? M0 : M0 - st, mR = d == 2 ? M1 : M0;
        const int u1 = d == 0 ? BX : (d == 1 ? mzp : 1), u2 = d == 0 ? mzp : (d == 1 ? 1 : BX);
        const int f1 = 3 * ((d + 1) % 3) * MS, f2 = 3 * ((d + 2) % 3) * MS;
        MetOff& m = met[s][d];
        m.sf = mR + 3 * d * MS;
        const int t1[4] = {mL + f1, mL + u1 + f1, mR + f1, mR + u1 + f1};
        const int t2[4] = {mL + f2, mL + u2 + f2, mR + f2, mR + u2 + f2};
        for (int i = 0; i < 4; ++i) {
          m.t1[i] = t1[i];
          m.t2[i] = t2[i];
        }
        m.vl = mL + 9 * MS;
        m.vr = mR + 9 * MS;
      }
  }
};
template <int NV, int BY>
__constant__ const FaceTab<NV, BY> face_tab{};

__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// named barriers between the warps that update and those that take the rates (stage 3)
__device__ __forceinline__ void named_arrive(int id, int n) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ void named_sync(int id, int n) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// 16 warps of 128 registers, one CTA per SM
template <bool VISC, int STAGE, int TYV>
__global__ void __launch_bounds__(512, 1) cstage_kernel(const GroupParams P) {
  constexpr bool LOADD = STAGE == 2 || STAGE == 3;
  using T = float;
  using PL = CPlan<VISC, TYV>;
  constexpr int TY = TYV, BY = PL::BY, NW = PL::NW, NT = 32 * NW, NITEM = 3 * TY + 2;
  constexpr int NST = PL::NST, NMS = PL::NMS, NV = PL::NV;
  constexpr int MS = BY * BX;
  // of the warps with one face item, WU update two rows each and the last WC convert
  constexpr int W1 = NITEM - NW, WU = TY / 2, WC = NW - W1 - WU;
  static_assert(TY % 2 == 0 && W1 >= TY && WC > 0, "two items and two rows a warp at most; rates by warps with two items");
  using Fm = VM<T>;

  extern __shared__ __align__(128) unsigned char smem[];
  T* ring = reinterpret_cast<T*>(smem + PL::ring);
  T* fxb = reinterpret_cast<T*>(smem + PL::fx);
  T* fyb = reinterpret_cast<T*>(smem + PL::fy);
  T* fzb = reinterpret_cast<T*>(smem + PL::fz);
  T* mring = reinterpret_cast<T*>(smem + PL::mring);
  double* red = reinterpret_cast<double*>(smem + PL::red);
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + PL::bar);
  int* slast = reinterpret_cast<int*>(smem + PL::misc);

  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // uniform: the stencil's offsets stay scalar
  const Physics& ph = P.ph;
  const PathK<T>& PK = path_k<T>(P);
  Consts<T> K;
  K.gm1 = PK.gm1;
  K.ggm1 = PK.ggm1;
  K.eps = PK.eps;
  K.mu = VISC ? PK.mu : T(0);
  K.kappa = VISC ? PK.kappa : T(0);
  K.lim = ph.limiter;
  const T gm1 = PK.gm1;
  const RateK<T> RK = {PK.gam, PK.vf};
  const T cflT = PK.cfl;

  if (tid == 0) {
    for (int s = 0; s < NST + NMS; ++s) mbar_init(&bar[s], 1);
    fence_barrier_init();
  }
  __syncthreads();

  const T dtT = STAGE == 0 ? T(0) : T(P.gctrl->dt);
  unsigned phase_bits = 0, mphase = 0;  // parity of each staging and metric slot (uniform across the CTA)
  unsigned pending = 0, mpending = 0;   // slots with a copy in flight (meaningful in thread 0)
  bool bad = false;                     // non-physical value met by this thread
  bool fail = false;                    // a copy did not arrive (uniform across the CTA)
  double nacc[5] = {0, 0, 0, 0, 0};     // FP64 sums of R^2 (stage 1)
  T rate_max = T(0);                    // stage 3

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
  const int lcta = (int)blockIdx.x - D->cta0, nctas = D->ctas;
  const long long W = D->units;
  const long long u_begin = (long long)lcta * W / nctas;
  const long long u_end = (long long)(lcta + 1) * W / nctas;
  constexpr unsigned QBYTES = 5u * MS * sizeof(T);

  auto rslot = [](int kp) { return (kp + 2) % PL::NR; };  // ring slot of plane kp (kp >= -2)
  auto sslot = [](int kp) { return (kp + 2) & (NST - 1); };
  auto mslot = [](int kp) { return (kp + 1) & (NMS - 1); };
  const Geometry g = D->g;

  // arrays of this stage
  const int cur = P.cur;
  const CUtensorMap* tmq = &D->tq[cur];
  const CUtensorMap* tmd = &D->td[STAGE == 3 ? 1 : 0];
  const double* qn = D->q[cur];
  const float* dprev = STAGE == 2 ? D->d[0] : (STAGE == 3 ? D->d[1] : nullptr);
  float* dout = STAGE == 1 ? D->d[0] : (STAGE == 2 ? D->d[1] : nullptr);
  double* qout = STAGE == 3 ? D->q[1 - cur] : nullptr;
  float* sout = STAGE == 3 ? D->sh[1 - cur] : nullptr;

  for (long long u = u_begin; u < u_end && !fail;) {
    const int nz = g.nz;
    const long long tile = u / nz;
    const int k0 = (int)(u - tile * nz);
    const int k1 = (int)min((long long)nz, (long long)k0 + (u_end - u));
    u += k1 - k0;
    const int tix = (int)(tile % D->ntx), tiy = (int)(tile / D->ntx);
    const int x0 = tix * TX, y0 = tiy * TY;  // storage coordinates of the box origin
    const int last_plane = k1 + 1;
    auto request = [&](int kp) {  // thread 0 only
      if (kp > last_plane) return;
      const int s = sslot(kp);
      mbar_expect_tx(&bar[s], QBYTES + (LOADD ? QBYTES : 0u));
      tma_load_4d(smem + PL::stq + s * PL::SLOT, tmq, &bar[s], x0, y0, kp + HALO, 0);
      if (LOADD) tma_load_4d(smem + PL::std_ + s * PL::SLOT, tmd, &bar[s], x0, y0, kp + HALO, 0);
      pending |= 1u << s;
    };
    auto mrequest = [&](int kp) {  // thread 0 only
      if (kp > k1) return;
      const int s = mslot(kp);
      mbar_expect_tx(&bar[NST + s], 10u * MS * sizeof(T));
      tma_load_4d(smem + PL::mring + s * PL::MSLOT, &D->tm, &bar[NST + s], x0, y0, kp + HALO, 0);
      mpending |= 1u << s;
    };
    // wait for plane kp and convert it, cells first, first + step, ... of the box, into its ring slot
    auto convert = [&](int kp, int first, int step) -> bool {
      const int s = sslot(kp);
      const bool ok = mbar_wait_bounded(&bar[s], (phase_bits >> s) & 1u);
      const T* sq = reinterpret_cast<const T*>(smem + PL::stq + s * PL::SLOT);
      const T* sd = reinterpret_cast<const T*>(smem + PL::std_ + s * PL::SLOT);
      T* rs = ring + (size_t)rslot(kp) * NV * MS;
      for (int c = first; c < MS; c += step) {
        const int cy = c / BX, cx = c - cy * BX;
        T q[5];
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          if constexpr (LOADD) q[v] = sq[v * MS + c] + sd[v * MS + c];
          else q[v] = sq[v * MS + c];
        }
        const bool valid = (x0 - HALO + cx < g.nx + HALO) && (y0 - HALO + cy < g.ny + HALO);
        T r = q[0];
        const T ir = Fm::rcp(r);
        const T uu = q[1] * ir, vv = q[2] * ir, ww = q[3] * ir;
        T p = gm1 * (q[4] - T(0.5) * r * (uu * uu + vv * vv + ww * ww));
        if (valid && !(r > T(0) && p > T(0))) bad = true;
        const bool fill = !valid || !(r > T(0) && p > T(0));
        rs[0 * MS + c] = fill ? T(1) : r;
        rs[1 * MS + c] = fill ? T(0) : uu;
        rs[2 * MS + c] = fill ? T(0) : vv;
        rs[3 * MS + c] = fill ? T(0) : ww;
        rs[4 * MS + c] = fill ? T(1) : p;
        if (VISC) rs[5 * MS + c] = fill ? T(1) : p * ir;
      }
      return ok;
    };
    // after a barrier behind which plane kp was converted: its slot is free for plane kp + NST
    auto converted = [&](int kp) {
      const unsigned b = 1u << sslot(kp);
      phase_bits ^= b;
      if (tid == 0) {
        pending &= ~b;
        fence_proxy_async();
        request(kp + NST);
      }
    };
    auto mwait = [&](int kp) -> bool { return mbar_wait_bounded(&bar[NST + mslot(kp)], (mphase >> mslot(kp)) & 1u); };
    auto mwaited = [&](int kp) {
      mphase ^= 1u << mslot(kp);
      mpending &= ~(1u << mslot(kp));
    };

    if (tid == 0) {
      tensormap_acquire(tmq);
      if (LOADD) tensormap_acquire(tmd);
      tensormap_acquire(&D->tm);
      fence_proxy_async();
      for (int kp = k0 - 2; kp <= k0 + 1; ++kp) request(kp);
      for (int kp = k0 - 1; kp <= k0 + 2; ++kp) mrequest(kp);
    }
    {
      bool ok = true;
      for (int kp = k0 - 2; kp <= k0 + 1; ++kp) ok = convert(kp, tid, NT) && ok;
      ok = mwait(k0 - 1) && ok;
      fail = __syncthreads_or(!ok);
      if (fail) break;
      for (int kp = k0 - 2; kp <= k0 + 1; ++kp) converted(kp);
      mwaited(k0 - 1);
    }

    // the update of rows row[0..1] of plane k, one cell of each a lane, side by side: a warp alone would
    // wait for most of its operations
    auto update = [&](int k, const int (&row)[2]) {
      const int ci = x0 + lane, ocx = lane + HALO, mk = mslot(k), mk1 = mslot(k + 1);
      bool live[2];
      long long o[2], of[2];
      double qo[2][5];
      float dp[2][5];
      T dtc[2];  // each cell's time step (its own one under local time stepping)
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int cj = y0 + row[i];  // interior coordinates
        live[i] = ci < g.nx && cj < g.ny;
        o[i] = gidx(g, ci, cj, k);
        of[i] = gidxf(g, ci, cj, k);
        dtc[i] = dtT;
        if constexpr (STAGE >= 1 && !VISC)  // local time steps: inviscid blocks only
          if (ph.local_dt && live[i]) dtc[i] = __ldg(static_cast<const T*>(D->dtl) + of[i]);
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          if constexpr (STAGE == 3) qo[i][v] = live[i] ? __ldg(qn + v * g.field + o[i]) : 1.0;
          if constexpr (LOADD) dp[i][v] = live[i] ? __ldg(dprev + v * g.fieldf + of[i]) : 0.0f;
        }
      }
      T R[2][5];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const T* fx = fxb + (k & 1) * PL::FX + row[i] * (TX + 1) + lane;
        const T* fy = fyb + (k & 1) * PL::FY + row[i] * TX + lane;
        const T* fzl = fzb + ((k + 3) % 3) * PL::FZ + row[i] * TX + lane;
        const T* fzu = fzb + ((k + 1) % 3) * PL::FZ + row[i] * TX + lane;
#pragma unroll
        for (int m = 0; m < 5; ++m) {
          const T ddx = fx[m * TY * (TX + 1) + 1] - fx[m * TY * (TX + 1)];
          const T ddy = fy[(m * (TY + 1) + 1) * TX] - fy[m * (TY + 1) * TX];
          R[i][m] = (ddx + ddy) + (fzu[m * TY * TX] - fzl[m * TY * TX]);  // face fluxes carry |S|; divided by V below
        }
        const T iv = Fm::rcp(mring[mb<BY>(mk, row[i] + HALO, ocx) + 9 * MS]);
#pragma unroll
        for (int m = 0; m < 5; ++m) R[i][m] = R[i][m] * iv;
      }
      if constexpr (STAGE == 0) {
        const long long n = (long long)g.nx * g.ny * g.nz;
#pragma unroll
        for (int i = 0; i < 2; ++i)
          if (live[i]) {
            const long long oc = ((long long)k * g.ny + y0 + row[i]) * g.nx + ci;
#pragma unroll
            for (int m = 0; m < 5; ++m) P.rout[m * n + oc] = double(R[i][m]);
          }
      } else {
        float inc[2][5];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int m = 0; m < 5; ++m) inc[i][m] = -dtc[i] * R[i][m];
        if constexpr (STAGE == 1 || STAGE == 2) {
#pragma unroll
          for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int m = 0; m < 5; ++m) {
              const float d = STAGE == 1 ? inc[i][m] : 0.25f * (dp[i][m] + inc[i][m]);
              if (live[i]) dout[m * g.fieldf + of[i]] = d;
            }
        } else {
          // a row's x-fluxes were read by this warp alone: their place takes its new state
          __syncwarp();
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            float qf[5];
            double dd[5];
#pragma unroll
            for (int m = 0; m < 5; ++m) {
              // (hardware conversions: the FP64 pipe has room, the issue slots do not)
              const float d = (2.0f / 3.0f) * (dp[i][m] + inc[i][m]);
              dd[m] = qo[i][m] + double(d);
              qf[m] = float(dd[m]);
            }
#pragma unroll
            for (int m = 0; m < 5; ++m) {
              if (live[i]) {
                qout[m * g.field + o[i]] = dd[m];
                sout[m * g.fieldf + of[i]] = qf[m];
              }
              fxb[(k & 1) * PL::FX + (m * TY + row[i]) * (TX + 1) + lane] = qf[m];
            }
          }
          named_arrive(1, 32 * (WU + TY));
        }
      }
      if constexpr (STAGE == 1) {
        // the residual norm is reduced in FP64: an FP32 residual's square is exact in FP64, so the sums
        // round only in the additions; it is widened on the integer pipe, one FP64 operation a variable
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int m = 0; m < 5; ++m) {
            const double r = f32_to_f64_bits(live[i] ? R[i][m] : 0.0f);
            nacc[m] = fma(r, r, nacc[m]);
          }
      }
    };

    // stage 3: the time-step rate of row `row` of plane k, from the state its update left in shared memory
    auto rate_row = [&](int k, int row) {
      const int ci = x0 + lane, cj = y0 + row, ocy = row + HALO, ocx = lane + HALO, mk = mslot(k), mk1 = mslot(k + 1);
      named_sync(1, 32 * (WU + TY));
      if (ci >= g.nx || cj >= g.ny) return;
      const T* qs = fxb + (k & 1) * PL::FX + row * (TX + 1) + lane;
      float qf[5];
#pragma unroll
      for (int m = 0; m < 5; ++m) qf[m] = qs[m * TY * (TX + 1)];
      const float ir = VM<float>::rcp(qf[0]);
      const float uu = qf[1] * ir, vv = qf[2] * ir, ww = qf[3] * ir;
      const float pp = gm1 * (qf[4] - 0.5f * qf[0] * (uu * uu + vv * vv + ww * ww));
      if (!(qf[0] > 0.0f && pp > 0.0f)) bad = true;
      T sb[9];
      cell_face_means<T, BY>(mring, mk, mk1, ocy, ocx, sb);
      const float rate =
          cell_rate_curvi<float>(qf[0], uu, vv, ww, pp, sb, mring[mb<BY>(mk, ocy, ocx) + 9 * MS], RK, ph.viscous);
      rate_max = fmax(rate_max, T(rate));
      if constexpr (!VISC)
        if (ph.local_dt) static_cast<float*>(D->dtl)[gidxf(g, ci, cj, k)] = cflT / rate;
    };

    // phase k: the faces of plane k (plane k0 - 1: its upper z-faces only), the update of plane k - 1 and
    // the conversion of plane k + 3
    for (int k = k0 - 1; k <= k1; ++k) {
      bool ok = true;
      if (warp >= W1 && warp < W1 + WU) {
        const int rows[2] = {warp - W1, warp - W1 + WU};
        if (k > k0) update(k - 1, rows);
      } else if (warp >= W1 + WU && k + 3 <= last_plane) {
        ok = convert(k + 3, tid - 32 * (W1 + WU), 32 * WC);
      }
      // what stage 3's update of plane k reads (60 bytes a cell): into L2 a phase ahead
      if (STAGE == 3 && warp >= W1 + WU && k >= k0 && k < k1)
#pragma unroll 1
        for (int row = warp - (W1 + WU); row < TY && y0 + row < g.ny; row += WC) {
          const int v = lane / 3, c = min(x0 + 16 * (lane % 3), g.nx - 1), cf = min(x0 + 31 * (lane % 3), g.nx - 1);
          if (lane < 15) prefetch_l2(qn + v * g.field + gidx(g, c, y0 + row, k));
          if (lane < 15 && lane % 3 < 2) prefetch_l2(dprev + v * g.fieldf + gidxf(g, cf, y0 + row, k));
        }
      if (k < k1) ok = mwait(k + 1) && ok;
      const int sk = rslot(k), mk = mslot(k);
      const int nitem = k == k1 ? 0 : (k < k0 ? TY : NITEM);
#pragma unroll 1
      for (int it = warp; it < nitem; it += NW) {
        const int d = it < TY ? 2 : (it < 2 * TY + 1 ? 1 : 0);
        const int fr = it < TY ? it : (it < 2 * TY + 1 ? it - TY : it - (2 * TY + 1));  // row; TY: the upper side
        // faces of cells of the block only (y and x: up to the upper face of its last cells)
        const bool side = d == 0 && fr == TY;
        const int ty = side ? lane : fr, tx = side ? TX : lane;
        if (side ? lane >= TY || x0 + TX > g.nx || y0 + lane >= g.ny : y0 + fr >= g.ny + (d == 1 ? 1 : 0)) continue;
        const int cell = (ty + HALO) * BX + tx + HALO;  // this lane's cell of the box
        const FaceOff& fo = face_tab<NV, BY>.face[sk][d];
        T F[5];
        face_flux_curvi<T, VISC, BY>(ring + cell, mring + cell, NV * MS, fo.sten, fo.tg, face_tab<NV, BY>.met[mk][d], K, F);
        T* out = d == 2 ? fzb + ((k + 1) % 3) * PL::FZ + ty * TX + tx
                        : (d == 1 ? fyb + (k & 1) * PL::FY + ty * TX + tx : fxb + (k & 1) * PL::FX + ty * (TX + 1) + tx);
        const int fs = d == 2 ? TY * TX : (d == 1 ? (TY + 1) * TX : TY * (TX + 1));
#pragma unroll
        for (int m = 0; m < 5; ++m) out[m * fs] = F[m];
      }
      if (STAGE == 3 && warp < TY && k > k0) rate_row(k - 1, warp);
      fail = __syncthreads_or(!ok);
      if (fail) break;
      if (k + 3 <= last_plane) converted(k + 3);
      if (k < k1) mwaited(k + 1);
      if (tid == 0 && k >= k0) {  // phase k was the last to read the metrics of plane k - 1
        fence_proxy_async();
        mrequest(k + 3);
      }
    }
  }

  // abort path: wait (bounded) for the copies still in flight, flag the timeout
  if (fail && tid == 0) {
    for (int s = 0; s < NST; ++s)
      if (pending & (1u << s)) mbar_wait_bounded(&bar[s], (phase_bits >> s) & 1u);
    for (int s = 0; s < NMS; ++s)
      if (mpending & (1u << s)) mbar_wait_bounded(&bar[NST + s], (mphase >> s) & 1u);
    atomicOr(&D->ctrl->flag, FLAG_TIMEOUT);
  }
  if (bad) atomicOr(&D->ctrl->flag, FLAG_NONPHYSICAL);

  if constexpr (STAGE == 1 || STAGE == 3)
    stage_reduce<STAGE, NW>(P, reinterpret_cast<double*>(smem + PL::ring), red, slast, nacc, double(rate_max));
}

// ---- launch helpers --------------------------------------------------------------------------
template <bool VISC, int STAGE, int TYV>
cudaError_t cstage_attr() {
  static std::atomic<unsigned long long> done{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 64 && ((done.load(std::memory_order_acquire) >> dev) & 1ull)) return cudaSuccess;
  e = cudaFuncSetAttribute(cstage_kernel<VISC, STAGE, TYV>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)CPlan<VISC, TYV>::bytes);
  if (e == cudaSuccess && dev < 64) done.fetch_or(1ull << dev, std::memory_order_acq_rel);
  return e;
}
template <bool VISC, int STAGE, int TYV>
cudaError_t cstage_go(const GroupParams& P, int grid, cudaStream_t s) {
  cudaError_t e = cstage_attr<VISC, STAGE, TYV>();
  if (e != cudaSuccess) return e;
  cstage_kernel<VISC, STAGE, TYV><<<grid, 512, CPlan<VISC, TYV>::bytes, s>>>(P);
  return cudaGetLastError();
}
template <bool VISC, int TYV>
cudaError_t cstage_prepare() {
  cudaError_t e = cstage_attr<VISC, 0, TYV>();
  if (e == cudaSuccess) e = cstage_attr<VISC, 1, TYV>();
  if (e == cudaSuccess) e = cstage_attr<VISC, 2, TYV>();
  if (e == cudaSuccess) e = cstage_attr<VISC, 3, TYV>();
  return e;
}
template <bool VISC, int TYV>
cudaError_t cstage_dispatch(int stage, const GroupParams& P, int grid, cudaStream_t s) {
  switch (stage) {
    case 0: return cstage_go<VISC, 0, TYV>(P, grid, s);
    case 1: return cstage_go<VISC, 1, TYV>(P, grid, s);
    case 2: return cstage_go<VISC, 2, TYV>(P, grid, s);
    case 3: return cstage_go<VISC, 3, TYV>(P, grid, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace gbcfd
