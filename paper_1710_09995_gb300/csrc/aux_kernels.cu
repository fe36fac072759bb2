// aux_kernels.cu -- halo exchange, state scatter/gather and time-step kernels.
#include <algorithm>

#include "launch.h"
#include "vmath.cuh"

namespace gbcfd {

// ---- halo exchange -------------------------------------------------------------------------
// One thread per halo cell of every block in the group.  The source of a halo cell is found by
// walking face neighbours: first along x, then along y in the block reached, then along z, so
// that edge and corner cells come from the diagonal neighbour.  A direction without a neighbour
// (a physical boundary) is skipped and its index stays outside: an edge cell next to a boundary
// face then copies the neighbour's boundary ghost, and a cell of the boundary face slab itself
// (no move at all) is left to the boundary kernel.  Each block's halo is the union of the
// z-slabs (k < 0 or k >= nz, all i, j), the y-slabs (0 <= k < nz, j outside, all i) and the
// x-slabs (inside k and j, i outside).
// Bound by latency: a few cells a thread, so what counts is the chain from the cell's number to its
// stores.  I: 32-bit unsigned wherever the cells' number allows (a 64-bit division is a subroutine of a
// hundred instructions, and there are six), and five variables are loaded before one is stored.
// Measured (one block, channel of 192 x 96 x 16): 7.5 -> 5.8 us.
template <typename T>
__device__ __forceinline__ void halo_copy(char* dst, const char* src, long long dfield, long long sfield, long long dof,
                                          long long sof, int nvar) {
  T* d = reinterpret_cast<T*>(dst) + dof;
  const T* s = reinterpret_cast<const T*>(src) + sof;
  for (int v0 = 0; v0 < nvar; v0 += 5) {
    T x[5];
#pragma unroll
    for (int v = 0; v < 5; ++v)
      if (v0 + v < nvar) x[v] = s[(v0 + v) * sfield];
#pragma unroll
    for (int v = 0; v < 5; ++v)
      if (v0 + v < nvar) d[(v0 + v) * dfield] = x[v];
  }
}
template <typename I>
__global__ void halo_kernel(const __grid_constant__ HaloGroup G) {
  const I stride = (I)gridDim.x * blockDim.x;
  for (I t = (I)blockIdx.x * blockDim.x + threadIdx.x; t < (I)G.total; t += stride) {
    int lo = 0, hi = G.n - 1;
    while (lo < hi) {  // last block whose prefix start <= t
      const int mid = (lo + hi + 1) >> 1;
      if (G.b[mid].first <= (long long)t) lo = mid; else hi = mid - 1;
    }
    const HaloBlock& B = G.b[lo];
    I h = t - (I)B.first;
    const int nx = B.nx, ny = B.ny, nz = B.nz;
    const I wx = nx + 2 * HALO, wy = ny + 2 * HALO;
    int i, j, k;
    const I zc = 2 * HALO * wx * wy, yc = (I)nz * (2 * HALO) * wx;
    if (h < zc) {
      const int kk = (int)(h / (wx * wy));
      const I r = h - kk * (wx * wy);
      k = kk < HALO ? kk - HALO : nz + kk - HALO;
      j = (int)(r / wx) - HALO;
      i = (int)(r % wx) - HALO;
    } else if ((h -= zc) < yc) {
      k = (int)(h / (2 * HALO * wx));
      const I r = h - k * (2 * HALO * wx);
      const int jj = (int)(r / wx);
      j = jj < HALO ? jj - HALO : ny + jj - HALO;
      i = (int)(r % wx) - HALO;
    } else {
      h -= yc;
      k = (int)(h / ((I)ny * (2 * HALO)));
      const I r = h - k * ((I)ny * (2 * HALO));
      j = (int)(r / (2 * HALO));
      const int ii = (int)(r % (2 * HALO));
      i = ii < HALO ? ii - HALO : nx + ii - HALO;
    }
    // walk to the source block (a missing neighbour leaves that index outside)
    int b = lo, si = i, sj = j, sk = k;
    bool moved = false;
    while (si < 0 && G.b[b].nbr[0] >= 0) { b = G.b[b].nbr[0]; si += G.b[b].nx; moved = true; }
    while (si >= G.b[b].nx && G.b[b].nbr[1] >= 0) { si -= G.b[b].nx; b = G.b[b].nbr[1]; moved = true; }
    while (sj < 0 && G.b[b].nbr[2] >= 0) { b = G.b[b].nbr[2]; sj += G.b[b].ny; moved = true; }
    while (sj >= G.b[b].ny && G.b[b].nbr[3] >= 0) { sj -= G.b[b].ny; b = G.b[b].nbr[3]; moved = true; }
    while (sk < 0 && G.b[b].nbr[4] >= 0) { b = G.b[b].nbr[4]; sk += G.b[b].nz; moved = true; }
    while (sk >= G.b[b].nz && G.b[b].nbr[5] >= 0) { sk -= G.b[b].nz; b = G.b[b].nbr[5]; moved = true; }
    // a source left outside a smaller neighbour's halo (only with blocks narrower than the halo)
    if (!moved || si < -HALO || si >= G.b[b].nx + HALO || sj < -HALO || sj >= G.b[b].ny + HALO ||
        sk < -HALO || sk >= G.b[b].nz + HALO)
      continue;
    const HaloBlock& S = G.b[b];
    const long long dplane = (long long)(ny + 2 * HALO) * B.pitch, dfield = dplane * (nz + 2 * HALO);
    const long long splane = (long long)(S.ny + 2 * HALO) * S.pitch, sfield = splane * (S.nz + 2 * HALO);
    const long long dof = (k + HALO) * dplane + (long long)(j + HALO) * B.pitch + (i + HALO);
    const long long sof = (sk + HALO) * splane + (long long)(sj + HALO) * S.pitch + (si + HALO);
    if (G.elem == 8) halo_copy<double>(B.base[0], S.base[0], dfield, sfield, dof, sof, G.nvar);
    else halo_copy<float>(B.base[0], S.base[0], dfield, sfield, dof, sof, G.nvar);
  }
}

cudaError_t launch_halo(const HaloGroup& G, cudaStream_t s) {
  if (G.total <= 0) return cudaSuccess;
  const int threads = 256;
  long long blocks = (G.total + threads - 1) / threads;
  if (blocks > 65535LL * 8) blocks = 65535LL * 8;
  // (32-bit numbers: the last stride may pass the total)
  if (G.total < (1LL << 30)) halo_kernel<unsigned><<<(unsigned)blocks, threads, 0, s>>>(G);
  else halo_kernel<unsigned long long><<<(unsigned)blocks, threads, 0, s>>>(G);
  return cudaGetLastError();
}

// ---- compact <-> padded state --------------------------------------------------------------
// shadow (may be null): the f32 rounding of the state, written alongside
// A CTA per row (v, k, j) of nx values: src is compact [5][nz][ny][nx] (device memory, or pinned
// host memory read over the host link), dst the padded f64 field; the mixed path's f32 shadow is
// rounded on the integer pipe (bitwise the hardware rounding, see vmath.cuh).
__global__ void scatter_kernel(Geometry g, const double* __restrict__ src, double* __restrict__ dst,
                               float* __restrict__ shadow) {
  const int rows = 5 * g.ny * g.nz;
  for (int row = blockIdx.x; row < rows; row += gridDim.x) {
    const int j = row % g.ny, r = row / g.ny, k = r % g.nz, v = r / g.nz;
    const double* s = src + (long long)row * g.nx;
    double* d = dst + v * g.field + gidx(g, 0, j, k);
    float* sh = shadow ? shadow + v * g.fieldf + gidxf(g, 0, j, k) : nullptr;
    for (int i = threadIdx.x; i < g.nx; i += blockDim.x) {
      const double x = s[i];
      d[i] = x;
      if (sh) sh[i] = f64_to_f32_bits(x);
    }
  }
}
// the reverse: padded f64 field -> compact [5][nz][ny][nx] (device memory or pinned host memory)
__global__ void gather_kernel(Geometry g, const double* __restrict__ src, double* __restrict__ dst) {
  const int rows = 5 * g.ny * g.nz;
  for (int row = blockIdx.x; row < rows; row += gridDim.x) {
    const int j = row % g.ny, r = row / g.ny, k = r % g.nz, v = r / g.nz;
    const double* s = src + v * g.field + gidx(g, 0, j, k);
    double* d = dst + (long long)row * g.nx;
    for (int i = threadIdx.x; i < g.nx; i += blockDim.x) d[i] = s[i];
  }
}
static unsigned grid_for(long long work, int threads) {
  long long b = (work + threads - 1) / threads;
  if (b > 65535LL * 16) b = 65535LL * 16;
  if (b < 1) b = 1;
  return (unsigned)b;
}
static unsigned row_grid(const Geometry& g) {
  const long long rows = 5LL * g.ny * g.nz;
  return (unsigned)std::min(rows, 65535LL * 16);
}
static int row_threads(const Geometry& g) { return g.nx >= 256 ? 256 : (g.nx >= 128 ? 128 : 64); }
cudaError_t launch_scatter(const Geometry& g, const double* src, double* dst, float* shadow, cudaStream_t s) {
  scatter_kernel<<<row_grid(g), row_threads(g), 0, s>>>(g, src, dst, shadow);
  return cudaGetLastError();
}
cudaError_t launch_gather(const Geometry& g, const double* src, double* dst, cudaStream_t s) {
  gather_kernel<<<row_grid(g), row_threads(g), 0, s>>>(g, src, dst);
  return cudaGetLastError();
}

// ---- time step -----------------------------------------------------------------------------
// rate = sum over directions of (|u_d| + c) / h_d (+ 4 max(4/3, gamma/Pr) mu / rho / h_d^2 when
// viscous); the CFL step is cfl / max(rate).  From the padded f64 state, in the path's flux
// precision T (the mixed path's time step is an f32 evaluation, like its fluxes).
// A warp takes a row of cells, or 2, 4 or 8 rows of at most 16, 8 or 4 (with a warp a row 28 lanes idled on blocks 4
// cells wide: setting the state of 4 x 512 x 512 cells took 750 us, now 574, against 663 with a thread a cell).  FP64 blocks
// evaluate it on the integer pipes (xfix.cuh).  The maxima are
// compared as bit patterns and the CTAs' folded by a warp of the last CTA: one thread walking all
// partial rows took most of the 60 us this pass cost a 32^3 block.
constexpr int RATE_THREADS = 256;
// log2 of the threads a row takes
__device__ __forceinline__ int row_shift(int nx) { return nx > 16 ? 5 : (nx > 8 ? 4 : (nx > 4 ? 3 : 2)); }
__device__ __forceinline__ void rate_fold(long long best, DevCtrl* ctrl, double* partial, double cfl) {
  __shared__ long long wmax[RATE_THREADS / 32];
  __shared__ int last;
  const int lane = threadIdx.x & 31;
  best = warp_max_bits(best);
  if (lane == 0) wmax[threadIdx.x >> 5] = best;
  __syncthreads();
  if (threadIdx.x < 32) {
    const long long m = warp_max_bits(lane < RATE_THREADS / 32 ? wmax[lane] : 0ll);
    if (lane == 0) {
      partial[(size_t)blockIdx.x * NPART + 5] = __longlong_as_double(m);
      __threadfence();
      last = (atomicAdd(&ctrl->counter, 1u) == gridDim.x - 1);
    }
  }
  __syncthreads();
  if (!last || threadIdx.x >= 32) return;
  __threadfence();
  long long m = 0;
#pragma unroll 4
  for (unsigned b = lane; b < gridDim.x; b += 32) {
    const long long v = __double_as_longlong(__ldcg(partial + (size_t)b * NPART + 5));
    m = v > m ? v : m;
  }
  m = warp_max_bits(m);
  if (lane == 0) {
    const double r = __longlong_as_double(m);
    ctrl->rate = r;
    ctrl->dt = cfl / r;
    ctrl->counter = 0u;
  }
}

// the mixed path's constants, formed on the host
struct RateConsts {
  float gam, gm1, f, mu4, fmu4, ihx, ihy, ihz, s2, cfl;
};
static RateConsts rate_consts(const Physics& ph) {
  const double f = std::max(4.0 / 3.0, ph.gamma / ph.Pr);
  return {float(ph.gamma), float(ph.gamma - 1.0), float(f), float(4.0 * ph.mu), float(4.0 * f * ph.mu), float(ph.ihx),
          float(ph.ihy), float(ph.ihz), float(ph.ihx * ph.ihx + ph.ihy * ph.ihy + ph.ihz * ph.ihz), float(ph.cfl)};
}

__global__ void __launch_bounds__(RATE_THREADS) init_rate_kernel(Geometry g, int viscous, RateConsts C, double cfl,
                                                                  const double* __restrict__ q, DevCtrl* ctrl,
                                                                  double* partial, float* dtl) {
  float best = 0.f;
  bool bad = false;
  const int rows = g.ny * g.nz, sh = row_shift(g.nx), per = RATE_THREADS >> sh;
  for (int row = blockIdx.x * per + (threadIdx.x >> sh); row < rows; row += gridDim.x * per) {
    const int j = row % g.ny, k = row / g.ny;
    for (int i = threadIdx.x & ((1 << sh) - 1); i < g.nx; i += 1 << sh) {
      const long long o = gidx(g, i, j, k);
      const float rho = float(q[o]), ir = 1.f / rho;
      const float u = float(q[g.field + o]) * ir, v = float(q[2 * g.field + o]) * ir, w = float(q[3 * g.field + o]) * ir;
      const float p = C.gm1 * (float(q[4 * g.field + o]) - 0.5f * rho * (u * u + v * v + w * w));
      const float a = sqrtf(C.gam * p * ir);
      float rate = (fabsf(u) + a) * C.ihx + (fabsf(v) + a) * C.ihy + (fabsf(w) + a) * C.ihz;
      if (viscous) rate += C.f * C.mu4 * ir * C.s2;
      if (dtl) dtl[gidxf(g, i, j, k)] = C.cfl / rate;
      if (!(rho > 0.f && p > 0.f)) bad = true;
      best = rate > best ? rate : best;
    }
  }
  if (bad) atomicOr(&ctrl->flag, FLAG_NONPHYSICAL);
  rate_fold(__double_as_longlong(double(best)), ctrl, partial, cfl);
}

// FP64: M = null on uniform grids, else the metric fields
template <bool VISC, bool CURVI>
__global__ void __launch_bounds__(RATE_THREADS) init_rate_x_kernel(Geometry g, Physics ph, XConsts K,
                                                                    const double* __restrict__ q,
                                                                    const double* __restrict__ M, DevCtrl* ctrl,
                                                                    double* partial, double* dtl) {
  __shared__ XVal h2[3], hsum, vs;  // vs: 4 max(4/3, gamma/Pr) mu (uniform: times the sum of 1 / h^2)
  if (threadIdx.x < 3) h2[threadIdx.x] = xdec_pos<62>(0.5 * (threadIdx.x == 0 ? ph.ihx : (threadIdx.x == 1 ? ph.ihy : ph.ihz)));
  if (threadIdx.x == 32) {
    hsum = xdec_pos<62>(ph.ihx + ph.ihy + ph.ihz);
    const double f = 4.0 * fmax(4.0 / 3.0, ph.gamma / ph.Pr) * ph.mu;
    vs = xdec_pos<62>(CURVI ? f : f * (ph.ihx * ph.ihx + ph.ihy * ph.ihy + ph.ihz * ph.ihz));
  }
  __syncthreads();
  long long best = 0;
  bool bad = false;
  const int rows = g.ny * g.nz, sh = row_shift(g.nx), per = RATE_THREADS >> sh;
  for (int row = blockIdx.x * per + (threadIdx.x >> sh); row < rows; row += gridDim.x * per) {
    const int j = row % g.ny, k = row / g.ny;
    for (int i = threadIdx.x & ((1 << sh) - 1); i < g.nx; i += 1 << sh) {
      const long long o = gidx(g, i, j, k);
      const double Q[5] = {q[o], q[g.field + o], q[2 * g.field + o], q[3 * g.field + o], q[4 * g.field + o]};
      XPrim W;
      const bool phys = xprim(Q, K, W);
      if (!phys) bad = true;
      const XVal c = xsound(W, K.gam);
      XVal rate;
      if constexpr (!CURVI) {
        rate = xrate<VISC>(W, c, h2, hsum, vs);
      } else {
        const XVal iv = xrcp(xdec_pos<62>(M[9 * g.field + o]));
        XVal f = {0, 0};
        if (VISC) f = {xmul(xmul(vs.m, W.ir.m) << 2, iv.m) << 2, vs.e + W.ir.e + iv.e + 2};
        const long long up[3] = {1, g.px, g.plane};
        XVal r[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          double lo[3], hi[3];
#pragma unroll
          for (int x = 0; x < 3; ++x) {
            lo[x] = M[(3 * d + x) * g.field + o];
            hi[x] = M[(3 * d + x) * g.field + o + up[d]];
          }
          r[d] = xradius<VISC>(W, c, lo, hi, f);
        }
        const XVal v = xsum3(r[0], r[1], r[2]);
        rate = xnormed(xmul(v.m, iv.m), v.e + iv.e + 3);
      }
      if (dtl) {
        const XVal ir = xrcp(rate);
        dtl[o] = ph.cfl * xenc(ir.m, ir.e);
      }
      const long long rb = __double_as_longlong(xenc(rate.m, rate.e));
      if (phys && rb > best) best = rb;
    }
  }
  if (bad) atomicOr(&ctrl->flag, FLAG_NONPHYSICAL);
  rate_fold(best, ctrl, partial, ph.cfl);
}

cudaError_t launch_init_rate(const Geometry& g, const Physics& ph, const double* q, DevCtrl* ctrl,
                             double* partial, int grid, int mixed, void* dtl, cudaStream_t s) {
  if (mixed)
    init_rate_kernel<<<grid, RATE_THREADS, 0, s>>>(g, ph.viscous, rate_consts(ph), ph.cfl, q, ctrl, partial,
                                                   static_cast<float*>(dtl));
  else if (ph.viscous)
    init_rate_x_kernel<true, false><<<grid, RATE_THREADS, 0, s>>>(g, ph, xconsts(ph.gamma, ph.eps), q, nullptr, ctrl,
                                                                  partial, static_cast<double*>(dtl));
  else
    init_rate_x_kernel<false, false><<<grid, RATE_THREADS, 0, s>>>(g, ph, xconsts(ph.gamma, ph.eps), q, nullptr, ctrl,
                                                                   partial, static_cast<double*>(dtl));
  return cudaGetLastError();
}

// ---- curvilinear metrics -------------------------------------------------------------------
// Per interior cell: the area vectors of its lower xi, eta, zeta faces, S = 1/2 (d1 x d2) over
// the face diagonals, oriented towards +xi, +eta, +zeta, and the volume by the divergence
// theorem, V = 1/3 sum over the six faces of (face centroid - first corner) . outward S.
// nodes: x[3][nz+1][ny+1][nx+1] (f64).  M: 10 padded fields, f64 or f32 (elem bytes).
__device__ __forceinline__ void vsub(const double* a, const double* b, double* c) {
  c[0] = a[0] - b[0]; c[1] = a[1] - b[1]; c[2] = a[2] - b[2];
}
__device__ __forceinline__ void half_cross(const double* a, const double* b, double* c) {
  c[0] = 0.5 * (a[1] * b[2] - a[2] * b[1]);
  c[1] = 0.5 * (a[2] * b[0] - a[0] * b[2]);
  c[2] = 0.5 * (a[0] * b[1] - a[1] * b[0]);
}

// node (i, j, k); indices beyond the block's nodes are extended by reflection through the
// boundary node along the grid line, X(-m) = 2 X(0) - X(m), X(n + m) = 2 X(n) - X(n - m), the
// x index first, then y, then z
__device__ __forceinline__ void node_in(const Geometry& g, const double* X, long long nn, int i, int j, int k,
                                        double* x) {
  const long long o = ((long long)k * (g.ny + 1) + j) * (g.nx + 1) + i;
  x[0] = X[o]; x[1] = X[nn + o]; x[2] = X[2 * nn + o];
}
__device__ __forceinline__ void node_k(const Geometry& g, const double* X, long long nn, int i, int j, int k,
                                       double* x) {
  if (k < 0 || k > g.nz) {
    const int e = k < 0 ? 0 : g.nz;
    double a[3], b[3];
    node_in(g, X, nn, i, j, e, a);
    node_in(g, X, nn, i, j, min(max(2 * e - k, 0), g.nz), b);  // clamp: blocks thinner than 2 cells
    for (int c = 0; c < 3; ++c) x[c] = __dsub_rn(2.0 * a[c], b[c]);
  } else {
    node_in(g, X, nn, i, j, k, x);
  }
}
__device__ __forceinline__ void node_jk(const Geometry& g, const double* X, long long nn, int i, int j, int k,
                                        double* x) {
  if (j < 0 || j > g.ny) {
    const int e = j < 0 ? 0 : g.ny;
    double a[3], b[3];
    node_k(g, X, nn, i, e, k, a);
    node_k(g, X, nn, i, min(max(2 * e - j, 0), g.ny), k, b);
    for (int c = 0; c < 3; ++c) x[c] = __dsub_rn(2.0 * a[c], b[c]);
  } else {
    node_k(g, X, nn, i, j, k, x);
  }
}
__device__ __forceinline__ void node_ext(const Geometry& g, const double* X, long long nn, int i, int j, int k,
                                         double* x) {
  if (i < 0 || i > g.nx) {
    const int e = i < 0 ? 0 : g.nx;
    double a[3], b[3];
    node_jk(g, X, nn, e, j, k, a);
    node_jk(g, X, nn, min(max(2 * e - i, 0), g.nx), j, k, b);
    for (int c = 0; c < 3; ++c) x[c] = __dsub_rn(2.0 * a[c], b[c]);
  } else {
    node_jk(g, X, nn, i, j, k, x);
  }
}

// every padded cell, halo included (halo nodes by reflection; the halo exchange then replaces
// the halo cells of connected faces with the neighbour's)
__global__ void metrics_kernel(Geometry g, const double* __restrict__ X, void* M, int elem) {
  const long long wx = g.nx + 2 * HALO, wy = g.ny + 2 * HALO;
  const long long n = wx * wy * (g.nz + 2 * HALO);
  const long long nn = (long long)(g.nx + 1) * (g.ny + 1) * (g.nz + 1);
  for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < n;
       c += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(c % wx) - HALO;
    const long long r = c / wx;
    const int j = (int)(r % wy) - HALO, k = (int)(r / wy) - HALO;
    double p[8][3];  // corner (di, dj, dk) at index di + 2 dj + 4 dk
    for (int q = 0; q < 8; ++q) node_ext(g, X, nn, i + (q & 1), j + ((q >> 1) & 1), k + (q >> 2), p[q]);
    // quadrilateral a, b, c, d in counter-clockwise order seen from the side S points to:
    // S = 1/2 (c - a) x (d - b)
    auto face = [&](int a, int b, int cc, int d, double* S, double* cen) {
      double d1[3], d2[3];
      vsub(p[cc], p[a], d1);
      vsub(p[d], p[b], d2);
      half_cross(d1, d2, S);
      for (int x = 0; x < 3; ++x) cen[x] = 0.25 * (p[a][x] + p[b][x] + p[cc][x] + p[d][x]) - p[0][x];
    };
    double S[6][3], C[6][3];
    face(0, 2, 6, 4, S[0], C[0]);  // lower xi   (eta, zeta plane at di = 0)
    face(1, 3, 7, 5, S[1], C[1]);  // upper xi
    face(0, 4, 5, 1, S[2], C[2]);  // lower eta  (zeta, xi plane at dj = 0)
    face(2, 6, 7, 3, S[3], C[3]);  // upper eta
    face(0, 1, 3, 2, S[4], C[4]);  // lower zeta (xi, eta plane at dk = 0)
    face(4, 5, 7, 6, S[5], C[5]);  // upper zeta
    double vol = 0.0;
    for (int f = 0; f < 6; ++f) {
      const double sgn = (f & 1) ? 1.0 : -1.0;
      vol += sgn * (C[f][0] * S[f][0] + C[f][1] * S[f][1] + C[f][2] * S[f][2]);
    }
    vol *= 1.0 / 3.0;
    const double out[10] = {S[0][0], S[0][1], S[0][2], S[2][0], S[2][1], S[2][2],
                            S[4][0], S[4][1], S[4][2], vol};
    if (elem == 8) {
      double* m = static_cast<double*>(M);
      const long long o = gidx(g, i, j, k);
      for (int v = 0; v < 10; ++v) m[v * g.field + o] = out[v];
    } else {
      float* m = static_cast<float*>(M);
      const long long o = gidxf(g, i, j, k);
      for (int v = 0; v < 10; ++v) m[v * g.fieldf + o] = float(out[v]);
    }
  }
}

cudaError_t launch_metrics(const Geometry& g, const double* nodes, void* M, int elem, cudaStream_t s) {
  const long long n = (long long)(g.nx + 2 * HALO) * (g.ny + 2 * HALO) * (g.nz + 2 * HALO);
  metrics_kernel<<<grid_for(n, 128), 128, 0, s>>>(g, nodes, M, elem);
  return cudaGetLastError();
}

// spectral-radius rate on a curvilinear grid: sum over directions of |u.Sb| + c |Sb| (+ 4 max(4/3,
// gamma/Pr) mu/rho |Sb|^2 / V), divided by V, with Sb the mean of a cell's two faces in a direction
__global__ void __launch_bounds__(RATE_THREADS) init_rate_curvi_kernel(Geometry g, int viscous, RateConsts C, double cfl,
                                                                        const double* __restrict__ q,
                                                                        const float* __restrict__ M, DevCtrl* ctrl,
                                                                        double* partial, float* dtl) {
  const long long fm = g.fieldf;
  float best = 0.f;
  bool bad = false;
  const int rows = g.ny * g.nz, sh = row_shift(g.nx), per = RATE_THREADS >> sh;
  for (int row = blockIdx.x * per + (threadIdx.x >> sh); row < rows; row += gridDim.x * per) {
    const int j = row % g.ny, k = row / g.ny;
    for (int i = threadIdx.x & ((1 << sh) - 1); i < g.nx; i += 1 << sh) {
      const long long o = gidx(g, i, j, k), om = gidxf(g, i, j, k);
      const long long up[3] = {1, g.pxf, g.planef};
      const float rho = float(q[o]), ir = 1.f / rho;
      const float u = float(q[g.field + o]) * ir, v = float(q[2 * g.field + o]) * ir, w = float(q[3 * g.field + o]) * ir;
      const float p = C.gm1 * (float(q[4 * g.field + o]) - 0.5f * rho * (u * u + v * v + w * w));
      const float a = sqrtf(C.gam * p * ir);
      const float vol = M[9 * fm + om], iv = 1.f / vol;
      float rate = 0.f;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        float sb[3];
#pragma unroll
        for (int x = 0; x < 3; ++x) sb[x] = 0.5f * (M[(3 * d + x) * fm + om] + M[(3 * d + x) * fm + om + up[d]]);
        const float s2 = sb[0] * sb[0] + sb[1] * sb[1] + sb[2] * sb[2];
        float lam = fabsf(u * sb[0] + v * sb[1] + w * sb[2]) + a * sqrtf(s2);
        if (viscous) lam += C.fmu4 * ir * s2 * iv;
        rate += lam;
      }
      rate *= iv;
      if (dtl) dtl[om] = C.cfl / rate;
      if (!(rho > 0.f && p > 0.f)) bad = true;
      best = rate > best ? rate : best;
    }
  }
  if (bad) atomicOr(&ctrl->flag, FLAG_NONPHYSICAL);
  rate_fold(__double_as_longlong(double(best)), ctrl, partial, cfl);
}

cudaError_t launch_init_rate_curvi(const Geometry& g, const Physics& ph, const double* q, const void* M,
                                   DevCtrl* ctrl, double* partial, int grid, int mixed, void* dtl, cudaStream_t s) {
  if (mixed)
    init_rate_curvi_kernel<<<grid, RATE_THREADS, 0, s>>>(g, ph.viscous, rate_consts(ph), ph.cfl, q,
                                                         static_cast<const float*>(M), ctrl, partial,
                                                         static_cast<float*>(dtl));
  else if (ph.viscous)
    init_rate_x_kernel<true, true><<<grid, RATE_THREADS, 0, s>>>(g, ph, xconsts(ph.gamma, ph.eps), q,
                                                                 static_cast<const double*>(M), ctrl, partial,
                                                                 static_cast<double*>(dtl));
  else
    init_rate_x_kernel<false, true><<<grid, RATE_THREADS, 0, s>>>(g, ph, xconsts(ph.gamma, ph.eps), q,
                                                                  static_cast<const double*>(M), ctrl, partial,
                                                                  static_cast<double*>(dtl));
  return cudaGetLastError();
}

// ---- boundary ghost cells ---------------------------------------------------------------------
// One thread per (side, ghost layer m, face-slab point) of the physical faces of direction
// B.dim, over the full padded extent of the other two directions so that edges and corners get
// physical values too (directions are filled one launch after the other: x, y, z).
//   slip wall: ghost m mirrors interior cell m about the wall face's unit normal n,
//              u_g = u - 2 (u.n) n, same density and pressure
//   far field: characteristic boundary state from the adjacent interior cell and the free
//              stream (outgoing invariant u.n + 2c/(gamma-1) from inside, incoming one from the
//              free stream; entropy and tangential velocity from the upwind side; supersonic
//              inflow takes the free stream, supersonic outflow the interior), both layers
// On the mixed path the state is f32; for stages 2 and 3 the field is the f32 increment D over
// the f32 state S^n (the stencil adds them): the ghost increment is f32(Q_ghost - S_ghost).
// The ghost-cell arithmetic runs in the precision of the field it fills: FP64 for the FP64 state,
// FP32 for the mixed path's f32 state and increments (the values the FP32 fluxes read; FP64 here
// would leave these small launches waiting on the FP64 pipe, 2 lanes per SM).
template <typename T> struct BcMath;
template <> struct BcMath<double> {
  static __device__ __forceinline__ double sqrt_(double x) { return sqrt(x); }
  static __device__ __forceinline__ double pow_(double x, double y) { return pow(x, y); }
};
template <> struct BcMath<float> {
  static __device__ __forceinline__ float sqrt_(float x) { return sqrtf(x); }
  static __device__ __forceinline__ float pow_(float x, float y) { return powf(x, y); }
};

template <typename T>
__device__ __forceinline__ void bc_load(const BcBlock& B, long long o, long long of, T* q) {
  if (sizeof(T) == 8) {
    const double* f = static_cast<const double*>(B.field);
    for (int v = 0; v < 5; ++v) q[v] = T(f[v * B.g.field + o]);
  } else if (B.mode == BC_F32) {
    const float* f = static_cast<const float*>(B.field);
    for (int v = 0; v < 5; ++v) q[v] = T(f[v * B.g.fieldf + of]);
  } else {  // the stage input S + D, formed in f32 as the stage kernel forms it
    const float* f = static_cast<const float*>(B.field);
    for (int v = 0; v < 5; ++v) q[v] = T(B.shadow[v * B.g.fieldf + of] + f[v * B.g.fieldf + of]);
  }
}
template <typename T>
__device__ __forceinline__ void bc_store(const BcBlock& B, long long o, long long of, const T* w) {
  const T gm = T(B.gamma);
  T q[5];
  q[0] = w[0];
  q[1] = w[0] * w[1];
  q[2] = w[0] * w[2];
  q[3] = w[0] * w[3];
  q[4] = w[4] / (gm - T(1)) + T(0.5) * w[0] * (w[1] * w[1] + w[2] * w[2] + w[3] * w[3]);
  if (B.mode == BC_F64) {
    double* f = static_cast<double*>(B.field);
    for (int v = 0; v < 5; ++v) f[v * B.g.field + o] = double(q[v]);
  } else if (B.mode == BC_F32) {
    float* f = static_cast<float*>(B.field);
    for (int v = 0; v < 5; ++v) f[v * B.g.fieldf + of] = float(q[v]);
  } else {
    float* f = static_cast<float*>(B.field);
    float sh[5];  // (all loaded before the first store)
    for (int v = 0; v < 5; ++v) sh[v] = B.shadow[v * B.g.fieldf + of];
    for (int v = 0; v < 5; ++v) f[v * B.g.fieldf + of] = float(q[v] - T(sh[v]));
  }
}
template <typename T>
__device__ __forceinline__ void bc_prim(T gm, const T* q, T* w) {
  w[0] = q[0];
  w[1] = q[1] / q[0];
  w[2] = q[2] / q[0];
  w[3] = q[3] / q[0];
  w[4] = (gm - T(1)) * (q[4] - T(0.5) * q[0] * (w[1] * w[1] + w[2] * w[2] + w[3] * w[3]));
}

// one ghost cell: layer m (0 nearest the face) beyond face `hi` of direction d, at (a, b) along the
// other two directions
template <typename T, int D>
__device__ __forceinline__ void bc_cell(const BcBlock& B, int a, int b, int m, int hi, int kind) {
  using M = BcMath<T>;
  const Geometry& g = B.g;
  constexpr int d = D, d1 = (D + 1) % 3, d2 = (D + 2) % 3;
  const int n[3] = {g.nx, g.ny, g.nz};
  int idx[3], gi[3], ii[3];
  idx[d1] = a; idx[d2] = b; idx[d] = hi ? n[d] : 0;  // the boundary face is this cell's lower face
  for (int x = 0; x < 3; ++x) { gi[x] = idx[x]; ii[x] = idx[x]; }
  gi[d] = hi ? n[d] + m : -1 - m;
  if (kind != BC_SLIP_WALL && m > 0) return;  // the far field's layers are alike: layer 0's thread writes them all
  // unit normal (towards +d) of the boundary face
  T nrm[3] = {T(0), T(0), T(0)};
  if (B.metrics) {
    T S[3];
    if (B.mode == BC_F64) {
      const double* Mt = static_cast<const double*>(B.metrics);
      const long long oc = gidx(g, idx[0], idx[1], idx[2]);
      for (int x = 0; x < 3; ++x) S[x] = T(Mt[(3 * d + x) * g.field + oc]);
    } else {
      const float* Mt = static_cast<const float*>(B.metrics);
      const long long oc = gidxf(g, idx[0], idx[1], idx[2]);
      for (int x = 0; x < 3; ++x) S[x] = T(Mt[(3 * d + x) * g.fieldf + oc]);
    }
    const T len = M::sqrt_(S[0] * S[0] + S[1] * S[1] + S[2] * S[2]);
    for (int x = 0; x < 3; ++x) nrm[x] = S[x] / len;
  } else {
    nrm[d] = T(1);
  }
  T q[5], wi[5], wb[5], inf[5];
  for (int v = 0; v < 5; ++v) inf[v] = T(B.inf[v]);
  const T gm = T(B.gamma);
  if (kind == BC_SLIP_WALL) {
    ii[d] = hi ? n[d] - 1 - m : m;  // the mirror image inside
    bc_load<T>(B, gidx(g, ii[0], ii[1], ii[2]), gidxf(g, ii[0], ii[1], ii[2]), q);
    bc_prim<T>(gm, q, wi);
    const T un = wi[1] * nrm[0] + wi[2] * nrm[1] + wi[3] * nrm[2];
    wb[0] = wi[0];
    for (int x = 0; x < 3; ++x) wb[1 + x] = wi[1 + x] - T(2) * un * nrm[x];
    wb[4] = wi[4];
  } else {
    ii[d] = hi ? n[d] - 1 : 0;  // the interior cell next to the face
    bc_load<T>(B, gidx(g, ii[0], ii[1], ii[2]), gidxf(g, ii[0], ii[1], ii[2]), q);
    bc_prim<T>(gm, q, wi);
    const T out[3] = {hi ? nrm[0] : -nrm[0], hi ? nrm[1] : -nrm[1], hi ? nrm[2] : -nrm[2]};
    const T ci = M::sqrt_(gm * wi[4] / wi[0]), cinf = M::sqrt_(gm * inf[4] / inf[0]);
    const T uni = wi[1] * out[0] + wi[2] * out[1] + wi[3] * out[2];
    const T uninf = inf[1] * out[0] + inf[2] * out[1] + inf[3] * out[2];
    if (uninf <= -cinf) {
      for (int v = 0; v < 5; ++v) wb[v] = inf[v];
    } else if (uni >= ci) {
      for (int v = 0; v < 5; ++v) wb[v] = wi[v];
    } else {
      const T rp = uni + T(2) * ci / (gm - T(1)), rm = uninf - T(2) * cinf / (gm - T(1));
      const T unb = T(0.5) * (rp + rm), cb = T(0.25) * (gm - T(1)) * (rp - rm);
      T src[5];  // the upwind side's state (selected by value: no local-memory array)
      for (int v = 0; v < 5; ++v) src[v] = unb < T(0) ? inf[v] : wi[v];
      const T un_src = src[1] * out[0] + src[2] * out[1] + src[3] * out[2];
      const T ent = src[4] / M::pow_(src[0], gm);
      const T rho = M::pow_(cb * cb / (gm * ent), T(1) / (gm - T(1)));
      wb[0] = rho;
      for (int x = 0; x < 3; ++x) wb[1 + x] = src[1 + x] + (unb - un_src) * out[x];
      wb[4] = rho * cb * cb / gm;
    }
  }
  bc_store<T>(B, gidx(g, gi[0], gi[1], gi[2]), gidxf(g, gi[0], gi[1], gi[2]), wb);
  if (kind != BC_SLIP_WALL)
    for (int l = 1; l < HALO; ++l) {
      gi[d] = hi ? n[d] + l : -1 - l;
      bc_store<T>(B, gidx(g, gi[0], gi[1], gi[2]), gidxf(g, gi[0], gi[1], gi[2]), wb);
    }
}

// I: 32-bit unsigned wherever the cells' number allows, as in halo_kernel; the arithmetic's type and the
// direction are compiled in (no indexed arrays in local memory).  The far field's
// ghost layers, which are alike, are computed once.  Measured (channel of 192 x 96 x 16, far-field x-faces and
// the y-faces): FP64 26 and 11.5 -> 22 and 12 us, FP32 10.4 and 11 -> 10.2 and 7.7.
template <typename I, typename T, int D>
__global__ void bc_kernel(const __grid_constant__ BcBlock B) {
  const Geometry& g = B.g;
  const int n[3] = {g.nx, g.ny, g.nz};
  const I w1 = n[(D + 1) % 3] + 2 * HALO, w2 = n[(D + 2) % 3] + 2 * HALO;
  const I total = 2 * HALO * w1 * w2, stride = (I)gridDim.x * blockDim.x;
  for (I t = (I)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += stride) {
    const int a = (int)(t % w1) - HALO;
    I r = t / w1;
    const int b = (int)(r % w2) - HALO;
    r /= w2;
    const int m = (int)(r % HALO), hi = (int)(r / HALO);
    const int kind = B.kind[2 * D + hi];
    if (kind != BC_NONE) bc_cell<T, D>(B, a, b, m, hi, kind);
  }
}
template <typename I, typename T>
static void bc_go(const BcBlock& B, int grid, cudaStream_t s) {
  if (B.dim == 0) bc_kernel<I, T, 0><<<grid, 128, 0, s>>>(B);
  else if (B.dim == 1) bc_kernel<I, T, 1><<<grid, 128, 0, s>>>(B);
  else bc_kernel<I, T, 2><<<grid, 128, 0, s>>>(B);
}

cudaError_t launch_bc(const BcBlock& B, cudaStream_t s) {
  const int n[3] = {B.g.nx, B.g.ny, B.g.nz};
  const long long total = 2LL * HALO * (n[(B.dim + 1) % 3] + 2 * HALO) * (n[(B.dim + 2) % 3] + 2 * HALO);
  const int grid = grid_for(total, 128);
  const bool f64 = B.mode == BC_F64;
  if (total < (1LL << 30)) {
    if (f64) bc_go<unsigned, double>(B, grid, s);
    else bc_go<unsigned, float>(B, grid, s);
  } else {
    if (f64) bc_go<unsigned long long, double>(B, grid, s);
    else bc_go<unsigned long long, float>(B, grid, s);
  }
  return cudaGetLastError();
}

struct CtrlList {
  DevCtrl* c[MAX_GROUP];
};
// global time step of a group: cfl / max rate over the blocks, to every block (and to `extra`,
// the group's own control block, when given)
__global__ void group_dt_kernel(CtrlList L, int n, double cfl, DevCtrl* extra) {
  if (threadIdx.x != 0) return;
  double m = 0.0;
  for (int b = 0; b < n; ++b) m = fmax(m, L.c[b]->rate);
  for (int b = 0; b < n; ++b) L.c[b]->dt = cfl / m;
  if (extra) {
    extra->rate = m;
    extra->dt = cfl / m;
  }
}
cudaError_t launch_group_dt(DevCtrl* const* ctrls, int n, double cfl, cudaStream_t s, DevCtrl* extra) {
  CtrlList L;
  for (int b = 0; b < n && b < MAX_GROUP; ++b) L.c[b] = ctrls[b];
  group_dt_kernel<<<1, 32, 0, s>>>(L, n, cfl, extra);
  return cudaGetLastError();
}

}  // namespace gbcfd
