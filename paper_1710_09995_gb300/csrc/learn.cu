// learn.cu -- kernels of the learned convergence accelerator (see learn.cuh): the weight gradient
// of the convolutions, Adam, weight packing, the loss, and the kernels that connect the network
// to a block.  The convolutions themselves (tcgen05 implicit GEMM) are in learn_tc.cu.
#include <atomic>

#include "internal.cuh"
#include "learn.cuh"

namespace gbcfd {
namespace learn {

using bf16 = __nv_bfloat16;

__device__ __forceinline__ float silu(float z) { return z / (1.0f + __expf(-z)); }
__device__ __forceinline__ float dsilu(float z) {
  const float s = 1.0f / (1.0f + __expf(-z));
  return s * (1.0f + z * (1.0f - s));
}

// tile -> (x0, y0, z, b)
__device__ __forceinline__ void tile_coords(long long tile, int X, int Y, int Z, int& x0, int& y0, int& z, int& b) {
  const int tx = (X + TILE_X - 1) / TILE_X, ty = (Y + TILE_Y - 1) / TILE_Y;
  x0 = (int)(tile % tx) * TILE_X;
  tile /= tx;
  y0 = (int)(tile % ty) * TILE_Y;
  tile /= ty;
  z = (int)(tile % Z);
  b = (int)(tile / Z);
}

// the input cells a tile reads: box cell (bx, by, bz) is volume cell (x0 + bx - 1, y0 + by - 1,
// z + bz - 1); zero outside in x and y, periodic (or zero) in z
__device__ __forceinline__ long long box_source(int x0, int y0, int z, int b, int cellb, int X, int Y, int Z,
                                                int zper) {
  const int bx = cellb % BOX_X, r = cellb / BOX_X, by = r % BOX_Y, bz = r / BOX_Y;
  const int gx = x0 + bx - 1, gy = y0 + by - 1;
  int gz = z + bz - 1;
  if (gx < 0 || gx >= X || gy < 0 || gy >= Y) return -1;
  if (zper) gz = (gz + Z) % Z;
  else if (gz < 0 || gz >= Z) return -1;
  return (((long long)b * Z + gz) * Y + gy) * X + gx;
}

// a kernel's dynamic shared-memory limit, set once per device
template <typename F>
static cudaError_t smem_attr(F* kernel, size_t bytes, std::atomic<unsigned long long>& done) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 64 && ((done.load(std::memory_order_acquire) >> dev) & 1ull)) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess && dev < 64) done.fetch_or(1ull << dev, std::memory_order_acq_rel);
  return e;
}

// partial rows of the weight gradients = CTAs: one per SM (the buffer holds two per SM)
static int wgrad_rows(const Net& n) { return n.wgrid / 2; }

// ---- weight gradient ---------------------------------------------------------------------------
// dW[o][c][t] = sum over cells of g[cell][o] a[cell + d_t][c], db[o] = sum of g[cell][o]: per tap a
// matrix product with the cells as its long dimension, g^T (outputs x cells) times the shifted a
// (cells x inputs).  Both operands are bf16 with the channels contiguous, so the cells' dimension
// is the strided one of either: fragments come from shared memory by ldmatrix.trans, and one warp
// per tap issues mma.sync m16n8k16 (f32 accumulation) on the whole [outputs][inputs] block.  (tcgen05
// has no use here: its smallest M is 64, the outputs are 5 to 32, and stacking taps in M needs
// operands whose rows lie at the taps' irregular shifts.)  27 tap warps share a tile of 32 x 4 cells
// and its 34 x 6 x 3 box of a, staged by cp.async one tile ahead; rows are padded by 16 bytes
// so that ldmatrix's eight rows fall into different banks.  A tile's products are summed on the
// tensor cores from zero and added to FP32 sums, so no chain is longer than 128 cells; a 28th warp
// sums the biases.  Each CTA writes its own partial row; launch_grad_reduce sums the rows in a
// fixed order (deterministic).  Measured (192 x 96 x 4 cells, batch 4), against one thread per weight with FP32
// operands in shared memory, two loads per multiply-add: a training step 25.9 -> 1.4 ms, 0.65 with the
// convolutions of today, 0.225 of it in the gradients; errors against 64-bit sums of the same bf16 products 0.8-1.0e-7 of
// the gradient, 1.2-2.8e-7 then.
constexpr int WG_THREADS = 28 * 32;
template <int P> constexpr int wg_pitch() { return 2 * P + 16; }  // bytes of a padded row of P channels

__device__ __forceinline__ void ldsm_t4(unsigned (&r)[4], unsigned addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
__device__ __forceinline__ void mma_bf16(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// stored channels: CIP of a (16 or 32), COPG of g (16 or 32); CI, CO of them are real
template <int CIP, int CI, int COPG, int CO>
struct WgPlan {
  static constexpr int PA = wg_pitch<CIP>(), PG = wg_pitch<COPG>();
  static constexpr int CELLS = TILE_X * TILE_Y;
  static constexpr size_t abytes = (size_t)BOX * PA, gbytes = (size_t)CELLS * PG, slot = abytes + gbytes;
  static constexpr size_t out = sizeof(float) * CO * CI * NTAP;  // the CTA's result, over the slots at the end
  static constexpr size_t bytes = 2 * slot > out ? 2 * slot : out;
};

template <int CIP, int CI, int COPG, int CO>
__global__ void __launch_bounds__(WG_THREADS, 1) wgrad_kernel(const bf16* __restrict__ a, const bf16* __restrict__ g,
                                                               float* __restrict__ part, int off_w, int off_b, int X,
                                                               int Y, int Z, int B, int zper) {
  using PL = WgPlan<CIP, CI, COPG, CO>;
  constexpr int MT = COPG / 16, NT = CIP / 8;  // 16-row and 8-column tiles
  extern __shared__ __align__(128) unsigned char smem[];
  const unsigned s0 = (unsigned)__cvta_generic_to_shared(smem);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const long long tiles = (long long)((X + TILE_X - 1) / TILE_X) * ((Y + TILE_Y - 1) / TILE_Y) * Z * B;

  // a tile's operands into a slot, 16 bytes per copy; cells outside the volume are zero
  auto stage = [&](long long tile, unsigned slot) {
    int x0, y0, z, b;
    tile_coords(tile, X, Y, Z, x0, y0, z, b);
    for (int i = tid; i < BOX * (CIP / 8); i += WG_THREADS) {
      const int cellb = i / (CIP / 8), q = i % (CIP / 8);
      const long long src = box_source(x0, y0, z, b, cellb, X, Y, Z, zper);
      const bf16* p = src >= 0 ? a + src * CIP + q * 8 : a;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(slot + (unsigned)(cellb * PL::PA + q * 16)),
                   "l"(p), "r"(src >= 0 ? 16 : 0)
                   : "memory");
    }
    for (int i = tid; i < PL::CELLS * (COPG / 8); i += WG_THREADS) {
      const int c = i / (COPG / 8), q = i % (COPG / 8);
      const int gx = x0 + c % TILE_X, gy = y0 + c / TILE_X;
      const bool in = gx < X && gy < Y;
      const bf16* p = in ? g + ((((long long)b * Z + z) * Y + gy) * X + gx) * COPG + q * 8 : g;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(
                       slot + (unsigned)(PL::abytes + c * PL::PG + q * 16)),
                   "l"(p), "r"(in ? 16 : 0)
                   : "memory");
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };

  float sum[MT][NT][4];
#pragma unroll
  for (int m = 0; m < MT; ++m)
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int q = 0; q < 4; ++q) sum[m][n][q] = 0.f;
  float bsum = 0.f;
  const int dz = warp / 9, dy = (warp / 3) % 3, dx = warp % 3;
  // this lane's row and column of the four 8 x 8 matrices of an ldmatrix: matrices 0, 1 are cells 0-7
  // and 8-15 of the first 8 channels for b, 0, 1 the first 8 and next 8 channels for g
  const int lr = lane & 7, lm = lane >> 3;

  if ((long long)blockIdx.x < tiles) stage(blockIdx.x, s0);
  int cur = 0;
  for (long long tile = blockIdx.x; tile < tiles; tile += gridDim.x, cur ^= 1) {
    const bool more = tile + gridDim.x < tiles;
    if (more) stage(tile + gridDim.x, s0 + (unsigned)((cur ^ 1) * PL::slot));
    if (more) asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    else asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();
    const unsigned as = s0 + (unsigned)(cur * PL::slot), gs = as + (unsigned)PL::abytes;
    if (warp < NTAP) {
      float acc[MT][NT][4];
#pragma unroll
      for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[m][n][q] = 0.f;
#pragma unroll 2
      for (int c0 = 0; c0 < PL::CELLS; c0 += 16) {
        const int cy = c0 / TILE_X, cx = c0 % TILE_X;
        unsigned ga[MT][4], bb[NT / 2][4];
#pragma unroll
        for (int m = 0; m < MT; ++m)  // A = g^T: (rows 0-7, 8-15) x (cells 0-7, 8-15)
          ldsm_t4(ga[m], gs + (unsigned)((c0 + lr + (lm >> 1) * 8) * PL::PG + (m * 16 + (lm & 1) * 8) * 2));
        const int base = (dz * BOX_Y + cy + dy) * BOX_X + cx + dx;
#pragma unroll
        for (int n = 0; n < NT / 2; ++n)  // B: (cells 0-7, 8-15) of two 8-column tiles
          ldsm_t4(bb[n], as + (unsigned)((base + lr + (lm & 1) * 8) * PL::PA + (n * 16 + (lm >> 1) * 8) * 2));
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
          for (int n = 0; n < NT; ++n) mma_bf16(acc[m][n], ga[m], bb[n / 2][(n & 1) * 2], bb[n / 2][(n & 1) * 2 + 1]);
      }
#pragma unroll
      for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
          for (int q = 0; q < 4; ++q) sum[m][n][q] += acc[m][n][q];
    } else if (lane < CO) {
      const bf16* gp = reinterpret_cast<const bf16*>(smem + cur * PL::slot + PL::abytes) + lane;
      float t = 0.f;
#pragma unroll 8
      for (int c = 0; c < PL::CELLS; ++c) t += __bfloat162float(gp[c * (PL::PG / 2)]);
      bsum += t;
    }
    __syncthreads();  // the slot is refilled by the next iteration's copies
  }
  // [o][c][t] through shared memory, so that the partial row is written in order
  float* out = reinterpret_cast<float*>(smem);
  if (warp < NTAP) {
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
      for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int o = m * 16 + (lane >> 2) + (q >> 1) * 8, c = n * 8 + (lane & 3) * 2 + (q & 1);
          if (o < CO && c < CI) out[(o * CI + c) * NTAP + warp] = sum[m][n][q];
        }
  } else if (lane < CO) {
    part[(size_t)blockIdx.x * NPARAM + off_b + lane] = bsum;
  }
  __syncthreads();
  for (int i = tid; i < CO * CI * NTAP; i += WG_THREADS) part[(size_t)blockIdx.x * NPARAM + off_w + i] = out[i];
}

template <int CIP, int CI, int COPG, int CO>
static cudaError_t wgrad_go(const bf16* a, const bf16* g, const Net& n, int off_w, int off_b, int X, int Y, int Z,
                            int B, int zper, cudaStream_t s) {
  constexpr size_t bytes = WgPlan<CIP, CI, COPG, CO>::bytes;
  static std::atomic<unsigned long long> done{0};
  cudaError_t e = smem_attr(wgrad_kernel<CIP, CI, COPG, CO>, bytes, done);
  if (e != cudaSuccess) return e;
  wgrad_kernel<CIP, CI, COPG, CO><<<wgrad_rows(n), WG_THREADS, bytes, s>>>(a, g, n.wpart, off_w, off_b, X, Y, Z, B,
                                                                            zper);
  return cudaGetLastError();
}

// layer 1: a = input features (16 ch, 10 used), g = dZ1 (32); layer 2: a = a1, g = dZ2; layer 3:
// a = a2, g = dY (16 ch, 5 used)
cudaError_t launch_wgrad(int layer, const bf16* a, const bf16* g, const Net& n, int X, int Y, int Z, int B, int zper,
                         cudaStream_t s) {
  if (layer == 1) return wgrad_go<P0, C0, P1, C1>(a, g, n, OFF_W1, OFF_B1, X, Y, Z, B, zper, s);
  if (layer == 2) return wgrad_go<P1, C1, P2, C2>(a, g, n, OFF_W2, OFF_B2, X, Y, Z, B, zper, s);
  if (layer == 3) return wgrad_go<P2, C2, 16, C3>(a, g, n, OFF_W3, OFF_B3, X, Y, Z, B, zper, s);
  return cudaErrorInvalidValue;
}

// 32 parameters per CTA, eight threads each: thread y sums rows y, y + 8, ..., then the eight in order
__global__ void grad_reduce_kernel(const float* __restrict__ part, int rows, float* __restrict__ grad) {
  __shared__ float red[8][32];
  const int o = blockIdx.x * 32 + threadIdx.x;
  float s = 0.f;
  if (o < NPARAM)
#pragma unroll 4
    for (int r = threadIdx.y; r < rows; r += 8) s += part[(size_t)r * NPARAM + o];
  red[threadIdx.y][threadIdx.x] = s;
  __syncthreads();
  if (threadIdx.y == 0 && o < NPARAM) {
    for (int y = 1; y < 8; ++y) s += red[y][threadIdx.x];
    grad[o] = s;
  }
}
cudaError_t launch_grad_reduce(const Net& n, cudaStream_t s) {
  grad_reduce_kernel<<<(NPARAM + 31) / 32, dim3(32, 8), 0, s>>>(n.wpart, wgrad_rows(n), n.grad);
  return cudaGetLastError();
}

// ---- Adam and packing ----------------------------------------------------------------------------
__global__ void adam_kernel(float* w, float* m, float* v, const float* g, float lr, float c1, float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= NPARAM) return;
  const float gi = g[i];
  const float mi = 0.9f * m[i] + 0.1f * gi;
  const float vi = 0.999f * v[i] + 0.001f * gi * gi;
  m[i] = mi;
  v[i] = vi;
  w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + 1e-8f);
}
cudaError_t launch_adam(const Net& n, float lr, int step, cudaStream_t s) {
  const float c1 = 1.0f - powf(0.9f, (float)step), c2 = 1.0f - powf(0.999f, (float)step);
  adam_kernel<<<(NPARAM + 255) / 256, 256, 0, s>>>(n.w, n.m, n.v, n.grad, lr, c1, c2);
  return cudaGetLastError();
}

// master weights -> bf16 GEMM layouts (forward [t][o][c], backward [t'][c][o] with t' = 26 - t)
// and padded biases; padding entries are zero
__global__ void pack_kernel(Net n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const float* w = n.w;
  if (i < NTAP * P1 * P0) {  // w1 [t][o<32][c<16]
    const int t = i / (P1 * P0), o = (i / P0) % P1, c = i % P0;
    n.w1[i] = __float2bfloat16(c < C0 ? w[OFF_W1 + (o * C0 + c) * NTAP + t] : 0.f);
  }
  if (i < NTAP * P2 * P1) {  // w2 [t][o][c], w2b [t'][c][o]
    const int t = i / (P2 * P1), o = (i / P1) % P2, c = i % P1;
    n.w2[i] = __float2bfloat16(w[OFF_W2 + (o * C1 + c) * NTAP + t]);
    const int tb = i / (P1 * P2), cb = (i / P2) % P1, ob = i % P2;  // w2b[tb][cb][ob] = W2[ob][cb][26 - tb]
    n.w2b[i] = __float2bfloat16(w[OFF_W2 + (ob * C1 + cb) * NTAP + (NTAP - 1 - tb)]);
  }
  if (i < NTAP * 16 * P2) {  // w3 [t][o<16][c<32] (the MMA is 16 wide; 5 used)
    const int t = i / (16 * P2), o = (i / P2) % 16, c = i % P2;
    n.w3[i] = __float2bfloat16(o < C3 ? w[OFF_W3 + (o * C2 + c) * NTAP + t] : 0.f);
  }
  if (i < NTAP * P2 * 16) {  // w3b [t'][c<32][o<16] = W3[o][c][26 - t']
    const int tb = i / (P2 * 16), cb = (i / 16) % P2, ob = i % 16;
    n.w3b[i] = __float2bfloat16(ob < C3 ? w[OFF_W3 + (ob * C2 + cb) * NTAP + (NTAP - 1 - tb)] : 0.f);
  }
  if (i < P1) n.b1[i] = w[OFF_B1 + i];
  if (i < P2) n.b2[i] = w[OFF_B2 + i];
  if (i < P3) n.b3[i] = i < C3 ? w[OFF_B3 + i] : 0.f;
}
cudaError_t launch_pack(const Net& n, cudaStream_t s) {
  pack_kernel<<<(NTAP * P2 * P1 + 255) / 256, 256, 0, s>>>(n);
  return cudaGetLastError();
}

// ---- loss: dY = 2 (y - t) / (5 cells) in bf16 (16 channels), per-CTA sums of (y - t)^2 ----------
__global__ void loss_kernel(const float* __restrict__ y, const float* __restrict__ t, bf16* __restrict__ dy,
                            double* __restrict__ partial, long long cells) {
  __shared__ double red[NTHREADS / 32];
  const double inv = 2.0 / (5.0 * (double)cells);
  double acc = 0.0;
  for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < cells; c += (long long)gridDim.x * blockDim.x) {
    __align__(16) bf16 out[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) out[k] = __float2bfloat16(0.f);
#pragma unroll
    for (int k = 0; k < C3; ++k) {
      const float d = y[c * P3 + k] - t[c * P3 + k];
      acc += (double)d * d;
      out[k] = __float2bfloat16((float)(inv * d));
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) reinterpret_cast<uint4*>(dy + c * 16)[k] = reinterpret_cast<const uint4*>(out)[k];
  }
  for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < NTHREADS / 32; ++w) s += red[w];
    partial[(size_t)blockIdx.x * NPART] = s;
  }
}
cudaError_t launch_loss(const float* y, const float* t, bf16* dy, double* partial, long long cells, int grid,
                        cudaStream_t s) {
  loss_kernel<<<grid, NTHREADS, 0, s>>>(y, t, dy, partial, cells);
  return cudaGetLastError();
}

// out[j] = sum over rows r < n of partial[r * NPART + j], j < nvals: a warp per value, lanes over the
// rows, folded in a fixed order
__global__ void sum_kernel(const double* __restrict__ partial, int n, double* __restrict__ out) {
  const int j = threadIdx.y, lane = threadIdx.x;
  double s = 0.0;
#pragma unroll 4
  for (int r = lane; r < n; r += 32) s += partial[(size_t)r * NPART + j];
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if (lane == 0) out[j] = s;
}
cudaError_t launch_sum(const double* partial, int n, int nvals, double* out, cudaStream_t s) {
  sum_kernel<<<1, dim3(32, nvals), 0, s>>>(partial, n, out);
  return cudaGetLastError();
}

// ---- block-facing kernels ----------------------------------------------------------------------
__device__ __forceinline__ long long vidx(const BlockView& v, int i, int j, int k) {
  return ((long long)(k + HALO) * (v.ny + 2 * HALO) + (j + HALO)) * v.px + (i + HALO);
}
__device__ __forceinline__ long long vidxf(const BlockView& v, int i, int j, int k) {
  return ((long long)(k + HALO) * (v.ny + 2 * HALO) + (j + HALO)) * v.pxf + (i + HALO);
}
__device__ __forceinline__ double cell_dt(const BlockView& v, int i, int j, int k) {
  if (!v.dtl) return *v.dt;
  return v.dtl_f32 ? (double)static_cast<const float*>(v.dtl)[vidxf(v, i, j, k)]
                   : static_cast<const double*>(v.dtl)[vidx(v, i, j, k)];
}

// per CTA: [0] sum over cells and variables of (dt R / ref)^2, [1] sum of R_rho^2
__global__ void feature_stats_kernel(BlockView v, const double* __restrict__ R, double* __restrict__ partial) {
  __shared__ double red[2][NTHREADS / 32];
  const long long n = (long long)v.nx * v.ny * v.nz;
  double s0 = 0.0, s1 = 0.0;
  for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(c % v.nx);
    const long long r = c / v.nx;
    const int j = (int)(r % v.ny), k = (int)(r / v.ny);
    const double dt = cell_dt(v, i, j, k);
    for (int m = 0; m < 5; ++m) {
      const double x = dt * R[m * n + c] / v.ref[m];
      s0 += x * x;
    }
    s1 += R[c] * R[c];
  }
  for (int off = 16; off > 0; off >>= 1) {
    s0 += __shfl_xor_sync(0xffffffffu, s0, off);
    s1 += __shfl_xor_sync(0xffffffffu, s1, off);
  }
  if ((threadIdx.x & 31) == 0) { red[0][threadIdx.x >> 5] = s0; red[1][threadIdx.x >> 5] = s1; }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0, b = 0.0;
    for (int w = 0; w < NTHREADS / 32; ++w) { a += red[0][w]; b += red[1][w]; }
    partial[(size_t)blockIdx.x * NPART] = a;
    partial[(size_t)blockIdx.x * NPART + 1] = b;
  }
}
cudaError_t launch_feature_stats(const BlockView& v, const double* R, double* partial, int grid, cudaStream_t s) {
  feature_stats_kernel<<<grid, NTHREADS, 0, s>>>(v, R, partial);
  return cudaGetLastError();
}

// x[cell] = (10 (Q - Q_inf) / ref, (-dt R / ref) / s, 0 x 6) in bf16; the compact state is saved
// (f64) for the prediction, the target and a revert.  s = sqrt(stats[0] / (5 cells)).
__global__ void features_kernel(BlockView v, const double* __restrict__ R, const double* __restrict__ stats,
                                bf16* __restrict__ x, double* __restrict__ qsave) {
  const long long n = (long long)v.nx * v.ny * v.nz;
  const double s = sqrt(stats[0] / (5.0 * (double)n));
  const double is = s > 0.0 ? 1.0 / s : 0.0;
  for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(c % v.nx);
    const long long r = c / v.nx;
    const int j = (int)(r % v.ny), k = (int)(r / v.ny);
    const long long o = vidx(v, i, j, k);
    const double dt = cell_dt(v, i, j, k);
    __align__(16) bf16 f[16];
#pragma unroll
    for (int m = 0; m < 5; ++m) {
      const double q = v.q[m * v.field + o];
      qsave[m * n + c] = q;
      f[m] = __double2bfloat16((double)STATE_GAIN * (q - v.qinf[m]) / v.ref[m]);
      f[5 + m] = __double2bfloat16(-dt * R[m * n + c] / v.ref[m] * is);
    }
#pragma unroll
    for (int m = 10; m < 16; ++m) f[m] = __float2bfloat16(0.f);
    reinterpret_cast<uint4*>(x + c * 16)[0] = reinterpret_cast<const uint4*>(f)[0];
    reinterpret_cast<uint4*>(x + c * 16)[1] = reinterpret_cast<const uint4*>(f)[1];
  }
}
cudaError_t launch_features(const BlockView& v, const double* R, const double* stats, bf16* x, double* qsave,
                            cudaStream_t s) {
  const long long n = (long long)v.nx * v.ny * v.nz;
  long long grid = (n + 255) / 256;
  if (grid > 65535LL * 8) grid = 65535LL * 8;
  features_kernel<<<(unsigned)grid, 256, 0, s>>>(v, R, stats, x, qsave);
  return cudaGetLastError();
}

// Q = Q_saved + alpha K s ref y (or Q_saved when revert), into the padded state and its f32 shadow
__global__ void apply_kernel(BlockView v, const float* __restrict__ y, const double* __restrict__ qsave,
                             const double* __restrict__ stats, int revert, double alpha) {
  const long long n = (long long)v.nx * v.ny * v.nz;
  const double s = alpha * sqrt(stats[0] / (5.0 * (double)n));
  for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(c % v.nx);
    const long long r = c / v.nx;
    const int j = (int)(r % v.ny), k = (int)(r / v.ny);
    const long long o = vidx(v, i, j, k);
#pragma unroll
    for (int m = 0; m < 5; ++m) {
      double q = qsave[m * n + c];
      if (!revert) q += (double)K_STEPS * s * v.ref[m] * (double)y[c * P3 + m];
      v.q[m * v.field + o] = q;
      if (v.sh) v.sh[m * v.fieldf + vidxf(v, i, j, k)] = (float)q;
    }
  }
}
cudaError_t launch_apply(const BlockView& v, const float* y, const double* qsave, const double* stats, int revert,
                         cudaStream_t s, double alpha) {
  const long long n = (long long)v.nx * v.ny * v.nz;
  long long grid = (n + 255) / 256;
  if (grid > 65535LL * 8) grid = 65535LL * 8;
  apply_kernel<<<(unsigned)grid, 256, 0, s>>>(v, y, qsave, stats, revert, alpha);
  return cudaGetLastError();
}

// t[cell][m] = (Q_now - Q_saved) / ref / (K s) (f32, 8 channels, 5 used)
__global__ void target_kernel(BlockView v, const double* __restrict__ qsave, const double* __restrict__ stats,
                              float* __restrict__ t) {
  const long long n = (long long)v.nx * v.ny * v.nz;
  const double s = sqrt(stats[0] / (5.0 * (double)n));
  const double is = s > 0.0 ? 1.0 / ((double)K_STEPS * s) : 0.0;
  for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(c % v.nx);
    const long long r = c / v.nx;
    const int j = (int)(r % v.ny), k = (int)(r / v.ny);
    const long long o = vidx(v, i, j, k);
#pragma unroll
    for (int m = 0; m < 5; ++m) t[c * P3 + m] = (float)((v.q[m * v.field + o] - qsave[m * n + c]) / v.ref[m] * is);
#pragma unroll
    for (int m = 5; m < P3; ++m) t[c * P3 + m] = 0.f;
  }
}
cudaError_t launch_target(const BlockView& v, const double* qsave, const double* stats, float* t, cudaStream_t s) {
  const long long n = (long long)v.nx * v.ny * v.nz;
  long long grid = (n + 255) / 256;
  if (grid > 65535LL * 8) grid = 65535LL * 8;
  target_kernel<<<(unsigned)grid, 256, 0, s>>>(v, qsave, stats, t);
  return cudaGetLastError();
}

}  // namespace learn
}  // namespace gbcfd
