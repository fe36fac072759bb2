// learn_tc.cu -- the accelerator's implicit-GEMM 3D convolution on the 5th-generation tensor
// cores: tcgen05.mma (kind::f16, bf16 x bf16 -> f32) issued by one thread, operands in shared
// memory in the canonical no-swizzle K-major layout, the 128 x N accumulator in tensor memory,
// read back with tcgen05.ld for the epilogue.
//
// A tile is 128 consecutive cells along x (one y, z, batch); GEMM view M = 128 cells,
// N = output channels (16 or 32), K = 27 taps x CIP input channels, issued as 27 x CIP/16 MMAs
// of K = 16.  A CTA takes a contiguous range of tiles with y fastest, so that consecutive tiles
// share six of their nine input rows: shared memory holds the weights and a ring of five y-rows
// (of the three z-planes each) of 130 cells, as 8 x 16-byte core matrices:
//   row    element (slot s, plane z, cell c, channel k) at (((3 s + z) CIP/8 + k / 8) RP + c) 8 + k % 8
//   weight element (tap t, out o, in k) at ((t CIP/8 + k / 8) N + o) 8 + k % 8
// so for tap t the A matrix of the tile starts at cell dx of plane dz of the slot of row y + dy - 1
// (rows = cells, 8 consecutive rows one 128-byte core matrix, SBO 128 B, LBO = RP x 16 B along K)
// and the B matrix at weight group t CIP/8 (SBO 128 B, LBO = N x 16 B).
//
// Warps: four per 16 output channels read the accumulators back (thread = TMEM lane = cell) and
// apply the epilogue, four load rows by cp.async (two groups of two warps, alternate rows), the last
// issues the MMAs: it walks and waits as a warp, so that the descriptors (a constant away from the three
// rows') stay in uniform registers, and one elected lane executes the MMA.  In a one-thread branch each
// descriptor was moved there anew, about 100 cycles an MMA (two tiles' MMAs in turn were no faster): layer 2
// 197 -> 121 us.  The warps meet only at mbarriers: a row landed, a tile's MMAs done (tcgen05.commit), an
// accumulator read back.  The first version copied a tile's nine rows anew by TMA, with the
// channel groups as 16-byte inner boxes: 36 copies of 130 such pieces a tile held it at 12 us
// (every unit below 30% busy); now a tile loads three rows, in pieces the threads copy whole cells
// at a time.  192 x 96 x 64 cells, three layers: 1.86 -> 0.34 ms.
#include <atomic>

#include "internal.cuh"
#include "learn.cuh"

namespace gbcfd {
namespace learn {

using bf16 = __nv_bfloat16;

constexpr int TC_M = 128, TC_BX = TC_M + 2, TC_NR = 5, TC_LOADERS = 64;
// cells a channel group's row is padded to: the four (two) groups of a cell fall into different banks
template <int CIP> struct TcPitch { static constexpr int value = CIP == 32 ? 138 : 140; };

__device__ __forceinline__ unsigned smem_u32(const void* p) {
  return static_cast<unsigned>(__cvta_generic_to_shared(p));
}

// shared-memory matrix descriptor: start, leading (K) and stride (M/N) byte offsets, no swizzle
__device__ __forceinline__ unsigned long long smem_desc(unsigned addr, unsigned lbo, unsigned sbo) {
  unsigned long long d = 0;
  d |= (unsigned long long)((addr >> 4) & 0x3FFFu);
  d |= (unsigned long long)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (unsigned long long)((sbo >> 4) & 0x3FFFu) << 32;
  d |= 1ull << 46;  // descriptor version for this architecture; base offset 0, layout: no swizzle
  return d;
}

// instruction descriptor, kind::f16: D f32, A and B bf16, both K-major, N, M = 128
__host__ __device__ constexpr unsigned instr_desc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(n >> 3) << 17) | ((unsigned)(TC_M >> 4) << 24);
}

__device__ __forceinline__ void tc_mma(unsigned tmem, unsigned long long a, unsigned long long b, unsigned idesc,
                                       unsigned accumulate) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.u32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ bool mbar_wait_limited(unsigned bar, unsigned parity) {
  const unsigned long long t0 = globaltimer_ns();
  while (true) {
    unsigned done;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
    if (globaltimer_ns() - t0 > 2000000000ull) return false;  // 2 s
  }
}

__device__ __forceinline__ void mbar_arrive1(unsigned bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}

// a CTA's range of tiles, walked in columns (x tile, z, b) of consecutive y
struct TcWalk {
  long long t, end;   // next tile, end of the range
  int x0, z, b, ya, n;  // the current column piece: rows ya .. ya + n - 1
  __device__ __forceinline__ bool next(const ConvArgs& A) {
    if (t >= end) return false;
    const int tx = (A.X + TC_M - 1) / TC_M;
    const long long col = t / A.Y;
    ya = (int)(t - col * A.Y);
    n = (int)min((long long)(A.Y - ya), end - t);
    x0 = (int)(col % tx) * TC_M;
    z = (int)((col / tx) % A.Z);
    b = (int)(col / tx / A.Z);
    t += n;
    return true;
  }
};

__device__ __forceinline__ bool elect_one() {
  unsigned p;
  asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
  return p != 0;
}

// the 27 x CIP/16 MMAs of one tile into the accumulator at tmem (one thread), then a commit;
// row[dy] = the descriptor of cell 0, plane 0 of the slot of row y + dy - 1, wdesc the weights'
template <int CIP, int N>
__device__ __forceinline__ void tc_issue(const unsigned long long (&row)[3], unsigned long long wdesc, unsigned tmem,
                                         unsigned bar) {
  constexpr unsigned idesc = instr_desc(N), RP = TcPitch<CIP>::value;
#pragma unroll
  for (int t = 0; t < NTAP; ++t) {
    const int dz = t / 9, dy = (t / 3) % 3, dx = t % 3;
#pragma unroll
    for (int kk = 0; kk < CIP / 16; ++kk)  // descriptor addresses count 16 bytes: one cell of a channel group
      tc_mma(tmem, row[dy] + (unsigned)((dz * (CIP / 8) + 2 * kk) * RP + dx),
             wdesc + (unsigned)((t * (CIP / 8) + 2 * kk) * N), idesc, (t | kk) != 0);
  }
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar) : "memory");
}

// NC output channels c0 .. c0 + NC - 1 of one cell: bias, SiLU (and the pre-activation kept for
// training), the linear output, or the product with SiLU' of the saved pre-activation
template <int COP, int NC, int MODE>
__device__ __forceinline__ void tc_epilogue(const ConvArgs& A, const float* bias, const float (&acc)[16], long long cell,
                                            int c0) {
  const long long at = cell * COP + c0;
  if constexpr (MODE == FWD_LINEAR) {
    float* out = static_cast<float*>(A.out) + at;
#pragma unroll
    for (int c = 0; c < NC; c += 4)
      *reinterpret_cast<float4*>(out + c) = make_float4(acc[c] + bias[c0 + c], acc[c + 1] + bias[c0 + c + 1],
                                                        acc[c + 2] + bias[c0 + c + 2], acc[c + 3] + bias[c0 + c + 3]);
  } else {
    __align__(16) bf16 o[NC];
#pragma unroll
    for (int c = 0; c < NC; c += 4) {
      if constexpr (MODE == FWD_SILU) {
        float v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          v[q] = acc[c + q] + bias[c0 + c + q];
          o[c + q] = __float2bfloat16(v[q] / (1.0f + __expf(-v[q])));
        }
        if (A.zsave) *reinterpret_cast<float4*>(A.zsave + at + c) = make_float4(v[0], v[1], v[2], v[3]);
      } else {
        const float4 z4 = *reinterpret_cast<const float4*>(A.zprev + at + c);
        const float zp[4] = {z4.x, z4.y, z4.z, z4.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float sg = 1.0f / (1.0f + __expf(-zp[q]));
          o[c + q] = __float2bfloat16(acc[c + q] * (sg * (1.0f + zp[q] * (1.0f - sg))));
        }
      }
    }
#pragma unroll
    for (int q = 0; q < NC / 8; ++q)
      reinterpret_cast<uint4*>(static_cast<bf16*>(A.out) + at)[q] = reinterpret_cast<const uint4*>(o)[q];
  }
}

// Steps (tiles) s = 0, 1, ... and rows g = 0, 1, ... of a CTA are counted over its columns; a column
// piece of n tiles has n + 2 rows, step i of it reads rows i, i + 1, i + 2.  Row g lives in slot g % 5
// (full[g % 5], phase g / 5); step s's accumulator is s % 2, its completion done[s % 4], phase s / 4;
// epi[s % 2] says the accumulator was read back.  A row may be loaded once the last step that read
// the row five before it is done: within a piece that is step i - 5 (of row i), which trails the
// steps that can have been issued by at most two, so four done barriers never wrap past a waiter.
// Every wait is bounded (2 s); a role that gives up flags the timeout and leaves, the others follow.
template <int N> struct TcWarps {  // epilogue warps, then four loaders, then the issuer
  static constexpr int epi = 4 * (N / 16), threads = 32 * (epi + 5);
};
template <int CIP, int N, int COP, int MODE>
__global__ void __launch_bounds__(TcWarps<N>::threads, CIP == 16 ? 2 : 1) conv_tc_kernel(const ConvArgs A, const bf16* __restrict__ wtc,
                                                             int* __restrict__ flag, long long ntiles) {
  constexpr int CG = CIP / 8, RP = TcPitch<CIP>::value, EPI = TcWarps<N>::epi, TC_THREADS = TcWarps<N>::threads;
  constexpr unsigned SLOTB = 3u * CG * RP * 16u;
  extern __shared__ __align__(128) unsigned char smem[];
  bf16* wsm = reinterpret_cast<bf16*>(smem + TC_NR * SLOTB);         // 27 x CIP x N
  float* bias = reinterpret_cast<float*>(wsm + NTAP * CIP * N);      // COP (FWD)
  unsigned long long* bar = reinterpret_cast<unsigned long long*>(bias + 32);  // full[5], done[4], epi[2]
  unsigned* tslot = reinterpret_cast<unsigned*>(bar + 11);
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // uniform: the issuer's branch and values
  constexpr unsigned COLW = N < 32 ? 32 : N, COLS = 2 * COLW;

  if (warp == EPI + 4) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tslot)),
                 "r"(COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  const unsigned rows0 = smem_u32(smem), w0 = smem_u32(wsm), full0 = smem_u32(bar), done0 = full0 + 5 * 8, epi0 = done0 + 4 * 8;
  if (tid == 0) {
    for (int j = 0; j < 11; ++j)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(full0 + 8u * j),
                   "r"(j < 5 ? TC_LOADERS : (j < 9 ? 1 : EPI * 32)));
    asm volatile("fence.mbarrier_init.release.cluster;\n");
  }
  for (int i = tid; i < NTAP * N * CG; i += TC_THREADS) {  // global [27][N][CIP] -> core matrices
    const int t = i / (N * CG), r = i % (N * CG), o = r / CG, kg = r % CG;
    const uint4 v = *reinterpret_cast<const uint4*>(wtc + ((size_t)t * N + o) * CIP + kg * 8);
    *reinterpret_cast<uint4*>(wsm + (((size_t)t * CG + kg) * N + o) * 8) = v;
  }
  if (MODE != BWD_DSILU && tid < COP) bias[tid] = A.bias[tid];
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const unsigned tmem0 = *tslot;
  TcWalk walk;
  walk.t = (long long)blockIdx.x * ntiles / gridDim.x;
  walk.end = (long long)(blockIdx.x + 1) * ntiles / gridDim.x;
  bool ok = true;

  if (warp >= EPI && warp < EPI + 4) {
    // ---- loaders: group 0 the even rows, group 1 the odd ones ----
    const int group = (warp - EPI) >> 1, lt = tid - 32 * EPI - group * TC_LOADERS;
    const int kg = lt % CG, c0 = lt / CG;  // a thread's channel group and first cell; then every TC_LOADERS / CG cells
    int g0 = 0, s0 = 0;
    while (ok && walk.next(A)) {
      const int cells = min(TC_BX, A.X - walk.x0 + 2);  // from x0 - 1 to the tile's or the volume's edge + 1
      for (int r = 0; r < walk.n + 2; ++r) {
        const int g = g0 + r;
        if ((g & 1) != group) continue;
        const int need = r >= TC_NR ? s0 + r - TC_NR : s0 - 1;  // the last step that read this slot
        if (need >= 0 && !(ok = mbar_wait_limited(done0 + 8u * (need & 3), (need >> 2) & 1))) break;
        const int y = walk.ya - 1 + r;
        const unsigned dst0 = rows0 + (unsigned)(g % TC_NR) * SLOTB;
        const bool iny = y >= 0 && y < A.Y;
#pragma unroll
        for (int pz = 0; pz < 3; ++pz) {
          int zz = walk.z + pz - 1;
          if (A.zper) zz = zz < 0 ? zz + A.Z : (zz >= A.Z ? zz - A.Z : zz);
          const bool inp = iny && zz >= 0 && zz < A.Z;
          const bf16* src = A.in + (inp ? ((((long long)walk.b * A.Z + zz) * A.Y + y) * A.X + walk.x0 - 1) * CIP + kg * 8 : 0);
          const unsigned dst = dst0 + (unsigned)((pz * CG + kg) * RP) * 16u;
#pragma unroll 3
          for (int c = c0; c < cells; c += TC_LOADERS / CG) {
            const int x = walk.x0 - 1 + c;
            const bool in = inp && x >= 0 && x < A.X;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst + c * 16u),
                         "l"(in ? src + (long long)c * CIP : A.in), "r"(in ? 16 : 0)
                         : "memory");
          }
        }
        asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");  // the tensor cores read it next
        mbar_arrive1(full0 + 8u * (g % TC_NR));
      }
      g0 += walk.n + 2;
      s0 += walk.n;
    }
  } else if (warp == EPI + 4) {
    // ---- MMA issue: the warp walks and waits as one, one elected lane issues ----
    const unsigned tm = __shfl_sync(0xffffffffu, tmem0, 0);
    const bool lead = elect_one();
    const unsigned long long rdesc = smem_desc(rows0, RP * 16u, 128u), wdesc = smem_desc(w0, N * 16u, 128u);
    int g0 = 0, s = 0;
    while (ok && walk.next(A)) {
      for (int r = 0; r < walk.n + 2 && ok; ++r) {
        const int g = g0 + r;
        ok = __all_sync(0xffffffffu, mbar_wait_limited(full0 + 8u * (g % TC_NR), (g / TC_NR) & 1));
        if (!ok || r < 2) continue;
        if (s >= 2 && !(ok = __all_sync(0xffffffffu, mbar_wait_limited(epi0 + 8u * (s & 1), ((s >> 1) - 1) & 1)))) break;
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        const unsigned long long row[3] = {rdesc + (unsigned)((g - 2) % TC_NR) * (SLOTB / 16u),
                                           rdesc + (unsigned)((g - 1) % TC_NR) * (SLOTB / 16u),
                                           rdesc + (unsigned)(g % TC_NR) * (SLOTB / 16u)};
        if (lead) tc_issue<CIP, N>(row, wdesc, tm + (s & 1) * COLW, done0 + 8u * (s & 3));
        __syncwarp();
        ++s;
      }
      g0 += walk.n + 2;
    }
    if (s > 0) mbar_wait_limited(done0 + 8u * ((s - 1) & 3), ((s - 1) >> 2) & 1);  // nothing in flight when it leaves
  } else if (warp < EPI) {
    // ---- epilogue: warps w and w + 4 the lanes of quarter w, 16 columns each ----
    const int lane_cell = tid & 127, c0 = (warp >> 2) * 16;
    int s = 0;
    while (ok && walk.next(A)) {
      for (int i = 0; i < walk.n; ++i, ++s) {
        ok = __all_sync(0xffffffffu, mbar_wait_limited(done0 + 8u * (s & 3), (s >> 2) & 1));
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        float acc[16];
        const unsigned taddr = tmem0 + (s & 1) * COLW + (unsigned)c0 + ((unsigned)((warp & 3) * 32) << 16);
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
            : "=f"(acc[0]), "=f"(acc[1]), "=f"(acc[2]), "=f"(acc[3]), "=f"(acc[4]), "=f"(acc[5]), "=f"(acc[6]),
              "=f"(acc[7]), "=f"(acc[8]), "=f"(acc[9]), "=f"(acc[10]), "=f"(acc[11]), "=f"(acc[12]), "=f"(acc[13]),
              "=f"(acc[14]), "=f"(acc[15])
            : "r"(taddr));
        asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
        mbar_arrive1(epi0 + 8u * (s & 1));  // in registers: the accumulator may be overwritten
        const int gx = walk.x0 + lane_cell;
        if (gx < A.X)
          tc_epilogue<COP, (COP < 16 ? COP : 16), MODE>(
              A, bias, acc, (((long long)walk.b * A.Z + walk.z) * A.Y + walk.ya + i) * A.X + gx, c0);
      }
    }
  }
  if (!ok) atomicOr(flag, FLAG_TIMEOUT);
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  __syncwarp();
  if (warp == EPI + 4) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem0), "r"(COLS));
}

template <int CIP, int N, int COP, int MODE>
static cudaError_t conv_tc_go(const ConvArgs& a, const bf16* wtc, int* flag, cudaStream_t s) {
  const size_t bytes = (size_t)TC_NR * 3 * (CIP / 8) * TcPitch<CIP>::value * 16 + (size_t)NTAP * CIP * N * sizeof(bf16) + 32 * sizeof(float) + 128;
  static std::atomic<unsigned long long> done{0};  // per-device bit; host threads may race here
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (!(dev < 64 && ((done.load(std::memory_order_acquire) >> dev) & 1ull))) {
    e = cudaFuncSetAttribute(conv_tc_kernel<CIP, N, COP, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)bytes);
    if (e != cudaSuccess) return e;
    if (dev < 64) done.fetch_or(1ull << dev, std::memory_order_acq_rel);
  }
  if (((uintptr_t)a.in & 15u) != 0) return cudaErrorMisalignedAddress;
  int nsm = 0;
  e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  // resident CTAs by the kernel's launch bounds and shared memory (228 KB an SM, 1 KB of it a CTA's own; the
  // occupancy query answered 1 for the two that ncu counts: layer 1 119 -> 82 us)
  constexpr int occ = CIP == 16 ? 2 : 1;
  const long long tiles = (long long)((a.X + TC_M - 1) / TC_M) * a.Y * a.Z * a.B;
  long long grid = (long long)nsm * occ;
  if (grid > tiles) grid = tiles;
  conv_tc_kernel<CIP, N, COP, MODE><<<(unsigned)grid, TcWarps<N>::threads, bytes, s>>>(a, wtc, flag, tiles);
  return cudaGetLastError();
}

// layers 1..3 forward; layers 3 and 2 backward-data (taps mirrored, channels swapped, x SiLU')
cudaError_t launch_conv(int layer, int mode, const ConvArgs& a, int* flag, cudaStream_t s) {
  if (mode == FWD_SILU && layer == 1) return conv_tc_go<P0, P1, P1, FWD_SILU>(a, a.w, flag, s);
  if (mode == FWD_SILU && layer == 2) return conv_tc_go<P1, P2, P2, FWD_SILU>(a, a.w, flag, s);
  if (mode == FWD_LINEAR && layer == 3) return conv_tc_go<P2, 16, P3, FWD_LINEAR>(a, a.w, flag, s);
  if (mode == BWD_DSILU && layer == 3) return conv_tc_go<16, P2, P2, BWD_DSILU>(a, a.w, flag, s);  // dY -> dZ2
  if (mode == BWD_DSILU && layer == 2) return conv_tc_go<P2, P1, P1, BWD_DSILU>(a, a.w, flag, s);  // dZ2 -> dZ1
  return cudaErrorInvalidValue;
}

}  // namespace learn
}  // namespace gbcfd
