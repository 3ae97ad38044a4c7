// BF16 implicit-GEMM 3D convolutions (FP32 accumulation) for the learned initial guess, plus
// the small kernels of its training step (input packing, loss gradient, Adam, prediction).
//
// Layout: activations channels-last BF16 [D][H][W][16] (channel counts padded to 16, padded
// channels are zero); weights BF16 [tap][co][ci] = [27][16][16], tap = 9(dz+1)+3(dy+1)+(dx+1);
// zero padding of 1 at the grid boundary.
//
// Forward / backward-data (conv3d_fwd): the tcgen05 tensor-core kernel below (TMA-staged
// input planes, one M128 N48 K16 MMA per (dy, dx) for the three dz, FP32 accumulators in tensor
// memory).  The backward-data pass is the same kernel on flipped, transposed weights with the ReLU
// mask of the layer input applied in the epilogue.
// Weight gradient (conv3d_wgrad): tcgen05 as well, (dy, dz, input channel) stacked into M and (dx,
// output channel) into N, K = voxels; each row's K-major operand is written once per run of rows
// with ldmatrix.trans / stmatrix (see k_conv3d_wgrad_tc), then a fixed-order reduction over blocks
// (deterministic).
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>

#include "pk_tile.cuh"

namespace pk {

constexpr int kCh = 16;         // channels (padded)

// Units [u, u1) of block b of G: equal shares, the first `units % G` blocks one more.
__device__ __forceinline__ void unit_share(int units, int& u, int& u1) {
  const int b = blockIdx.x, G = gridDim.x, base = units / G, rem = units - base * G;
  u = b * base + min(b, rem);
  u1 = u + base + (b < rem ? 1 : 0);
}

struct ConvArgs {
  const __nv_bfloat16* X;     // input activations [D][H][W][16]
  const __nv_bfloat16* Wt;    // weights [27][16 co][16 ci]
  const float* bias;          // [16] or null
  __nv_bfloat16* Y;           // output BF16 [D][H][W][16] (unless out_f32)
  float* Yf;                  // output FP32 channel 0 [D][H][W] (out_f32)
  const __nv_bfloat16* mask;  // ReLU mask source [D][H][W][16] or null
  int D, H, W;
  int relu;
  int out_f32;
};

// ---------------------------------------------------------------- tcgen05 forward kernel
// Implicit GEMM on the 5th-generation tensor cores: an M = 128 tile of voxels (8 along x by 16 along
// y at one z), K = 16 input channels per tap.  Input-stationary in z: the tile's input plane z (18
// rows x 10 voxels with the halo) is multiplied once with the taps of all three dz, N = 48 columns =
// (dz = -1, 0, +1) x 16 output channels, nine MMAs (dy, dx) per plane; column block dz is that
// plane's share of the outputs at z + 1, z and z - 1, and an output tile is the sum of three blocks
// of three neighbouring planes, added in the order dz = -1, 0, +1 (each block accumulates its nine
// taps in order: the same products and sums as one MMA per tap).  So a plane is staged once and its
// operand rows are read by 9 MMAs, where one MMA per tap and output tile staged every plane three
// times and read it 27 times: an M128 MMA reads 4 KB of A whatever N is, 32 clocks of shared-memory
// bandwidth, which bounds so narrow a product.
// A block takes a run of (column tile, z) units in z order; warp 0 issues the TMA copies (two
// [18][10][8] boxes per plane, the halo outside the grid filled with zeros), warps 1 and 2 the MMAs
// of every other plane (one warp's waits between two planes left the tensor pipe idle for as long as
// the nine MMAs take: 930 clocks per plane where the MMAs are 480), and two groups of four warps take
// the output tiles in turn (tcgen05.ld, bias, ReLU or mask, BF16 store).  Planes pass through
// kTcStages staging buffers and kTcSlots accumulator slots in tensor memory; a slot is free once the
// (up to three) output tiles that read it have.  One block per SM.
// Measured (launches back to back): 64^3 17.9 us before (one MMA per tap, two blocks per SM, plain
// launches), 10.6 now (with plain launches 12.2, and 14.7 with one MMA warp); 72^3: 22.9 -> 12.0; 32^3:
// 10.3 -> 10.6, which is the launch, the prologue (barriers, tensor memory, weights: 1.2 us) and one run's
// latency.  The 16.8 MB in and out take 2.4 us of memory time.
// A box lands in the no-swizzle K-major layout of the MMA's A operand: a core matrix is 8
// voxels consecutive in x (8 x 16 bytes), the two K halves are kTcHalf bytes apart (leading
// byte offset) and consecutive y rows kTcRow bytes apart (stride byte offset); a tap (dy, dx) is the
// same descriptor with its start moved.  Every mbarrier wait is bounded (2 s): a wait that runs out
// sets a device flag (pk_conv3d_check reports PK_TIMEOUT), and the block waits (bounded) for what it
// issued, frees its tensor memory and returns.

constexpr int kTcX = 8, kTcY = 16;                  // tile: 8 x 16 voxels = M 128
constexpr int kTcBx = kTcX + 2, kTcBy = kTcY + 2;   // staged block with the halo
constexpr int kTcRow = kTcBx * 16;                  // bytes between staged y rows (SBO)
constexpr int kTcBox = kTcBy * kTcRow;              // bytes of one [18][10][8] box (2880)
constexpr int kTcHalf = (kTcBox + 127) & ~127;      // box pitch, 128-byte aligned (LBO)
constexpr int kTcPlane = 2 * kTcHalf;               // one staged plane, 5,888 bytes
constexpr int kTcStages = 16;
constexpr int kTcN = 48;                            // (dz, output channel)
constexpr int kTcWTap = kTcN * 32;                  // weights of one (dy, dx): 48 rows x 16 channels
constexpr int kTcW = 9 * kTcWTap;                   // 13,824 bytes
constexpr int kTcSmem = kTcStages * kTcPlane + kTcW;
constexpr int kTcSlots = 10;                        // accumulators of 48 columns
constexpr uint32_t kTcCols = 512;                   // tensor memory (480 columns in use)
constexpr int kTcMma = 2;                            // MMA warps: planes in turn
constexpr int kTcThreads = 32 * (1 + kTcMma + 8);   // copies, MMAs, two epilogue groups of four warps

__device__ int g_conv_timeout = 0;

__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  // shared-memory matrix descriptor: start >> 4 (bits 0-13), LBO >> 4 (16-29), SBO >> 4
  // (32-45), fixed 0b001 (46-48), base offset 0, relative LBO, no swizzle (61-63 = 0)
  return (uint64_t)((saddr & 0x3FFFF) >> 4) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | (1ull << 46);
}

// instruction descriptor, kind::f16: D FP32 (bits 4-5 = 1), A and B BF16 (bits 7-9, 10-12 =
// 1), both K-major (bits 15, 16 = 0), N >> 3 (bits 17-22), M >> 4 (bits 24-28)
template <int M>
constexpr uint32_t kTcIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kTcN >> 3) << 17) |
                              ((uint32_t)(M >> 4) << 24);

template <int M = 128>
__device__ __forceinline__ void tc_mma(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(kTcIdesc<M>), "r"(accumulate)
      : "memory");
}

// One lane of a converged warp.  The MMA warps run their loops converged and issue under this
// predicate: descriptors and loop state then live in uniform registers, where a branch on the lane
// number costs a move per operand (measured: 146 clocks per MMA issued, 5 times what it takes).
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(p)::"memory");
  return p != 0;
}

__device__ __forceinline__ void tc_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   smem_addr(bar))
               : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void proxy_fence() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// 16 FP32 columns of this thread's tensor-memory lane.
__device__ __forceinline__ void tc_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int k = 0; k < 16; ++k) v[k] = __uint_as_float(r[k]);
}

// One [18][10][8] box of the channels-last input at (c, x, y, z) (x, y, z may lie outside
// the grid: zero fill) into shared memory, completion on `bar`.
__device__ __forceinline__ void tc_tma_box(uint32_t dst, const CUtensorMap* map, int c, int x, int y,
                                           int z, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, "
      "%4, %5}], [%6];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c), "r"(x), "r"(y), "r"(z), "r"(smem_addr(bar))
      : "memory");
}

__device__ __forceinline__ void mbar_arrive_n(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

// The runs of a block's units [u0, u1), unit = column tile * D + z: planes [za, zb) of one column.
struct TcRuns {
  int u, u1, D, col, za, zb;
  __device__ __forceinline__ TcRuns(int units, int D_) : D(D_) { unit_share(units, u, u1); }
  __device__ __forceinline__ bool next() {
    if (u >= u1) return false;
    col = u / D;
    za = u - col * D;
    zb = min(D, za + (u1 - u));
    u += zb - za;
    return true;
  }
};

__global__ void __launch_bounds__(kTcThreads, 1) k_conv3d_tc(const __grid_constant__ CUtensorMap xmap, ConvArgs a) {
  extern __shared__ __align__(1024) unsigned char smem_tc[];
  unsigned char* wsm = smem_tc + kTcStages * kTcPlane;     // weights [dy dx][k half][dz, co][8 ci]
  __shared__ __align__(8) uint64_t full_bar[kTcStages];    // plane loaded
  __shared__ __align__(8) uint64_t empty_bar[kTcStages];   // plane read by its MMAs
  __shared__ __align__(8) uint64_t done_bar[kTcSlots];     // accumulator complete
  __shared__ __align__(8) uint64_t free_bar[kTcSlots];     // accumulator read by its output tiles
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tx = (a.W + kTcX - 1) / kTcX, ty = (a.H + kTcY - 1) / kTcY;
  const int units = tx * ty * a.D;  // (< 2^31: checked by the host)
  // (one barrier per thread: initialised one after the other they took 0.5 us of every launch)
  if (threadIdx.x < kTcStages) {
    mbar_init(&full_bar[threadIdx.x], 1);
    mbar_init(&empty_bar[threadIdx.x], 1);
    if (threadIdx.x < kTcSlots) {
      mbar_init(&done_bar[threadIdx.x], 1);
      mbar_init(&free_bar[threadIdx.x], 3 * 4);  // three output tiles, a warp of four each
    }
    mbar_fence_init();
    if (threadIdx.x == 0) abort_flag = 0;
  }
  __syncthreads();  // the barriers are in place: the copies start while the other warps go on
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tmem_slot)),
                 "r"(kTcCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  griddep_wait();  // nothing in memory is read or written before
  for (int e = (int)threadIdx.x - 32; warp > 0 && e < 27 * kCh * 2; e += kTcThreads - 32) {
    const int half = e & 1, row = e >> 1, t = row / kCh, co = row % kCh;
    *reinterpret_cast<uint4*>(wsm + (t % 9) * kTcWTap + half * (kTcN * 16) + ((t / 9) * kCh + co) * 16) =
        __ldcg(reinterpret_cast<const uint4*>(a.Wt + row * kCh + 8 * half));
  }
  uint32_t tmem = 0;
  if (warp > 0) {
    proxy_fence();  // the weights are read by the tensor core (async proxy)
    tc_fence_before();
    asm volatile("bar.sync 1, %0;" ::"r"(kTcThreads - 32) : "memory");
    tc_fence_after();
    tmem = tmem_slot;
  }
  const uint32_t w_addr = smem_addr(wsm), s_base = smem_addr(smem_tc);
  volatile int* const stop = &abort_flag;
  TcRuns run(units, a.D);
  if (warp == 0) {
    if (lane == 0) {
      int q = 0;
      while (!*stop && run.next()) {
        const int x0 = (run.col % tx) * kTcX, y0 = (run.col / tx) * kTcY;
        for (int z = run.za - 1; z <= run.zb; ++z, ++q) {
          const int s = q % kTcStages;
          if (q >= kTcStages && !mbar_wait(&empty_bar[s], (q / kTcStages - 1) & 1)) {
            *stop = 1;
            break;
          }
          mbar_expect_tx(&full_bar[s], 2 * kTcBox);
          for (int h = 0; h < 2; ++h)
            tc_tma_box(s_base + s * kTcPlane + h * kTcHalf, &xmap, 8 * h, x0 - 1, y0 - 1, z, &full_bar[s]);
        }
      }
      // bounded waits for the copies in flight before the block leaves
      for (int p = max(0, q - kTcStages); p < q; ++p)
        if (!mbar_wait(&full_bar[p % kTcStages], (p / kTcStages) & 1)) *stop = 1;
    }
  } else if (warp <= kTcMma) {
    // descriptors differ by their start address (bits 0-13, in 16-byte units)
    const uint64_t wd = tc_desc(w_addr, kTcN * 16, 128), xd = tc_desc(s_base, kTcHalf, kTcRow);
    int q = 0, s = 0, d = 0, use_s = 0, use_d = 0;  // plane, its stage and slot and their uses so far
    int mine = -1;                                  // this warp's last plane
    bool ok = true;
    while (ok && run.next()) {
      for (int z = run.za - 1; z <= run.zb; ++z, ++q, s = s + 1 == kTcStages ? (++use_s, 0) : s + 1,
               d = d + 1 == kTcSlots ? (++use_d, 0) : d + 1) {
        if (q % kTcMma != warp - 1) continue;
        ok = mbar_wait(&full_bar[s], use_s & 1) && (use_d == 0 || mbar_wait(&free_bar[d], (use_d - 1) & 1));
        ok = !__any_sync(0xffffffffu, !ok || *stop);
        if (!ok) break;
        tc_fence_after();
        const uint64_t xs = xd + (uint64_t)(s * (kTcPlane >> 4));
        const uint32_t acc = tmem + d * kTcN;
        if (elect_one()) {
#pragma unroll
          for (int i = 0; i < 9; ++i)
            tc_mma(acc, xs + (((i / 3) * kTcRow + (i % 3) * 16) >> 4), wd + i * (kTcWTap >> 4), i > 0 ? 1u : 0u);
          tc_commit(&empty_bar[s]);
          tc_commit(&done_bar[d]);
        }
        __syncwarp();
        mine = q;
      }
    }
    if (!ok) *stop = 1;
    // the last commit covers every MMA this warp issued
    if (mine >= 0 && !mbar_wait(&done_bar[mine % kTcSlots], (mine / kTcSlots) & 1)) *stop = 1;
  } else {
    const int grp = (warp - 1 - kTcMma) >> 2, quarter = warp & 3;  // a warp reads its quarter of the lanes
    const float bl = a.bias && lane < 16 ? __ldcg(a.bias + lane) : 0.f;
    float bias[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) bias[c] = __shfl_sync(0xffffffffu, bl, c);
    const int m = 32 * quarter + lane;
    int q0 = 0, k = 0;  // first plane of the run, output tiles so far
    while (!__any_sync(0xffffffffu, *stop) && run.next()) {
      const int x = (run.col % tx) * kTcX + m % kTcX, y = (run.col / tx) * kTcY + m / kTcX;
      const int c0 = q0 + 1, c1 = q0 + run.zb - run.za;  // planes at the centre of the output tiles
      for (int c = c0; c <= c1; ++c, ++k) {
        if ((k & 1) != grp) continue;
        for (int p = c - 1; p <= c + 1; ++p)
          if (!mbar_wait(&done_bar[p % kTcSlots], (p / kTcSlots) & 1)) *stop = 1;
        if (__any_sync(0xffffffffu, *stop)) break;
        tc_fence_after();
        float o[16];
        {
          // the three partial sums (taps with dz = -1, 0, +1), added in that order
          const uint32_t row = tmem + ((uint32_t)(32 * quarter) << 16);
          float p1[16], p2[16];
          tc_ld16(row + ((c - 1) % kTcSlots) * kTcN, o);
          tc_ld16(row + (c % kTcSlots) * kTcN + 16, p1);
          tc_ld16(row + ((c + 1) % kTcSlots) * kTcN + 32, p2);
#pragma unroll
          for (int j = 0; j < 16; ++j) o[j] = (o[j] + p1[j]) + p2[j];
        }
        tc_fence_before();
        __syncwarp();
        if (lane < 3) {
          // slot of plane p: read by the output tiles centred at p - 1, p, p + 1 of this run; the
          // first of them arrives for those that the run does not have
          const int p = c - 1 + lane, lo = max(c0, p - 1), hi = min(c1, p + 1);
          mbar_arrive_n(&free_bar[p % kTcSlots], c == lo ? 1 + (3 - (hi - lo + 1)) : 1);
        }
        const int z = run.za + (c - c0);
        if (y < a.H && x < a.W) {
          const size_t v = ((size_t)z * a.H + y) * a.W + x;
          if (a.out_f32) {
            a.Yf[v] = o[0] + bias[0];
          } else {
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              o[j] += bias[j];
              if (a.relu) o[j] = fmaxf(o[j], 0.f);
            }
            if (a.mask) {
              const uint4 m0 = __ldcg(reinterpret_cast<const uint4*>(a.mask + v * kCh));
              const uint4 m1 = __ldcg(reinterpret_cast<const uint4*>(a.mask + v * kCh + 8));
              const __nv_bfloat16* mb0 = reinterpret_cast<const __nv_bfloat16*>(&m0);
              const __nv_bfloat16* mb1 = reinterpret_cast<const __nv_bfloat16*>(&m1);
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                if (!(__bfloat162float(mb0[j]) > 0.f)) o[j] = 0.f;
                if (!(__bfloat162float(mb1[j]) > 0.f)) o[8 + j] = 0.f;
              }
            }
            uint4 p0, p1;
            __nv_bfloat162* r0 = reinterpret_cast<__nv_bfloat162*>(&p0);
            __nv_bfloat162* r1 = reinterpret_cast<__nv_bfloat162*>(&p1);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              r0[j] = __floats2bfloat162_rn(o[2 * j], o[2 * j + 1]);
              r1[j] = __floats2bfloat162_rn(o[8 + 2 * j], o[8 + 2 * j + 1]);
            }
            *reinterpret_cast<uint4*>(a.Y + v * kCh) = p0;
            *reinterpret_cast<uint4*>(a.Y + v * kCh + 8) = p1;
          }
        }
      }
      q0 += run.zb - run.za + 2;
    }
  }
  tc_fence_before();
  __syncthreads();
  griddep_trigger();
  if (threadIdx.x == 0 && abort_flag) atomicExch(&g_conv_timeout, 1);
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTcCols) : "memory");
  }
}

// ---------------------------------------------------------------- tcgen05 weight gradient
// dW[tap][co][ci] = sum_v G[v][co] A[v + s][ci] (s the tap's shift) as implicit GEMMs on the tensor
// cores, K = voxels.  With s = (dz, dy, dx), sum_v G[v] A[v + s] = sum_k A[k + (dz, dy, 0)]
// G[k - (0, 0, dx)]: a product of M rows (dy, dz, ci) and N = 48 columns (dx, co) per 16 voxels.
// A block walks y along runs of rows (z, y) of a 64-voxel x segment.  A row of A is an operand row
// group of 16 channels x 64 voxels (2 KB); the groups of a run lie in y order, three (dz) per y, so
// the nine groups around row y are consecutive and the next y uses six of them again: each row of A
// is transposed once per run where a separate operand per output row transposed eight.  One MMA of
// M = 128 takes the first eight groups, a second one of M = 64 (whose other rows are not read) the
// ninth, (1, 1); both accumulate in tensor memory over the block's rows.
// A loader warp brings the rows (three of A and one of G per step, 66 voxels with the x halo, zeros
// outside the grid) as two TMA boxes into a staging ring (a copy per row, issued by a lane each, took
// 950 clocks per step and set the pace); two groups of eight warps take the steps in turn (a step is a
// chain of some 1,200 clocks of waits, loads, stores, fence and arrivals, twice what its MMAs take) and
// write the operands with ldmatrix.trans + stmatrix, which turn [voxel][channel] 8 x 8 blocks into the
// [channel][voxel] core matrices of the no-swizzle K-major layout (K-adjacent core matrices 128 bytes
// apart, M- or N-adjacent 1 KB).  (Loading the fragments from global memory instead, 4 bytes of a voxel
// per thread, took 560 clocks of issue per step.)  Two warps issue the MMAs of every other output row,
// each into accumulators of its own (one warp's waits and issue took 1,000 clocks per row).  Runs have
// at most kWgRun rows: two run buffers alternate, and four buffers of G (its three dx shifts) rotate.
// One more warp sums the block's part of db from global memory, over segments b, b + G, b + 2 G, ... of
// the whole grid instead of the rows that the block multiplies.  G of a loss sums to nearly nothing over
// the grid and is smooth along it: the sum over a run of neighbouring rows is large and of one sign, over
// rows from everywhere it has cancelled already, and what the block sums are rounded to is what db is off
// by.  (Runs of rows moved db of the last layer by up to 6e-5 of itself against these sums, in the worst of
// 400 random boxes of 12 to 72 voxels a side.)
// Every wait is bounded (a wait that runs out sets the device flag that pk_conv3d_check reports, and
// the block waits, bounded, for what it issued before it frees its tensor memory).  At the end each
// thread reads its accumulator lane into the block's partial; a fixed-order reduction over blocks
// follows.
// Measured with that reduction (64^3, launches back to back with programmatic launches): 32.9 us before
// (an im2col operand per 64-voxel segment, plain launches), 17.5 us now; 72^3 (two segments per row, the
// second mostly empty): 68.7 -> 34.6; 32^3: 14.4 -> 11.4.  The rest is issue and wait latency: tensor pipe
// and memory are idle for most of it.
constexpr int kWgSeg = 64;                       // voxels (K) per segment
constexpr int kWgRun = 10;                       // output rows per run
constexpr int kWgSlots = kWgRun + 2;             // y rows of A per run
constexpr int kWgRowOp = 2048;                   // one operand row group: 16 channels x 64 voxels
constexpr int kWgA = kWgSlots * 3 * kWgRowOp;    // a run's A operand (72 KB)
constexpr int kWgG = 3 * kWgRowOp;               // G of a row, three dx shifts (6 KB)
constexpr int kWgGs = 4;                         // (even: see below)
constexpr int kWgRow = (kWgSeg + 2) * 32;        // a staged row: 66 voxels x 16 channels BF16
constexpr int kWgStageG = (3 * kWgRow + 127) & ~127;  // A at dz = -1, 0, +1, then G, 128-byte aligned
constexpr int kWgStage = (kWgStageG + kWgRow + 127) & ~127;
constexpr int kWgStages = 6;
constexpr int kWgSmem = 2 * kWgA + kWgGs * kWgG + kWgStages * kWgStage;  // (the second MMA reads 6 KB past a run)
constexpr int kWgReady = 16;                     // ready barriers (the writers are at most 8 steps ahead)
constexpr int kWgMaxBlocks = 256;
constexpr int kWgMma = 2;                        // MMA warps: output rows in turn, accumulators of their own
constexpr uint32_t kWgCols = 128 * kWgMma;       // tensor memory: 48 columns at 0 and at 64 for each
constexpr int kWgWarps = 8;                      // warps that write a step's operands
constexpr int kWgGroups = 2;                     // groups of them, fill steps in turn
constexpr int kWgThreads = 32 * kWgWarps * kWgGroups;
constexpr int kWgBlock = kWgThreads + 32 * (2 + kWgMma);  // ... the loader warp, the MMA warps, the warp of db
constexpr int kWgDbRows = 16;                    // chains of db per channel
static_assert(kWgDbRows * kCh == 32 * 8 && kWgSeg % kWgDbRows == 0, "a lane of the db warp: 8 channels of a chain");
// A group's steps with an output row are every other row, the rows of one MMA warp, and an even number
// of G buffers keeps a buffer with that pair: its phases complete in order, and no wait can take the
// phase before the last for the one it needs.
static_assert(kWgGroups == kWgMma && kWgGs % kWgGroups == 0 && kWgStages % kWgGroups == 0, "buffers and their pairs");
static_assert(kWgGs * kWgG >= 3 * kWgRowOp && kWgSmem <= 226 * 1024, "the second MMA's unused rows stay in bounds");

__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}

__device__ __forceinline__ void stsm4(uint32_t addr, const uint32_t (&r)[4]) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(r[0]), "r"(r[1]),
               "r"(r[2]), "r"(r[3])
               : "memory");
}

// The fill steps of a block's units [u, u1), unit = (segment * D + z) * H + y: per run of L rows
// from ya, steps t = 0 .. L + 1 bring row ya - 1 + t of A and, from t = 2 on, row ya + t - 2 of G,
// after which that output row can be multiplied.
struct WgSteps {
  int u, u1, D, H;
  int seg, z, ya, L, t, run;
  __device__ __forceinline__ WgSteps(int units, int D_, int H_) : D(D_), H(H_), L(0), t(1), run(-1) {
    unit_share(units, u, u1);
  }
  __device__ __forceinline__ bool next() {
    if (++t < L + 2) return true;
    if (u >= u1) return false;
    const int zs = u / H;
    ya = u - zs * H;
    seg = zs / D;
    z = zs - seg * D;
    L = min(kWgRun, min(H - ya, u1 - u));
    u += L;
    t = 0;
    ++run;
    return true;
  }
};

// The block's part of db, in one warp: chain i = 0 .. 15 of a channel adds voxels i, i + 16, i + 32, i + 48
// of segments b, b + G, ... (unit numbers (z, y, segment), the segment fastest) one after the other.  A
// lane holds 8 channels of a chain, so a load of the warp is 16 voxels, 512 bytes.  One segment in flight:
// the warp keeps pace with the MMAs (1,100 clocks a row), and two or four in flight raise the kernel's
// registers from 54 to 80 and 96 (64^3: 17.5, 17.6 and 18.3 us; the sums in the writer warps 18.5).
__device__ __forceinline__ void wg_db(const __nv_bfloat16* G, int D, int H, int W, float (*dbs)[kCh]) {
  const int lane = threadIdx.x & 31, i = lane >> 1, c8 = 8 * (lane & 1);
  const int nseg = (W + kWgSeg - 1) / kWgSeg;
  const int64_t units = (int64_t)nseg * D * H;
  float db[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
  for (int64_t c = blockIdx.x; c < units; c += gridDim.x) {
    const int64_t zy = c / nseg;
    const int x0 = (int)(c - zy * nseg) * kWgSeg + i;
    uint4 g[kWgSeg / kWgDbRows];
#pragma unroll
    for (int k = 0; k < kWgSeg / kWgDbRows; ++k)
      g[k] = x0 + kWgDbRows * k < W
                 ? __ldcg(reinterpret_cast<const uint4*>(G + (zy * W + x0 + kWgDbRows * k) * kCh + c8))
                 : make_uint4(0, 0, 0, 0);
#pragma unroll
    for (int k = 0; k < kWgSeg / kWgDbRows; ++k) {
      const __nv_bfloat16* v = reinterpret_cast<const __nv_bfloat16*>(&g[k]);
#pragma unroll
      for (int q = 0; q < 8; ++q) db[q] += __bfloat162float(v[q]);
    }
  }
#pragma unroll
  for (int q = 0; q < 8; ++q) dbs[i][c8 + q] = db[q];
}

__global__ void __launch_bounds__(kWgBlock, 1) k_conv3d_wgrad_tc(const __grid_constant__ CUtensorMap amap,
                                                                 const __grid_constant__ CUtensorMap gmap,
                                                                 const __nv_bfloat16* G, float* partial,
                                                                 float* partial_db, int D, int H, int W) {
  extern __shared__ __align__(1024) unsigned char smem_wg[];
  __shared__ __align__(8) uint64_t full_bar[kWgStages];  // staging buffer loaded
  __shared__ __align__(8) uint64_t empty_bar[kWgStages]; // staging buffer read (8 warps)
  __shared__ __align__(8) uint64_t ready_bar[kWgReady];  // a fill step is written (8 warps)
  __shared__ __align__(8) uint64_t gfree_bar[kWgGs];     // a G buffer is read (MMA commit)
  __shared__ __align__(8) uint64_t afree_bar[2];         // a run buffer is read
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  __shared__ float dbs[kWgDbRows][kCh];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nseg = (W + kWgSeg - 1) / kWgSeg;
  const int units = nseg * D * H;  // (< 2^31: checked by the host)
  if (threadIdx.x < kWgReady) {
    const int k = threadIdx.x;
    mbar_init(&ready_bar[k], kWgWarps);
    if (k < kWgStages) mbar_init(&full_bar[k], 1);
    if (k < kWgStages) mbar_init(&empty_bar[k], kWgWarps);
    if (k < kWgGs) mbar_init(&gfree_bar[k], 1);
    if (k < 2) mbar_init(&afree_bar[k], kWgMma);
    mbar_fence_init();
    if (k == 0) abort_flag = 0;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tmem_slot)),
                 "r"(kWgCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const uint32_t base = smem_addr(smem_wg);
  volatile int* const stop = &abort_flag;
  griddep_wait();  // nothing in memory is read or written before
  WgSteps step(units, D, H);
  if (warp == kWgBlock / 32 - 1) {
    wg_db(G, D, H, W, dbs);
  } else if (warp > kWgThreads / 32) {
    // MMA warps: per output row 4 x 2 MMAs
    const int me = warp - kWgThreads / 32 - 1;
    const uint32_t acc = tmem + 128 * me;
    int last = -1;  // this warp's last row
    const uint64_t sd = tc_desc(base, 128, 1024);  // (start address in 16-byte units, bits 0-13)
    int f = 0, j = -1, jg = kWgGs - 1;  // fill steps, output row, j % kWgGs
    bool ok = true;
    while (step.next()) {
      if (step.t >= 2) {
        ++j;
        if (++jg == kWgGs) jg = 0;
      }
      ok = ok && mbar_wait(&ready_bar[f % kWgReady], (f / kWgReady) & 1);  // (of every step)
      ++f;
      if (step.t < 2 || j % kWgMma != me) {
        if (step.t == step.L + 1 && elect_one()) tc_commit(&afree_bar[step.run & 1]);
        continue;
      }
      ok = !__any_sync(0xffffffffu, !ok || *stop);
      if (!ok) break;
      tc_fence_after();
      const uint64_t ad = sd + (uint64_t)(((step.run & 1) * kWgA + (step.t - 2) * 3 * kWgRowOp) >> 4);
      const uint64_t gd = sd + (uint64_t)((2 * kWgA + jg * kWgG) >> 4);
      const uint32_t more = last >= 0 ? 1u : 0u;
      if (elect_one()) {
#pragma unroll
        for (int ks = 0; ks < kWgSeg / 16; ++ks) {
          tc_mma(acc, ad + ks * 16, gd + ks * 16, ks > 0 ? 1u : more);
          tc_mma<64>(acc + 64, ad + ((8 * kWgRowOp) >> 4) + ks * 16, gd + ks * 16, ks > 0 ? 1u : more);
        }
        tc_commit(&gfree_bar[jg]);
        if (step.t == step.L + 1) tc_commit(&afree_bar[step.run & 1]);
      }
      __syncwarp();
      last = j;
    }
    if (!ok) *stop = 1;
    // the last commit covers every MMA this warp issued
    if (last >= 0 && !mbar_wait(&gfree_bar[last % kWgGs], (last / kWgGs) & 1)) *stop = 1;
  } else if (warp == kWgThreads / 32) {
    // loader warp: one box of A's three rows (dz) and one of G's row per step
    if (lane == 0) {
      int f = 0, sb = 0, use = 0;
      while (!*stop && step.next()) {
        if (use > 0 && !mbar_wait(&empty_bar[sb], (use - 1) & 1)) {
          *stop = 1;
          break;
        }
        const int x0 = step.seg * kWgSeg - 1, y = step.ya - 1 + step.t;
        const uint32_t dst = base + 2 * kWgA + kWgGs * kWgG + sb * kWgStage;
        mbar_expect_tx(&full_bar[sb], step.t < 2 ? 3 * kWgRow : 4 * kWgRow);
        tc_tma_box(dst, &amap, 0, x0, y, step.z - 1, &full_bar[sb]);
        if (step.t >= 2) tc_tma_box(dst + kWgStageG, &gmap, 0, x0, y - 1, step.z, &full_bar[sb]);
        ++f;
        if (++sb == kWgStages) sb = 0, ++use;
      }
      // bounded waits for the copies in flight before the block leaves
      for (int p = max(0, f - kWgStages); p < f; ++p)
        if (!mbar_wait(&full_bar[p % kWgStages], (p / kWgStages) & 1)) *stop = 1;
    }
  } else {
    // writers: three jobs of four 8 x 8 blocks per fill step and warp, of the 12 of A (dz, channel
    // half, voxel half) and the 12 of G (dx, channel half, voxel half); warps 0 .. 3: A dz = -1, A
    // dz = +1, G dx = 0; warps 4 .. 7: A dz = 0, G dx = -1, G dx = +1
    const int grp = warp / kWgWarps;
    const bool low = (warp & 7) < 4;
    const int h = (warp >> 1) & 1, kg = 4 * (warp & 1);
    // this lane addresses row lane % 8 of block lane / 8: the voxel of the loads, the channel of the
    // stores
    const int vox = (kg + (lane >> 3)) * 8 + (lane & 7);
    const uint32_t dst = h * 1024 + (kg + (lane >> 3)) * 128 + (lane & 7) * 16;
    const uint32_t src = base + 2 * kWgA + kWgGs * kWgG + h * 16 + (vox + 1) * 32;  // (voxel -1 comes first)
    int f = 0, j = 0;
    for (; step.next(); j += step.t >= 2, ++f) {
      if (f % kWgGroups != grp) continue;
      const int sb = f % kWgStages;
      // the step's rows, the run's buffer (a group's first step of the run) and G buffer j
      bool ok = mbar_wait(&full_bar[sb], (f / kWgStages) & 1);
      if (step.t < kWgGroups && step.run >= 2) ok = ok && mbar_wait(&afree_bar[step.run & 1], (step.run / 2 - 1) & 1);
      if (step.t >= 2 && j >= kWgGs) ok = ok && mbar_wait(&gfree_bar[j % kWgGs], (j / kWgGs - 1) & 1);
      if (__any_sync(0xffffffffu, !ok || *stop)) {
        *stop = 1;
        break;
      }
      const uint32_t st = src + sb * kWgStage, sg = st + kWgStageG;
      const uint32_t ab = base + (step.run & 1) * kWgA + step.t * 3 * kWgRowOp + dst;
      const uint32_t gb = base + 2 * kWgA + (j % kWgGs) * kWgG + dst;
      const bool g = step.t >= 2;
      uint32_t r[3][4];
      if (low) {
        ldsm4t(r[0], st);
        ldsm4t(r[1], st + 2 * kWgRow);
        if (g) ldsm4t(r[2], sg);
        stsm4(ab, r[0]);
        stsm4(ab + 2 * kWgRowOp, r[1]);
        if (g) stsm4(gb + kWgRowOp, r[2]);
      } else {
        ldsm4t(r[0], st + kWgRow);
        if (g) ldsm4t(r[1], sg + 32);  // dx = -1: G at k + 1
        if (g) ldsm4t(r[2], sg - 32);  // dx = +1: G at k - 1
        stsm4(ab + kWgRowOp, r[0]);
        if (g) stsm4(gb, r[1]);
        if (g) stsm4(gb + 2 * kWgRowOp, r[2]);
      }
      proxy_fence();  // the operands are read by the tensor core (async proxy)
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&ready_bar[f % kWgReady]);
        mbar_arrive(&empty_bar[sb]);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  griddep_trigger();
  float* P = partial + (size_t)blockIdx.x * 27 * kCh * kCh;
  if (!abort_flag && warp < kWgThreads / 32) {
    // warps 0 .. 3: lanes 32 w .. + 31 of the first accumulator, row m = (group, ci); warp 4: lanes
    // 0 .. 15 of the second (group 8); the two MMA warps' sums are added (a block of one row has the
    // first alone).  Group g is (dy, dz) = (g / 3 - 1, g % 3 - 1); columns (dx, co)
    const int m = 32 * (warp & 3) + lane, ci = m & 15, g = warp < 4 ? m >> 4 : 8;
    int u0, u1;
    unit_share(units, u0, u1);
    const bool two = u1 - u0 >= kWgMma;
    if (warp <= 4) {
#pragma unroll 1
      for (int dx = 0; dx < 3; ++dx) {
        float v[16], v2[16];
        const uint32_t at = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (warp < 4 ? 0 : 64) + dx * 16;
        tc_ld16(at, v);
        tc_ld16(at + 128, v2);
        if (two) {
#pragma unroll
          for (int co = 0; co < 16; ++co) v[co] += v2[co];
        }
        const int tap = 9 * (g % 3) + 3 * (g / 3) + dx;
        if (warp < 4 || lane < 16) {
#pragma unroll
          for (int co = 0; co < 16; ++co) P[(tap * kCh + co) * kCh + ci] = v[co];
        }
      }
    }
    if (threadIdx.x < kCh) {
      float t = 0.f;
      for (int k = 0; k < kWgDbRows; ++k) t += dbs[k][threadIdx.x];
      partial_db[blockIdx.x * kCh + threadIdx.x] = t;
    }
  } else if (abort_flag && threadIdx.x == 0) {
    atomicExch(&g_conv_timeout, 1);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kWgCols) : "memory");
  }
}

// dW = sum over blocks of the partials (deterministic): a block of 8 warps per 32 outputs;
// warp w adds blocks w, w + 8, ... in order (their loads in flight together), then the 8 sums
// are added in warp order.
__global__ void __launch_bounds__(256) k_conv3d_wgrad_reduce(const float* partial, const float* partial_db,
                                                             int nblk, float* dW, float* db) {
  __shared__ float part[8][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int e = blockIdx.x * 32 + lane;
  constexpr int nw = 27 * kCh * kCh;
  float s = 0.f;
  griddep_trigger();
  griddep_wait();
  if (e < nw + kCh) {
    const float* src = e < nw ? partial + e : partial_db + (e - nw);
    const size_t stride = e < nw ? (size_t)nw : (size_t)kCh;
    constexpr int kPer = (kWgMaxBlocks + 7) / 8;  // every load of the thread in flight at once
    float v[kPer];
#pragma unroll
    for (int q = 0; q < kPer; ++q) v[q] = warp + 8 * q < nblk ? __ldcg(src + (size_t)(warp + 8 * q) * stride) : 0.f;
#pragma unroll
    for (int q = 0; q < kPer; ++q)
      if (warp + 8 * q < nblk) s += v[q];
  }
  part[warp][lane] = s;
  __syncthreads();
  if (warp == 0 && e < nw + kCh) {
    float t = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) t += part[w][lane];
    if (e < nw) dW[e] = t;
    else db[e - nw] = t;
  }
}

// Wf[26 - t][ci][co] = W[t][co][ci]: the weights of the backward-data convolution.
__global__ void k_conv3d_flip(const __nv_bfloat16* W, __nv_bfloat16* Wf) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= 27 * kCh * kCh) return;
  const int t = e / (kCh * kCh), co = (e / kCh) % kCh, ci = e % kCh;
  Wf[((26 - t) * kCh + ci) * kCh + co] = W[e];
}

// ------------------------------------------------------------------ training-step helpers

// Deterministic two-stage sums of up to 3 FP64 values over n (scratch: 3 x gridDim doubles,
// then the arrival counter as an unsigned at scratch[3 * gridDim]).
template <int NV, class F>
__device__ __forceinline__ void grid_sums(int n, double* scratch, F&& f, double (&out)[NV], bool& last) {
  double v[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) v[k] = 0.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) f(i, v);
  block_partials<NV>(v, scratch);
  unsigned int* counter = reinterpret_cast<unsigned int*>(scratch + 3 * gridDim.x);
  last = arrive_last(counter);
  if (last) {
    final_sums<NV>(scratch, out);
    __syncthreads();
    if (threadIdx.x == 0) *counter = 0;
  }
}

// A voxel's 16 channels: three given, the others zero.  Two 16-byte stores where the voxel is aligned.
__device__ __forceinline__ void ws_voxel(__nv_bfloat16* o, __nv_bfloat16 c0, __nv_bfloat16 c1, __nv_bfloat16 c2) {
  if (((uintptr_t)o & 15) == 0) {
    __nv_bfloat162 q[2];
    q[0].x = c0;
    q[0].y = c1;
    q[1].x = c2;
    q[1].y = __float2bfloat16_rn(0.f);
    uint4 lo = make_uint4(*reinterpret_cast<const unsigned int*>(&q[0]), *reinterpret_cast<const unsigned int*>(&q[1]), 0, 0);
    reinterpret_cast<uint4*>(o)[0] = lo;
    reinterpret_cast<uint4*>(o)[1] = make_uint4(0, 0, 0, 0);
  } else {
    o[0] = c0;
    o[1] = c1;
    o[2] = c2;
    for (int c = 3; c < kCh; ++c) o[c] = __float2bfloat16_rn(0.f);
  }
}

constexpr int kWsGrid = 608;  // four blocks per SM: a row's loads are a chain that many warps hide

// Residual of the linear extrapolation e = 2 x_{t-1} - x_{t-2} in row i:
// r = b_i - sum_j a_ij e_j (left to right, four entries' loads in flight); d = a_ii (1 where the row
// has no nonzero diagonal entry).
__device__ __forceinline__ void ws_row(const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                                       const double* __restrict__ va, const double* __restrict__ xm1,
                                       const double* __restrict__ xm2, const double* __restrict__ b, int i,
                                       double& r, double& d) {
  double s = 0.0;
  d = 0.0;
  const int j1 = __ldg(rp + i + 1);
  for (int j = __ldg(rp + i); j < j1; j += 4) {
    int c[4];
    double v[4], p[4], q[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      c[k] = j + k < j1 ? __ldg(ci + j + k) : -1;
      v[k] = j + k < j1 ? __ldg(va + j + k) : 0.0;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      p[k] = c[k] >= 0 ? __ldg(xm1 + c[k]) : 0.0;
      q[k] = c[k] >= 0 ? __ldg(xm2 + c[k]) : 0.0;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (c[k] >= 0) {
        s = fma(v[k], 2.0 * p[k] - q[k], s);
        if (c[k] == i) d = v[k];
      }
  }
  r = b[i] - s;
  if (d == 0.0) d = 1.0;
}

// What k_ws_rms leaves for k_ws_pack in the 32 bytes of a voxel of X16: r / d, r, d.
struct WsStash {
  double z, r, d, unused;
};
static_assert(sizeof(WsStash) == kCh * sizeof(__nv_bfloat16), "a voxel's 16 channels");

// scales = rms of (r / d, r, d) (1 where zero).  stash: X16 where it is 8-byte aligned, else null.
// Bound by FP64 issue: 26 operations per row of seven entries (11 us at 64^3), which the second pass
// over the rows that k_ws_pack made before doubled.
__global__ void __launch_bounds__(kBlock) k_ws_rms(int n, const int32_t* rp, const int32_t* ci,
                                                   const double* va, const double* xm1,
                                                   const double* xm2, const double* b,
                                                   double* scales, double* scratch, WsStash* stash) {
  double out[3];
  bool last;
  grid_sums<3>(n, scratch, [&](int i, double (&v)[3]) {
    double r, d;
    ws_row(rp, ci, va, xm1, xm2, b, i, r, d);
    const double z = r / d;
    if (stash) {
      stash[i].z = z;
      stash[i].r = r;
      stash[i].d = d;
    }
    v[0] = fma(z, z, v[0]);
    v[1] = fma(r, r, v[1]);
    v[2] = fma(d, d, v[2]);
  }, out, last);
  if (last && threadIdx.x == 0) {
    for (int k = 0; k < 3; ++k) {
      const double s = sqrt(out[k] / n);
      scales[k] = s > 0 ? s : 1.0;
    }
  }
}

// X16[v] = bf16((r/d)/s0, r/s1, d/s2, 0, ..., 0): the Jacobi-scaled residual of the
// extrapolation, the residual itself and the diagonal, each channel of order one.  The quotients by
// the scales are products with their reciprocals (formed once per block: an FP64 division is nine
// operations of the narrow FP64 pipe; the product is rounded to 24 and then 8 bits).
__global__ void k_ws_pack(int n, const int32_t* rp, const int32_t* ci, const double* va,
                          const double* xm1, const double* xm2, const double* b,
                          const double* scales, __nv_bfloat16* X16, int stashed) {
  __shared__ double inv[3];
  if (threadIdx.x < 3) inv[threadIdx.x] = 1.0 / scales[threadIdx.x];
  __syncthreads();
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  __nv_bfloat16* o = X16 + (size_t)v * kCh;
  double z, r, d;
  if (stashed) {
    const WsStash s = *reinterpret_cast<const WsStash*>(o);
    z = s.z;
    r = s.r;
    d = s.d;
  } else {
    ws_row(rp, ci, va, xm1, xm2, b, v, r, d);
    z = r / d;
  }
  const __nv_bfloat16 c[3] = {__float2bfloat16_rn((float)(z * inv[0])), __float2bfloat16_rn((float)(r * inv[1])),
                              __float2bfloat16_rn((float)(d * inv[2]))};
  ws_voxel(o, c[0], c[1], c[2]);
}

// target y = (x_t - 2 x_{t-1} + x_{t-2}) / s0 (what linear extrapolation misses, in units of
// the Jacobi-scaled residual); G[v][0] = bf16(2 (out - y) / n); loss = mean((out - y)^2).
__global__ void __launch_bounds__(kBlock) k_ws_loss(int n, const float* __restrict__ out, const double* __restrict__ xt,
                                                    const double* __restrict__ xm1, const double* __restrict__ xm2,
                                                    const double* scales, __nv_bfloat16* G,
                                                    double* loss, double* scratch) {
  const double is = 1.0 / scales[0], gn = 2.0 / n;
  const __nv_bfloat16 zero = __float2bfloat16_rn(0.f);
  double sum[1];
  bool last;
  grid_sums<1>(n, scratch, [&](int i, double (&v)[1]) {
    const double d = (double)out[i] - (xt[i] - 2.0 * xm1[i] + xm2[i]) * is;
    v[0] = fma(d, d, v[0]);
    ws_voxel(G + (size_t)i * kCh, __float2bfloat16_rn((float)(gn * d)), zero, zero);
  }, sum, last);
  if (last && threadIdx.x == 0) *loss = sum[0] / n;
}

// x_hat = 2 x_{t-1} - x_{t-2} + s0 out (out == nullptr: the extrapolation alone).
__global__ void k_ws_apply(int n, const float* out, const double* xm1, const double* xm2,
                           const double* scales, double* xhat) {
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  const double e = 2.0 * xm1[v] - xm2[v];
  xhat[v] = out ? fma(scales[0], (double)out[v], e) : e;
}

// The energy step along the network's correction: d = s0 out, r = b - A e,
// gamma = <r, d> / <d, A d> -- the step from e along d that minimises the A-norm of the error
// (<x_t - e - gamma d, A (x_t - e - gamma d)> is a parabola in gamma with its minimum there,
// because A (x_t - e) = r).  Row i adds r_i d_i and d_i (A d)_i; d is formed at every gathered
// column from out.  gamma = 0 when <d, A d> <= 0 or is not finite (the extrapolation alone).
__global__ void __launch_bounds__(kBlock) k_ws_energy(int n, const int32_t* rp, const int32_t* ci,
                                                      const double* va, const float* out,
                                                      const double* xm1, const double* xm2,
                                                      const double* b, const double* scales,
                                                      double* gamma, double* scratch) {
  const double s0 = scales[0];
  double sums[2];
  bool last;
  grid_sums<2>(n, scratch, [&](int i, double (&v)[2]) {
    double se = 0.0, sd = 0.0;
    for (int j = rp[i]; j < rp[i + 1]; ++j) {
      const int c = ci[j];
      se = fma(va[j], 2.0 * xm1[c] - xm2[c], se);
      sd = fma(va[j], s0 * (double)out[c], sd);
    }
    const double r = b[i] - se, d = s0 * (double)out[i];
    v[0] = fma(r, d, v[0]);
    v[1] = fma(d, sd, v[1]);
  }, sums, last);
  if (last && threadIdx.x == 0) {
    const double g = sums[0] / sums[1];
    gamma[0] = sums[1] > 0.0 && isfinite(g) ? g : 0.0;
  }
}

// x_hat = 2 x_{t-1} - x_{t-2} + gamma s0 out.
__global__ void k_ws_apply_gamma(int n, const float* out, const double* xm1, const double* xm2,
                                 const double* scales, const double* gamma, double* xhat) {
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  const double e = 2.0 * xm1[v] - xm2[v];
  xhat[v] = fma(gamma[0], scales[0] * (double)out[v], e);
}

// One damped Jacobi sweep from a starting guess: xout_i = x_i + omega (b_i - sum_j a_ij x_j) / d_i,
// d_i = a_ii (1 where the row has no nonzero diagonal entry); the row's products are summed
// left to right.  Applied to the learned guess it damps the rough part of the guess's error,
// the part CG removes slowest on this operator.
__global__ void k_ws_relax(int n, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                           const double* __restrict__ va, const double* __restrict__ b,
                           const double* __restrict__ x, double omega, double* __restrict__ xout) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double s = 0.0, d = 0.0;
  for (int j = rp[i]; j < rp[i + 1]; ++j) {
    const int c = ci[j];
    s = fma(va[j], x[c], s);
    if (c == i) d = va[j];
  }
  if (d == 0.0) d = 1.0;
  xout[i] = fma(omega, (b[i] - s) / d, x[i]);
}

// Loss of the learned guess after damped Jacobi sweeps (training through the sweeps).  The
// guess's error in units of s0 is delta = out - (x_t - 2 x_{t-1} + x_{t-2}) / s0; a sweep maps
// an error e to P e = e - omega D^-1 A e; the loss is mean((P^s delta)^2) and its gradient
// (2/n) (P^T)^s P^s delta, P^T g = g - omega A (D^-1 g) for a symmetric A.
// d_i = a_ii (1 where the row has no nonzero diagonal entry).
__global__ void k_ws_diag(int n, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                          const double* __restrict__ va, double* __restrict__ d) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double di = 1.0;
  for (int j = rp[i]; j < rp[i + 1]; ++j)
    if (ci[j] == i && va[j] != 0.0) di = va[j];
  d[i] = di;
}

__global__ void k_ws_delta(int n, const float* __restrict__ out, const double* __restrict__ xt,
                           const double* __restrict__ xm1, const double* __restrict__ xm2,
                           const double* __restrict__ scales, double* __restrict__ e) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  e[i] = (double)out[i] - (xt[i] - 2.0 * xm1[i] + xm2[i]) / scales[0];
}

// eout = e - omega D^-1 A e (one sweep's error propagator)
__global__ void k_ws_prop(int n, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                          const double* __restrict__ va, const double* __restrict__ d, double omega,
                          const double* __restrict__ e, double* __restrict__ eout) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double s = 0.0;
  for (int j = rp[i]; j < rp[i + 1]; ++j) s = fma(va[j], e[ci[j]], s);
  eout[i] = fma(omega, (0.0 - s) / d[i], e[i]);
}

// gout = g - omega A (D^-1 g) (its transpose, A symmetric)
__global__ void k_ws_prop_t(int n, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                            const double* __restrict__ va, const double* __restrict__ d, double omega,
                            const double* __restrict__ g, double* __restrict__ gout) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double s = 0.0;
  for (int j = rp[i]; j < rp[i + 1]; ++j) {
    const int c = ci[j];
    s = fma(va[j], g[c] / d[c], s);
  }
  gout[i] = fma(-omega, s, g[i]);
}

// *loss = mean(e^2)
__global__ void __launch_bounds__(kBlock) k_ws_sq_mean(int n, const double* e, double* loss, double* scratch) {
  double sum[1];
  bool last;
  grid_sums<1>(n, scratch, [&](int i, double (&v)[1]) { v[0] = fma(e[i], e[i], v[0]); }, sum, last);
  if (last && threadIdx.x == 0) *loss = sum[0] / n;
}

// G[v][0] = bf16(2 g_v / n), other channels 0
__global__ void k_ws_grad_pack(int n, const double* __restrict__ g, __nv_bfloat16* __restrict__ G) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  __nv_bfloat16* gi = G + (size_t)i * kCh;
  gi[0] = __float2bfloat16_rn((float)(2.0 * g[i] / n));
  for (int c = 1; c < kCh; ++c) gi[c] = __float2bfloat16_rn(0.f);
}

// One parameter of Adam (FP32 master, optional BF16 copy).
__device__ __forceinline__ __nv_bfloat16 adam_one(int e, float* p, const float* grad, float* m, float* v, float lr, float b1,
                                                  float b2, float eps, float c1, float c2) {
  const float gr = grad[e];
  const float mm = b1 * m[e] + (1.f - b1) * gr;
  const float vv = b2 * v[e] + (1.f - b2) * gr * gr;
  m[e] = mm;
  v[e] = vv;
  const float mh = mm / c1, vh = vv / c2;
  const float np = p[e] - lr * mh / (sqrtf(vh) + eps);
  p[e] = np;
  return __float2bfloat16_rn(np);
}

__global__ void k_adam(int count, float* p, const float* grad, float* m, float* v, float lr,
                       float b1, float b2, float eps, float c1, float c2, __nv_bfloat16* p16) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= count) return;
  const __nv_bfloat16 np = adam_one(e, p, grad, m, v, lr, b1, b2, eps, c1, c2);
  if (p16) p16[e] = np;
}

// The same for all tensors of a network in one launch (a step of the four-layer network was eight
// launches of k_adam and four of k_conv3d_flip, 3.3 us each whatever their size).
struct AdamTensor {
  float* p;
  const float* grad;
  float* m;
  float* v;
  __nv_bfloat16* p16;
  __nv_bfloat16* flipped;
  int count, block0;  // elements; the tensor's first block
};
struct AdamTensors {
  AdamTensor t[PK_ADAM_MAX_TENSORS];
};

__global__ void k_adam_many(const __grid_constant__ AdamTensors a, int tensors, float lr, float b1, float b2, float eps,
                            float c1, float c2) {
  int k = 0;
  while (k + 1 < tensors && (int)blockIdx.x >= a.t[k + 1].block0) ++k;
  const AdamTensor& t = a.t[k];
  const int e = ((int)blockIdx.x - t.block0) * blockDim.x + threadIdx.x;
  if (e >= t.count) return;
  const __nv_bfloat16 np = adam_one(e, t.p, t.grad, t.m, t.v, lr, b1, b2, eps, c1, c2);
  if (t.p16) t.p16[e] = np;
  if (t.flipped) {
    const int tap = e / (kCh * kCh), co = (e / kCh) % kCh, ci = e % kCh;
    t.flipped[((26 - tap) * kCh + ci) * kCh + co] = np;
  }
}

// Tensor map of a channels-last BF16 activation [D][H][W][16] for the TMA boxes of the convolution
// kernels: dimensions (channel, x, y, z), box (bc, bx, by, bz), zero fill outside.
using EncodeTiled = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                 const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                 CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                 CUtensorMapFloatOOBfill);

static pk_status input_map(CUtensorMap* map, const __nv_bfloat16* X, int D, int H, int W, int bc,
                             int bx, int by, int bz) {
  static EncodeTiled encode = nullptr;
  if (!encode) {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) !=
            cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !fn) {
      set_error("cuTensorMapEncodeTiled is not available");
      return PK_ERR_CUDA;
    }
    encode = reinterpret_cast<EncodeTiled>(fn);
  }
  if (reinterpret_cast<uintptr_t>(X) & 15) {
    set_error("pk_conv3d: activations and gradients must be 16-byte aligned");
    return PK_ERR_ARG;
  }
  const cuuint64_t dims[4] = {(cuuint64_t)kCh, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)D};
  const cuuint64_t strides[3] = {(cuuint64_t)kCh * 2, (cuuint64_t)W * kCh * 2, (cuuint64_t)H * W * kCh * 2};
  const cuuint32_t box[4] = {(cuuint32_t)bc, (cuuint32_t)bx, (cuuint32_t)by, (cuuint32_t)bz};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  const CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<__nv_bfloat16*>(X), dims,
                            strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                            CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    set_error("pk_conv3d: cuTensorMapEncodeTiled failed");
    return PK_ERR_CUDA;
  }
  return PK_OK;
}

static pk_status conv_setup() {
  static bool done = false;
  if (!done) {
    PK_CUDA(cudaFuncSetAttribute(k_conv3d_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, kTcSmem));
    PK_CUDA(cudaFuncSetAttribute(k_conv3d_wgrad_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, kWgSmem));
    done = true;
  }
  return PK_OK;
}

}  // namespace pk

using namespace pk;

extern "C" {

pk_status pk_conv3d_fwd(const void* X, const void* Wt, const float* bias, void* Y, int32_t D,
                        int32_t H, int32_t W, int32_t relu, int32_t out_f32, const void* mask,
                        void* stream) {
  if (!X || !Wt || !Y || D <= 0 || H <= 0 || W <= 0 ||
      (int64_t)D * ((H + kTcY - 1) / kTcY) * ((W + kTcX - 1) / kTcX) >= (int64_t(1) << 31)) {
    set_error("pk_conv3d_fwd: bad arguments");
    return PK_ERR_ARG;
  }
  pk_status e = conv_setup();
  if (e) return e;
  ConvArgs a;
  a.X = static_cast<const __nv_bfloat16*>(X);
  a.Wt = static_cast<const __nv_bfloat16*>(Wt);
  a.bias = bias;
  a.Y = out_f32 ? nullptr : static_cast<__nv_bfloat16*>(Y);
  a.Yf = out_f32 ? static_cast<float*>(Y) : nullptr;
  a.mask = static_cast<const __nv_bfloat16*>(mask);
  a.D = D;
  a.H = H;
  a.W = W;
  a.relu = relu;
  a.out_f32 = out_f32;
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    PK_CUDA(cudaGetDevice(&dev));
    PK_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  }
  CUtensorMap map;
  if ((e = input_map(&map, a.X, D, H, W, 8, kTcBx, kTcBy, 1))) return e;
  // one block per SM (it takes all of the tensor memory), at most one per (column tile, z) unit
  const int64_t units = (int64_t)D * ((H + kTcY - 1) / kTcY) * ((W + kTcX - 1) / kTcX);
  launch_pdl(k_conv3d_tc, (int)std::min<int64_t>(units, sms), kTcThreads, kTcSmem, (cudaStream_t)stream, map, a);
  PK_CUDA(cudaGetLastError());
  return PK_OK;
}

pk_status pk_conv3d_check(void* stream) {
  int flag = 0, zero = 0;
  cudaStream_t s = (cudaStream_t)stream;
  PK_CUDA(cudaMemcpyFromSymbolAsync(&flag, g_conv_timeout, sizeof(int), 0, cudaMemcpyDeviceToHost, s));
  PK_CUDA(cudaMemcpyToSymbolAsync(g_conv_timeout, &zero, sizeof(int), 0, cudaMemcpyHostToDevice, s));
  PK_CUDA(cudaStreamSynchronize(s));
  if (flag) {
    set_error("a tensor-core convolution timed out waiting for its MMAs");
    return PK_TIMEOUT;
  }
  return PK_OK;
}

// Blocks of the weight-gradient launch: one per SM (its shared memory allows one), at most
// one per segment and at most kWgMaxBlocks (the scratch size).
static int wgrad_blocks(int32_t D, int32_t H, int32_t W, int sms) {
  const int64_t chunks = (int64_t)D * H * ((W + kWgSeg - 1) / kWgSeg);
  return (int)std::max<int64_t>(1, std::min<int64_t>(chunks, std::min(sms, kWgMaxBlocks)));
}

int64_t pk_conv3d_wgrad_scratch_floats(int32_t D, int32_t H, int32_t W) {
  return (int64_t)wgrad_blocks(D, H, W, kWgMaxBlocks) * (27 * kCh * kCh + kCh);
}

pk_status pk_conv3d_wgrad(const void* A, const void* G, float* scratch, float* dW, float* db,
                          int32_t D, int32_t H, int32_t W, void* stream) {
  if (!A || !G || !scratch || !dW || !db || D <= 0 || H <= 0 || W <= 0 ||
      (int64_t)D * H * ((W + kWgSeg - 1) / kWgSeg) >= (int64_t(1) << 31)) {
    set_error("pk_conv3d_wgrad: bad arguments");
    return PK_ERR_ARG;
  }
  pk_status e = conv_setup();
  if (e) return e;
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    PK_CUDA(cudaGetDevice(&dev));
    PK_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  }
  const int nblk = wgrad_blocks(D, H, W, sms);
  // partials laid out for the scratch size's block count (the launch may use fewer blocks)
  const int nmax = wgrad_blocks(D, H, W, kWgMaxBlocks);
  float* partial = scratch;
  float* partial_db = scratch + (size_t)nmax * 27 * kCh * kCh;
  cudaStream_t s = (cudaStream_t)stream;
  CUtensorMap amap, gmap;
  if ((e = input_map(&amap, static_cast<const __nv_bfloat16*>(A), D, H, W, kCh, kWgSeg + 2, 1, 3))) return e;
  if ((e = input_map(&gmap, static_cast<const __nv_bfloat16*>(G), D, H, W, kCh, kWgSeg + 2, 1, 1))) return e;
  launch_pdl(k_conv3d_wgrad_tc, nblk, kWgBlock, kWgSmem, s, amap, gmap, static_cast<const __nv_bfloat16*>(G), partial,
             partial_db, D, H, W);
  launch_pdl(k_conv3d_wgrad_reduce, (27 * kCh * kCh + kCh + 31) / 32, 256, 0, s, (const float*)partial,
             (const float*)partial_db, nblk, dW, db);
  PK_CUDA(cudaGetLastError());
  return PK_OK;
}

pk_status pk_conv3d_flip(const void* W, void* Wf, void* stream) {
  if (!W || !Wf) { set_error("pk_conv3d_flip: NULL"); return PK_ERR_ARG; }
  k_conv3d_flip<<<(27 * kCh * kCh + 255) / 256, 256, 0, (cudaStream_t)stream>>>(
      static_cast<const __nv_bfloat16*>(W), static_cast<__nv_bfloat16*>(Wf));
  PK_CUDA(cudaGetLastError());
  return PK_OK;
}

int64_t pk_warmstart_scratch_doubles(void) { return 3 * kWsGrid + 8; }

pk_status pk_warmstart_input(pk_csr* A, const double* xm1, const double* xm2, const double* b,
                             void* X16, double* scales, double* scratch, void* stream) {
  if (!A || !xm1 || !xm2 || !b || !X16 || !scales || !scratch) {
    set_error("pk_warmstart_input: bad arguments");
    return PK_ERR_ARG;
  }
  const int n = A->n;
  cudaStream_t s = (cudaStream_t)stream;
  PK_CUDA(cudaMemsetAsync(scratch + 3 * kWsGrid, 0, sizeof(double), s));
  WsStash* stash = (reinterpret_cast<uintptr_t>(X16) & 7) == 0 ? static_cast<WsStash*>(X16) : nullptr;
  k_ws_rms<<<kWsGrid, kBlock, 0, s>>>(n, A->rp, A->ci, A->va, xm1, xm2, b, scales, scratch, stash);
  k_ws_pack<<<(n + 255) / 256, 256, 0, s>>>(n, A->rp, A->ci, A->va, xm1, xm2, b, scales,
                                             static_cast<__nv_bfloat16*>(X16), stash != nullptr);
  PK_CUDA(cudaGetLastError());
  return PK_OK;
}

pk_status pk_warmstart_loss(int64_t n, const float* out, const double* xt, const double* xm1,
                            const double* xm2, const double* scales, void* G, double* loss,
                            double* scratch, void* stream) {
  if (n <= 0 || n >= (int64_t(1) << 31) || !out || !xt || !xm1 || !xm2 || !scales || !G || !loss ||
      !scratch) {
    set_error("pk_warmstart_loss: bad arguments");
    return PK_ERR_ARG;
  }
  cudaStream_t s = (cudaStream_t)stream;
  PK_CUDA(cudaMemsetAsync(scratch + 3 * kWsGrid, 0, sizeof(double), s));
  k_ws_loss<<<kWsGrid, kBlock, 0, s>>>((int)n, out, xt, xm1, xm2, scales,
                                       static_cast<__nv_bfloat16*>(G), loss, scratch);
  PK_CUDA(cudaGetLastError());
  return PK_OK;
}

pk_status pk_warmstart_apply(int64_t n, const float* out, const double* xm1, const double* xm2,
                             const double* scales, double* xhat, void* stream) {
  if (n <= 0 || n >= (int64_t(1) << 31) || !xm1 || !xm2 || !scales || !xhat) {
    set_error("pk_warmstart_apply: bad arguments");
    return PK_ERR_ARG;
  }
  k_ws_apply<<<(int)((n + 255) / 256), 256, 0, (cudaStream_t)stream>>>((int)n, out, xm1, xm2,
                                                                       scales, xhat);
  PK_CUDA(cudaGetLastError());
  return PK_OK;
}

pk_status pk_warmstart_apply_energy(pk_csr* A, const float* out, const double* xm1, const double* xm2,
                                    const double* b, const double* scales, double* xhat, double* gamma,
                                    double* scratch, void* stream) {
  if (!A || !out || !xm1 || !xm2 || !b || !scales || !xhat || !gamma || !scratch) {
    set_error("pk_warmstart_apply_energy: bad arguments");
    return PK_ERR_ARG;
  }
  const int n = A->n;
  if (n == 0) return PK_OK;
  cudaStream_t s = (cudaStream_t)stream;
  PK_CUDA(cudaMemsetAsync(scratch + 3 * kWsGrid, 0, sizeof(double), s));
  k_ws_energy<<<kWsGrid, kBlock, 0, s>>>(n, A->rp, A->ci, A->va, out, xm1, xm2, b, scales, gamma, scratch);
  k_ws_apply_gamma<<<(n + 255) / 256, 256, 0, s>>>(n, out, xm1, xm2, scales, gamma, xhat);
  PK_CUDA(cudaGetLastError());
  return PK_OK;
}

pk_status pk_warmstart_relax(pk_csr* A, const double* b, const double* x, double omega, double* xout,
                             void* stream) {
  if (!A || !b || !x || !xout || !(omega > 0.0 && omega < 2.0)) {
    set_error("pk_warmstart_relax: bad arguments (omega must lie in (0, 2))");
    return PK_ERR_ARG;
  }
  if (x == xout) {
    set_error("pk_warmstart_relax: xout must not be x (rows read x at other rows' columns)");
    return PK_ERR_ARG;
  }
  const int n = A->n;
  if (n == 0) return PK_OK;
  k_ws_relax<<<(n + 255) / 256, 256, 0, (cudaStream_t)stream>>>(n, A->rp, A->ci, A->va, b, x, omega, xout);
  PK_CUDA(cudaGetLastError());
  return PK_OK;
}

pk_status pk_warmstart_loss_swept(pk_csr* A, const float* out, const double* xt, const double* xm1,
                                  const double* xm2, const double* scales, double omega, int32_t sweeps,
                                  void* G, double* loss, double* work, double* scratch, void* stream) {
  if (!A || !out || !xt || !xm1 || !xm2 || !scales || !G || !loss || !work || !scratch ||
      !(omega > 0.0 && omega < 2.0) || sweeps < 0 || sweeps > PK_WS_MAX_SWEEPS || A->n == 0) {
    set_error("pk_warmstart_loss_swept: bad arguments (omega in (0, 2), sweeps in [0, 8], n > 0)");
    return PK_ERR_ARG;
  }
  const int n = A->n;
  const int nb = (n + 255) / 256;
  cudaStream_t s = (cudaStream_t)stream;
  double* d = work;
  double* buf[2] = {work + n, work + 2 * (size_t)n};
  k_ws_diag<<<nb, 256, 0, s>>>(n, A->rp, A->ci, A->va, d);
  k_ws_delta<<<nb, 256, 0, s>>>(n, out, xt, xm1, xm2, scales, buf[0]);
  int cur = 0;
  for (int k = 0; k < sweeps; ++k, cur ^= 1)
    k_ws_prop<<<nb, 256, 0, s>>>(n, A->rp, A->ci, A->va, d, omega, buf[cur], buf[cur ^ 1]);
  PK_CUDA(cudaMemsetAsync(scratch + 3 * kWsGrid, 0, sizeof(double), s));
  k_ws_sq_mean<<<kWsGrid, kBlock, 0, s>>>(n, buf[cur], loss, scratch);
  for (int k = 0; k < sweeps; ++k, cur ^= 1)
    k_ws_prop_t<<<nb, 256, 0, s>>>(n, A->rp, A->ci, A->va, d, omega, buf[cur], buf[cur ^ 1]);
  k_ws_grad_pack<<<nb, 256, 0, s>>>(n, buf[cur], static_cast<__nv_bfloat16*>(G));
  PK_CUDA(cudaGetLastError());
  return PK_OK;
}

pk_status pk_adam_step(int64_t count, float* p, const float* grad, float* m, float* v, float lr,
                       float beta1, float beta2, float eps, int32_t step, void* p_bf16, void* stream) {
  if (count <= 0 || !p || !grad || !m || !v || step < 1) {
    set_error("pk_adam_step: bad arguments");
    return PK_ERR_ARG;
  }
  const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
  k_adam<<<(int)((count + 255) / 256), 256, 0, (cudaStream_t)stream>>>(
      (int)count, p, grad, m, v, lr, beta1, beta2, eps, c1, c2, static_cast<__nv_bfloat16*>(p_bf16));
  PK_CUDA(cudaGetLastError());
  return PK_OK;
}

pk_status pk_adam_step_many(int32_t tensors, const int64_t* counts, float* const* p, const float* const* grad,
                            float* const* m, float* const* v, void* const* p_bf16, void* const* flipped, float lr,
                            float beta1, float beta2, float eps, int32_t step, void* stream) {
  if (tensors < 1 || tensors > PK_ADAM_MAX_TENSORS || !counts || !p || !grad || !m || !v || step < 1) {
    set_error("pk_adam_step_many: bad arguments");
    return PK_ERR_ARG;
  }
  AdamTensors a;
  int64_t blocks = 0;
  for (int k = 0; k < tensors; ++k) {
    AdamTensor& t = a.t[k];
    t.p16 = p_bf16 ? static_cast<__nv_bfloat16*>(p_bf16[k]) : nullptr;
    t.flipped = flipped ? static_cast<__nv_bfloat16*>(flipped[k]) : nullptr;
    if (counts[k] <= 0 || counts[k] >= (int64_t(1) << 31) || !p[k] || !grad[k] || !m[k] || !v[k] ||
        (t.flipped && counts[k] != 27 * kCh * kCh)) {
      set_error("pk_adam_step_many: bad tensor");
      return PK_ERR_ARG;
    }
    t.p = p[k];
    t.grad = grad[k];
    t.m = m[k];
    t.v = v[k];
    t.count = (int)counts[k];
    t.block0 = (int)blocks;
    blocks += (counts[k] + 255) / 256;
  }
  if (blocks >= (int64_t(1) << 31)) { set_error("pk_adam_step_many: too many parameters"); return PK_ERR_ARG; }
  const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
  k_adam_many<<<(int)blocks, 256, 0, (cudaStream_t)stream>>>(a, tensors, lr, beta1, beta2, eps, c1, c2);
  PK_CUDA(cudaGetLastError());
  return PK_OK;
}

}  // extern "C"
