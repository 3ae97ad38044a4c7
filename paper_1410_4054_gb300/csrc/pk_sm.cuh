// Solver loops with the matrix resident in shared memory ("SM loops"): device primitives.
//
// A system of up to a few hundred thousand rows fits the shared memory of the 152 SMs (34 MB):
// its values, 16-bit column indices and solver vectors are loaded once and the whole iteration
// loop runs in one cooperative launch.  Block b owns the rows of tile block b of the launched
// kernels and computes them with the same schedule (tile_rows), so per iteration no matrix byte
// leaves the SM; what remains is the FP64 work and two kinds of exchange between blocks through
// L2, both of 16-byte words that carry their own epoch, so that neither needs a fence or a flag
// (a reader polls the data itself and each 8-byte half is valid once its epoch matches; the steps are
// those of the publicly documented low-latency protocol of collective libraries, NCCL's LL: data and flag
// in one 8-byte store):
//   - the gathered vector: every block publishes its rows, and fetches the rows it gathers from
//     other blocks (its halo, a sorted list built with the plan) into shared memory, where the
//     product's gathers find own and halo rows by one 16-bit index;
//   - inner products: every block sends its block sums to block 0, which adds them in the order
//     of the launched kernels' second stage, does the scalar work (divisions, convergence test)
//     and broadcasts the result.  Measured on GB300 for three sums from 304 blocks: every block
//     polling every slot takes 5.8 us (contention on the slots' lines), through block 0 about half.
// Buffers alternate by epoch parity: between two uses of one buffer lies a reduction that every
// block enters after it has read the earlier contents.  Every wait is bounded by the solve's
// wait_ns; a block that gives up records PK_TIMEOUT and leaves, and the others then do the same.
#pragma once

#include "pk_tile.cuh"

namespace pk {

constexpr int kSmThreads = kConsumers;  // 256: the consumer threads of the launched kernels
constexpr int kSmMaxBlocks = 320;
constexpr size_t kSmBytesMax = 225 * 1024;  // dynamic shared memory of a block (227 KB less the static part)
constexpr size_t kSmBytesPair = 113 * 1024;  // ... of each of two blocks on an SM (228 KB, 1 KB of each reserved)
// Up to kSmFineRows rows blocks of kSmFineWork FMAs (see sm_tiles).  Measured (us per iteration, 800 / 1200 /
// 1600 / 2400 / 3200 FMAs, and the launched kernels' blocks): CG 150^2 7.2 7.2 7.2 7.5 7.1, 8.4; 40^3 7.5 in
// all five, 9.2; P1 elasticity 4,752 rows 8.6 8.6 9.6 8.2 10.6, 11.9; SPD power law 20,000 rows 11.7 11.7 11.6
// 11.7 13.1, 15.7; BiCGStab 32^3 14.8 14.9 14.8 14.8 15.5, 17.9; GMRES 32^3 12.5 12.5 12.5 12.5 13.9, 17.9: flat
// up to 2,400.  The row limit: 250^2 8.0 against 7.5 with the launched blocks, 40^3 (64,000 rows) 7.5 against
// 9.2; beyond it the launched kernels have a block for nearly every SM (41^3 9.4 against 9.5).
constexpr int kSmFineRows = 65536;
constexpr int kSmFineWork = 1600;
constexpr int kSmSums = 4;              // block sums per reduction
constexpr int kSmWords = 4;             // scalars broadcast per reduction
constexpr int kSmCopies = 16;           // copies of the broadcast (blocks share them out)
constexpr size_t kSmSlotWords = (size_t)2 * kSmSums * kSmMaxBlocks;
constexpr size_t kSmBcWords = (size_t)2 * kSmCopies * kSmWords;
constexpr size_t kSmColWords = (size_t)2 * 65 * (kSmMaxBlocks + 8);

struct SmArgs {
  CsrTiles T;
  const int32_t* rows;      // block b owns rows [rows[b], rows[b + 1])
  const uint16_t* ci16;     // column of every entry: own row offset, or hoff + halo position
  const int32_t* halo;      // halo columns of block b: [halo_ptr[b], halo_ptr[b + 1]), ascending
  const int32_t* halo_ptr;
  ulonglong2* vex;          // [2][n] published vector
  ulonglong2* slots;        // [2][kSmSums][kSmMaxBlocks]
  ulonglong2* bc;           // [2][kSmCopies][kSmWords]
  ulonglong2* col;          // GMRES: column sums and their broadcast (kSmColWords)
  int32_t n;
  int32_t max_rows, max_nnz, max_halo;  // shared memory layout
  uint32_t ep0;             // epochs of this launch start above ep0
  DevState* st;
};

__device__ __forceinline__ void ll_put(ulonglong2* a, double v, uint32_t ep) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v), e = (unsigned long long)ep << 32;
  asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(a), "l"((b & 0xffffffffull) | e), "l"((b >> 32) | e)
               : "memory");
}

__device__ __forceinline__ ulonglong2 ll_load(const ulonglong2* a) {
  ulonglong2 w;
  asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(w.x), "=l"(w.y) : "l"(a) : "memory");
  return w;
}

__device__ __forceinline__ bool ll_valid(const ulonglong2& w, uint32_t ep) {
  return (uint32_t)(w.x >> 32) == ep && (uint32_t)(w.y >> 32) == ep;
}

__device__ __forceinline__ double ll_value(const ulonglong2& w) {
  return __longlong_as_double((long long)((w.x & 0xffffffffull) | (w.y << 32)));
}

// Bounded waits: polls between two looks at the clock and at the other blocks' timeout flag.
struct SmWait {
  DevState* st;
  unsigned long long t0 = 0;
  int polls = 0;
  __device__ __forceinline__ explicit SmWait(DevState* s) : st(s) {}
  // After an unsuccessful poll: false once the wait's bound has passed.
  __device__ __forceinline__ bool again() { return (++polls & 63) != 0 || look(); }
  __device__ __noinline__ bool look() {
    const unsigned long long now = global_ns();
    if (!t0) t0 = now;
    else if (now - t0 > st->wait_ns || __ldcg(&st->timeout)) {
      report_timeout(st);
      return false;
    }
    return true;
  }
};

// Words at addr(u), u < n <= N, each polled until it carries epoch ep and then given to
// take(u, value); all N loads in flight together.  false: gave up.
template <int N, class Addr, class Take>
__device__ __forceinline__ bool ll_wait(Addr&& addr, int n, uint32_t ep, DevState* st, Take&& take) {
  SmWait w(st);
  unsigned todo = (1u << n) - 1u;
  while (todo) {
    ulonglong2 x[N];
#pragma unroll
    for (int u = 0; u < N; ++u)
      if (todo >> u & 1) x[u] = ll_load(addr(u));
#pragma unroll
    for (int u = 0; u < N; ++u)
      if ((todo >> u & 1) && ll_valid(x[u], ep)) {
        take(u, ll_value(x[u]));
        todo &= ~(1u << u);
      }
    if (todo && !w.again()) return false;
  }
  return true;
}

// Shared-memory layout of a block.
struct SmLayout {
  double* va;
  double* vec[7];   // vec[0] has max_rows + max_halo elements (the gathered vector), the others max_rows
  int32_t* rp;      // max_rows + 1, relative to the block's first entry
  uint16_t* ci;
};

__host__ __device__ inline int sm_even(int v) { return (v + 3) & ~3; }

__host__ __device__ inline size_t sm_bytes(int max_rows, int max_nnz, int max_halo, int nvec, int ngather) {
  const size_t r = sm_even(max_rows), h = sm_even(max_halo);
  return 8 * ((size_t)sm_even(max_nnz) + (r + h) * ngather + r * (nvec - ngather)) + 4 * (r + 4) +
         2 * (size_t)sm_even(max_nnz);
}

// NVEC vectors, the first NGATHER of them with room for the halo.
template <int NVEC, int NGATHER>
__device__ __forceinline__ SmLayout sm_layout(unsigned char* smem, const SmArgs& a) {
  static_assert(NVEC <= 7, "SmLayout::vec");
  SmLayout L;
  const int r = sm_even(a.max_rows), h = sm_even(a.max_halo), z = sm_even(a.max_nnz);
  double* d = reinterpret_cast<double*>(smem);
  L.va = d;
  d += z;
#pragma unroll
  for (int k = 0; k < NVEC; ++k) {
    L.vec[k] = d;
    d += k < NGATHER ? r + h : r;
  }
  L.rp = reinterpret_cast<int32_t*>(d);
  L.ci = reinterpret_cast<uint16_t*>(L.rp + r + 4);
  return L;
}

// The last `missing` vectors have no room in shared memory: rp and ci follow the last one that has.
__device__ __forceinline__ void sm_shorten(SmLayout& L, const SmArgs& a, int missing) {
  const int skip = missing * sm_even(a.max_rows);
  L.rp -= 2 * skip;
  L.ci -= 4 * skip;
}

struct SmemVec {
  const double* p;
};
template <>
struct GatherShared<SmemVec> {
  static constexpr bool value = true;
};
__device__ __forceinline__ double gather(SmemVec x, int c) { return x.p[c]; }

// Two row products with the gathered vector in shared memory, each summed left to right.  Four
// entries of both rows at a time: a gather is a shared-memory load, so there is no L2 latency to
// cover, and the registers of an eight-entry batch would spill.  The FMAs issued are those of the
// warp's longest batch (a predicated-off FP64 instruction still takes a slot of the pipe).
template <int M>
__device__ __forceinline__ void fma4(const double (&v)[4], const double (&xv)[4], int m, double& s) {
#pragma unroll
  for (int k = 0; k < M; ++k)
    if (k < m) s = fma(v[k], xv[k], s);
}

__device__ __forceinline__ void fma4n(int mx, const double (&v)[4], const double (&xv)[4], int m, double& s) {
  switch (mx) {
    case 1: fma4<1>(v, xv, m, s); break;
    case 2: fma4<2>(v, xv, m, s); break;
    case 3: fma4<3>(v, xv, m, s); break;
    case 4: fma4<4>(v, xv, m, s); break;
    default: break;
  }
}

template <class CI>
__device__ __forceinline__ void row_pair(const double* sva, const CI* sci, int ja, int ja1, int jb, int jb1,
                                         SmemVec x, double& sa, double& sb) {
  sa = 0.0;
  sb = 0.0;
  for (;;) {
    const int ma = min(4, ja1 - ja), mb = min(4, jb1 - jb);
    if (ma <= 0 && mb <= 0) break;
    double va[4], vb[4], xa[4], xb[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      va[k] = k < ma ? sva[ja + k] : 0.0;
      xa[k] = k < ma ? x.p[sci[ja + k]] : 0.0;
      vb[k] = k < mb ? sva[jb + k] : 0.0;
      xb[k] = k < mb ? x.p[sci[jb + k]] : 0.0;
    }
    const unsigned conv = __activemask();
    fma4n(__reduce_max_sync(conv, max(ma, 0)), va, xa, ma, sa);
    fma4n(__reduce_max_sync(conv, max(mb, 0)), vb, xb, mb, sb);
    ja += ma > 0 ? ma : 0;
    jb += mb > 0 ? mb : 0;
  }
}

// The rows of a grouped tile, G lanes per row, in the order of group_rows<G>.  G stays a runtime
// value and a batch holds four entries: one copy of the loop instead of four eight-entry ones (the
// loops' code must fit the instruction cache).
template <class CI, class XP, class RowDone>
__device__ __forceinline__ void group_rows_shared(int G, const int32_t* srp, const double* sva, const CI* sci, int R0,
                                                  int R1, XP x, RowDone& row_done) {
  const int lg = __ffs(G) - 1, ng = kConsumers >> lg;
  const int gid = (int)threadIdx.x >> lg, q = (int)threadIdx.x & (G - 1);
  const int rounds = (R1 - R0 + ng - 1) / ng;
#pragma unroll 1
  for (int k = 0; k < rounds; ++k) {
    const int r = R0 + gid + k * ng;
    int j = r < R1 ? srp[r] + q : 0;
    const int j1 = r < R1 ? srp[r + 1] : 0;
    double s = 0.0;
    for (;;) {
      const int m = j < j1 ? min(4, (j1 - j + G - 1) >> lg) : 0;
      const int mx = __reduce_max_sync(0xffffffffu, m);
      if (mx == 0) break;
      double v[4], xv[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        v[u] = u < m ? sva[j + u * G] : 0.0;
        xv[u] = u < m ? x.p[sci[j + u * G]] : 0.0;
      }
      fma4n(mx, v, xv, m, s);
      j += 4 * G;
    }
#pragma unroll 1
    for (int o = G >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (r < R1 && q == 0) row_done(r, s);
  }
}

// What a block knows about its part of the system.
struct SmBlock {
  int b, G, r0, rows, t0, t1, nh;
  int hoff;   // index of the first halo element: rows rounded up
  int stall;  // PK_FLAG_TEST_STALL: no block sum is sent, so block 0's wait runs out (GMRES: no column sum)
  const int32_t* halo;
};

// Loads the block's matrix into shared memory (before the first barrier).
__device__ __forceinline__ SmBlock sm_begin(const SmArgs& a, const SmLayout& L) {
  SmBlock B;
  B.b = blockIdx.x;
  B.G = gridDim.x;
  B.r0 = a.rows[B.b];
  B.rows = a.rows[B.b + 1] - B.r0;
  B.t0 = a.T.blk_tile[B.b];
  B.t1 = a.T.blk_tile[B.b + 1];
  B.hoff = sm_even(B.rows);
  B.stall = a.st->stall_test;
  const int h0 = a.halo_ptr[B.b];
  B.nh = a.halo_ptr[B.b + 1] - h0;
  B.halo = a.halo + h0;
  const int z0 = a.T.rp[B.r0], z1 = a.T.rp[B.r0 + B.rows];
#pragma unroll 1
  for (int k = threadIdx.x; k <= B.rows; k += kSmThreads) L.rp[k] = a.T.rp[B.r0 + k] - z0;
  for (int z = threadIdx.x; z < z1 - z0; z += kSmThreads) {
    L.va[z] = a.T.va[z0 + z];
    L.ci[z] = a.ci16[z0 + z];
  }
  return B;
}

// y = (A v)_row for the block's rows, v in shared memory with its halo.
template <bool IRR, class RowDone>
__device__ __forceinline__ void sm_product(const SmArgs& a, const SmLayout& L, const SmBlock& B, const double* v,
                                           RowDone&& row_done) {
#pragma unroll 1
  for (int t = B.t0; t < B.t1; ++t) {
    const int R0 = __ldg(a.T.tile_row + t), R1 = __ldg(a.T.tile_row + t + 1);
    const int G = IRR ? (int)__ldg(a.T.tile_grp + t) : 1;
    const int16_t* perm = IRR && G == 32 && a.T.tile_perm ? a.T.tile_perm + (size_t)t * kTileRows : nullptr;
    tile_rows<IRR>(R0, R1, G, perm, L.rp - B.r0, L.va, L.ci, SmemVec{v}, row_done);
  }
}

// The start of an iteration count, opaque to the compiler: it would peel the first iteration
// (which skips the convergence test) and double a loop body whose size the instruction cache feels.
__device__ __forceinline__ int sm_zero() {
  int z = 0;
  asm volatile("" : "+r"(z));
  return z;
}

__device__ __forceinline__ void sm_publish(const SmArgs& a, int row, double v, uint32_t ep) {
  ll_put(a.vex + (size_t)(ep & 1) * a.n + row, v, ep);
}

// The halo of exchange ep behind the own rows of v (SCALE: times `scale`); a barrier must follow.
// false: gave up (this thread).
template <bool SCALE = false>
__device__ __forceinline__ bool sm_fetch(const SmArgs& a, const SmBlock& B, double* v_own, uint32_t ep,
                                         double scale = 1.0) {
  constexpr int N = 4;
  double* dst = v_own + B.hoff;
  const ulonglong2* src = a.vex + (size_t)(ep & 1) * a.n;
#pragma unroll 1
  for (int k0 = threadIdx.x; k0 < B.nh; k0 += N * kSmThreads) {
    int c[N];
#pragma unroll
    for (int u = 0; u < N; ++u) c[u] = k0 + u * kSmThreads < B.nh ? __ldg(B.halo + k0 + u * kSmThreads) : 0;
    if (!ll_wait<N>([&](int u) { return src + c[u]; }, min(N, (B.nh - k0 + kSmThreads - 1) / kSmThreads), ep, a.st,
                    [&](int u, double v) { dst[k0 + u * kSmThreads] = SCALE ? v * scale : v; }))
      return false;
  }
  return true;
}

// One reduction (epoch ep): block sums of v to block 0, their totals in the order of final_sums,
// decide(total, word) in every lane of block 0's warp 0 (the same values in each; a division can
// take one lane per quotient), the words broadcast to every thread of every block,
// then record(total, word) in block 0's thread 0 (the solver state and the trace: global stores
// and the loads they need stay behind the broadcast, off every block's critical path).
// word[NW - 1] carries the decision (kRunning: go on).  Returns the decision, or PK_TIMEOUT.
template <int NV, int NW, class Decide, class Record>
__device__ __forceinline__ int sm_reduce(const SmArgs& a, const SmBlock& B, double (&v)[NV], uint32_t ep,
                                         double (&word)[NW], Decide&& decide, Record&& record) {
  static_assert(NV <= kSmSums && NW <= kSmWords, "exchange layout");
  __shared__ double gs[NV][kSmMaxBlocks / 32];
  __shared__ double sw[NW];
  __shared__ int bad;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  ulonglong2* slots = a.slots + (size_t)(ep & 1) * kSmSums * kSmMaxBlocks;
  ulonglong2* bc = a.bc + (size_t)(ep & 1) * kSmCopies * kSmWords;
  if (threadIdx.x == 0) bad = 0;
  block_sums<NV, kSmThreads / 32>(v, [&](int k, double t) {
    if (!B.stall) ll_put(slots + k * kSmMaxBlocks + B.b, t, ep);
  });
  if (B.b == 0) {
    // thread t takes slot t of every sum (and slot t + 256): a warp's slots are a group of 32
    const int ng = (B.G + 31) >> 5;
#pragma unroll 1
    for (int g = warp; g < ng; g += kSmThreads / 32) {
      const int c = g * 32 + lane;
      double t[NV];
#pragma unroll
      for (int k = 0; k < NV; ++k) t[k] = 0.0;
      if (!ll_wait<NV>([&](int k) { return slots + k * kSmMaxBlocks + c; }, c < B.G ? NV : 0, ep, a.st,
                       [&](int k, double u) { t[k] = u; }))
        bad = 1;
      __syncwarp();
      warp_sums<NV>(t);
      if (lane == 0) {
#pragma unroll
        for (int k = 0; k < NV; ++k) gs[k][g] = t[k];
      }
    }
    __syncthreads();
    if (warp == 0) {
      double t[NV];
#pragma unroll
      for (int k = 0; k < NV; ++k) t[k] = lane < ng ? gs[k][lane] : 0.0;
      warp_sums<NV>(t);
      decide(t, word);
      if (bad) word[NW - 1] = (double)PK_TIMEOUT;
#pragma unroll
      for (int k = 0; k < NW; ++k) {
        if (lane < kSmCopies) ll_put(bc + lane * kSmWords + k, word[k], ep);
        if (lane == 0) sw[k] = word[k];
      }
      if (lane == 0 && !bad) record(t, word);
    }
  } else if (warp == 0) {
    double w = 0.0;
    const ulonglong2* mine = bc + (B.b % kSmCopies) * kSmWords;
    const bool ok = ll_wait<1>([&](int) { return mine + lane; }, lane < NW ? 1 : 0, ep, a.st, [&](int, double t) { w = t; });
    if (!ok) bad = 1;
    __syncwarp();
    if (lane < NW) sw[lane] = w;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < NW; ++k) word[k] = sw[k];
  const int sts = bad ? PK_TIMEOUT : (int)word[NW - 1];
  __syncthreads();  // (sw, gs, bad are rewritten by the next reduction)
  return sts;
}

// ------------------------------------------------------------------ host side (pk_sm_plan.cu)

// The plan of A for this device (built on first use, kept with the handle): false if A does not
// fit.  columns: GMRES's column exchange too.
pk_status sm_prepare(pk_csr* A, cudaStream_t s, bool* usable, bool columns = false);
// Whether the system is small enough for one thread-block cluster to beat the SM loops.  Measured
// on GB300 (us per iteration, cluster / SM loop; work = nnz + 6 n): CG 64x64 (45k) 4.3 / 5.4, 16^3
// (52k) 4.6 / 6.3, 24^3 (176k) 7.2 / 6.6, 32^3 (420k) 11.0 / 6.4, 256x256 (720k) 16.0 / 6.7, P1
// elasticity 4,752 rows (214k) 13.0 / 9.2; BiCGStab 16^3 10.2 / 12.5, 24^3 17.2 / 12.4, 32^3
// 23.7 / 13.6: the cluster's 16 SMs slow down with the FP64 work, the SM loop hardly does.
inline bool cluster_size_work(const pk_csr* A) { return (int64_t)A->nnz + 6 * (int64_t)A->n <= 120000; }

// Blocks and tiles of A's SM loops (pk_csr.cu); those of a system of rows of at most eight entries on `blocks`
// blocks, formed on the device when the plan is built (pk_sm_plan.cu).
pk_status sm_tiles(pk_csr* A, int sms, cudaStream_t s);
constexpr int kSmFineBlocks = 256;  // blocks that sm_tiles_short takes: one per thread of its kernel
pk_status sm_tiles_short(pk_csr* A, int blocks);
// GMRES's column exchange, on first use; usable = false: no memory for it.
pk_status sm_columns(pk_csr* A, cudaStream_t s, bool* usable);
// Whether a block of `kernel` with nvec vectors (ngather gathered) fits, with every block resident.
bool sm_fits(const pk_csr* A, const void* kernel, int nvec, int ngather, size_t* smem);
// Arguments of one launch whose epochs stay below ep0 + epochs.
pk_status sm_args(pk_csr* A, uint64_t epochs, cudaStream_t s, SmArgs* out);
// Cooperative launch of an SM loop: `kernel` takes SmArgs and `extra` by value.  Its blocks take every SM
// and wait for one another; a cooperative launch starts once all of them can be resident, so it queues
// behind whatever holds the SMs, another such loop included, and no two of them each hold a part.  Seen on
// GB300: 64^3 (every SM) beside a GMRES loop that kept 16 SMs for 0.7 s waited for it with wait_ns at
// 20 ms; eight threads with a loop each (seven of this kind, one grid-resident) for 12 s at 100 ms: 1,544
// solves, none timed out, all with the bits of a solve alone.
template <class Kernel, class Extra>
pk_status sm_launch(pk_csr* A, Kernel kernel, size_t smem, const SmArgs& a, const Extra& extra, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(A->sm_grid);
  cfg.blockDim = dim3(kSmThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;  // every block resident at once (they wait on each other)
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  PK_CUDA(cudaLaunchKernelEx(&cfg, kernel, a, extra));
  return PK_OK;
}
// v as the first exchange of the launch (epoch a.ep0), by a kernel before the loop.
void launch_sm_publish(const SmArgs& a, const double* v, cudaStream_t s);
// After the solve: `epochs` were used (0: unknown, the exchange buffers are cleared next time).
void sm_done(pk_csr* A, uint64_t epochs);

}  // namespace pk
