// Plan of the shared-memory-resident solver loops (pk_sm.cuh): which columns every block gathers
// from other blocks, and every entry's column as a 16-bit index into the block's own rows or its
// halo.  Built on the device from the tile schedule, once per handle.
#include <algorithm>
#include <vector>

#include "pk_guard.cuh"
#include "pk_sm.cuh"

namespace pk {

namespace {

constexpr int kPlanThreads = 1024;
constexpr size_t kColBytes = sizeof(ulonglong2) * kSmColWords;

// The columns of block b's rows outside [r0, r1) as a bitmap, then their ranks.  EMIT = false:
// cnt[b] = their number; true: the ascending list at halo + ptr[b], and ci16 of the block's entries.
template <bool EMIT>
__global__ void __launch_bounds__(kPlanThreads) k_sm_plan(const int32_t* rp, const int32_t* ci, const int32_t* rows,
                                                          int words, int32_t* cnt, const int32_t* ptr, int32_t* halo,
                                                          uint16_t* ci16) {
  extern __shared__ uint32_t bits[];  // words bitmap words, then words ranks
  uint32_t* rank = bits + words;
  __shared__ int wsum[kPlanThreads / 32];
  const int b = blockIdx.x, r0 = rows[b], r1 = rows[b + 1];
  const int z0 = rp[r0], z1 = rp[r1];
  for (int w = threadIdx.x; w < words; w += kPlanThreads) bits[w] = 0;
  __syncthreads();
  for (int z = z0 + threadIdx.x; z < z1; z += kPlanThreads) {
    const int c = ci[z];
    if (c < r0 || c >= r1) atomicOr(bits + (c >> 5), 1u << (c & 31));
  }
  __syncthreads();
  // ranks: each thread counts a run of words, then an exclusive scan over the threads
  const int per = (words + kPlanThreads - 1) / kPlanThreads;
  const int w0 = min(words, (int)threadIdx.x * per), w1 = min(words, w0 + per);
  int mine = 0;
  for (int w = w0; w < w1; ++w) mine += __popc(bits[w]);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int inc = mine;
  for (int o = 1; o < 32; o <<= 1) {
    const int up = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += up;
  }
  if (lane == 31) wsum[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    int t = wsum[lane];
    for (int o = 1; o < 32; o <<= 1) {
      const int up = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += up;
    }
    wsum[lane] = t;
  }
  __syncthreads();
  int at = inc - mine + (warp ? wsum[warp - 1] : 0);
  if (!EMIT) {
    if (threadIdx.x == kPlanThreads - 1) cnt[b] = wsum[kPlanThreads / 32 - 1];
    return;
  }
  int32_t* out = halo + ptr[b];
  for (int w = w0; w < w1; ++w) {
    rank[w] = at;
    for (uint32_t m = bits[w]; m; m &= m - 1) out[at++] = 32 * w + __ffs(m) - 1;
  }
  __syncthreads();
  const int hoff = sm_even(r1 - r0);
  for (int z = z0 + threadIdx.x; z < z1; z += kPlanThreads) {
    const int c = ci[z];
    ci16[z] = (uint16_t)(c >= r0 && c < r1 ? c - r0
                                           : hoff + (int)rank[c >> 5] + __popc(bits[c >> 5] & ((1u << (c & 31)) - 1u)));
  }
}

__global__ void __launch_bounds__(kBlock) k_sm_publish(SmArgs a, const double* v) {
  if (state_done(a.st)) return;
  const int row = blockIdx.x * kBlock + threadIdx.x;
  if (row < a.n) sm_publish(a, row, v[row], a.ep0);
}

// What build_plan (pk_csr.cu) gives G blocks of a system whose rows have at most eight entries: block b's rows
// start at the first row with rp[row] + 2 row >= wtot b / G, rounded down to a warp, and its tiles are
// kTileRows rows each.  A thread per block.  most: the rows and entries of the largest block.
__global__ void __launch_bounds__(kSmFineBlocks) k_sm_short_tiles(const int32_t* rp, int n, int G, double wtot,
                                                                  int32_t* blk_row, int32_t* blk_tile,
                                                                  int32_t* tile_row, int32_t* most) {
  __shared__ int row[kSmFineBlocks + 1], wsum[kSmFineBlocks / 32], wmax[2][kSmFineBlocks / 32];
  const int b = threadIdx.x, lane = b & 31, warp = b >> 5;
  if (b < G) {
    const double target = wtot * b / G;
    int lo = 0, hi = n;
    while (b && lo < hi) {
      const int mid = (lo + hi) / 2;
      if ((double)rp[mid] + 2.0 * (double)mid < target) lo = mid + 1;
      else hi = mid;
    }
    row[b] = lo / 32 * 32;
  }
  if (b == 0) row[G] = n;
  __syncthreads();
  const int r0 = b < G ? row[b] : 0, rows = b < G ? row[b + 1] - r0 : 0;
  const int tiles = (rows + kTileRows - 1) / kTileRows;
  int inc = tiles, mr = rows, mz = rows ? rp[r0 + rows] - rp[r0] : 0;
  for (int o = 1; o < 32; o <<= 1) {
    const int up = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += up;
    mr = max(mr, __shfl_xor_sync(0xffffffffu, mr, o));
    mz = max(mz, __shfl_xor_sync(0xffffffffu, mz, o));
  }
  if (lane == 31) wsum[warp] = inc;
  if (lane == 0) {
    wmax[0][warp] = mr;
    wmax[1][warp] = mz;
  }
  __syncthreads();
  int first = inc - tiles;
  for (int w = 0; w < warp; ++w) first += wsum[w];
  if (b < G) {
    blk_row[b] = r0;
    blk_tile[b] = first;
    for (int t = 0; t < tiles; ++t) tile_row[first + t] = r0 + t * kTileRows;
    if (b == G - 1) {
      blk_row[G] = n;
      blk_tile[G] = first + tiles;
      tile_row[first + tiles] = n;
    }
  }
  if (b < 2) {
    int m = 0;
    for (int w = 0; w < kSmFineBlocks / 32; ++w) m = max(m, wmax[b][w]);
    most[b] = m;
  }
}

size_t exchange_bytes(const pk_csr* A) {
  return sizeof(ulonglong2) * (2 * (size_t)A->n + kSmSlotWords + kSmBcWords);
}

// Whether the loops may fit, by what the handle knows without a plan: the matrix and three vectors, without
// their halos, in blocks that are all resident, without rows longer than a tile.
bool may_fit(const pk_csr* A, int sms) {
  if (!A->tma_ok || A->tile_z0 || A->n > kSmMaxRows || A->grid_tma > kSmMaxBlocks || A->grid_tma > 2 * sms) return false;
  const size_t most = A->grid_tma > sms ? kSmBytesPair : kSmBytesMax;
  return sm_bytes(A->blk_rows_max, A->blk_nnz_max, 0, 3, 1) <= most;
}

pk_status build(pk_csr* A, bool columns, cudaStream_t s) {
  const int G = A->sm_grid, words = (A->n + 31) / 32;
  const size_t smem = sizeof(uint32_t) * 2 * (size_t)words;
  for (auto k : {k_sm_plan<false>, k_sm_plan<true>})
    PK_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  std::vector<int32_t> ptr(G + 2, 0);
  if (pk_status e = ensure_state(A)) return e;
  // the counts in the reductions' scratch (three sums per block), the largest block's rows and entries after
  // them; one allocation, one wait: a handle's first solve pays for them
  int32_t* cnt = reinterpret_cast<int32_t*>(A->partials);
  const bool tiles_due = A->sm_rows_max == 0;  // (see sm_tiles_short)
  if (tiles_due) {
    k_sm_short_tiles<<<1, kSmFineBlocks, 0, s>>>(A->rp, A->n, G, (double)A->nnz + 2.0 * (double)A->n,
                                                 const_cast<int32_t*>(A->sm_blk_row),
                                                 const_cast<int32_t*>(A->sm_blk_tile),
                                                 const_cast<int32_t*>(A->sm_tile_row), cnt + G);
    PK_CUDA(cudaGetLastError());
  }
  k_sm_plan<false><<<G, kPlanThreads, smem, s>>>(A->rp, A->ci, A->sm_blk_row, words, cnt, nullptr, nullptr, nullptr);
  PK_CUDA(cudaGetLastError());
  PK_CUDA(cudaMemcpyAsync(ptr.data(), cnt, sizeof(int32_t) * (G + 2), cudaMemcpyDeviceToHost, s));
  PK_CUDA(cudaStreamSynchronize(s));
  if (tiles_due) {
    A->sm_rows_max = ptr[G];
    A->sm_nnz_max = ptr[G + 1];
  }
  int sum = 0, most = 0;
  for (int b = 0; b < G; ++b) {
    const int c = ptr[b];
    ptr[b] = sum;
    sum += c;
    most = std::max(most, c);
  }
  ptr[G] = sum;
  A->sm_halo_max = most;
  size_t need = 0;
  if (sm_even(A->sm_rows_max) + most > 65535) return PK_OK;
  need = sm_bytes(A->sm_rows_max, A->sm_nnz_max, most, 3, 1);
  if (need > kSmBytesMax) return PK_OK;  // no loop fits
  const auto up = [](size_t b) { return (b + 255) & ~size_t(255); };
  const size_t bx = up(exchange_bytes(A)), b0 = bx + (columns ? up(kColBytes) : 0), b1 = up(sizeof(int32_t) * (G + 1)), b2 = up(sizeof(int32_t) * std::max(1, sum));
  PK_CUDA(cudaMalloc(&A->sm_exchange, b0 + b1 + b2 + sizeof(uint16_t) * ((size_t)A->nnz + 64)));
  char* d = reinterpret_cast<char*>(A->sm_exchange);
  if (columns) A->sm_col = d + bx;
  A->sm_halo_ptr = reinterpret_cast<int32_t*>(d + b0);
  A->sm_halo = reinterpret_cast<int32_t*>(d + b0 + b1);
  A->sm_ci16 = reinterpret_cast<uint16_t*>(d + b0 + b1 + b2);
  // (from pageable memory: staged before the call returns)
  PK_CUDA(cudaMemcpyAsync(A->sm_halo_ptr, ptr.data(), sizeof(int32_t) * (G + 1), cudaMemcpyHostToDevice, s));
  k_sm_plan<true><<<G, kPlanThreads, smem, s>>>(A->rp, A->ci, A->sm_blk_row, words, nullptr, A->sm_halo_ptr, A->sm_halo,
                                                 A->sm_ci16);
  PK_CUDA(cudaGetLastError());
  A->sm_state = 1;
  return PK_OK;
}

}  // namespace

pk_status sm_prepare(pk_csr* A, cudaStream_t s, bool* usable, bool columns) {
  *usable = A->sm_state == 1;
  if (A->sm_state) return PK_OK;
  A->sm_state = -1;
  int coop = 0, sms = 1;
  PK_CUDA(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, A->device));
  PK_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, A->device));
  if (!coop || !may_fit(A, sms)) return PK_OK;
  // (guarded here and not only at the entry: a failed host allocation is no reason to fail the solve)
  const pk_status e = guarded([&]() -> pk_status {
    const pk_status t = sm_tiles(A, sms, s);
    return t ? t : build(A, columns, s);
  });
  if (e == PK_ERR_OOM) {  // no memory for the plan: the launched loop needs none
    cudaGetLastError();
    if (A->sm_own) cudaFree(A->sm_own);
    A->sm_own = nullptr;
    A->sm_state = -1;
    return PK_OK;
  }
  *usable = A->sm_state == 1;
  return e;
}

// A handle's first solve pays for its plan, so a small system's is short: with the row pointers copied back,
// shared out by the host and the blocks copied down again, and with GMRES's column exchange (680 KB) in every
// solver's allocation, the first solve of few iterations on a new handle took up to 120 us longer than on the
// launched loop.  Measured (us of the first solve, 6 to 10 iterations; launched loop / plan by the host /
// this): CG 150^2 241 / 347 / 233, 250^2 304 / 406 / 324, 32^3 296 / 427 / 315, 40^3 397 / 475 / 316,
// BiCGStab 32^3 352 / 462 / 402; the second solve there 201 / 143 / 142, 264 / 147 / 149, 181 / 136 / 136,
// 238 / 145 / 141 and 229 / 153 / 164.
pk_status sm_tiles_short(pk_csr* A, int blocks) {
  auto up = [](size_t b) { return (b + 63) & ~size_t(63); };
  const size_t w0 = up(blocks + 1), w1 = up(blocks + 1), w2 = (size_t)A->n / kTileRows + blocks + 2;
  PK_CUDA(cudaMalloc(&A->sm_own, sizeof(int32_t) * (w0 + w1 + w2)));
  int32_t* d = static_cast<int32_t*>(A->sm_own);
  A->sm_grid = blocks;
  A->sm_blk_row = d;
  A->sm_blk_tile = d + w0;
  A->sm_tile_row = d + w0 + w1;
  A->sm_tile_grp = nullptr;
  A->sm_tile_perm = nullptr;
  A->sm_irregular = false;
  A->sm_rows_max = A->sm_nnz_max = 0;  // with the blocks, when the plan is built
  return PK_OK;
}

pk_status sm_columns(pk_csr* A, cudaStream_t s, bool* usable) {
  if (A->sm_col) return PK_OK;
  const cudaError_t e = cudaMalloc(&A->sm_col_own, kColBytes);
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    A->sm_col_own = nullptr;
    *usable = false;
    return PK_OK;
  }
  PK_CUDA(e);
  PK_CUDA(cudaMemsetAsync(A->sm_col_own, 0, kColBytes, s));
  A->sm_col = A->sm_col_own;
  return PK_OK;
}

// By the handle alone, not by a plan that an earlier solve may have made: a graph solve gives the same bits
// whatever ran before it.  Only where the loop may fit: tile blocks share out nonzeros, and their rows differ
// where row lengths change along the numbering.  600,000 rows, 3 entries in the first half and 61 in the
// second (13,440 rows in the longest block): the update kernel 29.5 us on them, 17.3 us on equal chunks.
bool rows_by_tile_block(const pk_csr* A) {
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, A->device) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return may_fit(A, sms);
}

bool sm_fits(const pk_csr* A, const void* kernel, int nvec, int ngather, size_t* smem) {
  *smem = sm_bytes(A->sm_rows_max, A->sm_nnz_max, A->sm_halo_max, nvec, ngather);
  if (*smem > kSmBytesMax) return false;
  int sms = 1, per = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, A->device) != cudaSuccess ||
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmBytesMax) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, kSmThreads, *smem) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return per * sms >= A->sm_grid;
}

pk_status sm_args(pk_csr* A, uint64_t epochs, cudaStream_t s, SmArgs* out) {
  // epochs are 32 bits and only compared for equality: start over before they wrap, and after a
  // solve that did not say how many it used
  if (A->sm_epoch == 0 || A->sm_epoch + epochs >= (1ull << 32)) {
    PK_CUDA(cudaMemsetAsync(A->sm_exchange, 0, exchange_bytes(A), s));
    if (A->sm_col) PK_CUDA(cudaMemsetAsync(A->sm_col, 0, kColBytes, s));
    A->sm_epoch = 1;
  }
  SmArgs a;
  a.T = csr_tiles_of(A);
  a.T.tile_row = A->sm_tile_row;
  a.T.blk_tile = A->sm_blk_tile;
  a.T.tile_grp = A->sm_tile_grp;
  a.T.tile_perm = A->sm_tile_perm;
  a.rows = A->sm_blk_row;
  a.ci16 = A->sm_ci16;
  a.halo = A->sm_halo;
  a.halo_ptr = A->sm_halo_ptr;
  a.vex = reinterpret_cast<ulonglong2*>(A->sm_exchange);
  a.slots = a.vex + 2 * (size_t)A->n;
  a.bc = a.slots + kSmSlotWords;
  a.col = static_cast<ulonglong2*>(A->sm_col);
  a.n = A->n;
  a.max_rows = A->sm_rows_max;
  a.max_nnz = A->sm_nnz_max;
  a.max_halo = A->sm_halo_max;
  a.ep0 = (uint32_t)A->sm_epoch;
  a.st = A->st;
  *out = a;
  A->sm_epoch_next = A->sm_epoch;
  A->sm_epoch = 0;  // unknown until sm_done
  return PK_OK;
}

void launch_sm_publish(const SmArgs& a, const double* v, cudaStream_t s) {
  k_sm_publish<<<(a.n + kBlock - 1) / kBlock, kBlock, 0, s>>>(a, v);
}

void sm_done(pk_csr* A, uint64_t epochs) { A->sm_epoch = epochs ? A->sm_epoch_next + epochs : 0; }

}  // namespace pk
