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

size_t exchange_bytes(const pk_csr* A) {
  return sizeof(ulonglong2) * (2 * (size_t)A->n + kSmSlotWords + kSmBcWords + kSmColWords);
}

// Whether the loops may fit, by what the handle knows without a plan: the matrix and three vectors, without
// their halos, in blocks that are all resident, without rows longer than a tile.
bool may_fit(const pk_csr* A, int sms) {
  if (!A->tma_ok || A->tile_z0 || A->n > kSmMaxRows || A->grid_tma > kSmMaxBlocks || A->grid_tma > 2 * sms) return false;
  const size_t most = A->grid_tma > sms ? kSmBytesPair : kSmBytesMax;
  return sm_bytes(A->blk_rows_max, A->blk_nnz_max, 0, 3, 1) <= most;
}

pk_status build(pk_csr* A, cudaStream_t s) {
  const int G = A->sm_grid, words = (A->n + 31) / 32;
  const size_t smem = sizeof(uint32_t) * 2 * (size_t)words;
  for (auto k : {k_sm_plan<false>, k_sm_plan<true>})
    PK_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  std::vector<int32_t> ptr(G + 1, 0);
  if (pk_status e = ensure_state(A)) return e;
  // the counts in the reductions' scratch (three sums per block); one allocation, one wait: a handle's
  // first solve pays for them
  int32_t* cnt = reinterpret_cast<int32_t*>(A->partials);
  k_sm_plan<false><<<G, kPlanThreads, smem, s>>>(A->rp, A->ci, A->sm_blk_row, words, cnt, nullptr, nullptr, nullptr);
  PK_CUDA(cudaGetLastError());
  PK_CUDA(cudaMemcpyAsync(ptr.data(), cnt, sizeof(int32_t) * G, cudaMemcpyDeviceToHost, s));
  PK_CUDA(cudaStreamSynchronize(s));
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
  const size_t b0 = up(exchange_bytes(A)), b1 = up(sizeof(int32_t) * (G + 1)), b2 = up(sizeof(int32_t) * std::max(1, sum));
  PK_CUDA(cudaMalloc(&A->sm_exchange, b0 + b1 + b2 + sizeof(uint16_t) * ((size_t)A->nnz + 64)));
  char* d = reinterpret_cast<char*>(A->sm_exchange);
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

pk_status sm_prepare(pk_csr* A, cudaStream_t s, bool* usable) {
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
    return t ? t : build(A, s);
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
  a.col = a.bc + kSmBcWords;
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
