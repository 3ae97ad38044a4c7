// Restarted pipelined GMRES(m) (Alg. 6, Sec. 3.3) with the matrix in shared memory (pk_sm.cuh): one
// cooperative launch for the whole solve.  The launched form has four kernels per Arnoldi step; here
// a step has one vector exchange and two grid-wide reductions:
//   w = A v_{i-1}; partial <v_j, w>, j < i, and xi_{i-1} of the step before;
//   columns: the total of column j is formed by block j (all columns at once; one block adding 30
//   columns of 304 slots would take 4 us) and broadcast; block 0 takes xi_{i-1}, the residual estimate
//   and the end-of-cycle decision, so a cycle's last product may be unused;
//   w -= sum R_{j,i} v_j, publish w, reduce ||w||^2: R_{i,i} and the breakdown test in block 0;
//   v_i = w / R_{i,i}; halo elements are scaled when they are fetched (the same product as the
//   owner's, so the same bits), which lets the exchange travel during the reduction.
// The basis stays in global memory (L2); every block touches its own rows only.  R and xi go to the
// handle's scratch; block 0 solves R eta = xi at the end of a cycle and broadcasts eta.
// Sums are the integer ones (warp_sums), where the launched form keeps FP64 trees (pk_gmres.cu): trees here
// cost 10 % of a step (64^3, m = 30: 8.87 against 9.73 ms a solve) and are no closer to the oracle.  Largest
// deviation of xi_i over the first cycle, integer / trees / launched form, on a 2D Laplacian with three rows
// of 4,000 couplings among rows of 5 (four such matrices, one right-hand side): 2.2e-10 / 4.3e-10 / 2.2e-10,
// 2.2e-10 / 1.8e-10 / 2.2e-10, 4.4e-10 / 4.5e-10 / 4.3e-10, 4.6e-10 / 4.4e-10 / 4.6e-10; the first with rows
// and columns scaled by up to 100: 4.8e-12 / 4.8e-12 / 2.5e-12.  Classical Gram-Schmidt makes that of any
// rounding; the one matrix where it passed a bar has rows longer than a tile, which this loop does not take.
#include "pk_sm.cuh"

namespace pk {

namespace {

constexpr int kSgLd = 65;                // leading dimension of R (restart length up to 64)
constexpr int kSgCopies = 8;             // copies of a column's broadcast
constexpr double kSgEstFloor = 1e-12;    // below it the estimate is rounding (as in the launched form)
constexpr int kCycleEnd = 65;            // decision: the cycle ends here
static_assert(kSmColWords >= 2 * kSgLd * kSmMaxBlocks + 2 * kSgCopies * kSgLd, "column exchange");

struct SmGm {
  const double* b;
  const double* r;  // r_0 (setup kernel; published by k_sm_publish)
  double* x;
  double* V;        // basis, column j at V + j * ld
  int64_t ld;
  double* Rout;     // R[j * kSgLd + i]
  double* xiout;
  int m;
  int nvec;         // 2: w in shared memory, 1: w in its basis column
};

template <bool IRR>
__global__ void __launch_bounds__(kSmThreads, 2) k_sm_gm(SmArgs a, SmGm g) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ double Rc[kSgLd + 1];   // column i: [j] = R_{j,i}, j < i; [i] = R_{i,i}; [0]: the decision
  __shared__ double eta[kSgLd + 1];  // eta; the parts of the inner products before
  __shared__ double gs[kSmMaxBlocks / 32];
  __shared__ double start[2];
  DevState* st = a.st;
  if (state_done(st)) return;  // decided by the setup kernel, the same for every block
  SmLayout L = sm_layout<2, 1>(smem, a);
  sm_shorten(L, a, 2 - g.nvec);
  SmBlock B = sm_begin(a, L);
  const int stall = B.stall;  // (the columns' waits; the other loops run out sm_reduce's)
  B.stall = 0;
  double* const cur = L.vec[0];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int maxit = st->maxit, trace_cap = st->trace_cap, m = g.m;
  double* const trace = st->trace;
  ulonglong2* const mslots = a.col;
  ulonglong2* const mbc = a.col + (size_t)2 * kSgLd * kSmMaxBlocks;
  auto vcol = [&](int j) { return g.V + (size_t)j * g.ld + B.r0; };
  auto wcol = [&](int i) { return g.nvec > 1 ? L.vec[1] : vcol(i); };
  // scalar state of block 0's warp 0; the counters are the same in every thread
  const double thr2 = st->thr2;
  double rr = st->rr, sumxi2 = 0.0, rii = 0.0;
  int total = 0, cycle = 0, k = 0, status = kRunning;
  uint32_t xe = a.ep0, se = a.ep0, me = a.ep0;  // epochs: vector, scalars, columns
  if (threadIdx.x == 0) {
    start[0] = sqrt(rr);
    start[1] = 1.0 / start[0];
  }
  __syncthreads();
  double rho = start[0], scale = start[1], xip = 0.0, rho0 = rho;
#pragma unroll 1
  for (int l = threadIdx.x; l < B.rows; l += kSmThreads) {
    const double t = g.r[B.r0 + l] * scale;
    vcol(0)[l] = t;
    cur[l] = t;
  }
  for (int i = 1 + sm_zero();;) {
    // i = 1 .. m: step i (no product is due after the last one); i = 0: x and the true residual at a
    // restart
    const bool last = i > m || (i >= 1 && total >= maxit);
    double* const w = wcol(i <= m ? i : 0);
    if (i == 0) {
#pragma unroll 1
      for (int l = threadIdx.x; l < B.rows; l += kSmThreads) {
        const double xv = g.x[B.r0 + l];
        cur[l] = xv;
        sm_publish(a, B.r0 + l, xv, xe);
      }
      scale = 1.0;
    }
    double v[1] = {0.0};
    if (!last) {
      if (!__syncthreads_and(sm_fetch<true>(a, B, cur, xe, scale))) { status = PK_TIMEOUT; break; }
      sm_product<IRR>(a, L, B, cur, [&](int row, double y) {
        const int l = row - B.r0;
        if (i == 0) {
          y = __ldg(g.b + row) - y;
          sm_publish(a, row, y, xe + 1);
          v[0] = fma(y, y, v[0]);
        }
        w[l] = y;
      });
    }
    if (i == 0) {
      double c[3];  // rho0, 1 / rho0, decision
      const int sts = sm_reduce<1, 3>(a, B, v, se++, c, [&](const double (&t)[1], double (&word)[3]) {
        rr = t[0];
        int dec = kRunning;
        if (!isfinite(rr)) dec = PK_ERR_NAN;
        else if (rr <= thr2) dec = PK_OK;
        else if (total >= maxit) dec = PK_NOT_CONVERGED;
        else if (k == 0) dec = PK_BREAKDOWN;
        rho0 = sqrt(rr);
        sumxi2 = 0.0;
        word[0] = rho0;
        word[1] = 1.0 / rho0;
        word[2] = (double)dec;
      }, [&](const double (&)[1], const double (&)[3]) {});
      if (sts != kRunning) { status = sts; break; }
      rho = c[0];
      scale = c[1];
      double* const v0 = vcol(0);
#pragma unroll 1
      for (int l = threadIdx.x; l < B.rows; l += kSmThreads) {
        const double t = w[l] * scale;
        v0[l] = t;
        cur[l] = t;
      }
      xe += 1;
      k = 0;
      i = 1;
      continue;
    }
    int dec = kRunning;
    if (i >= 2) {
      // ---- columns: xi_{i-1} (index 0) and <v_j, w>, j = 1 .. i - 1
      const int nc = last ? 0 : i - 1, par = me & 1;
      ulonglong2* const slots = mslots + (size_t)par * kSgLd * kSmMaxBlocks;
      ulonglong2* const bc = mbc + (size_t)par * kSgCopies * kSgLd;
      double p[1] = {xip};
      block_sums<1, kSmThreads / 32>(p, [&](int, double t) {
        if (!stall) ll_put(slots + B.b, t, me);
      });  // (a barrier inside: w is complete)
      // a warp per column, or per part of one while there are fewer columns than warps
      const int lc = nc == 1 ? 3 : nc == 2 ? 2 : nc <= 4 ? 1 : 0, step = 32 << lc;
#pragma unroll 1
      for (int t = warp; t < nc << lc; t += kSmThreads / 32) {
        const double* vj = vcol(1 + (t >> lc));
        double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
        int l = lane + 32 * (t & ((1 << lc) - 1));
#pragma unroll 1
        for (; l + 3 * step < B.rows; l += 4 * step) {
          const double a0 = vj[l], a1 = vj[l + step], a2 = vj[l + 2 * step], a3 = vj[l + 3 * step];
          s0 = fma(a0, w[l], s0);
          s1 = fma(a1, w[l + step], s1);
          s2 = fma(a2, w[l + 2 * step], s2);
          s3 = fma(a3, w[l + 3 * step], s3);
        }
#pragma unroll 1
        for (; l < B.rows; l += step) s0 = fma(vj[l], w[l], s0);
        const double s = warp_sum((s0 + s1) + (s2 + s3));
        if (lane == 0) eta[t] = s;
      }
      __syncthreads();
      if ((int)threadIdx.x < nc) {
        double s = eta[threadIdx.x << lc];
        for (int c = 1; c < 1 << lc; ++c) s += eta[(threadIdx.x << lc) + c];
        ll_put(slots + (threadIdx.x + 1) * kSmMaxBlocks + B.b, s, me);
      }
      // totals: column j by block j (mod the grid)
      const int ng = (B.G + 31) >> 5;
      bool ok = true;
#pragma unroll 1
      for (int j = B.b; j <= nc; j += B.G) {
        const ulonglong2* sj = slots + j * kSmMaxBlocks;
#pragma unroll 1
        for (int q = warp; q < ng; q += kSmThreads / 32) {
          double t = 0.0;
          ok &= ll_wait<1>([&](int) { return sj + q * 32 + lane; }, q * 32 + lane < B.G ? 1 : 0, me, st,
                           [&](int, double u) { t = u; });
          __syncwarp();
          t = warp_sum(t);
          if (lane == 0) gs[q] = t;
        }
        const bool all = __syncthreads_and(ok);
        if (warp == 0) {
          double t = warp_sum(lane < ng ? gs[lane] : 0.0);
          const double xi = t;
          double est = 0.0;
          if (j == 0) {
            // step i - 1 is done: the residual estimate rho0 sqrt(1 - sum xi^2), the end of the cycle
            sumxi2 += xi * xi;
            double rel2 = 1.0 - sumxi2;
            if (rel2 < 0.0) rel2 = 0.0;
            est = rho0 * sqrt(rel2);
            t = (double)kRunning;
            if (!all) t = (double)PK_TIMEOUT;
            else if (!isfinite(xi)) t = (double)PK_ERR_NAN;
            else if (est * est <= thr2 || rel2 <= kSgEstFloor || i - 1 >= m || total >= maxit) t = (double)kCycleEnd;
          }
          if (lane < kSgCopies) ll_put(bc + lane * kSgLd + j, t, me);
          if (j == 0) {
            const int s = i - 1, row = total - 1;
            for (int c = 1 + lane; c <= s; c += 32) g.Rout[c * kSgLd + s] = Rc[c];
            if (lane == 0) {
              g.xiout[s] = xi;
              if (trace && row < trace_cap) {
                trace[(size_t)row * 4 + 0] = s >= 2 ? Rc[s - 1] : 0.0;
                trace[(size_t)row * 4 + 1] = Rc[s];
                trace[(size_t)row * 4 + 2] = xi;
                trace[(size_t)row * 4 + 3] = est;
              }
            }
          }
        }
        __syncthreads();  // (gs is reused; Rc is rewritten below)
      }
      if ((int)threadIdx.x <= nc)
        ok &= ll_wait<1>([&](int) { return bc + (B.b % kSgCopies) * kSgLd + threadIdx.x; }, 1, me, st,
                         [&](int, double u) { Rc[threadIdx.x] = u; });
      if (!__syncthreads_and(ok)) { status = PK_TIMEOUT; break; }
      me += 1;
      dec = (int)Rc[0];
    } else {
      __syncthreads();  // w is complete
    }
    if (dec == kRunning) {
      // ---- w -= sum_j R_{j,i} v_j (j = 1, 2, ... in order), ||w||^2; eight basis values in flight
      double p[1] = {0.0};
#pragma unroll 1
      for (int l = threadIdx.x; l < B.rows; l += kSmThreads) {
        double t = w[l];
        const double* vl = vcol(1) + l;
        int j = 1;
#pragma unroll 1
        for (; j + 8 <= i; j += 8) {
          double vv[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) vv[q] = vl[(size_t)(j - 1 + q) * g.ld];
#pragma unroll
          for (int q = 0; q < 8; ++q) t = fma(-Rc[j + q], vv[q], t);
        }
#pragma unroll 1
        for (; j <= i - 1; ++j) t = fma(-Rc[j], vl[(size_t)(j - 1) * g.ld], t);
        w[l] = t;
        sm_publish(a, B.r0 + l, t, xe + 1);
        p[0] = fma(t, t, p[0]);
      }
      double c[2];  // 1 / R_{i,i}, decision
      dec = sm_reduce<1, 2>(a, B, p, se++, c, [&](const double (&t)[1], double (&word)[2]) {
        // R_{i,i} = ||w||, the lucky-breakdown test against ||A v_{i-1}||
        double r2 = 0.0;
        for (int j = 1 + lane; j <= i - 1; j += 32) r2 = fma(Rc[j], Rc[j], r2);
        r2 = t[0] + warp_sum(r2);
        const double root = sqrt((threadIdx.x & 1) ? r2 : t[0]);
        rii = __shfl_sync(0xffffffffu, root, 0);
        const double col = __shfl_sync(0xffffffffu, root, 1);
        word[0] = 1.0 / rii;
        word[1] = (double)(!isfinite(rii)                         ? PK_ERR_NAN
                           : rii == 0.0 || rii <= 1e-14 * col ? kCycleEnd
                                                              : kRunning);
      }, [&](const double (&)[1], const double (&)[2]) { Rc[i] = rii; });
      if (dec == kRunning) {
        // ---- v_i = w / R_{i,i}; this thread's part of xi_i = <v_0, v_i>
        scale = c[0];
        xip = 0.0;
        const double* v0 = vcol(0);
        double* const vi = vcol(i);
#pragma unroll 1
        for (int l = threadIdx.x; l < B.rows; l += kSmThreads) {
          const double t = w[l] * scale;
          vi[l] = t;
          cur[l] = t;
          xip = fma(v0[l], t, xip);
        }
        xe += 1;
        total += 1;
        k = i;
        i += 1;
        continue;
      }
      xe += 1;  // (w was published)
    }
    if (dec != kCycleEnd) { status = dec; break; }
    // ---- cycle end: R eta = xi in block 0's warp 0, x += rho0 (eta_1 v_0 + sum_{i >= 2} eta_i v_{i-1})
    if (k > 0) {
      ulonglong2* const bc = mbc + (size_t)(me & 1) * kSgCopies * kSgLd;
      __syncthreads();
      if (B.b == 0 && warp == 0) {
        for (int ii = k; ii >= 1; --ii) {
          double s = 0.0;
          for (int j = ii + 1 + lane; j <= k; j += 32) s = fma(g.Rout[ii * kSgLd + j], eta[j], s);
          s = warp_sum(s);
          if (lane == 0) eta[ii] = (g.xiout[ii] - s) / g.Rout[ii * kSgLd + ii];
          __syncwarp();
        }
        for (int ii = 1 + lane; ii <= k; ii += 32)
          for (int c = 0; c < kSgCopies; ++c) ll_put(bc + c * kSgLd + ii, eta[ii], me);
      }
      bool ok = true;
      if ((int)threadIdx.x >= 1 && (int)threadIdx.x <= k)
        ok = ll_wait<1>([&](int) { return bc + (B.b % kSgCopies) * kSgLd + threadIdx.x; }, 1, me, st,
                        [&](int, double u) { if (B.b) eta[threadIdx.x] = u; });
      if (!__syncthreads_and(ok)) { status = PK_TIMEOUT; break; }
      me += 1;
#pragma unroll 1
      for (int l = threadIdx.x; l < B.rows; l += kSmThreads) {
        const double* vl = vcol(0) + l;
        double acc = 0.0;
        int ii = 1;
#pragma unroll 1
        for (; ii + 8 <= k + 1; ii += 8) {
          double vv[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) vv[q] = vl[(size_t)(ii - 1 + q) * g.ld];
#pragma unroll
          for (int q = 0; q < 8; ++q) acc = fma(eta[ii + q], vv[q], acc);
        }
#pragma unroll 1
        for (; ii <= k; ++ii) acc = fma(eta[ii], vl[(size_t)(ii - 1) * g.ld], acc);
        g.x[B.r0 + l] = fma(rho, acc, g.x[B.r0 + l]);
      }
      __syncthreads();  // (eta is rewritten by the next cycle)
    }
    cycle += 1;
    xip = 0.0;
    xe += 1;  // (epoch xe holds v_k)
    i = 0;
  }
  if (B.b == 0 && threadIdx.x == 0) {
    st->iter = total;
    st->rr = rr;
    st->gm_cycle = cycle;
    st->status = status;
    st->done = 1;
  }
}

const void* sm_gm_kernel(const pk_csr* A) {
  return A->sm_irregular ? (const void*)k_sm_gm<true> : (const void*)k_sm_gm<false>;
}

int sm_gm_vectors(const pk_csr* A, size_t* smem) {
  for (int nv = 2; nv >= 1; --nv)
    if (sm_fits(A, sm_gm_kernel(A), nv, 1, smem)) return nv;
  return 0;
}

}  // namespace

pk_status sm_gmres_usable(pk_csr* A, cudaStream_t s, bool* usable) {
  pk_status e = sm_prepare(A, s, usable, true);
  if (e || !*usable) return e;
  size_t smem;
  *usable = sm_gm_vectors(A, &smem) > 0;
  return *usable ? sm_columns(A, s, usable) : PK_OK;
}

// Epochs that a solve of `iters` steps in `cycles` cycles uses at most, of each kind.
uint64_t sm_gmres_epochs(uint64_t iters, uint64_t cycles) { return 2 * iters + 3 * cycles + 16; }

// The loop, after the setup kernel (r_0, <r_0,r_0>, <b,b>).  Two launches: r_0 to the exchange buffer,
// then the loop.
pk_status launch_sm_gmres(pk_csr* A, const double* b, const double* r, double* x, int m, double* V, int64_t ld,
                          double* Rout, double* xiout, int maxit, cudaStream_t s) {
  SmArgs a;
  // (a cycle that takes no step ends the solve, so there are at most maxit + 2 cycles)
  pk_status e = sm_args(A, sm_gmres_epochs((uint64_t)maxit, (uint64_t)maxit + 2), s, &a);
  if (e) return e;
  size_t smem;
  const int nv = sm_gm_vectors(A, &smem);
  launch_sm_publish(a, r, s);
  PK_CUDA(cudaGetLastError());
  return sm_launch(A, A->sm_irregular ? k_sm_gm<true> : k_sm_gm<false>, smem, a,
                   SmGm{b, r, x, V, ld, Rout, xiout, m, nv}, s);
}

}  // namespace pk
