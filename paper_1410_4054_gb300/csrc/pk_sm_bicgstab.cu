// Pipelined BiCGStab (Alg. 4, Sec. 3.2, r0* = r0) with the matrix in shared memory (pk_sm.cuh):
// one cooperative launch for the whole solve.  The launched form has four kernels and four
// grid-wide reductions per iteration; here there are two reductions, each joined to a product:
//   fetch p, Ap, reduce (<r,r0*>, <r,r> of the last update, <Ap,r0*>): convergence test, alpha;
//   s = r - alpha Ap, publish s, fetch s, As, reduce (<s,s>, <As,s>, <As,As>, <As,r0*>): the early
//   exit on ||s||, omega, beta;
//   x, r, p, publish p.
// So the tests come one product later than in the launched form; iterates and counts are the same.
// Shared memory holds the matrix, the gathered vector with its halo, p, r (s in its place between
// the two updates) and Ap; As, r0* and x too where there is room, else they stay in global
// memory (L2), where only the owning block reads them.
#include "pk_sm.cuh"

namespace pk {

namespace {

constexpr int kSmBiMin = 4, kSmBiMax = 7;  // vectors in shared memory
constexpr int kEarly = 64;                 // decision: ||s|| small, x += alpha p ends the solve

struct SmBi {
  double* x;
  const double* r;
  const double* r0s;
  double* as;  // global room for As
  int nvec;    // vectors in shared memory, kSmBiMin .. kSmBiMax
};

template <bool IRR>
__global__ void __launch_bounds__(kSmThreads, 2) k_sm_bi(SmArgs a, SmBi g) {
  extern __shared__ __align__(16) unsigned char smem[];
  DevState* st = a.st;
  if (state_done(st)) return;  // decided by the setup kernel, the same for every block
  SmLayout L = sm_layout<kSmBiMax, 1>(smem, a);
  sm_shorten(L, a, kSmBiMax - g.nvec);
  const SmBlock B = sm_begin(a, L);
  double *sg = L.vec[0], *sp = L.vec[1], *sr = L.vec[2], *sap = L.vec[3];
  double* as = g.nvec > 4 ? L.vec[4] : g.as + B.r0;
  const double* z = g.nvec > 5 ? L.vec[5] : g.r0s + B.r0;
  double* x = g.nvec > 6 ? L.vec[6] : g.x + B.r0;
  for (int l = threadIdx.x; l < B.rows; l += kSmThreads) {
    const double r0 = g.r[B.r0 + l];
    sg[l] = sp[l] = sr[l] = r0;  // p0 = r0 (published by k_sm_publish)
    if (g.nvec > 5) L.vec[5][l] = g.r0s[B.r0 + l];
    if (g.nvec > 6) L.vec[6][l] = g.x[B.r0 + l];
  }
  const int maxit = st->maxit, trace_cap = st->trace_cap;
  double* const trace = st->trace;
  const double thr2 = st->thr2;
  double rr0s = st->s[0], apr0s = 0.0;  // (block 0's warp 0)
  double alpha = 0.0;
  double q[4] = {0.0, 0.0, 0.0, 0.0};
  uint32_t ep = a.ep0;
  // half iterations h = 2 i (p -> alpha -> s) and 2 i + 1 (s -> omega, beta -> p): one copy of the
  // exchange, the product and the reduction for both (the loop must fit the instruction cache)
#pragma unroll 1
  for (int h = sm_zero();; ++h, ++ep) {
    const int i = h >> 1;
    const bool second = h & 1;
    if (!__syncthreads_and(sm_fetch(a, B, sg, ep))) break;
    double* const out = second ? as : sap;
    sm_product<IRR>(a, L, B, sg, [&](int row, double y) {
      const int l = row - B.r0;
      out[l] = y;
      q[2] = fma(y, z[l], q[2]);
      if (second) {
        q[1] = fma(y, sg[l], q[1]);
        q[3] = fma(y, y, q[3]);
      }
    });
    double w[3];  // alpha | omega, beta; decision
    const int sts = sm_reduce<4, 3>(a, B, q, ep, w, [&](const double (&t)[4], double (&word)[3]) {
      int status = kRunning;
      double num0 = 0.0, den0 = 1.0, num1 = 0.0, den1 = 1.0;
      if (!second) {  // <r,r0*>, <r,r> of the last update; <Ap,r0*>
        if (i >= 1) {
          rr0s = t[0];
          if (!isfinite(t[0]) || !isfinite(t[1])) status = PK_ERR_NAN;
          else if (t[1] <= thr2) status = PK_OK;
          else if (i >= maxit) status = PK_NOT_CONVERGED;
        }
        if (status == kRunning) {
          apr0s = t[2];
          if (!isfinite(apr0s)) status = PK_ERR_NAN;
          else if (apr0s == 0.0 || rr0s == 0.0) status = PK_BREAKDOWN;
        }
        num0 = rr0s;
        den0 = apr0s;
      } else {  // <s,s>, <As,s>, <As,r0*>, <As,As>
        if (!isfinite(t[0])) status = PK_ERR_NAN;
        else if (t[0] <= thr2) status = kEarly;
        else if (!isfinite(t[1]) || !isfinite(t[2]) || !isfinite(t[3])) status = PK_ERR_NAN;
        else if (t[3] == 0.0) status = PK_BREAKDOWN;
        num0 = t[1];
        den0 = t[3];
        num1 = -t[2];
        den1 = apr0s;
      }
      // one lane per quotient (an FP64 division is about 500 clocks)
      const bool odd = threadIdx.x & 1;
      const double d = (odd ? num1 : num0) / (odd ? den1 : den0);
      word[0] = __shfl_sync(0xffffffffu, d, 0);
      word[1] = __shfl_sync(0xffffffffu, d, 1);
      word[2] = (double)status;
    }, [&](const double (&t)[4], const double (&word)[3]) {
      const int status = (int)word[2];
      if (!second) {
        if (i >= 1) {
          st->iter = i;
          st->rr = t[1];
          st->s[0] = t[0];
          if (trace && i - 1 < trace_cap) trace[(size_t)(i - 1) * 4 + 3] = t[1];
        }
        if (status == kRunning) {
          st->s[1] = apr0s;
          st->alpha = word[0];
          if (trace && i < trace_cap) trace[(size_t)i * 4 + 0] = word[0];
        }
      } else {
        st->s[2] = t[0];
        if (status == kEarly) {
          st->iter = i + 1;
          st->rr = t[0];
          if (trace && i < trace_cap) trace[(size_t)i * 4 + 3] = t[0];
        } else if (status == kRunning) {
          st->omega = word[0];
          st->beta = word[1];
          if (trace && i < trace_cap) {
            trace[(size_t)i * 4 + 1] = word[1];
            trace[(size_t)i * 4 + 2] = word[0];
          }
        }
      }
      if (status != kRunning) finish(st, status == kEarly ? PK_OK : status);
    });
    q[0] = q[1] = q[2] = q[3] = 0.0;
    if (sts == kEarly)
      for (int l = threadIdx.x; l < B.rows; l += kSmThreads) x[l] = fma(alpha, sp[l], x[l]);
    if (sts != kRunning) break;
    if (!second) {
      alpha = w[0];
      // s_i = r_i - alpha_i Ap_i, in r's place
#pragma unroll 1
      for (int l = threadIdx.x; l < B.rows; l += kSmThreads) {
        const double s = fma(-alpha, sap[l], sr[l]);
        sm_publish(a, B.r0 + l, s, ep + 1);
        sr[l] = s;
        sg[l] = s;
        q[0] = fma(s, s, q[0]);
      }
    } else {
      const double omega = w[0], beta = w[1];
#pragma unroll 1
      for (int l = threadIdx.x; l < B.rows; l += kSmThreads) {
        const double pk = sp[l], sk = sr[l];
        const double rn = fma(-omega, as[l], sk);
        const double pn = fma(beta, fma(-omega, sap[l], pk), rn);
        sm_publish(a, B.r0 + l, pn, ep + 1);
        sg[l] = pn;
        sp[l] = pn;
        sr[l] = rn;
        x[l] = fma(omega, sk, fma(alpha, pk, x[l]));
        q[0] = fma(rn, z[l], q[0]);
        q[1] = fma(rn, rn, q[1]);
      }
    }
  }
  __syncthreads();
  if (g.nvec > 6)
    for (int l = threadIdx.x; l < B.rows; l += kSmThreads) g.x[B.r0 + l] = x[l];
}

const void* sm_bi_kernel(const pk_csr* A) {
  return A->sm_irregular ? (const void*)k_sm_bi<true> : (const void*)k_sm_bi<false>;
}

// The most vectors in shared memory that still fit (0: none).
int sm_bi_vectors(const pk_csr* A, size_t* smem) {
  for (int nv = kSmBiMax; nv >= kSmBiMin; --nv)
    if (sm_fits(A, sm_bi_kernel(A), nv, 1, smem)) return nv;
  return 0;
}

}  // namespace

pk_status sm_bicgstab_usable(pk_csr* A, cudaStream_t s, bool* usable) {
  pk_status e = sm_prepare(A, s, usable);
  if (e || !*usable) return e;
  size_t smem;
  *usable = sm_bi_vectors(A, &smem) > 0;
  return PK_OK;
}

// The loop, after the setup kernel (r0, r0*, <r0,r0*>, <b,b>); as: global room for one vector.
// Two launches: p0 to the exchange buffer, then the loop.
pk_status launch_sm_bicgstab(pk_csr* A, double* x, const double* r, const double* r0s, double* as, int maxit,
                             cudaStream_t s) {
  SmArgs a;
  pk_status e = sm_args(A, 2 * (uint64_t)maxit + 8, s, &a);
  if (e) return e;
  size_t smem;
  const int nv = sm_bi_vectors(A, &smem);
  launch_sm_publish(a, r, s);
  PK_CUDA(cudaGetLastError());
  return sm_launch(A, A->sm_irregular ? k_sm_bi<true> : k_sm_bi<false>, smem, a, SmBi{x, r, r0s, as, nv}, s);
}

}  // namespace pk
