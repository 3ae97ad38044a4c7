// Pipelined CG (Alg. 2, Sec. 3.1) with the matrix in shared memory (pk_sm.cuh): one cooperative
// launch for the whole solve of a system that the SMs hold, between the thread-block cluster's
// sizes and a few hundred thousand rows.
//
// Iteration i:
//   fetch   the halo of p_i;
//   S_i     Ap_i with the block's parts of <Ap_i, Ap_i>, <p_i, Ap_i> (and of <r_i, r_i> from U_i);
//   reduce  block 0: convergence test on <r_i, r_i>, then alpha_i, beta_i by Eq. (3), broadcast;
//   U_i+1   r, p, publish p, then x and the part of <r, r> (while p travels).
// The launched form tests <r_i, r_i> before A p_i; here the test joins the reduction after it, so
// the last product of a solve is unused and an iteration has one grid-wide exchange instead of two.
// Rows, threads and summation orders are those of the launched kernels (the update kernel takes
// the same row blocks for systems of this size), so both give the same bits.
// JAC: with the Jacobi preconditioner (pk_pcg.cu): p = M^-1 r + beta p, and <r, M^-1 r>,
// <Ap, M^-1 Ap> in the place of <r, r>, <Ap, Ap> in Eq. (3); <r, r> still decides.
#include "pk_sm.cuh"

namespace pk {

namespace {

struct SmCg {
  double* x;
  const double* r;
  const double* p;
  const double* dinv;  // JAC
  int x_shared;        // x has room in shared memory (else only its owner reads it from global memory)
};

template <bool IRR, bool JAC>
__global__ void __launch_bounds__(kSmThreads, 2) k_sm_cg(SmArgs a, SmCg g) {
  extern __shared__ __align__(16) unsigned char smem[];
  DevState* st = a.st;
  if (state_done(st)) return;  // decided by the setup kernel, the same for every block
  constexpr int NV = JAC ? 4 : 3;
  constexpr int NVEC = JAC ? 5 : 4;
  SmLayout L = sm_layout<NVEC, 1>(smem, a);
  sm_shorten(L, a, g.x_shared ? 0 : 1);
  const SmBlock B = sm_begin(a, L);
  double *sp = L.vec[0], *sr = L.vec[1], *sa = L.vec[2], *sd = JAC ? L.vec[3] : nullptr, *sx = L.vec[NVEC - 1];
  double* const gx = g.x + B.r0;
  uint32_t ep = a.ep0;
#pragma unroll 1
  for (int l = threadIdx.x; l < B.rows; l += kSmThreads) {
    const double pv = g.p[B.r0 + l];
    sm_publish(a, B.r0 + l, pv, ep);
    sp[l] = pv;
    if (g.x_shared) sx[l] = gx[l];
    sr[l] = g.r[B.r0 + l];
    if (JAC) sd[l] = g.dinv[B.r0 + l];
  }
  const int maxit = st->maxit, trace_cap = st->trace_cap;
  double* const trace = st->trace;
  const double thr2 = st->thr2;
  // gamma: <r, M^-1 r> (without preconditioner <r, r> itself); vr, vz: this thread's parts
  double rr = st->rr, gamma = JAC ? st->s[0] : rr, vr = 0.0, vz = 0.0;
  for (int i = sm_zero();; ++i, ++ep) {
    if (!__syncthreads_and(sm_fetch(a, B, sp, ep))) break;
    double v[NV];
    v[0] = vr;
    v[1] = v[2] = 0.0;
    if (JAC) v[NV - 1] = vz;
    sm_product<IRR>(a, L, B, sp, [&](int row, double y) {
      const int l = row - B.r0;
      sa[l] = y;
      v[1] = fma(JAC ? y * sd[l] : y, y, v[1]);
      v[2] = fma(sp[l], y, v[2]);
    });
    double w[3];  // alpha, beta, decision
    const int sts = sm_reduce<NV, 3>(a, B, v, ep, w, [&](const double (&t)[NV], double (&word)[3]) {
      int status = kRunning;
      double alpha = 0.0, beta = 0.0;
      if (i >= 1) {
        rr = t[0];
        gamma = JAC ? t[NV - 1] : rr;
      }
      if (i >= 1 && (!isfinite(rr) || !isfinite(gamma))) status = PK_ERR_NAN;
      else if (i >= 1 && rr <= thr2) status = PK_OK;
      else if (i >= 1 && i >= maxit) status = PK_NOT_CONVERGED;
      else if (!isfinite(t[1]) || !isfinite(t[2])) status = PK_ERR_NAN;
      else if (t[2] <= 0.0) status = PK_NOT_SPD;
      else cg_coefficients_warp(gamma, t[1], t[2], alpha, beta);
      word[0] = alpha;
      word[1] = beta;
      word[2] = (double)status;
    }, [&](const double (&)[NV], const double (&word)[3]) {
      if (i >= 1) {
        st->iter = i;
        st->rr = rr;
        if (JAC) st->s[0] = gamma;
        if (trace && i - 1 < trace_cap) trace[(size_t)(i - 1) * 4 + 3] = rr;
      }
      if ((int)word[2] != kRunning) {
        finish(st, (int)word[2]);
        return;
      }
      st->alpha = word[0];
      st->beta = word[1];
      if (trace && i < trace_cap) {
        trace[(size_t)i * 4 + 0] = word[0];
        trace[(size_t)i * 4 + 1] = word[1];
      }
    });
    if (sts != kRunning) break;
    const double alpha = w[0], beta = w[1];
    // U_{i+1}: thread t takes the row pairs of K-CG-U; p first, x and <r, r> while it travels
    vr = vz = 0.0;
#pragma unroll 1
    for (int base = 0; base < B.rows; base += 2 * kStreamRows) {
      double2 pk[2], rn[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int l = base + 2 * ((int)threadIdx.x + u * kSmThreads);
        if (l < B.rows) {
          pk[u] = ld2(sp + l);
          const double2 ak = ld2(sa + l), rq = ld2(sr + l);
          rn[u].x = fma(-alpha, ak.x, rq.x);
          rn[u].y = fma(-alpha, ak.y, rq.y);
          double2 zn = rn[u], pn;
          if (JAC) {
            const double2 dk = ld2(sd + l);
            zn.x *= dk.x;
            zn.y *= dk.y;
          }
          pn.x = fma(beta, pk[u].x, zn.x);
          pn.y = fma(beta, pk[u].y, zn.y);
          sm_publish(a, B.r0 + l, pn.x, ep + 1);
          if (l + 1 < B.rows) sm_publish(a, B.r0 + l + 1, pn.y, ep + 1);
          st2(sp + l, pn);
          st2(sr + l, rn[u]);
          if (JAC) {
            vz = fma(rn[u].x, zn.x, vz);
            if (l + 1 < B.rows) vz = fma(rn[u].y, zn.y, vz);
          }
        }
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int l = base + 2 * ((int)threadIdx.x + u * kSmThreads);
        if (l < B.rows) {
          if (g.x_shared) {
            double2 xk = ld2(sx + l);
            xk.x = fma(alpha, pk[u].x, xk.x);
            xk.y = fma(alpha, pk[u].y, xk.y);
            st2(sx + l, xk);
          } else {  // (a caller's x need not be 16-byte aligned)
            gx[l] = fma(alpha, pk[u].x, gx[l]);
            if (l + 1 < B.rows) gx[l + 1] = fma(alpha, pk[u].y, gx[l + 1]);
          }
          vr = fma(rn[u].x, rn[u].x, vr);
          if (l + 1 < B.rows) vr = fma(rn[u].y, rn[u].y, vr);
        }
      }
    }
  }
  __syncthreads();
  if (g.x_shared)
#pragma unroll 1
    for (int l = threadIdx.x; l < B.rows; l += kSmThreads) gx[l] = sx[l];
}

using SmCgKernel = void (*)(SmArgs, SmCg);

SmCgKernel sm_cg_kernel(const pk_csr* A, bool jac) {
  return A->sm_irregular ? (jac ? k_sm_cg<true, true> : k_sm_cg<true, false>)
                         : (jac ? k_sm_cg<false, true> : k_sm_cg<false, false>);
}

}  // namespace

// Vectors in shared memory: all, or all but x; 0: does not fit.
static int sm_cg_vectors(const pk_csr* A, bool jac, size_t* smem) {
  const int all = jac ? 5 : 4;
  for (int nv = all; nv >= all - 1; --nv)
    if (sm_fits(A, (const void*)sm_cg_kernel(A, jac), nv, 1, smem)) return nv;
  return 0;
}

// Whether pipelined CG on A (jac: with the Jacobi preconditioner) can run as an SM loop here.
pk_status sm_cg_usable(pk_csr* A, bool jac, cudaStream_t s, bool* usable) {
  pk_status e = sm_prepare(A, s, usable);
  if (e || !*usable) return e;
  size_t smem;
  *usable = sm_cg_vectors(A, jac, &smem) > 0;
  return PK_OK;
}

// The loop, after the setup kernel (r0, p0, <r0,r0>, <b,b>; with dinv: <r0, M^-1 r0> too).
pk_status launch_sm_cg(pk_csr* A, double* x, const double* r, const double* p, const double* dinv, int maxit,
                       cudaStream_t s) {
  SmArgs a;
  pk_status e = sm_args(A, (uint64_t)maxit + 8, s, &a);
  if (e) return e;
  size_t smem;
  const int nv = sm_cg_vectors(A, dinv != nullptr, &smem);
  return sm_launch(A, sm_cg_kernel(A, dinv != nullptr), smem, a, SmCg{x, r, p, dinv, nv == (dinv ? 5 : 4)}, s);
}

}  // namespace pk
