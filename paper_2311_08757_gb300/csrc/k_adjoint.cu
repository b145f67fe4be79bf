// Projected PCG of the potential gradient: (A - lambda M) w = r with r orthogonal to phi and w
// M-orthogonal to phi, z = Pi M^{-1} r, Pi = I - phi (M phi)^T (see adjoint_pcg in api.cu).
// All scalars stay on the device: c->st holds rho = (r, Pi z), pq, alpha, beta, rr, the tolerance and
// the done flag that the preconditioner's kernels test; AdjScal the projections' coefficients.
// An iteration is four kernels beside the preconditioner.  Both projections are folded into the
// updates through scalars that the reductions yield anyway:
//   r <- r - alpha q - tp u   with tp = (phi, r - alpha q) = (phi, r) - alpha (phi, q)
//   p <- (z - t phi) + beta p with t = (u, z), (Pi z, y) = (z, y) - t (phi, y) for y = r, q
// The projected residual's (phi, r), of the size of rounding, is measured afresh in every
// iteration, so its drift does not accumulate.  Bound by latency (L = 256, n = 32: 2 MB per vector,
// all in L2).  The form before this took twenty launches and six host reads per iteration (about
// 190 us there, 60 of them kernels; 72 iterations per gradient); forward and backward together
// went from 32.8 to 24.9 ms.
#include "dd_common.cuh"

namespace dd {

namespace {
// blocks of the reducing passes: two entries per thread, at most three blocks per SM (76 registers)
int adj_blocks(const dd_ctx* c) { return grid_blocks(c->g.plen / 2, kThreads, 3); }
}  // namespace

// rr0 = (r, r), phr = (phi, r); tol2 = rtol^2 rr0 (rtol^2 preset in tol2 by the host)
__global__ void __launch_bounds__(kThreads) k_adj_init(long long n, const double2* __restrict__ r,
                                                       const double2* __restrict__ phi, PcgState* st, AdjScal* as,
                                                       double* partials, unsigned* counter) {
  double acc[2] = {0.0, 0.0};
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n / 2;
       t += (long long)gridDim.x * blockDim.x) {
    const double2 a = r[t], f = phi[t];
    acc[0] = fma(a.x, a.x, acc[0]);
    acc[0] = fma(a.y, a.y, acc[0]);
    acc[1] = fma(f.x, a.x, acc[1]);
    acc[1] = fma(f.y, a.y, acc[1]);
  }
  double tot[2];
  if (grid_sum_last<2>(acc, partials, counter, tot) && threadIdx.x == 0) {
    st->rr0 = st->rr = tot[0];
    st->tol2 *= tot[0];
    as->phr = tot[1];
    if (!isfinite(tot[0])) {
      st->status = DD_ENAN;
      st->done = 1;
    } else if (tot[0] == 0.0) {
      st->done = 1;
    }
  }
}

// p <- (z - t phi) + beta p
__global__ void __launch_bounds__(kThreads) k_adj_pupdate(long long n, const double2* __restrict__ z,
                                                          const double2* __restrict__ phi, double2* __restrict__ p,
                                                          const PcgState* st, const AdjScal* as) {
  if (st->done) return;
  const double t1 = as->t, beta = st->beta;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n / 2;
       t += (long long)gridDim.x * blockDim.x) {
    const double2 a = z[t], f = phi[t];
    double2 v = p[t];
    v.x = fma(beta, v.x, fma(-t1, f.x, a.x));
    v.y = fma(beta, v.y, fma(-t1, f.y, a.y));
    p[t] = v;
  }
}

// q = T p (T = A - lambda M), pq = (p, q), phq = (phi, q); alpha and tp
template <int P>
__global__ void __launch_bounds__(kThreads) k_adj_stencil(Geo g, const double* __restrict__ tab,
                                                          const double* __restrict__ p,
                                                          const double* __restrict__ phi, double* __restrict__ q,
                                                          PcgState* st, AdjScal* as, double* partials,
                                                          unsigned* counter) {
  if (st->done) return;
  const long long total = (long long)g.nxi * (P == 2 ? g.nxi : 1) * g.Ypad;
  double acc[2] = {0.0, 0.0};
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const Node nd = node_of<P>(g, t);
    const double v = stencil_at<P>(g, tab, p, nd.idx, cls_of<P>(g, nd));
    q[nd.idx] = v;
    acc[0] = fma(p[nd.idx], v, acc[0]);
    acc[1] = fma(phi[nd.idx], v, acc[1]);
  }
  double tot[2];
  if (grid_sum_last<2>(acc, partials, counter, tot) && threadIdx.x == 0) {
    if (!(tot[0] > 0.0)) {
      st->status = isfinite(tot[0]) ? DD_ENOTSPD : DD_ENAN;
      st->done = 1;
      return;
    }
    st->pq = tot[0];
    st->alpha = st->rho / tot[0];
    as->phq = tot[1];
    as->tp = fma(-st->alpha, tot[1], as->phr);
  }
}

// x += alpha p, r <- r - alpha q - tp u, rr = (r, r), phr = (phi, r); stop test
__global__ void __launch_bounds__(kThreads) k_adj_update(long long n, const double2* __restrict__ p,
                                                         const double2* __restrict__ q, const double2* __restrict__ u,
                                                         const double2* __restrict__ phi, double2* __restrict__ x,
                                                         double2* __restrict__ r, PcgState* st, AdjScal* as,
                                                         double* partials, unsigned* counter) {
  if (st->done) return;
  const double alpha = st->alpha, tp = as->tp;
  double acc[2] = {0.0, 0.0};
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n / 2;
       t += (long long)gridDim.x * blockDim.x) {
    const double2 pv = p[t], qv = q[t], uv = u[t], f = phi[t];
    double2 xv = x[t], rv = r[t];
    xv.x = fma(alpha, pv.x, xv.x);
    xv.y = fma(alpha, pv.y, xv.y);
    x[t] = xv;
    rv.x = fma(-tp, uv.x, fma(-alpha, qv.x, rv.x));
    rv.y = fma(-tp, uv.y, fma(-alpha, qv.y, rv.y));
    r[t] = rv;
    acc[0] = fma(rv.x, rv.x, acc[0]);
    acc[0] = fma(rv.y, rv.y, acc[0]);
    acc[1] = fma(f.x, rv.x, acc[1]);
    acc[1] = fma(f.y, rv.y, acc[1]);
  }
  double tot[2];
  if (grid_sum_last<2>(acc, partials, counter, tot) && threadIdx.x == 0) {
    st->rr = tot[0];
    st->iter += 1;
    as->phr = tot[1];
    if (!isfinite(tot[0])) {
      st->status = DD_ENAN;
      st->done = 1;
    } else if (tot[0] <= st->tol2) {
      st->done = 1;
    } else if (st->iter >= st->maxit) {
      st->status = DD_EMAXIT;
      st->done = 1;
    }
  }
}

// t = (u, z), rho = (r, Pi z) and, after the start, the Polak-Ribiere beta
// (Pi z_{k+1}, r_{k+1} - r_k) / (Pi z_k, r_k) = -(Pi z_{k+1}, q_k) / pq_k
__global__ void __launch_bounds__(kThreads) k_adj_dots(long long n, const double2* __restrict__ z,
                                                       const double2* __restrict__ u, const double2* __restrict__ r,
                                                       const double2* __restrict__ q, int start, PcgState* st,
                                                       AdjScal* as, double* partials, unsigned* counter) {
  if (st->done) return;
  double acc[3] = {0.0, 0.0, 0.0};
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n / 2;
       t += (long long)gridDim.x * blockDim.x) {
    const double2 a = z[t], uv = u[t], rv = r[t], qv = start ? make_double2(0.0, 0.0) : q[t];
    acc[0] = fma(uv.x, a.x, acc[0]);
    acc[0] = fma(uv.y, a.y, acc[0]);
    acc[1] = fma(rv.x, a.x, acc[1]);
    acc[1] = fma(rv.y, a.y, acc[1]);
    acc[2] = fma(qv.x, a.x, acc[2]);
    acc[2] = fma(qv.y, a.y, acc[2]);
  }
  double tot[3];
  if (grid_sum_last<3>(acc, partials, counter, tot) && threadIdx.x == 0) {
    const double t1 = tot[0];
    as->t = t1;
    st->rho = fma(-t1, as->phr, tot[1]);
    st->beta = start ? 0.0 : -fma(-t1, as->phq, tot[2]) / st->pq;
  }
}

void launch_adj_init(dd_ctx* c, const double* r, const double* phi, cudaStream_t s) {
  (k_adj_init<<<adj_blocks(c), kThreads, 0, s>>>(c->g.plen, (const double2*)r, (const double2*)phi, c->st, c->adj, c->red,
                                                 c->cnt + CNT_GRAD),
   dd::note_launch());
  DD_CUDA(cudaGetLastError());
}

void launch_adj_pupdate(dd_ctx* c, const double* phi, double* p, cudaStream_t s) {
  (k_adj_pupdate<<<grid_blocks(c->g.plen / 2, kThreads), kThreads, 0, s>>>(c->g.plen, (const double2*)c->z,
                                                                           (const double2*)phi, (double2*)p, c->st,
                                                                           c->adj),
   dd::note_launch());
  DD_CUDA(cudaGetLastError());
}

void launch_adj_stencil(dd_ctx* c, const double* tab, const double* p, const double* phi, double* q, cudaStream_t s) {
  const Geo& g = c->g;
  const int nb = grid_blocks((long long)g.nxi * (g.p == 2 ? g.nxi : 1) * g.Ypad, kThreads, 4);
  if (g.p == 1)
    (k_adj_stencil<1><<<nb, kThreads, 0, s>>>(g, tab, p, phi, q, c->st, c->adj, c->red, c->cnt + CNT_GRAD),
     dd::note_launch());
  else
    (k_adj_stencil<2><<<nb, kThreads, 0, s>>>(g, tab, p, phi, q, c->st, c->adj, c->red, c->cnt + CNT_GRAD),
     dd::note_launch());
  DD_CUDA(cudaGetLastError());
}

void launch_adj_update(dd_ctx* c, const double* p, const double* q, const double* u, const double* phi, double* x,
                       double* r, cudaStream_t s) {
  (k_adj_update<<<adj_blocks(c), kThreads, 0, s>>>(c->g.plen, (const double2*)p, (const double2*)q, (const double2*)u,
                                                   (const double2*)phi, (double2*)x, (double2*)r, c->st, c->adj, c->red,
                                                   c->cnt + CNT_GRAD),
   dd::note_launch());
  DD_CUDA(cudaGetLastError());
}

void launch_adj_dots(dd_ctx* c, const double* u, const double* r, const double* q, int start, cudaStream_t s) {
  (k_adj_dots<<<adj_blocks(c), kThreads, 0, s>>>(c->g.plen, (const double2*)c->z, (const double2*)u, (const double2*)r,
                                                 (const double2*)q, start, c->st, c->adj, c->red, c->cnt + CNT_GRAD),
   dd::note_launch());
  DD_CUDA(cudaGetLastError());
}

}  // namespace dd
