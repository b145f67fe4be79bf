// Right-preconditioned restarted GMRES (flexible form: the preconditioned directions z_j are
// kept, so a rounded preconditioner is allowed) for A_sigma x = b with the two-level Schwarz
// preconditioner, the Krylov method paired with the restricted M_RAS2^{-1} (Sec. 2.2).
// Arnoldi by classical Gram-Schmidt applied twice, three passes over the basis (k_gm_pass).  The
// Givens rotations of the Hessenberg column and the triangular solve run on the device; the host
// reads only the residual estimate, one step behind the launches.
#include <algorithm>

#include "dd_common.cuh"

namespace dd {

namespace {
constexpr int kGmThreads = 512, kGmWarps = kGmThreads / 32;
constexpr int kGmMaxBlocks = 152;   // one block per SM
constexpr int kGmMaxBasis = 201;    // restart length at most 200, and one

// sums of a and b over the warp: the first exchange leaves a to the lower half and b to the
// upper, so both take five FP64 warp instructions together (the pipe charges whole ones);
// lane 0 returns a's sum, lane 16 b's
__device__ __forceinline__ double warp_sum_pair(double a, double b) {
  const bool up = (threadIdx.x & 16) != 0;
  double v = (up ? b : a) + __shfl_xor_sync(kFull, up ? a : b, 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}
}  // namespace

// One pass of the Gram-Schmidt of w against V_0 .. V_{nv-1}.  A block owns a run of seg entries;
// its warps take one vector (or, for few vectors, one part of one) each, so a projection costs
// seg / 32 FMAs and half a shuffle tree per block, and the run of w and its part of the
// basis are read from L2 once for both halves of the pass.
//   MODE 0: out[i] = h_i = (V_i, w)
//   MODE 1: w -= sum coef_i V_i, then out[i] = (V_i, w) and col[i] = coef_i + out_i
//   MODE 2: w -= sum coef_i V_i, then out[0] = ||w||^2, out[1] = 1 / ||w|| (0 for w = 0), col[nv] = ||w||
// Bound by the FP64 pipe (2 lanes per clock and SM): 4 n FMAs per basis vector and step over the
// three passes.  73.8k entries (L = 96, n = 24), average over a cycle of 30: 9.1, 11.3 and 8.5 us for
// the three modes, of which the FMAs take 8 us in all; the rest is the latency of a block's loads,
// its sums and the last block's.  Before, projections summed every value by a tree in every one of
// 304 blocks (15.5 us each) and eight launches made the step.
template <int MODE>
__global__ void __launch_bounds__(kGmThreads) k_gm_pass(long long n, int seg, int nv,
                                                        const double* const* __restrict__ V,
                                                        const double* __restrict__ coef, double* w,
                                                        double* __restrict__ partial, unsigned* counter,
                                                        double* __restrict__ out, double* __restrict__ col) {
  __shared__ const double* vp[kGmMaxBasis];
  __shared__ double cf[kGmMaxBasis], sp[kGmMaxBasis];
  __shared__ int s_last;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nb = gridDim.x;
  const long long t0 = blockIdx.x * (long long)seg;
  const long long t1 = min(n, t0 + seg);
  for (int i = threadIdx.x; i < nv; i += kGmThreads) {
    vp[i] = V[i];
    if (MODE > 0) cf[i] = coef[i];
  }
  __syncthreads();
  double nrm = 0.0;
  if (MODE > 0) {
    for (long long t = t0 + threadIdx.x; t < t1; t += kGmThreads) {
      double acc = 0.0;
#pragma unroll 8
      for (int i = 0; i < nv; ++i) acc = fma(cf[i], __ldg(vp[i] + t), acc);
      const double wv = w[t] - acc;
      w[t] = wv;
      if (MODE == 2) nrm = fma(wv, wv, nrm);
    }
    __syncthreads();   // the block's run of w is complete
  }
  if (MODE == 2) {
    nrm = warp_sum(nrm);
    if (lane == 0) sp[wid] = nrm;
    __syncthreads();
    if (wid == 0) {
      const double v = warp_sum(lane < kGmWarps ? sp[lane] : 0.0);
      if (lane == 0) partial[blockIdx.x] = v;
    }
  } else {
    // up to eight vectors: several warps per vector, each with a part of the run
    const int parts = nv <= kGmWarps / 2 ? kGmWarps / nv : 1;
    const long long len = t1 - t0, plen = ((len + parts - 1) / parts + 31) & ~31LL;
    for (int q = wid; q < nv * parts; q += 2 * kGmWarps) {
      const int i = q % nv, part = q / nv;
      const bool two = q + kGmWarps < nv * parts;   // only with parts == 1
      const double* va = vp[i];
      const double* vb = vp[two ? i + kGmWarps : i];
      const long long e0 = t0 + part * plen, e1 = min(t1, e0 + plen);
      double a = 0.0, b = 0.0;
      if (two) {
#pragma unroll 4
        for (long long t = e0 + lane; t < e1; t += 32) {
          const double wv = w[t];
          a = fma(__ldg(va + t), wv, a);
          b = fma(__ldg(vb + t), wv, b);
        }
      } else {
#pragma unroll 4
        for (long long t = e0 + lane; t < e1; t += 32) a = fma(__ldg(va + t), w[t], a);
      }
      a = warp_sum_pair(a, b);
      if (lane == 0) sp[q] = a;
      if (lane == 16 && two) sp[q + kGmWarps] = a;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nv; i += kGmThreads) {
      double v = sp[i];
      for (int k = 1; k < parts; ++k) v += sp[k * nv + i];
      partial[(size_t)i * nb + blockIdx.x] = v;
    }
  }
  // the last block adds the blocks' partial sums in block order
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(counter, 1u) == (unsigned)nb - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const int nsum = MODE == 2 ? 1 : nv;
  for (int i = wid; i < nsum; i += 2 * kGmWarps) {
    const bool two = i + kGmWarps < nsum;
    double a = 0.0, b = 0.0;
    for (int k = lane; k < nb; k += 32) {
      a += __ldcg(partial + (size_t)i * nb + k);
      if (two) b += __ldcg(partial + (size_t)(i + kGmWarps) * nb + k);
    }
    a = warp_sum_pair(a, b);
    const int e = lane == 0 ? i : i + kGmWarps;
    if (lane == 0 || (lane == 16 && two)) {
      out[e] = a;
      if (MODE == 1) col[e] = cf[e] + a;
      if (MODE == 2) {
        const double nrm = sqrt(a);
        col[nv] = nrm;
        out[1] = nrm > 0.0 ? 1.0 / nrm : 0.0;
      }
    }
  }
  if (threadIdx.x == 0) *counter = 0u;
}

// w[t] -= sum_i coef[i] V_i[t]   (sign = -1), or x[t] += sum_i coef[i] V_i[t] (sign = +1)
__global__ void __launch_bounds__(kThreads) k_multiaxpy(long long n, int nv, const double* const* __restrict__ V,
                                                        const double* __restrict__ coef, double sign, double* w) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x) {
    double acc = 0.0;
    for (int i = 0; i < nv; ++i) acc = fma(__ldg(coef + i), V[i][t], acc);
    w[t] = fma(sign, acc, w[t]);
  }
}

// v = w / ||w||: nrm2 holds ||w||^2 and, with have_inv, 1 / ||w|| behind it (a square root and a
// division by every thread took most of the 4.1 us of a pass over 73.8k entries)
__global__ void __launch_bounds__(kThreads) k_scale_by_norm(long long n, const double* __restrict__ w,
                                                            const double* __restrict__ nrm2, int have_inv, double* v) {
  double s;
  if (have_inv) {
    s = nrm2[1];
  } else {
    const double nv = sqrt(*nrm2);
    s = nv > 0.0 ? 1.0 / nv : 0.0;
  }
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x)
    v[t] = w[t] * s;
}

// Column j of the Hessenberg matrix (its entries 0 .. j + 1 written by the Gram-Schmidt passes):
// apply the earlier rotations, form the new one, update g; res[0] = |g[j+1]| (residual estimate).
// H is column-major with leading dimension ld = restart + 1.  One warp; the rotations are a
// serial chain of one thread over values staged in shared memory.
__global__ void k_givens(int j, int ld, double* H, double* cs, double* sn, double* g, double* res) {
  __shared__ double sc[kGmMaxBasis], ss[kGmMaxBasis], sh[kGmMaxBasis + 1];
  double* col = H + (size_t)j * ld;
  for (int i = threadIdx.x; i <= j + 1; i += blockDim.x) {
    sh[i] = col[i];
    if (i < j) {
      sc[i] = cs[i];
      ss[i] = sn[i];
    }
  }
  const double gj = g[j];
  __syncwarp();
  if (threadIdx.x == 0) {
    double a = sh[0];
    for (int i = 0; i < j; ++i) {
      const double nx = sh[i + 1], t = sc[i] * a + ss[i] * nx;
      a = -ss[i] * a + sc[i] * nx;
      sh[i] = t;
    }
    const double b = sh[j + 1];
    const double den = hypot(a, b);
    const double c = den > 0.0 ? a / den : 1.0, s = den > 0.0 ? b / den : 0.0;
    cs[j] = c;
    sn[j] = s;
    sh[j] = den;
    sh[j + 1] = 0.0;
    g[j + 1] = -s * gj;
    g[j] = c * gj;
    res[0] = fabs(s * gj);
  }
  __syncwarp();
  for (int i = threadIdx.x; i <= j + 1; i += blockDim.x) col[i] = sh[i];
}

// y = R^{-1} g (R the rotated Hessenberg, m x m upper triangle), column by column: y_i from the
// diagonal, then rows above it less R_ki y_i by the lanes.  One warp; with FITS the triangle is
// staged in shared memory first, so that a step is not a round trip to L2 (m = 30: one thread
// took 41 us).
template <bool FITS>
__global__ void k_backsolve(int m, int ld, const double* __restrict__ H, const double* __restrict__ g, double* y) {
  extern __shared__ double R[];
  __shared__ double acc[kGmMaxBasis];
  if (FITS)
    for (int i = threadIdx.x; i < m * m; i += 32) {
      const int c = i / m, r = i - c * m;
      if (r <= c) R[i] = H[(size_t)c * ld + r];
    }
  for (int i = threadIdx.x; i < m; i += 32) acc[i] = g[i];
  __syncwarp();
  for (int i = m - 1; i >= 0; --i) {
    const double* col = FITS ? R + (size_t)i * m : H + (size_t)i * ld;
    const double yi = acc[i] / col[i];
    __syncwarp();
    for (int k = threadIdx.x; k < i; k += 32) acc[k] = fma(-col[k], yi, acc[k]);
    if (threadIdx.x == 0) y[i] = yi;
    __syncwarp();
  }
}

// g = (beta, 0, ...) with beta = sqrt(nrm2)
__global__ void k_gmres_start(const double* __restrict__ nrm2, double* g, int len) {
  for (int i = threadIdx.x; i < len; i += blockDim.x) g[i] = (i == 0) ? sqrt(*nrm2) : 0.0;
}

// The two Gram-Schmidt passes of step j on w = W against V_0 .. V_j and the norm of what is left:
// h and the Hessenberg column j (unrotated, its last entry ||w||) on the device, ||w||^2 and 1 / ||w|| in
// nrm2.
// One block per SM and at least 128 entries each.  L = 96, n = 24, TF32, one GMRES solve of 69
// steps: 9.2 -> 5.2 ms with the host's read of the estimate one step behind the launches.
void launch_gm_orthogonalise(dd_ctx* c, int j, double* w, double* nrm2, cudaStream_t s) {
  const long long n = c->g.plen;
  const int nv = j + 1, ld = c->gm_restart + 1;
  long long seg = (n + kGmMaxBlocks - 1) / kGmMaxBlocks;
  seg = std::max(128LL, (seg + 31) & ~31LL);
  const int nb = (int)((n + seg - 1) / seg);
  double *h = c->gm_h, *h2 = c->gm_h + ld, *col = c->gm_H + (size_t)j * ld;
  const double* const* V = c->gm_Vptr;
  unsigned* cnt = c->cnt + CNT_GMRES;
  (k_gm_pass<0><<<nb, kGmThreads, 0, s>>>(n, (int)seg, nv, V, nullptr, w, c->gm_part, cnt, h, nullptr),
   dd::note_launch());
  (k_gm_pass<1><<<nb, kGmThreads, 0, s>>>(n, (int)seg, nv, V, h, w, c->gm_part, cnt, h2, col), dd::note_launch());
  (k_gm_pass<2><<<nb, kGmThreads, 0, s>>>(n, (int)seg, nv, V, h2, w, c->gm_part, cnt, nrm2, col), dd::note_launch());
  DD_CUDA(cudaGetLastError());
}

void launch_multiaxpy(dd_ctx* c, int nv, const double* const* V, const double* coef, double sign, double* w,
                      cudaStream_t s) {
  const long long n = c->g.plen;
  (k_multiaxpy<<<grid_blocks(n, kThreads), kThreads, 0, s>>>(n, nv, V, coef, sign, w), dd::note_launch());
  DD_CUDA(cudaGetLastError());
}

void launch_scale_by_norm(dd_ctx* c, const double* w, const double* nrm2, bool have_inv, double* v, cudaStream_t s) {
  const long long n = c->g.plen;
  (k_scale_by_norm<<<grid_blocks(n, kThreads), kThreads, 0, s>>>(n, w, nrm2, have_inv ? 1 : 0, v), dd::note_launch());
  DD_CUDA(cudaGetLastError());
}

void launch_givens(dd_ctx* c, int j, double* res, cudaStream_t s) {
  const int ld = c->gm_restart + 1;
  (k_givens<<<1, 32, 0, s>>>(j, ld, c->gm_H, c->gm_cs, c->gm_sn, c->gm_g, res), dd::note_launch());
  DD_CUDA(cudaGetLastError());
}

void launch_backsolve(dd_ctx* c, int m, cudaStream_t s) {
  const int ld = c->gm_restart + 1;
  const size_t sm = sizeof(double) * (size_t)m * m;
  if (sm <= 40 * 1024)
    (k_backsolve<true><<<1, 32, sm, s>>>(m, ld, c->gm_H, c->gm_g, c->gm_y), dd::note_launch());
  else
    (k_backsolve<false><<<1, 32, 0, s>>>(m, ld, c->gm_H, c->gm_g, c->gm_y), dd::note_launch());
  DD_CUDA(cudaGetLastError());
}

void launch_gmres_start(dd_ctx* c, const double* nrm2, cudaStream_t s) {
  (k_gmres_start<<<1, 64, 0, s>>>(nrm2, c->gm_g, c->gm_restart + 1), dd::note_launch());
  DD_CUDA(cudaGetLastError());
}

}  // namespace dd
