// FP64 local solves of the plain method: y_i = A_{sigma,i}^{-1} R_i r for every subdomain
// (Sec. 3.1), A_{sigma,i} = R_i A_sigma R_i^T on the interior nodes of the open overlapping box.
//
// All subdomains with the same clipping (left / interior / right per axis) have the same
// matrix, so it is factored once per type.  Cut into the node planes c1 = 0 .. K-1 along x_1
// (m = w2 nyi unknowns each) it is block tridiagonal with couplings B that are themselves
// stencils (3 taps per node for p = 1, 9 for p = 2).  It is eliminated from both ends towards
// the plane t = K / 2 (a twisted block LDL^T):
//   S_0 = D_0,  S_k = D_k - B_{k,k-1} S_{k-1}^{-1} B_{k-1,k}        k = 1 .. t-1 (left side)
//   the mirror image for k = K-1 .. t+1 (right side), and S_t takes both contributions.
// Stored are the dense inverses S_k^{-1}, so a solve is
//   h_k = S_k^{-1} (f_k - B h_{k -+ 1})  towards t,   x_t = h_t,   x_k = h_k - S_k^{-1} (B x_{k +- 1})
// away from it: K steps of one dense m x m product each, where the banded triangular sweeps
// took 2 K m dependent steps.  The work is 2 m^2 multiply-adds per plane and sweep pair
// against 2 m (m + 1) for the banded factor.  On the pipe the rows come in warps of 32 and the columns in
// chunks of 8 (4 for planes of at most 32 unknowns); the sweeps paid by the band's warps of 32.
#include <algorithm>

#include "dd_async.cuh"

namespace dd {

// Planes of the types' local boxes: type ty has K = w1 planes of m = w2 nyi unknowns; inverse
// Schur complements are ms x ms, ms the largest m (mmax) rounded up to whole warps (rows and columns
// past m hold the identity).
struct BlkGeo {
  int ntypes, ms, mmax, kmax;
  int w1[kMaxTypes], w2[kMaxTypes], lo1[kMaxTypes], lo2[kMaxTypes];
};

__device__ __forceinline__ const double* blk_inverse(const BlkGeo& B, const double* Sinv, int ty, int k) {
  return Sinv + ((size_t)ty * B.kmax + k) * B.ms * B.ms;
}

// sum over the taps with x_1 offset d1 of A_sigma(row, neighbour) v(neighbour), row (plane k,
// local column c2, slot sj) of type ty; neighbours outside the box are left out (homogeneous
// Dirichlet on its boundary)
template <int P>
__device__ __forceinline__ double blk_couple(const Geo& g, const double* __restrict__ tabS, const BlkGeo& B, int ty,
                                             int k, int c2, int sj, int d1, const double* v) {
  const int a1 = (B.lo1[ty] + k) % g.n;
  const int cls = (P == 1 ? a1 : a1 * g.n + (B.lo2[ty] + c2) % g.n) * g.Ypad + sj;
  const int row = c2 * g.nyi + sj;
  double s = 0.0;
#pragma unroll
  for (int d2 = (P == 1 ? 0 : -1); d2 <= (P == 1 ? 0 : 1); ++d2)
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy) {
      const int tap = (P == 1) ? (d1 + 1) * 3 + dy + 1 : ((d1 + 1) * 3 + d2 + 1) * 3 + dy + 1;
      const bool in = sj + dy >= 0 && sj + dy < g.nyi && (P == 1 || (c2 + d2 >= 0 && c2 + d2 < B.w2[ty]));
      if (in) s = fma(__ldg(tabS + (size_t)tap * g.ncls + cls), v[row + d2 * g.nyi + dy], s);
    }
  return s;
}

// ----------------------------------------------------------------------------------------
// Set-up.  Step s of the two-sided recursion works on every chain (type, side) at once:
// k_schur_form writes S_k, then one k_gj_panel launch per 32 pivots inverts it in place (block
// Gauss-Jordan without pivoting: S_k is a Schur complement of a positive definite matrix), from
// one buffer into another, the last one into Sinv.
// ----------------------------------------------------------------------------------------
struct BlkChain {
  int ty, k, prev_l, prev_r;   // plane to form, planes it takes contributions from (-1: none)
};

// chain ch at step s (s < 0: the meeting planes); ty < 0 where the chain has ended
__device__ __forceinline__ BlkChain blk_chain(const BlkGeo& B, int ch, int s) {
  if (s < 0) {
    const int K = B.w1[ch], t = K / 2;
    return BlkChain{ch, t, t > 0 ? t - 1 : -1, t + 1 < K ? t + 1 : -1};
  }
  const int ty = ch >> 1, K = B.w1[ty], t = K / 2;
  if (ch & 1) return s < K - 1 - t ? BlkChain{ty, K - 1 - s, -1, s > 0 ? K - s : -1} : BlkChain{-1, 0, -1, -1};
  return s < t ? BlkChain{ty, s, s > 0 ? s - 1 : -1, -1} : BlkChain{-1, 0, -1, -1};
}

// rows i of S_k, one block per row: T = B(i, :) S_prev^{-1} in shared memory, then
// S(i, j) = D(i, j) - sum_v T(v) B(j, v).  81 (p = 2) multiply-adds per entry done as 9 + 9.
template <int P>
__global__ void k_schur_form(Geo g, BlkGeo B, const double* __restrict__ tabS, const double* __restrict__ Sinv, int s,
                             double* __restrict__ out) {
  extern __shared__ double T[];
  const BlkChain c = blk_chain(B, blockIdx.y, s);
  if (c.ty < 0) return;
  const int ms = B.ms, m = B.w2[c.ty] * g.nyi, i = blockIdx.x;
  double* row = out + ((size_t)blockIdx.y * ms + i) * ms;
  if (i >= m) {
    for (int j = threadIdx.x; j < ms; j += blockDim.x) row[j] = (i == j) ? 1.0 : 0.0;
    return;
  }
  const int c2i = i / g.nyi, sji = i % g.nyi;
  const int a1 = (B.lo1[c.ty] + c.k) % g.n;
  const int cls = (P == 1 ? a1 : a1 * g.n + (B.lo2[c.ty] + c2i) % g.n) * g.Ypad + sji;
  for (int side = 0; side < 2; ++side) {
    const int prev = side ? c.prev_r : c.prev_l, d1 = side ? 1 : -1;
    __syncthreads();
    if (prev < 0) {
      for (int v = threadIdx.x; v < m; v += blockDim.x) T[side * ms + v] = 0.0;
      continue;
    }
    const double* Sp = blk_inverse(B, Sinv, c.ty, prev);
    for (int v = threadIdx.x; v < m; v += blockDim.x) {
      double t = 0.0;
      for (int d2 = (P == 1 ? 0 : -1); d2 <= (P == 1 ? 0 : 1); ++d2)
        for (int dy = -1; dy <= 1; ++dy) {
          if (sji + dy < 0 || sji + dy >= g.nyi || (P == 2 && (c2i + d2 < 0 || c2i + d2 >= B.w2[c.ty]))) continue;
          const int tap = (P == 1) ? (d1 + 1) * 3 + dy + 1 : ((d1 + 1) * 3 + d2 + 1) * 3 + dy + 1;
          t = fma(__ldg(tabS + (size_t)tap * g.ncls + cls), Sp[(size_t)(i + d2 * g.nyi + dy) * ms + v], t);
        }
      T[side * ms + v] = t;
    }
  }
  __syncthreads();
  for (int j = threadIdx.x; j < ms; j += blockDim.x) {
    double v = 0.0;
    if (j < m) {
      const int c2j = j / g.nyi, sjj = j % g.nyi;
      const int d2 = c2j - c2i, dy = sjj - sji;
      if (d2 >= -1 && d2 <= 1 && dy >= -1 && dy <= 1 && (P == 2 || d2 == 0)) {
        const int tap = (P == 1) ? 3 + dy + 1 : (3 + d2 + 1) * 3 + dy + 1;
        v = tabS[(size_t)tap * g.ncls + cls];
      }
      if (c.prev_l >= 0) v -= blk_couple<P>(g, tabS, B, c.ty, c.k, c2j, sjj, -1, T);
      if (c.prev_r >= 0) v -= blk_couple<P>(g, tabS, B, c.ty, c.k, c2j, sjj, 1, T + ms);
    }
    row[j] = v;
  }
}

// Pivots I = 32 p .. 32 p + 31 of the in-place inversion, one block per 32-column tile J and
// chain.  Every block inverts the 32 x 32 pivot block itself (the blocks need not wait on one
// another), then, from the old matrix A to the new one:
//   J = I:   A(I, I) = P,  A(K, I) = -A(K, I) P          (P the inverse of A(I, I))
//   J != I:  A(I, J) = P A(I, J) = U,  A(K, J) -= A(K, I) U
constexpr int kGjThreads = 256;
__global__ void __launch_bounds__(kGjThreads) k_gj_panel(Geo g, BlkGeo B, const double* __restrict__ in,
                                                         double* __restrict__ out, double* __restrict__ Sinv, int s,
                                                         int p, int* flag) {
  __shared__ double Pm[32][33], U[32][33], C[32][33];
  __shared__ double s_inv;
  const BlkChain c = blk_chain(B, blockIdx.y, s);
  if (c.ty < 0) return;
  const int ms = B.ms, jt = blockIdx.x, tid = threadIdx.x, col = tid & 31, r0 = tid >> 5;
  const double* A = in + (size_t)blockIdx.y * ms * ms;
  double* O = (Sinv != nullptr) ? Sinv + ((size_t)c.ty * B.kmax + c.k) * ms * ms : out + (size_t)blockIdx.y * ms * ms;
  for (int q = 0; q < 4; ++q) {
    const int r = r0 + 8 * q;
    Pm[r][col] = A[(size_t)(32 * p + r) * ms + 32 * p + col];
    U[r][col] = A[(size_t)(32 * p + r) * ms + 32 * jt + col];
  }
  __syncthreads();
  const int npiv = min(32, B.w2[c.ty] * g.nyi - 32 * p);   // pivots past m are rows of the identity
  for (int k = 0; k < npiv; ++k) {
    if (r0 == 0) {
      double piv = Pm[k][k];
      if (!(piv > 0.0)) {
        if (col == 0) atomicOr(flag, 1);
        piv = 1.0;
      }
      piv = 1.0 / piv;
      if (col == 0) s_inv = piv;
    }
    __syncthreads();
    const double iv = s_inv;
    double nv[4];
    for (int q = 0; q < 4; ++q) {
      const int r = r0 + 8 * q;
      if (r == k) nv[q] = (col == k) ? iv : Pm[k][col] * iv;
      else nv[q] = (col == k) ? -Pm[r][k] * iv : fma(-Pm[r][k] * iv, Pm[k][col], Pm[r][col]);
    }
    __syncthreads();
    for (int q = 0; q < 4; ++q) Pm[r0 + 8 * q][col] = nv[q];
    __syncthreads();
  }
  // U = P A(I, J) (J != I), or P itself for the tile that holds the pivots
  if (jt != p) {
    double u[4] = {0.0, 0.0, 0.0, 0.0};
    for (int l = 0; l < 32; ++l)
      for (int q = 0; q < 4; ++q) u[q] = fma(Pm[r0 + 8 * q][l], U[l][col], u[q]);
    __syncthreads();
    for (int q = 0; q < 4; ++q) U[r0 + 8 * q][col] = u[q];
  } else {
    for (int q = 0; q < 4; ++q) U[r0 + 8 * q][col] = Pm[r0 + 8 * q][col];
  }
  __syncthreads();
  for (int kt = 0; kt < ms / 32; ++kt) {
    if (kt == p) {
      for (int q = 0; q < 4; ++q) O[(size_t)(32 * p + r0 + 8 * q) * ms + 32 * jt + col] = U[r0 + 8 * q][col];
      continue;
    }
    double a[4];
    for (int q = 0; q < 4; ++q) {
      C[r0 + 8 * q][col] = A[(size_t)(32 * kt + r0 + 8 * q) * ms + 32 * p + col];
      a[q] = (jt != p) ? A[(size_t)(32 * kt + r0 + 8 * q) * ms + 32 * jt + col] : 0.0;
    }
    __syncthreads();
#pragma unroll 8
    for (int l = 0; l < 32; ++l)
      for (int q = 0; q < 4; ++q) a[q] = fma(-C[r0 + 8 * q][l], U[l][col], a[q]);
    for (int q = 0; q < 4; ++q) O[(size_t)(32 * kt + r0 + 8 * q) * ms + 32 * jt + col] = a[q];
    __syncthreads();
  }
}

static BlkGeo blk_geo(const dd_ctx* c) {
  BlkGeo B{};
  B.ntypes = c->ntypes;
  B.mmax = 1;
  for (int t = 0; t < c->ntypes; ++t) {
    B.w1[t] = c->type_w1[t];
    B.w2[t] = c->type_w2[t];
    B.kmax = std::max(B.kmax, B.w1[t]);
    B.mmax = std::max(B.mmax, B.w2[t] * c->g.nyi);
    const Sub& s = c->subs_h[c->rep_of_type[t]];
    B.lo1[t] = s.lo1;
    B.lo2[t] = s.lo2;
  }
  B.ms = (B.mmax + 31) / 32 * 32;
  return B;
}

// forms and inverts the Schur complements of every type; *flag is set on a non-positive pivot
void block_factor(dd_ctx* c, int* flag) {
  const Geo& g = c->g;
  const BlkGeo B = blk_geo(c);
  if (sizeof(double) * 2 * B.ms > 220 * 1024) throw Error(DD_EINVAL, "fixed direction too long for the FP64 local solves");
  const size_t blk = (size_t)B.ms * B.ms;
  cudaStream_t st = c->stream;
  if (!c->blkS) c->blkS = (double*)dev_alloc(c, sizeof(double) * blk * B.ntypes * B.kmax);
  double* buf = nullptr;
  DD_CUDA(cudaMallocAsync(&buf, sizeof(double) * blk * 4 * B.ntypes, st));
  double* half[2] = {buf, buf + blk * 2 * B.ntypes};
  const int np = B.ms / 32;
  const size_t smem = sizeof(double) * 2 * B.ms;
  auto step = [&](int s, int chains) {
    if (g.p == 1) (k_schur_form<1><<<dim3(B.ms, chains), 128, smem, st>>>(g, B, c->tabS, c->blkS, s, half[0]), note_launch());
    else (k_schur_form<2><<<dim3(B.ms, chains), 128, smem, st>>>(g, B, c->tabS, c->blkS, s, half[0]), note_launch());
    for (int p = 0; p < np; ++p)
      (k_gj_panel<<<dim3(np, chains), kGjThreads, 0, st>>>(g, B, half[p & 1], half[(p + 1) & 1], p + 1 == np ? c->blkS : nullptr,
                                                           s, p, flag),
       note_launch());
  };
  if (smem > 48 * 1024) {
    DD_CUDA(cudaFuncSetAttribute(k_schur_form<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
    DD_CUDA(cudaFuncSetAttribute(k_schur_form<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
  }
  for (int s = 0; s < B.kmax / 2; ++s) step(s, 2 * B.ntypes);
  step(-1, B.ntypes);
  DD_CUDA(cudaGetLastError());
  DD_CUDA(cudaFreeAsync(buf, st));
}

// ----------------------------------------------------------------------------------------
// The solves.  A cluster of 2 CR blocks takes R subdomains of one type; its first CR blocks
// walk the planes from the left, the others from the right, and they meet at plane t through
// distributed shared memory.  With CR > 1 the rows of a plane's product are divided among the
// side's blocks (each writes its rows of h into all of them).  Inside a block, a warp takes 32
// rows and one of PW column ranges of the product for one subdomain.
//
// One DFMA occupies an SM's FP64 pipe for 16 clocks (64 for a warp alone on its sub-partition),
// so the products are bound by that pipe as soon as every sub-partition has a warp; loads of
// S_k^{-1} are 8 columns ahead (across planes too) and cost nothing.
// ----------------------------------------------------------------------------------------
struct BlkShape {
  int R, PW, RW, rgl;   // subdomains, column ranges and row warps per block; row groups per block
  int nch, cpp;         // chunks of eight columns and columns of a range: the PW ranges cover mmax, not
                        // ms, whose further columns meet zeros
};

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync_all() {
  cluster_arrive();
  cluster_wait();
}
// store to the same shared-memory variable of block `rank` of the cluster
__device__ __forceinline__ void dsm_store(double* local, unsigned rank, double v) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(local);
  unsigned ra;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(rank));
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(ra), "d"(v) : "memory");
}

// arrive at the mbarrier at the same place in block `rank` of the cluster, after this thread's
// stores into that block; mbar_wait_cluster waits for such arrivals (bounded, as mbar_wait)
__device__ __forceinline__ void dsm_arrive(uint32_t local_bar, unsigned rank) {
  uint32_t ra;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(local_bar), "r"(rank));
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(ra) : "memory");
}
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t a, uint32_t parity, int* err, int code) {
  for (long long i = 0; i < (1LL << 26); ++i) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(a), "r"(parity)
        : "memory");
    if (ok) return true;
    if (i > 256) __nanosleep(64);
  }
  atomicOr(err, code);
  return false;
}

// Planes of more than 7040 unknowns (three planes at most, the local vectors were bounded before) keep
// the block's vectors in global memory (GLOB: 4 R ms doubles per block at `scratch`).
template <int P, int CR, bool GLOB>
__global__ void __launch_bounds__(1024) k_block_solve(Geo g, BlkGeo B, BlkShape sh, const Sub* __restrict__ subs,
                                                      const int2* __restrict__ groups,
                                                      const int* __restrict__ sub_of_slot,
                                                      const double* __restrict__ r, const double* __restrict__ tabS,
                                                      const double* __restrict__ Sinv, double* __restrict__ Y, int kpad,
                                                      const PcgState* st, double* scratch) {
  if (st != nullptr && st->done) return;
  cluster_arrive();   // waited for before the first store into another block's shared memory
  extern __shared__ double s_blk[];
  const unsigned rank = cluster_rank();
  const size_t vlen = (size_t)4 * sh.R * B.ms;
  double* const sm = GLOB ? scratch + blockIdx.x * vlen : s_blk;
  // store to the same variable of block `to` of the cluster
  auto remote = [&](double* local, unsigned to, double v) {
    if (GLOB) local[((long long)to - (long long)rank) * (long long)vlen] = v;
    else dsm_store(local, to, v);
  };
  const int side = (int)rank / CR, cr = (int)rank % CR;
  const int2 grp = groups[blockIdx.x / (2 * CR)];
  const int ms = B.ms, R = sh.R;
  const int ntr = (int)blockDim.x / R;              // threads of one subdomain
  const int rr = (int)threadIdx.x / ntr, tr = (int)threadIdx.x - rr * ntr;
  const bool live = rr < grp.y;
  const Sub sb = subs[sub_of_slot[grp.x + (live ? rr : 0)]];
  const int ty = sb.type, K = B.w1[ty], w2 = B.w2[ty], nyi = g.nyi, m = w2 * nyi, t = K / 2;
  const int nmine = side ? K - 1 - t : t, k0 = side ? K - 1 : 0, dir = side ? -1 : 1;
  // shared memory: the product's argument, h (two planes in turn), the right side's
  // contribution to plane t, the column ranges' partial sums
  double* gv = sm + (size_t)rr * ms;
  double* hb[2] = {sm + (size_t)(R + rr) * ms, sm + (size_t)(2 * R + rr) * ms};
  double* ub = sm + (size_t)(3 * R + rr) * ms;
  double* part = (GLOB ? s_blk : sm + (size_t)4 * R * ms) + (size_t)rr * sh.PW * sh.rgl * 32;
  const int lane = tr & 31, w = tr >> 5, rw = w % sh.RW, pw = w / sh.RW;
  const int cpp = sh.cpp, nch = sh.nch;             // columns and 8-column chunks of this warp's range
  const int rg_first = cr * sh.rgl + rw, rg_end = min((cr + 1) * sh.rgl, ms >> 5);
  const long long cstride = (P == 1) ? g.Ypad : (long long)g.ncx * g.Ypad;
  const double* rb = r + ((P == 1) ? (long long)sb.lo1 * g.Ypad : ((long long)sb.lo1 * g.ncx + sb.lo2) * g.Ypad);
  double* yb = Y + (size_t)(grp.x + (live ? rr : 0)) * kpad;
  auto barrier = [&]() {
    if (CR > 1) cluster_sync_all();
    else __syncthreads();
  };
  // f_k at row (0 past the plane)
  auto load_f = [&](int k, int row) -> double {
    if (!live || row >= m) return 0.0;
    const int c2 = (P == 1) ? 0 : row / nyi, sj = row - c2 * nyi;
    return rb[(long long)k * cstride + (long long)c2 * g.Ypad + sj];
  };
  double nx[8];   // the next chunk of S^{-1}, loaded ahead of its use
  auto load8 = [&](const double* p) {
#pragma unroll
    for (int q = 0; q < 8; ++q) nx[q] = __ldg(p + (size_t)q * ms);
  };
  auto chunk0 = [&](int k, int rg) { return blk_inverse(B, Sinv, ty, k) + (size_t)pw * cpp * ms + rg * 32 + lane; };
  // h = S_k^{-1} gv by this block's warps; emit(row, h) runs in the column range 0 warps.  knext:
  // the plane whose first chunk is loaded before returning (-1: none).
  auto product = [&](int k, int knext, auto&& emit) {
    for (int rg = rg_first; rg < rg_end; rg += sh.RW) {
      double acc = 0.0;
      const double* base = chunk0(k, rg);
      for (int ch = 0; ch < nch; ++ch) {
        double cu[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) cu[q] = nx[q];
        if (ch + 1 < nch) load8(base + (size_t)(ch + 1) * 8 * ms);
        else if (rg + sh.RW < rg_end) load8(chunk0(k, rg + sh.RW));
        else if (knext >= 0) load8(chunk0(knext, rg_first));
        const double* a = gv + pw * cpp + ch * 8;
#pragma unroll
        for (int q = 0; q < 8; ++q) acc = fma(cu[q], a[q], acc);
      }
      if (sh.PW == 1) emit(rg * 32 + lane, acc);
      else part[((size_t)pw * sh.rgl + (rg - cr * sh.rgl)) * 32 + lane] = acc;
    }
    if (sh.PW > 1) {
      __syncthreads();
      if (pw == 0)
        for (int rg = rg_first; rg < rg_end; rg += sh.RW) {
          double acc = part[(size_t)(rg - cr * sh.rgl) * 32 + lane];
          for (int j = 1; j < sh.PW; ++j) acc += part[((size_t)j * sh.rgl + (rg - cr * sh.rgl)) * 32 + lane];
          emit(rg * 32 + lane, acc);
        }
    }
  };
  // hb[b](row) = v in every block of this side
  auto share = [&](double* h, int row, double v) {
    if (CR == 1) h[row] = v;
    else
#pragma unroll
      for (int q = 0; q < CR; ++q) remote(h + row, side * CR + q, v);
  };
  auto ypos = [&](int k, int row) -> size_t {
    const int c2 = (P == 1) ? 0 : row / nyi;
    return (size_t)(k * w2 + c2) * g.Ypad + (row - c2 * nyi);
  };
  const int smax = (CR > 1) ? t : nmine;   // left steps t >= right steps: equal barrier counts
  if (nmine > 0 && rg_first < rg_end) load8(chunk0(k0, rg_first));
  for (int row = tr; row < ms; row += ntr) gv[row] = load_f(nmine > 0 ? k0 : t, row);
  __syncthreads();
  cluster_wait();
  // ---- towards plane t
  for (int s = 0; s < smax; ++s) {
    const bool on = s < nmine;
    const int k = k0 + dir * s;
    double* h = hb[s & 1];
    double fn = 0.0;   // f of the next plane, loaded beside the product
    if (on) {
      if (s + 1 < nmine) fn = load_f(k + dir, tr);
      product(k, s + 1 < nmine ? k + dir : t, [&](int row, double v) {
        share(h, row, v);
        if (live && row < m) yb[ypos(k, row)] = v;
      });
    }
    barrier();
    if (on && s + 1 < nmine) {
      for (int row = tr; row < ms; row += ntr) {
        double v = 0.0;
        if (row < m) {
          const int c2 = (P == 1) ? 0 : row / nyi;
          v = (row == tr ? fn : load_f(k + dir, row)) -
              blk_couple<P>(g, tabS, B, ty, k + dir, c2, row - c2 * nyi, -dir, h);
        }
        gv[row] = v;
      }
      __syncthreads();
    }
  }
  // ---- plane t: the right side sends B h_{t+1}, the left side solves and sends x_t back
  if (side == 1)
    for (int row = tr; row < ms; row += ntr) {
      const int c2 = (P == 1) ? 0 : row / nyi;
      const double v = (row < m && nmine > 0)
                           ? blk_couple<P>(g, tabS, B, ty, t, c2, row - c2 * nyi, 1, hb[(nmine - 1) & 1]) : 0.0;
      remote(ub + row, cr, v);
    }
  cluster_sync_all();
  int cur = t & 1;   // the buffer that takes x_t: the left side has just read the other one
  if (side == 0) {
    for (int row = tr; row < ms; row += ntr) {
      double v = 0.0;
      if (row < m) {
        const int c2 = (P == 1) ? 0 : row / nyi;
        v = load_f(t, row) - ub[row];
        if (nmine > 0) v -= blk_couple<P>(g, tabS, B, ty, t, c2, row - c2 * nyi, -1, hb[(nmine - 1) & 1]);
      }
      gv[row] = v;
    }
    __syncthreads();
    if (nmine == 0 && rg_first < rg_end) load8(chunk0(t, rg_first));
    product(t, nmine > 0 ? t - 1 : -1, [&](int row, double v) {
#pragma unroll
      for (int q = 0; q < 2 * CR; ++q) remote(hb[cur] + row, q, v);
      if (live && row < m) yb[ypos(t, row)] = v;
    });
  } else if (nmine > 0 && rg_first < rg_end) {
    load8(chunk0(t + 1, rg_first));
  }
  cluster_sync_all();
  // ---- away from plane t
  for (int s = smax - 1; s >= 0; --s) {
    const bool on = s < nmine;
    const int k = k0 + dir * s;
    if (on) {
      for (int row = tr; row < ms; row += ntr) {
        const int c2 = (P == 1) ? 0 : row / nyi;
        gv[row] = (row < m) ? blk_couple<P>(g, tabS, B, ty, k, c2, row - c2 * nyi, dir, hb[cur]) : 0.0;
      }
      __syncthreads();
      double* h = hb[cur ^ 1];
      product(k, s > 0 ? k - dir : -1, [&](int row, double v) {
        double x = 0.0;
        if (row < m && live) {
          double* y = yb + ypos(k, row);   // h_k, stored by this thread on the way in
          x = *y - v;
          *y = x;
        }
        share(h, row, x);
      });
      cur ^= 1;
    }
    barrier();
  }
}

// Planes of at most 32 unknowns (ms = 32): a lane holds a row, so the couplings are shuffles and a
// product needs no shared memory but its argument.  PW warps take one subdomain; each forms the
// product over its share of the columns, and all of them add the PW partial sums and form the
// next argument themselves (the sub-partitions are idle then, and one barrier per plane is
// enough).  A plane's S^{-1} is one 8 KB block; a warp of its own brings the planes into a ring
// by bulk copies ahead of their use.  f, h_k and (p = 1) the coupling coefficients are loaded two
// planes ahead.  The two sides meet through one mbarrier per subdomain.
//
// With one warp per subdomain the FP64 pipe bounds long boxes, and thin planes leave most of it to
// padding; there the form above cost more than the banded sweeps it replaced.
// TRIM (planes of at most 28 unknowns): the products end at the plane's own columns, inside a group of
// four.  us per launch at L = 2048, banded / groups of four / TRIM: 19 unknowns (n = 20) 170 / 157 / 137, 23 (n = 24)
// 249 / 223 / 198, 27 (n = 14) 153 / 135 / 122; the same at L = 400.  29 unknowns and more have at most three columns to
// leave out: 31 (n = 32) 440 / 334 / 335, at L = 400 381 / 94 / 101.
// HALF (planes of at most 16 unknowns, TRIM too): a warp takes two subdomains, each half of it one's rows, so
// every instruction works for both; the pair reads the same S^{-1}.  us per launch, banded / TRIM / HALF: 15 unknowns
// (n = 16) L = 310 99 / 36 / 35, L = 2048 113 / 97 / 58, L = 8000 371 / 344 / 193; 5 (n = 12) L = 4000 60 / 82 / 47; 3 (n = 4)
// L = 20000 111 / 135 / 83.
constexpr int ERR_BLK_WAIT = 1 << 8;   // error-word bit: a plane of S^{-1} or the other side did not arrive in time
constexpr int row_stages(int PW) { return PW == 1 ? 3 : 6; }
constexpr size_t row_smem(int PW) { return row_stages(PW) * 32 * 32 * sizeof(double); }

constexpr int kRowTrimMax = 28, kRowHalfMax = 16;
template <int P, int PW, bool TRIM = false, bool HALF = false>
__global__ void __launch_bounds__(160, P == 1 && PW == 1 ? 7 : 3) k_block_solve_row(Geo g, BlkGeo B, const Sub* __restrict__ subs,
                                                         const int2* __restrict__ groups,
                                                         const int* __restrict__ sub_of_slot,
                                                         const double* __restrict__ r, const double* __restrict__ tabS,
                                                         const double* __restrict__ Sinv, double* __restrict__ Y,
                                                         int kpad, const PcgState* st, int* err) {
  constexpr int CPP = HALF ? 16 : 32 / PW, MS = 32, NT = (P == 1) ? 3 : 9, D = row_stages(PW);
  if (st != nullptr && st->done) return;
  extern __shared__ __align__(128) double s_ring[];  // [D][32][32]
  __shared__ __align__(16) double s_g[4][32];        // per warp: the product's argument
  __shared__ double s_part[2][4][32];                // partial sums, alternating
  __shared__ double s_mid[4][32];                    // left side: B h_{t+1}; right side: x_t
  __shared__ __align__(8) unsigned long long s_bar[2 * D + 4];   // full, empty, meeting
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (int)(blockDim.x >> 5) - 1;   // nw working warps
  const uint32_t bar = smem_u32(s_bar);
  // The barriers exist before any thread arrives, so the cluster barrier's release and acquire show
  // them to both blocks: the other side's first arrival at the meeting may follow its wait at once.
  if (threadIdx.x == 0) {
    for (int i = 0; i < D; ++i) {
      mbar_init(bar + 8 * i, 1);
      mbar_init(bar + 8 * (D + i), nw);
    }
    for (int i = 0; i < 4; ++i) mbar_init(bar + 8 * (2 * D + i), 32);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  cluster_arrive();
  const int side = (int)cluster_rank();
  const int2 grp = groups[blockIdx.x >> 1];
  const int ty = subs[sub_of_slot[grp.x]].type, K = B.w1[ty], t = K / 2;
  const int nmine = side ? K - 1 - t : t, k0 = side ? K - 1 : 0, dir = side ? -1 : 1;
  const int nprod = 2 * nmine + (side ? 0 : 1);      // products: inwards, plane t (left side), outwards
  cluster_wait();
  if (w == nw) {   // the ring's producer
    if (lane == 0) {
      // the columns that the shares cover, in whole groups of four
      const uint32_t bytes = PW * (((B.w2[ty] * g.nyi + PW - 1) / PW + 3) & ~3) * MS * sizeof(double);
      int q = 0;
      for (; q < nprod; ++q) {
        const int sl = q % D;
        if (q >= D && !mbar_wait(bar + 8 * (D + sl), (uint32_t)(q / D - 1) & 1u, err, ERR_BLK_WAIT)) break;
        const int i = q < nmine ? q : 2 * nmine - q - (side ? 1 : 0);   // plane i from this side's end (nmine: t)
        mbar_expect_tx(bar + 8 * sl, bytes);
        bulk_g2s(smem_u32(s_ring + sl * MS * MS), blk_inverse(B, Sinv, ty, k0 + dir * i), bytes, bar + 8 * sl);
      }
      // the last copy into each slot: a warp that gave up has not waited for it
      for (int k = max(0, q - D); k < q; ++k) mbar_wait(bar + 8 * (k % D), (uint32_t)(k / D) & 1u, err, ERR_BLK_WAIT);
    }
    return;
  }
  const int ws = w / PW, pw = w % PW;                // the warps of one subdomain (HALF: of a pair of them)
  const int half = HALF ? lane & 16 : 0, row = lane - half;
  const int rr = HALF ? 2 * ws + (half >> 4) : ws;
  const bool live = rr < grp.y;
  const Sub sb = subs[sub_of_slot[grp.x + (live ? rr : 0)]];
  const int w2 = B.w2[ty], nyi = g.nyi, m = w2 * nyi;
  const int cpp = ((m + PW - 1) / PW + 3) & ~3;      // columns of this warp's share (S and g are 0 past m)
  const bool in = row < m;
  const int c2 = (P == 1) ? 0 : row / nyi, sj = row - c2 * nyi;
  const long long cstride = (P == 1) ? g.Ypad : (long long)g.ncx * g.Ypad;
  const double* rb = r + ((P == 1) ? (long long)sb.lo1 * g.Ypad : ((long long)sb.lo1 * g.ncx + sb.lo2) * g.Ypad) +
                     (long long)c2 * g.Ypad + sj;
  double* yb = Y + (size_t)(grp.x + (live ? rr : 0)) * kpad + c2 * g.Ypad + sj;
  const int ystride = w2 * g.Ypad;
  bool dead = false;   // a wait gave up: the error word tells the host, later waits are skipped
  auto wait = [&](uint32_t b, uint32_t parity) {
    if (!dead && !mbar_wait(b, parity, err, ERR_BLK_WAIT)) dead = true;
  };
  auto load_f = [&](int k) -> double { return (live && in) ? rb[(long long)k * cstride] : 0.0; };
  // coefficients of this row's couplings to the plane at offset d1 of plane k (0 outside the box)
  const double* tb = tabS + ((P == 1) ? 0 : (B.lo2[ty] + c2) % g.n * g.Ypad) + sj;
  const int clsn = (P == 1) ? g.Ypad : g.n * g.Ypad;
  auto load_cf = [&](int k, int d1, double (&cf)[NT]) {
    const double* q = tb + (size_t)((B.lo1[ty] + k) % g.n) * clsn;
#pragma unroll
    for (int e = 0; e < NT; ++e) {
      const int d2 = (P == 1) ? 0 : e / 3 - 1, dy = e % 3 - 1;
      const bool ok = in && sj + dy >= 0 && sj + dy < nyi && (P == 1 || (c2 + d2 >= 0 && c2 + d2 < w2));
      cf[e] = ok ? __ldg(q + (size_t)((d1 + 1) * NT + e) * g.ncls) : 0.0;
    }
  };
  // v - sum of the couplings times the neighbour rows' h
  auto less_coupling = [&](double v, const double (&cf)[NT], double h) -> double {
    double hn[NT];
#pragma unroll
    for (int e = 0; e < NT; ++e) {
      const int off = (P == 1) ? e - 1 : (e / 3 - 1) * nyi + e % 3 - 1;
      hn[e] = __shfl_sync(kFull, h, HALF ? half + ((row + off) & 15) : (lane + off) & 31);
    }
#pragma unroll
    for (int e = 0; e < NT; ++e) v = fma(-cf[e], hn[e], v);
    return v;
  };
  int buf = 0, q = 0, sl = 0, ph = 0;   // product q reads ring slot sl at parity ph
  // init + S_k^{-1} g (this lane's row) for the next plane in turn
  auto product = [&](double gl, double init) -> double {
    double* gs = s_g[w];
    __syncwarp();
    gs[lane] = gl;
    __syncwarp();
    wait(bar + 8 * sl, (uint32_t)ph);
    const double* Sp = s_ring + sl * MS * MS + pw * cpp * MS + row;
    const double2* ga = reinterpret_cast<const double2*>(gs + half + pw * cpp);
    double acc = init;
    // four columns at a time, the next four loaded beside them
    double a0 = Sp[0], a1 = Sp[MS], a2 = Sp[2 * MS], a3 = Sp[3 * MS];
    double2 u = ga[0], v = ga[1];
#pragma unroll
    for (int b = 0; b < CPP; b += 4) {
      if (b < cpp) {
        double n0 = 0.0, n1 = 0.0, n2 = 0.0, n3 = 0.0;
        double2 nu = u, nv = v;
        if (b + 4 < CPP) {   // (columns past the share are in range and not used)
          n0 = Sp[(b + 4) * MS];
          n1 = Sp[(b + 5) * MS];
          n2 = Sp[(b + 6) * MS];
          n3 = Sp[(b + 7) * MS];
          nu = ga[b / 2 + 2];
          nv = ga[b / 2 + 3];
        }
        acc = fma(a0, u.x, acc);
        if (!TRIM || b + 1 < m) acc = fma(a1, u.y, acc);
        if (!TRIM || b + 2 < m) acc = fma(a2, v.x, acc);
        if (!TRIM || b + 3 < m) acc = fma(a3, v.y, acc);
        a0 = n0; a1 = n1; a2 = n2; a3 = n3;
        u = nu; v = nv;
      }
    }
    if (PW > 1) s_part[buf][w][lane] = acc;
    __syncwarp();
    if (lane == 0) mbar_arrive(bar + 8 * (D + sl));
    if (++sl == D) {
      sl = 0;
      ph ^= 1;
    }
    if (PW == 1) return acc;
    asm volatile("bar.sync %0, %1;" ::"r"(1 + ws), "n"(32 * PW) : "memory");
    double p[PW];
#pragma unroll
    for (int j = 0; j < PW; ++j) p[j] = s_part[buf][ws * PW + j][lane];
    acc = p[0];
#pragma unroll
    for (int j = 1; j < PW; ++j) acc += p[j];
    buf ^= 1;
    return acc;
  };
  // plane i (0 .. nmine - 1) of this side counted from its end; plane nmine is t
  auto pl = [&](int i) { return k0 + dir * i; };
  double h = 0.0, gl = load_f(pl(0)), f1 = load_f(pl(min(1, nmine))), f2 = load_f(pl(min(2, nmine)));
  double c1[NT], c2n[NT], c3[NT];
  load_cf(pl(min(1, nmine)), -dir, c1);
  if (P == 1) load_cf(pl(min(2, nmine)), -dir, c2n);
  // ---- towards plane t; after the last product h couples to plane t
  for (int i = 0; i < nmine; ++i) {
    const int k = pl(i), k3 = pl(min(i + 3, nmine));
    const double f3 = load_f(k3);
    if (P == 1) load_cf(k3, -dir, c3);
    h = product(gl, 0.0);
    if (pw == 0 && live && in) yb[(size_t)k * ystride] = h;
    // the right side leaves f_t to the left one and sends its coupling alone
    gl = less_coupling((side && i + 1 == nmine) ? 0.0 : f1, c1, h);
    f1 = f2;
    f2 = f3;
    if (P == 1) {
#pragma unroll
      for (int e = 0; e < NT; ++e) {
        c1[e] = c2n[e];
        c2n[e] = c3[e];
      }
    } else {
      load_cf(pl(min(i + 2, nmine)), -dir, c1);
    }
  }
  // ---- plane t: the right side's first warp sends its coupling, the left side's x_t
  const uint32_t meet = bar + 8 * (2 * D + ws);
  auto send = [&](double v) {
    if (pw != 0) return;
    dsm_store(&s_mid[ws][lane], side ^ 1, v);
    dsm_arrive(meet, side ^ 1);
  };
  auto receive = [&]() -> double {
    if (!dead && !mbar_wait_cluster(meet, 0, err, ERR_BLK_WAIT)) dead = true;
    return s_mid[ws][lane];
  };
  if (side == 1) send(nmine > 0 ? gl : 0.0);
  // h_k is read back by the warp that stored it
  const bool mine = pw == 0 && live && in;
  auto load_h = [&](int i) -> double { return (mine && i >= 0) ? yb[(size_t)pl(i) * ystride] : 0.0; };
  double h1 = load_h(nmine - 1), h2 = load_h(nmine - 2);
  if (nmine > 0) load_cf(pl(nmine - 1), dir, c1);
  if (P == 1) load_cf(pl(max(nmine - 2, 0)), dir, c2n);
  const double other = receive();   // left: the right side's coupling; right: x_t
  double x = other;
  if (side == 0) {
    x = product(gl + other, 0.0);
    send(x);
    if (mine) yb[(size_t)t * ystride] = x;
  }
  // ---- away from it: x_k = h_k - S_k^{-1} (B x), h_k the initial value of the product
  for (int i = nmine - 1; i >= 0; --i) {
    const int k = pl(i);
    const double h3 = load_h(i - 2);
    if (P == 1) load_cf(pl(max(i - 2, 0)), dir, c3);
    gl = less_coupling(0.0, c1, x);
    x = product(gl, h1);
    if (mine) yb[(size_t)k * ystride] = x;
    h1 = h2;
    h2 = h3;
    if (P == 1) {
#pragma unroll
      for (int e = 0; e < NT; ++e) {
        c1[e] = c2n[e];
        c2n[e] = c3[e];
      }
    } else {
      load_cf(pl(max(i - 1, 0)), dir, c1);
    }
  }
  // A thread that has seen the meeting complete knows that the other block stores no more into this one.
  // One whose wait gave up (it ran through the remaining, meaningless work without waiting) keeps the
  // block alive until every thread of the other has ended or is here too (ended threads count as
  // arrived); a barrier for all on every path cost 2% at L = 2048.
  if (dead) cluster_sync_all();
}

// The launch shape.  Planes of at most 32 unknowns: PW warps per subdomain and side, 4 while every
// sub-partition gets one of them at most (2 nsub PW warps over 4 per SM: 76 subdomains), 2 while it gets
// two (304), then 1.  A warp alone leaves most of its pipe idle, so two half-length products beside each other beat
// one of full length, but a third starts another round (us per launch for 1 / 2 / 4: h = 1/32, L = 64
// 72 / 48 / 42, L = 100 71 / 50 / 55, L = 301 84 / 66 / 123, L = 350 87 / 121 / 124; h = 1/20, l = 1.5,
// L = 301 48 / 43 / 79, L = 350 49 / 76 / 78; h = 1/12, L = 200 24 / 22 / 30).  With PW = 1 the
// blocks take 1, 2 or 4 subdomains: small blocks spread evenly over few rounds (us per launch for
// 1 / 2 / 4 at h = 1/32: L = 512 88 / 96 / 96, L = 1000 187 / 158 / 177, L = 2048 361 / 353 / 319,
// where four warps also share each plane's copy); pairs of subdomains per warp (HALF) by the same rule.
// Larger planes (k_block_solve): a warp per 32 rows, up to 4 subdomains and 32 warps per block, up to 4 column
// ranges while that leaves an SM sub-partition at most 5 warps, up to 4 blocks per side while the grid
// does not fill the SMs.  The results do not depend on the subdomains per block.
//
// Measured against the banded triangular sweeps this replaced (one warp per one or two
// subdomains, 2 n_loc dependent steps; us per application by events, the coarse branch beside it): p = 1,
// h = 1/32, delta = 4: L = 37 375 -> 41, L = 512 390 -> 98, L = 2048 440 -> 328 (295 in the trace of a solve; the
// FP64 pipe needs 288 for its instructions); ell = 2, L = 301 1335 -> 216; p = 2, h = 1/16, delta = 2 (planes of
// 285): L = 6 5678 -> 298 (204 in a solve), L = 16 5689 -> 1604 (pipe floor of the banded flops 1330).
// Planes of m unknowns stored as ms x ms, banded / all ms columns / the mmax columns that are there: m = 35, ms = 64
// (h = 1/24, ell = 1.5, delta = 3) L = 64 561 / 82 / 83, L = 512 565 / 279 / 205, L = 2048 655 / 903 / 595; m = 47,
// ms = 64 (ell = 2) L = 2048 848 / 904 / 699; m = 71, ms = 96 (ell = 3) L = 2048 3923 / 1943 / 1494.
void block_groups(dd_ctx* c, int want) {
  const BlkGeo B = blk_geo(c);
  const int RG = B.ms / 32, N = c->g.nsub, sms = 152;
  int cr = 1, PW = 1, RW = 1, rgl = 1, R = 1;
  bool glob = false, half = false;
  if (RG == 1) {
    PW = 8 * N <= 4 * sms ? 4 : (4 * N <= 8 * sms ? 2 : 1);
    half = c->g.p == 1 && PW == 1 && B.mmax <= kRowHalfMax;
    const int pair = half ? 2 : 1;                     // subdomains per warp
    const double x = 2.0 * N / (4 * sms * pair);       // warps with a half chain per sub-partition
    R = std::min(want > 0 ? want : pair * (x <= 2.0 ? 1 : (x <= 5.0 ? 2 : 4)), pair * 4 / PW);
  } else {
    while (cr < 4 && 2 * cr <= RG && (long long)2 * N * cr * 2 <= sms) cr *= 2;
    while (cr < 4 && (RG + cr - 1) / cr > 32) cr *= 2;
    rgl = (RG + cr - 1) / cr;
    RW = std::min(rgl, 32);
    const long long warps = (long long)2 * N * cr * RW;
    while (PW < 4 && warps * PW * 2 <= 4 * sms * 5 && RW * PW * 2 <= 32) PW *= 2;
    R = want > 0 ? want : std::max(1, 4 / (PW * RW));
    while (R > 1 && R * RW * PW > 32) R /= 2;
    const size_t per = sizeof(double) * ((size_t)4 * B.ms + (PW > 1 ? (size_t)PW * rgl * 32 : 0));
    while (R > 1 && per * R > 200 * 1024) R /= 2;
    glob = per * R > 220 * 1024;
  }
  c->blk_cr = cr;
  c->blk_R = R;
  c->blk_PW = PW;
  c->blk_RW = RW;
  c->blk_rgl = rgl;
  std::vector<int2> grp;
  for (int t = 0; t < c->ntypes; ++t)
    for (int j = 0; j < c->type_count[t]; j += R)
      grp.push_back(make_int2(c->type_first[t] + j, std::min(R, c->type_count[t] - j)));
  c->ngroups = (int)grp.size();
  c->blk_half = half;
  c->blk_glob = glob;   // R = 1 and cr = 4 then, whatever was asked for: allocated once
  if (glob && !c->blk_vec) c->blk_vec = (double*)dev_alloc(c, sizeof(double) * 4 * B.ms * (size_t)grp.size() * 2 * cr);
  DD_CUDA(cudaMemcpyAsync(c->groups, grp.data(), sizeof(int2) * grp.size(), cudaMemcpyHostToDevice, c->stream));
  DD_CUDA(cudaStreamSynchronize(c->stream));   // grp is a temporary
}

template <typename... KArgs, typename... Args>
static void launch_cluster(void (*kern)(KArgs...), int blocks, int threads, size_t smem, int cluster, cudaStream_t s,
                           Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cluster;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  DD_CUDA(cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...));
  note_launch();
}

template <int P, int CR, bool GLOB = false>
static void launch_block_solve_t(dd_ctx* c, const BlkGeo& B, const double* r, cudaStream_t s) {
  const int nch = (B.mmax + 8 * c->blk_PW - 1) / (8 * c->blk_PW);
  const BlkShape sh{c->blk_R, c->blk_PW, c->blk_RW, c->blk_rgl, nch, 8 * nch};
  static PerDeviceOnce attr;
  once_per_device(attr, [] {
    DD_CUDA(cudaFuncSetAttribute(k_block_solve<P, CR, GLOB>, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
  });
  const size_t smem = sizeof(double) * sh.R * ((GLOB ? 0 : (size_t)4 * B.ms) + (sh.PW > 1 ? (size_t)sh.PW * sh.rgl * 32 : 0));
  launch_cluster(k_block_solve<P, CR, GLOB>, c->ngroups * 2 * CR, 32 * sh.R * sh.PW * sh.RW, smem, 2 * CR, s, c->g, B, sh,
                 (const Sub*)c->subs, (const int2*)c->groups, (const int*)c->sub_of_slot, r, (const double*)c->tabS,
                 (const double*)c->blkS, c->Y64, c->kpad, (const PcgState*)c->st, c->blk_vec);
}

template <int P>
static void launch_block_solve_p(dd_ctx* c, const double* r, cudaStream_t s) {
  const BlkGeo B = blk_geo(c);
  if (B.ms == 32) {
    static PerDeviceOnce attr;   // static + dynamic shared memory above 48 KB
    once_per_device(attr, [] {
      DD_CUDA(cudaFuncSetAttribute(k_block_solve_row<P, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024));
      DD_CUDA(cudaFuncSetAttribute(k_block_solve_row<P, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024));
    });
    auto kern = c->blk_PW == 1 ? k_block_solve_row<P, 1> : (c->blk_PW == 2 ? k_block_solve_row<P, 2> : k_block_solve_row<P, 4>);
    if (c->blk_half) kern = k_block_solve_row<1, 1, true, true>;
    else if (P == 1 && c->blk_PW == 1 && B.mmax <= kRowTrimMax) kern = k_block_solve_row<1, 1, true>;
    const int warps = c->blk_half ? (c->blk_R + 1) / 2 : c->blk_R * c->blk_PW;
    launch_cluster(kern, c->ngroups * 2, 32 * (warps + 1), row_smem(c->blk_PW), 2, s, c->g, B, (const Sub*)c->subs,
                   (const int2*)c->groups, (const int*)c->sub_of_slot, r, (const double*)c->tabS,
                   (const double*)c->blkS, c->Y64, c->kpad, (const PcgState*)c->st, c->dev_err + 8);
  } else if (c->blk_glob) {
    launch_block_solve_t<P, 4, true>(c, B, r, s);
  } else if (c->blk_cr == 1) {
    launch_block_solve_t<P, 1>(c, B, r, s);
  } else if (c->blk_cr == 2) {
    launch_block_solve_t<P, 2>(c, B, r, s);
  } else {
    launch_block_solve_t<P, 4>(c, B, r, s);
  }
}

void launch_block_solve(dd_ctx* c, const double* r, cudaStream_t s) {
  if (c->g.p == 1) launch_block_solve_p<1>(c, r, s);
  else launch_block_solve_p<2>(c, r, s);
}

}  // namespace dd
