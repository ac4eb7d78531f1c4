// Batched GMRES on the stacked real and imaginary parts (Sec. 4.1, Sec. 4.3:
// "Call GMRES with b = -iFQ").  The operator is only real-linear (it contains
// a complex conjugation), so the unknown is x = [Re S; Im S] in R^{2 N^2} and
// every inner product is <a, b> = Re sum conj(a) b; all Krylov coefficients
// are real.
//
// Each slot (one value of k) runs its own Arnoldi process; all slots advance
// in lock step and a per-slot flag masks slots whose cycle has finished.
// Orthogonalisation is classical Gram-Schmidt: one pass of dot products
// against all basis vectors, one update pass.  Basis vectors are stored
// unnormalised (v~_i) with a per-slot scale sigma_i = 1/||v~_i|| applied by
// every reader, which saves a normalisation pass.
//
// Reductions are two-level with a fixed order (per-block partials in FP64,
// then a single block per slot), so a slot's result does not depend on which
// other slots share the launch.
#pragma once
#include "passes.cuh"

namespace dbar {

// Block sum of per-thread partials: within each warp in the partials' own
// precision (FP32 for the inner solve: GB300's FP64 pipe cannot keep up with
// one FP64 operation per element at HBM speed), across warps in FP64.
template <typename T>
__device__ __forceinline__ double block_sum_256(T v, double* sh) {
  v = warp_sum_t(v, 32);
  const int w = threadIdx.x >> 5;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[w] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += sh[i];
  return s;  // valid in thread 0
}

// part[slot][i][chunk] = <v~_i, w>, w = sigma_j v~_j + KS, i = 0..j
template <typename T>
__global__ void __launch_bounds__(KR_THREADS) k_dots(const KryArgs a, const cx<T>* __restrict__ V,
                                                      long long vss, const cx<T>* __restrict__ KS,
                                                      long long kss, int j) {
  __shared__ double red[KR_THREADS / 32][129];
  const int slot = blockIdx.y;
  if (!a.run[slot]) return;
  const long long len = box_len(a.box, slot, a.n);
  const long long base = (long long)blockIdx.x * KR_CHUNK + threadIdx.x;
  const cx<T>* Vs = V + (size_t)slot * vss;
  const T sj = (T)a.sigma[(size_t)slot * a.mp1 + j];
  cx<T> w[KR_EPT];
#pragma unroll
  for (int e = 0; e < KR_EPT; ++e) {
    const long long idx = base + (long long)e * KR_THREADS;
    if (idx < len) {
      const cx<T> vj = ldg(Vs + (size_t)j * a.n + idx);
      const cx<T> ks = ldg(KS + (size_t)slot * kss + idx);
      w[e] = mkc(sj * vj.re + ks.re, sj * vj.im + ks.im);
    } else {
      w[e] = mkc((T)0, (T)0);
    }
  }
  const int wid = threadIdx.x >> 5;
  for (int i = 0; i <= j; ++i) {
    T s = 0;
#pragma unroll
    for (int e = 0; e < KR_EPT; ++e) {
      const long long idx = base + (long long)e * KR_THREADS;
      if (idx < len) {
        const cx<T> vi = ldg(Vs + (size_t)i * a.n + idx);
        s += vi.re * w[e].re + vi.im * w[e].im;
      }
    }
    const T d = warp_sum_t(s, 32);
    if ((threadIdx.x & 31) == 0) red[wid][i] = (double)d;
  }
  __syncthreads();
  for (int i = threadIdx.x; i <= j; i += blockDim.x) {
    double s = 0.0;
    for (int w2 = 0; w2 < KR_THREADS / 32; ++w2) s += red[w2][i];
    a.part[((size_t)slot * a.mp1 + i) * a.nchunk + blockIdx.x] = s;
  }
}

// H[slot][j][i] = h_i = sigma_i sum_chunks part;  coef[slot][i] = h_i sigma_i
// One warp per slot (KR_THREADS / 32 slots per block): the j + 1 reductions are
// warp shuffles, not block barriers, and thousands of small slots share blocks.
static __global__ void __launch_bounds__(KR_THREADS) k_finalize_h(const KryArgs a, double* H, int j, int nslots) {
  const int slot = blockIdx.x * (KR_THREADS / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (slot >= nslots || !a.run[slot]) return;
  for (int i = 0; i <= j; ++i) {
    double s = 0.0;
    const double* p = a.part + ((size_t)slot * a.mp1 + i) * a.nchunk;
    for (int c = lane; c < a.nchunk; c += 32) s += p[c];
    s = warp_sum(s, 32);
    if (lane == 0) {
      const double sg = a.sigma[(size_t)slot * a.mp1 + i];
      const double h = s * sg;
      H[((size_t)slot * (a.mp1 - 1) + j) * a.mp1 + i] = h;
      a.coef[(size_t)slot * a.mp1 + i] = h * sg;
    }
  }
}

// v~_{j+1} = sigma_j v~_j + KS - sum_i coef_i v~_i ; part2 = ||v~_{j+1}||^2 partials
template <typename T>
__global__ void __launch_bounds__(KR_THREADS) k_update(const KryArgs a, cx<T>* __restrict__ V, long long vss,
                                                        const cx<T>* __restrict__ KS, long long kss, int j) {
  __shared__ double sh[KR_THREADS / 32];
  const int slot = blockIdx.y;
  if (!a.run[slot]) return;
  const long long len = box_len(a.box, slot, a.n);
  const long long base = (long long)blockIdx.x * KR_CHUNK + threadIdx.x;
  cx<T>* Vs = V + (size_t)slot * vss;
  const T sj = (T)a.sigma[(size_t)slot * a.mp1 + j];
  cx<T> w[KR_EPT];
#pragma unroll
  for (int e = 0; e < KR_EPT; ++e) {
    const long long idx = base + (long long)e * KR_THREADS;
    if (idx < len) {
      const cx<T> vj = ldg(Vs + (size_t)j * a.n + idx);
      const cx<T> ks = ldg(KS + (size_t)slot * kss + idx);
      w[e] = mkc(sj * vj.re + ks.re, sj * vj.im + ks.im);
    } else {
      w[e] = mkc((T)0, (T)0);
    }
  }
  for (int i = 0; i <= j; ++i) {
    const T c = (T)a.coef[(size_t)slot * a.mp1 + i];
#pragma unroll
    for (int e = 0; e < KR_EPT; ++e) {
      const long long idx = base + (long long)e * KR_THREADS;
      if (idx < len) {
        const cx<T> vi = ldg(Vs + (size_t)i * a.n + idx);
        w[e] = mkc(w[e].re - c * vi.re, w[e].im - c * vi.im);
      }
    }
  }
  T s = 0;
#pragma unroll
  for (int e = 0; e < KR_EPT; ++e) {
    const long long idx = base + (long long)e * KR_THREADS;
    if (idx < len) {
      Vs[(size_t)(j + 1) * a.n + idx] = w[e];
      s += w[e].re * w[e].re + w[e].im * w[e].im;
    }
  }
  const double tot = block_sum_256(s, sh);
  if (threadIdx.x == 0) a.part2[(size_t)slot * a.nchunk + blockIdx.x] = tot;
}


// Givens step for Hessenberg column j of a slot whose rows 0..j+1 are in Hc:
// applies the earlier rotations, forms rotation j, updates g and the step
// counters; returns true when the slot's cycle stops after this column
// (residual estimate below the threshold, cycle full, iteration cap, or a
// zero subdiagonal: the Krylov space is invariant).
__device__ inline bool givens_column(const CycleState& c, int slot, int j, double* Hc) {
  const int m = c.m;
  const double sub = Hc[j + 1];
  double* cs = c.cs + (size_t)slot * m;
  double* sn = c.sn + (size_t)slot * m;
  double* g = c.g + (size_t)slot * (m + 1);
  for (int i = 0; i < j; ++i) {
    const double t0 = cs[i] * Hc[i] + sn[i] * Hc[i + 1];
    Hc[i + 1] = -sn[i] * Hc[i] + cs[i] * Hc[i + 1];
    Hc[i] = t0;
  }
  const double rho = hypot(Hc[j], Hc[j + 1]);
  double cj = 1.0, sj = 0.0;
  if (rho > 0.0) {
    cj = Hc[j] / rho;
    sj = Hc[j + 1] / rho;
  }
  cs[j] = cj;
  sn[j] = sj;
  Hc[j] = rho;
  Hc[j + 1] = 0.0;
  g[j + 1] = -sj * g[j];
  g[j] = cj * g[j];
  c.nsteps[slot] = j + 1;
  c.itot[slot] += 1;
  return fabs(g[j + 1]) <= c.thr[slot] || j + 1 >= m || sub == 0.0 || c.itot[slot] - c.cit[slot] >= c.max_iter;
}

// Norm of the new vector, Givens rotation of column j, residual estimate.
// One warp per slot, as k_finalize_h.
static __global__ void __launch_bounds__(KR_THREADS) k_givens(const KryArgs a, CycleState c, int j, int nslots) {
  const int slot = blockIdx.x * (KR_THREADS / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (slot >= nslots || !c.run[slot]) return;
  double s = 0.0;
  for (int q = lane; q < a.nchunk; q += 32) s += a.part2[(size_t)slot * a.nchunk + q];
  s = warp_sum(s, 32);
  if (lane != 0) return;
  const int m = c.m;
  const double nrm = sqrt(s);
  double* Hc = c.H + ((size_t)slot * m + j) * (m + 1);
  Hc[j + 1] = nrm;
  c.sigma[(size_t)slot * (m + 1) + j + 1] = nrm > 0.0 ? 1.0 / nrm : 0.0;
  if (givens_column(c, slot, j, Hc)) c.run[slot] = 0;
}

// y = R^{-1} g (back substitution), ycoef_i = y_i sigma_i.
static __global__ void k_solve_y(CycleState c, int nslots) {
  const int slot = blockIdx.x * blockDim.x + threadIdx.x;
  if (slot >= nslots) return;
  const int ns = c.active[slot] ? c.nsteps[slot] : 0;
  const int m = c.m;
  double* y = c.ycoef + (size_t)slot * (m + 1);
  const double* g = c.g + (size_t)slot * (m + 1);
  for (int i = ns - 1; i >= 0; --i) {
    double s = g[i];
    for (int l = i + 1; l < ns; ++l) s -= c.H[((size_t)slot * m + l) * (m + 1) + i] * y[l];
    const double d = c.H[((size_t)slot * m + i) * (m + 1) + i];
    y[i] = d != 0.0 ? s / d : 0.0;
  }
  for (int i = 0; i < ns; ++i) y[i] *= c.sigma[(size_t)slot * (m + 1) + i];
  c.nsteps[slot] = ns;
}

// x += sum_i ycoef_i v~_i   (basis in T; x stored as XS: FP64, or double-float
// pairs for the mixed path's double-float residual).  The correction is
// accumulated in T (it carries the precision of the basis) and added to x once.
__device__ __forceinline__ cx<double> xadd(cx<double> x, cx<double> d) { return x + d; }
__device__ __forceinline__ cx<double> xadd(cx<double> x, cx<float> d) { return x + ccast<double>(d); }
__device__ __forceinline__ cx<dd> xadd(cx<dd> x, cx<float> d) { return mkc(x.re + dd(d.re), x.im + dd(d.im)); }
template <typename T, typename XS>
__global__ void __launch_bounds__(KR_THREADS) k_xupdate(long long n, const int4* box, int mp1, const int* __restrict__ nsteps,
                                                         const double* __restrict__ ycoef,
                                                         const cx<T>* __restrict__ V, long long vss,
                                                         cx<XS>* __restrict__ X, long long xss) {
  const int slot = blockIdx.y;
  const int ns = nsteps[slot];
  if (ns == 0) return;
  const long long len = box_len(box, slot, n);
  const long long base = (long long)blockIdx.x * KR_CHUNK + threadIdx.x;
  const cx<T>* Vs = V + (size_t)slot * vss;
  cx<T> acc[KR_EPT];
#pragma unroll
  for (int e = 0; e < KR_EPT; ++e) acc[e] = mkc((T)0, (T)0);
  for (int i = 0; i < ns; ++i) {
    const T cf = (T)ycoef[(size_t)slot * mp1 + i];
#pragma unroll
    for (int e = 0; e < KR_EPT; ++e) {
      const long long idx = base + (long long)e * KR_THREADS;
      if (idx < len) {
        const cx<T> vi = ldg(Vs + (size_t)i * n + idx);
        acc[e] = mkc(acc[e].re + cf * vi.re, acc[e].im + cf * vi.im);
      }
    }
  }
#pragma unroll
  for (int e = 0; e < KR_EPT; ++e) {
    const long long idx = base + (long long)e * KR_THREADS;
    if (idx < len) {
      cx<XS>* xp = X + (size_t)slot * xss + idx;
      *xp = xadd(*xp, acc[e]);
    }
  }
}

// FP64 copy of double-float fields (solution read-out)
// Start of a cycle from a squared-norm partial sum over nblk blocks:
// beta = ||r||, sigma_0 = 1/beta, g = beta e_1, stop threshold, flags.
// first != 0: the vector is b itself (records ||b||).  mask (nullable): only the
// slots with mask[slot] != 0 (slots being started while others run).
// first = 1: a new solve from x = 0 (part holds |b|^2: sets ||b|| and the
// counters); 0: the next cycle of a running solve; 2: a new solve from a given
// x (after a first = 1 launch on b; part holds |b - A x|^2: the counters stay
// as that launch set them).
// box: nblk partials per box column, slots part_ss apart (allcols_N > 0: per column of the grid).
static __global__ void __launch_bounds__(KR_THREADS) k_cycle_start(CycleState c, const double* part, int nblk,
                                                             int first, const int* mask, const int4* box,
                                                             long long part_ss, int allcols_N) {
  __shared__ double sh[KR_THREADS / 32];
  const int slot = blockIdx.x;
  if (mask && !mask[slot]) return;
  if (first != 1 && !c.active[slot]) return;
  double s = 0.0;
  if (box) {
    const int4 b = box[slot];
    nblk *= allcols_N > 0 ? allcols_N : b.y - b.x;
  } else {
    part_ss = nblk;
  }
  for (int q = threadIdx.x; q < nblk; q += blockDim.x) s += part[(size_t)slot * part_ss + q];
  s = block_sum_256(s, sh);
  if (threadIdx.x != 0) return;
  const int m = c.m;
  const double beta = sqrt(s);
  if (first == 1) {
    c.bnorm[slot] = beta;
    // a normal FP32 number for FP64 right-hand sides beyond FP32's range too
    c.nscale[slot] = beta > 0.0 ? (float)exp2(-(double)max(-126, min(126, ilogb(beta)))) : 1.f;
    c.itot[slot] = c.cit[slot] = 0;
    c.ncyc[slot] = c.ccyc[slot] = 0;
  }
  const double bn = c.bnorm[slot];
  const double rel = bn > 0.0 ? beta / bn : 0.0;
  c.resid[slot] = rel;
  const int act = (bn > 0.0) && (rel > c.tol) && (c.itot[slot] - c.cit[slot] < c.max_iter) &&
                  (c.ncyc[slot] - c.ccyc[slot] < c.max_outer);
  c.active[slot] = act;
  c.run[slot] = act;
  c.nsteps[slot] = 0;
  c.sigma[(size_t)slot * (m + 1)] = beta > 0.0 ? 1.0 / beta : 0.0;
  double* g = c.g + (size_t)slot * (m + 1);
  g[0] = beta;
  for (int i = 1; i <= m; ++i) g[i] = 0.0;
  double thr = 0.5 * c.tol * bn;
  if (c.inner_tol > 0.0) thr = fmax(thr, c.inner_tol * beta);
  c.thr[slot] = thr;
  if (act && first != 2) c.ncyc[slot] += 1;
  if (first == 2 && !act) c.ncyc[slot] = 0;  // x already meets tol: no cycle runs
}

// ---------------------------------------------------------------------------
// s-step (block) Arnoldi.  The Krylov space and the GMRES minimisation are the
// ones of the step-by-step process above; only the order of the work changes,
// so that each sweep over the stored basis serves S new directions instead of
// one (the basis sweeps are HBM-bound).  From the last basis vector
// v_{J-1} a block forms the monomial chain in K = A - I,
//     p_0 = v_{J-1},  p_{i+1} = K p_i   (i < S, stored raw in basis slots J+i),
// so A p_i = p_i + p_{i+1}.  One sweep then yields C = V^T p (J x S) and the
// Gram matrix p^T p (S x S); a per-slot FP64 step normalises the chain
// (p^_i = p_i / ||p_i||), forms G = p^T p - C^T C, its Cholesky factor R (the
// block's orthonormalisation, CholQR), and from A P^ = P^ B (B unit lower
// bidiagonal up to the normalisation) the S new columns of the Hessenberg
// matrix,  H_new = (T B - [H_prev Z; 0]) U^{-1},  where T holds the chain's
// coordinates in the new orthonormal basis, U its part on v_{J-1}..v_{J+S-2}
// and Z its part on v_0..v_{J-2}.  A second sweep writes the new basis vectors
// Q = (P^ - V C) R^{-1} over the chain.  A pivot of G below kBlockPivot ends
// the cycle after the columns it still supports (the outer refinement
// continues from the true residual).
// ---------------------------------------------------------------------------
// Elements per thread and chunk of the block sweeps: one for short vectors (N <= 128: a single
// vector is then 4 to 64 chunks and spreads over as many SMs; the FP64 sweeps of one 64^2 vector ran
// on 4 SMs), else KB_EPT.  From the grid size alone: the same order of sums in every batch.
__host__ __device__ constexpr int block_ept(long long n) { return n / KB_CHUNK < 32 ? 1 : KB_EPT; }

// Chunks per dot-sweep block, and the blocks that have any, from a vector's chunks alone: a
// slot's summation order does not depend on the batch, and no block has a short share when the
// chunks do not divide by the block limit.
__host__ __device__ __forceinline__ int bdot_share(int nwork) {
  return (nwork + kBlockDotBlocks - 1) / kBlockDotBlocks;
}
__device__ __forceinline__ int bdot_blocks(int nwork) {
  const int c = bdot_share(nwork);
  return c > 0 ? (nwork + c - 1) / c : 0;
}

// A thread's EPT elements of the chunk at c0: FP32 pairs of complex values as one 16-byte load (len
// is even: a box is a multiple of 2 columns wide), else one complex value each; 0 beyond len.
template <int EPT>
__device__ __forceinline__ void bd_load(const cx<float>* v, long long c0, long long len, cx<float> (&o)[EPT]) {
  if constexpr (EPT == 1) {
    o[0] = ldg_if(v + c0 + threadIdx.x, c0 + threadIdx.x < len);
  } else {
#pragma unroll
    for (int e = 0; e < EPT / 2; ++e) {
      const long long i = c0 + 2 * (e * KR_THREADS + threadIdx.x);
      const float4 f = i < len ? __ldg(reinterpret_cast<const float4*>(v + i)) : make_float4(0.f, 0.f, 0.f, 0.f);
      o[2 * e] = mkc(f.x, f.y);
      o[2 * e + 1] = mkc(f.z, f.w);
    }
  }
}
template <int EPT>
__device__ __forceinline__ void bd_load(const cx<double>* v, long long c0, long long len, cx<double> (&o)[EPT]) {
#pragma unroll
  for (int e = 0; e < EPT; ++e) {
    const long long i = c0 + e * KR_THREADS + threadIdx.x;
    o[e] = ldg_if(v + i, i < len);
  }
}
// RB x S dot products of one chunk: per-thread sums, one reduce-scatter, added to red[r0*S ..]
template <typename T, int S, int EPT, int RB>
__device__ __forceinline__ void bd_dots(const cx<T> (&v)[RB][EPT], const cx<T> (&w)[S][EPT], T* red, int r0, int lane) {
  T s[RB * S];
#pragma unroll
  for (int k = 0; k < RB; ++k)
#pragma unroll
    for (int i = 0; i < S; ++i) {
      T d = 0;
#pragma unroll
      for (int e = 0; e < EPT; ++e) d += v[k][e].re * w[i][e].re + v[k][e].im * w[i][e].im;
      s[k * S + i] = d;
    }
  const T d = warp_reduce_scatter<RB * S>(s, lane);
  if ((lane & (32 / (RB * S) - 1)) == 0) red[r0 * S + lane / (32 / (RB * S))] += d;
}
// the S (S + 1) / 2 products <p_i, p_l>, added to red[J*S ..]
template <typename T, int S, int EPT>
__device__ __forceinline__ void bd_gram(const cx<T> (&w)[S][EPT], T* red, int J, int lane) {
  constexpr int NG = S * (S + 1) / 2, NP = S == 4 ? 16 : 4;  // padded to a power of two
  T g[NP];
#pragma unroll
  for (int q = 0; q < NP; ++q) g[q] = 0;
  int it = 0;
#pragma unroll
  for (int i = 0; i < S; ++i)
#pragma unroll
    for (int l = i; l < S; ++l) {
      T d = 0;
#pragma unroll
      for (int e = 0; e < EPT; ++e) d += w[i][e].re * w[l][e].re + w[i][e].im * w[l][e].im;
      g[it] = d;
      ++it;
    }
  const T d = warp_reduce_scatter<NP>(g, lane);
  const int q = lane / (32 / NP);
  if ((lane & (32 / NP - 1)) == 0 && q < NG) red[J * S + q] += d;
}
// block totals of the warps' sums -> part
template <typename T>
__device__ __forceinline__ void bd_store(const BlockArgs& a, const T* redf, int nit, int slot) {
  __syncthreads();
  for (int q = threadIdx.x; q < nit; q += blockDim.x) {
    T s = 0;
    for (int w2 = 0; w2 < KR_THREADS / 32; ++w2) s += redf[w2 * nit + q];
    a.part[((size_t)slot * a.nitem + q) * a.nchunk + blockIdx.x] = (double)s;
  }
}

// part[slot][r*S+i][block] = <v~_r, p_{i+1}> (r < J); then <p_i, p_l>, i <= l.  The FP64 sweep, bound
// by the FP64 pipe: basis vectors in groups of RB, loaded together, one reduce-scatter per group.
template <typename T, int S, int EPT>
__global__ void __launch_bounds__(KR_THREADS) k_bdots(const BlockArgs a, const cx<T>* __restrict__ V, long long vss,
                                                       int J) {
  constexpr int RB = 4, CH = KR_THREADS * EPT;
  // [KR_THREADS / 32][nit] warp totals in T
  extern __shared__ __align__(16) unsigned char bd_smem[];
  T* redf = reinterpret_cast<T*>(bd_smem);
  const int slot = blockIdx.y;
  if (!a.run[slot]) return;
  const long long len = box_len(a.box, slot, a.n);
  const int nwork = (int)((len + CH - 1) / CH), share = bdot_share(nwork);
  const int ch0 = blockIdx.x * share, ch1 = ch0 + share < nwork ? ch0 + share : nwork;
  if (ch0 >= nwork) return;
  const int nit = block_items(J, S);
  const cx<T>* Vs = V + (size_t)slot * vss;
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // each warp accumulates its own row of red over the block's chunks
  for (int q = threadIdx.x; q < (KR_THREADS / 32) * nit; q += blockDim.x) redf[q] = 0;
  __syncthreads();
  T* red = redf + wid * nit;
  for (int ch = ch0; ch < ch1; ++ch) {
    const long long c0 = (long long)ch * CH;
    cx<T> w[S][EPT];
#pragma unroll
    for (int i = 0; i < S; ++i) bd_load<EPT>(Vs + (size_t)(J + i) * a.n, c0, len, w[i]);
    int r = 0;
    for (; r + RB <= J; r += RB) {
      cx<T> v[RB][EPT];
#pragma unroll
      for (int k = 0; k < RB; ++k) bd_load<EPT>(Vs + (size_t)(r + k) * a.n, c0, len, v[k]);
      bd_dots<T, S, EPT, RB>(v, w, red, r, lane);
    }
    for (; r < J; ++r) {
      cx<T> v[1][EPT];
      bd_load<EPT>(Vs + (size_t)r * a.n, c0, len, v[0]);
      bd_dots<T, S, EPT, 1>(v, w, red, r, lane);
    }
    bd_gram<T, S, EPT>(w, red, J, lane);
  }
  bd_store<T>(a, redf, nit, slot);
}

// Per-slot FP64 step of a block, one CTA per slot.  Latency-bound: a chain of small dense steps, and
// on GB300 a warp's FP64 instruction holds the narrow FP64 pipe for 64 cycles whatever its active
// lanes, a division for some twenty of them (reciprocal square roots stand in for most).  So what has a
// free index runs one element per lane or per warp (the dot partials, C^T C, the product with the
// earlier Hessenberg columns, the earlier rotations with one new column per lane, the back
// substitution with one row per lane), all of it in shared memory, and only the S x S Cholesky factor
// and the S new rotations are serial: 25 us at restart 32, 72-81 us with one warp and divisions.  Writes the block's Hessenberg columns J-1..
// (unrotated into Hraw, rotated into c.H), the sweep coefficients, the scales of the new vectors,
// and upd[slot]: 1 for every slot that ran the block (its new vectors need the update sweep even
// when it stops here), 2 for one that ends its cycle.
// shared doubles: val[items], W[J][S], X[J + S][S], rotations cs, sn[m], g[m + 1]
__host__ __device__ constexpr int bscalar_smem(int J, int S, int m) {
  return block_items(J, S) + J * S + (J + S) * S + 3 * m + 1;
}
template <int S>
static __global__ void __launch_bounds__(KR_THREADS) k_bscalar(BlockArgs a, CycleState c, double* __restrict__ Hraw,
                                                               double* __restrict__ bcoef, int* __restrict__ upd,
                                                               int J) {
  extern __shared__ double sm[];
  constexpr int NG = S * (S + 1) / 2, NW = KR_THREADS / 32;
  __shared__ double Sg[S + 1], iS[S + 1], GC[NG], sRi[S][S];
  const int slot = blockIdx.x;
  if (!c.run[slot]) {
    if (threadIdx.x == 0) upd[slot] = 0;
    return;
  }
  const int m = c.m, rows = J + S, nit = block_items(J, S);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  double* val = sm;
  double* Wm = val + nit;
  double* X = Wm + J * S;
  double* scs = X + rows * S;
  double* ssn = scs + m;
  double* sg_ = ssn + m;  // g
  double* sg = c.sigma + (size_t)slot * (m + 1);
  // the dot sweep's partials, four items per warp at a time (a fixed order of sums)
  const int npart = bdot_blocks((int)((box_len(a.box, slot, a.n) + a.chunk - 1) / a.chunk));
  for (int q0 = wid * 4; q0 < nit; q0 += NW * 4) {
    double s[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      s[u] = 0.0;
      if (q0 + u < nit) {
        const double* p = a.part + ((size_t)slot * a.nitem + q0 + u) * a.nchunk;
        for (int ch = lane; ch < npart; ch += 32) s[u] += p[ch];
      }
    }
    const double d = warp_reduce_scatter<4>(s, lane);
    if ((lane & 7) == 0 && q0 + (lane >> 3) < nit) val[q0 + (lane >> 3)] = d;
  }
  // the cycle's rotations and right-hand side so far
  for (int q = threadIdx.x; q < J - 1; q += blockDim.x) {
    scs[q] = c.cs[(size_t)slot * m + q];
    ssn[q] = c.sn[(size_t)slot * m + q];
  }
  for (int q = threadIdx.x; q <= m; q += blockDim.x) sg_[q] = c.g[(size_t)slot * (m + 1) + q];
  __syncthreads();
  // chain norms Sg[i] = ||p_i|| (Sg[0] = 1: v_{J-1} has unit norm); the diagonal items
  // of p^T p follow the J S items of V^T p
  if (threadIdx.x <= S) {
    const int i = threadIdx.x - 1;
    const double q = threadIdx.x == 0 ? 1.0 : fmax(val[J * S + i * S - i * (i - 1) / 2], 0.0);
    const double is = q > 0.0 ? rsqrt(q) : 0.0;
    iS[threadIdx.x] = is;  // 1 / Sg, 0 for a zero vector
    Sg[threadIdx.x] = q * is;
  }
  __syncthreads();
  // C^ = coordinates of p^_{i+1} on v_r (in place in val), one item per thread
  for (int q = threadIdx.x; q < J * S; q += blockDim.x) {
    const int r = q / S, i = q - r * S;
    val[q] *= sg[r] * iS[i + 1];
  }
  __syncthreads();
  // C^T C, one entry per warp; W = H_prev Z (Z: the chain's part on v_0..v_{J-2}), one item per thread
  for (int e = wid; e < NG; e += NW) {
    int i = 0, l = e;
    while (l >= S - i) l -= S - i++;
    l += i;
    double s = 0.0;
    for (int r = lane; r < J; r += 32) s += val[r * S + i] * val[r * S + l];
    s = warp_sum(s, 32);
    if (lane == 0) GC[e] = s;
  }
  for (int q = threadIdx.x; q < J * (S - 1); q += blockDim.x) {
    const int i = q / J, r = q - i * J;  // column i + 1; neighbouring threads read neighbouring rows
    double s = 0.0;
    const double* Hp = Hraw + (size_t)slot * m * (m + 1) + r;
#pragma unroll 8
    for (int p = (r > 0 ? r - 1 : 0); p < J - 1; ++p) s += Hp[(size_t)p * (m + 1)] * val[p * S + i];
    Wm[r * S + i + 1] = s;
  }
  __syncthreads();
  int ncols = 0;
  if (wid == 0) {
    // G = p^T p (normalised) - C^T C, Cholesky G = R^T R, R^{-1} on the accepted columns; every lane
    // computes all of it (the same cost as one lane)
    double R[S][S], Ri[S][S];
#pragma unroll
    for (int i = 0; i < S; ++i)
#pragma unroll
      for (int l = 0; l < S; ++l) R[i][l] = Ri[i][l] = 0.0;
    int nok = S;
#pragma unroll
    for (int i = 0; i < S; ++i) {
      if (nok == S) {
#pragma unroll
        for (int l = 0; l < S; ++l) {
          if (l < i || nok < S) continue;
          const int e = i * S - i * (i - 1) / 2 + l - i;
          double gv = val[J * S + e] * (iS[i + 1] * iS[l + 1]) - GC[e];
#pragma unroll
          for (int q = 0; q < S; ++q)
            if (q < i) gv -= R[q][i] * R[q][l];
          if (l == i) {
            if (!(gv > kBlockPivot) || Sg[i + 1] == 0.0) {
              nok = i;
            } else {
              Ri[i][i] = rsqrt(gv);
              R[i][i] = gv * Ri[i][i];
            }
          } else {
            R[i][l] = gv * Ri[i][i];
          }
        }
      }
    }
    ncols = nok > 0 ? nok : 1;  // nok = 0: p_1 lies in span(V), a happy breakdown column
#pragma unroll
    for (int i = 0; i < S; ++i)
      if (i < nok) {
#pragma unroll
        for (int q = S - 1; q >= 0; --q)
          if (q < i) {
            double s = 0.0;
#pragma unroll
            for (int l = 0; l < S; ++l)
              if (l > q && l <= i) s += R[q][l] * Ri[l][i];
            Ri[q][i] = -s * Ri[q][q];
          }
      }
    if (lane == 0)
#pragma unroll
      for (int i = 0; i < S; ++i)
#pragma unroll
        for (int l = 0; l < S; ++l) sRi[i][l] = Ri[i][l];
    // T[r][k]: coordinates of p^_k on v_0..v_{J+S-1}; H_new = (T B - [W; 0]) U^{-1}, one row per lane
    double bsub[S];
#pragma unroll
    for (int i = 0; i < S; ++i) bsub[i] = i < ncols ? Sg[i + 1] * iS[i] : 0.0;
    for (int r = lane; r < rows; r += 32) {
      double x[S], T[S + 1];
      T[0] = r == J - 1 ? 1.0 : 0.0;
#pragma unroll
      for (int k = 1; k <= S; ++k) {
        double t = 0.0;
        if (r < J) t = val[r * S + k - 1];
        else
#pragma unroll
          for (int q = 0; q < S; ++q)
            if (r - J == q && q <= k - 1) t = R[q][k - 1];
        T[k] = t;
      }
#pragma unroll
      for (int i = 0; i < S; ++i) {
        x[i] = 0.0;
        if (i < ncols) {
          double v = T[i] + T[i + 1] * bsub[i];
          if (r < J && i > 0) v -= Wm[r * S + i];
#pragma unroll
          for (int l = 0; l < S; ++l)
            if (l < i) v -= x[l] * (l == 0 ? val[(J - 1) * S + i - 1] : R[l > 0 ? l - 1 : 0][i > 0 ? i - 1 : 0]);
          const double ui = i == 0 ? 1.0 : Ri[i > 0 ? i - 1 : 0][i > 0 ? i - 1 : 0];
          x[i] = r <= J + i ? v * ui : 0.0;
          if (r <= J + i) Hraw[((size_t)slot * m + J - 1 + i) * (m + 1) + r] = x[i];
        }
        X[r * S + i] = x[i];
      }
    }
  }
  __syncthreads();
  if (wid > 0) {
    // sweep coefficients: Q = P^ R^{-1} - V C^ R^{-1}, on the raw stored vectors
    double* bc = bcoef + (size_t)slot * (S * S + (m + 1) * S);
    for (int q = threadIdx.x - 32; q < S * S + J * S; q += KR_THREADS - 32) {
      if (q < S * S) {
        const int k = q / S, i = q - k * S;
        bc[q] = sRi[k][i] * iS[k + 1];
      } else {
        const int r = (q - S * S) / S, i = q - S * S - r * S;
        double s = 0.0;
        for (int k = 0; k <= i; ++k) s += val[r * S + k] * sRi[k][i];
        bc[q] = -s * sg[r];
      }
    }
    return;
  }
  // warp 0.  The earlier rotations on the new columns, one column per lane
  if (lane < ncols) {
    double h0 = X[lane];
#pragma unroll 4
    for (int k = 0; k < J - 1; ++k) {
      const double h1 = X[(k + 1) * S + lane], ck = scs[k], sk = ssn[k];
      X[k * S + lane] = ck * h0 + sk * h1;
      h0 = ck * h1 - sk * h0;
    }
    X[(J - 1) * S + lane] = h0;
  }
  __syncwarp();
  // the new rotations: column i's own from its last two entries, applied to the columns after it
  const double thr = c.thr[slot];
  const int last = c.max_iter + c.cit[slot];
  int itot = c.itot[slot], done = 0;
  double gj = sg_[J - 1];
  bool stop = false;
  for (int i = 0; i < ncols && !stop; ++i) {
    const int j = J - 1 + i;
    const double hj = X[j * S + i], sub = X[(j + 1) * S + i];
    // rho = |(hj, sub)|; outside the range where its square is safe (never for a scaled basis), hypot
    const double r2 = hj * hj + sub * sub;
    double rho = 0.0, cj = 1.0, sj = 0.0;
    if (r2 > 1e-280 && r2 < 1e280) {
      const double ir = rsqrt(r2);
      rho = r2 * ir;
      cj = hj * ir;
      sj = sub * ir;
    } else if ((rho = hypot(hj, sub)) > 0.0) {
      cj = hj / rho;
      sj = sub / rho;
    }
    __syncwarp();
    if (lane > i && lane < ncols) {
      const double h0 = X[j * S + lane], h1 = X[(j + 1) * S + lane];
      X[j * S + lane] = cj * h0 + sj * h1;
      X[(j + 1) * S + lane] = cj * h1 - sj * h0;
    } else if (lane == i) {
      X[j * S + i] = rho;
      X[(j + 1) * S + i] = 0.0;
      c.cs[(size_t)slot * m + j] = cj;
      c.sn[(size_t)slot * m + j] = sj;
    }
    const double gn = -sj * gj;
    if (lane == 0) sg_[j] = cj * gj;
    gj = gn;
    ++itot;
    done = i + 1;
    stop = fabs(gn) <= thr || j + 1 >= m || sub == 0.0 || itot >= last;
    __syncwarp();
  }
  const int ns = J - 1 + done;
  if (lane == 0) {
    sg_[ns] = gj;
    c.nsteps[slot] = ns;
    c.itot[slot] = itot;
    upd[slot] = 1;
  }
  if (lane < S) sg[J + lane] = 1.0;
  __syncwarp();
  for (int q = lane; q < done * (J + S); q += 32) {  // rotated columns
    const int i = q / (J + S), r = q - i * (J + S);
    if (r <= J + i) c.H[((size_t)slot * m + J - 1 + i) * (m + 1) + r] = X[r * S + i];
  }
  for (int q = J - 1 + lane; q <= ns; q += 32) c.g[(size_t)slot * (m + 1) + q] = sg_[q];
  if (ncols < S || J - 1 + 2 * S > m) stop = true;
  if (!stop) return;
  // last block of this slot's cycle: y = R^{-1} g on the rotated columns (row r of the remaining
  // right-hand side on lane r mod 32, column i + 1 loaded ahead), and ycoef_i = y_i sigma_i, so that
  // the update sweep also adds V y to x
  __syncwarp();
  const double* H = c.H + (size_t)slot * m * (m + 1);
  double* inv = scs;  // reciprocal diagonal (the rotations are not needed any more)
  for (int i = lane; i < ns; i += 32) {
    const double d = H[(size_t)i * (m + 1) + i];
    inv[i] = d != 0.0 ? 1.0 / d : 0.0;
  }
  __syncwarp();
  double* y = c.ycoef + (size_t)slot * (m + 1);
  double hn = ns > 1 && lane < ns - 1 ? H[(size_t)(ns - 1) * (m + 1) + lane] : 0.0;
  for (int i = ns - 1; i >= 0; --i) {
    const double h = hn;
    hn = i > 1 && lane < i - 1 ? H[(size_t)(i - 1) * (m + 1) + lane] : 0.0;
    const double yi = sg_[i] * inv[i];
    __syncwarp();
    if (lane < i) sg_[lane] -= h * yi;
    for (int r = lane + 32; r < i; r += 32) sg_[r] -= H[(size_t)i * (m + 1) + r] * yi;
    if (lane == 0) ssn[i] = yi;
    __syncwarp();
  }
  for (int i = lane; i <= m; i += 32) y[i] = i < ns ? ssn[i] * sg[i] : 0.0;
  if (lane == 0) {
    upd[slot] = 2;
    c.run[slot] = 0;
  }
}

// ---------------------------------------------------------------------------
// Block update: Q_i = sum_k bcoef_ki p_{k+1} + sum_r bcoef'_ri v~_r, written over the chain (basis
// slots J..J+S-1); slots with upd[slot] != 0 only.  upd[slot] == 2 (the slot's last block of the
// cycle): also x += sum_r ycoef_r v~_r + sum_i ycoef_{J+i} Q_i, accumulated in T and added to x
// once (no separate pass over the basis).  The basis is streamed through shared memory by bulk
// asynchronous copies (cp.async.bulk, completion counted on an mbarrier):
// KB_STAGES chunks of basis vectors are in flight per CTA while the threads
// work on an earlier one, so a CTA keeps ~KB_STAGES x 8 KB of reads
// outstanding with no registers held for them.  Every wait is bounded: when one runs out the CTA
// sets *a.err, stops computing, drains its own copies (bounded) and returns.
// n is a multiple of every chunk (N >= 32).
// ---------------------------------------------------------------------------
// stages per CTA: 32 KB of shared memory for either element size
template <typename T>
struct KBStages {
  static constexpr int value = sizeof(cx<T>) == 8 ? 4 : 2;
};
constexpr int kWaitLimit = 1 << 18;  // try_wait rounds before a wait is declared lost (~1 s on GB300)

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
// one arrival that also announces the bytes the next copy will deliver
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}
// By a stage's readers, before the barrier after which the stage is refilled: the barrier alone does not
// order their reads (generic proxy) before the bulk copy's write (async proxy).
__device__ __forceinline__ void stage_release() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
// true once the barrier's phase with the given parity has completed; false after kWaitLimit rounds
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  const uint32_t addr = smem_u32(bar);
  for (int i = 0; i < kWaitLimit; ++i) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(addr), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

// The FP32 dot sweep (k_bdots' sums) with the basis streamed through shared memory by bulk copies in
// groups of four vectors, KD_STAGES groups (96 KB at four elements per thread) in flight per CTA: the
// register version kept too few loads in flight, at one slot (a chain of load latencies: 42 us a
// sweep at 1024^2, J = 16) and at many (5.9 TB/s).  Bounded waits as in k_bupdate_bulk.
constexpr int KD_STAGES = 3;
template <int EPT>
__host__ __device__ constexpr int bdots_stage_bytes() { return 4 * KR_THREADS * EPT * (int)sizeof(cx<float>); }
template <int S, int EPT>
__global__ void __launch_bounds__(KR_THREADS) k_bdots_bulk(const BlockArgs a, const cx<float>* __restrict__ V,
                                                            long long vss, int J) {
  constexpr int RB = 4, CH = KR_THREADS * EPT;
  constexpr uint32_t kBytes = CH * sizeof(cx<float>);
  extern __shared__ __align__(128) unsigned char kd_raw[];
  cx<float>* stage = reinterpret_cast<cx<float>*>(kd_raw);  // [KD_STAGES][RB][CH]
  float* redf = reinterpret_cast<float*>(kd_raw + KD_STAGES * bdots_stage_bytes<EPT>());
  __shared__ __align__(8) uint64_t bar[KD_STAGES];
  __shared__ int lost;
  const int slot = blockIdx.y;
  if (!a.run[slot]) return;
  const long long len = box_len(a.box, slot, a.n);
  const int nwork = (int)((len + CH - 1) / CH), share = bdot_share(nwork);
  const int ch0 = blockIdx.x * share, ch1 = ch0 + share < nwork ? ch0 + share : nwork;
  if (ch0 >= nwork) return;
  const int ngrp = (J + RB - 1) / RB, total = (ch1 - ch0) * ngrp;
  const int nit = block_items(J, S);
  const cx<float>* Vs = V + (size_t)slot * vss;
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  auto issue = [&](int i) {  // thread 0: group i of the flattened (chunk, group) sequence
    const int ch = ch0 + i / ngrp, g = i % ngrp, st = i % KD_STAGES;
    const int nv = J - RB * g < RB ? J - RB * g : RB;
    mbar_expect_tx(&bar[st], nv * kBytes);
    for (int k = 0; k < nv; ++k)
      bulk_g2s(stage + (size_t)(st * RB + k) * CH, Vs + (size_t)(RB * g + k) * a.n + (long long)ch * CH, kBytes, &bar[st]);
  };
  if (threadIdx.x == 0) {
    lost = 0;
    for (int s = 0; s < KD_STAGES; ++s) mbar_init(&bar[s], 1);
    mbar_fence_init();
    for (int i = 0; i < KD_STAGES && i < total; ++i) issue(i);
  }
  for (int q = threadIdx.x; q < (KR_THREADS / 32) * nit; q += blockDim.x) redf[q] = 0.f;
  __syncthreads();
  float* red = redf + wid * nit;
  cx<float> w[S][EPT];
  int i = 0;
  for (; i < total; ++i) {
    const int ch = ch0 + i / ngrp, g = i % ngrp, st = i % KD_STAGES;
    const long long c0 = (long long)ch * CH;
    if (g == 0)
#pragma unroll
      for (int k = 0; k < S; ++k) bd_load<EPT>(Vs + (size_t)(J + k) * a.n, c0, len, w[k]);
    if (!mbar_wait(&bar[st], (uint32_t)((i / KD_STAGES) & 1))) lost = 1;
    __syncthreads();  // every thread has waited (and sees `lost`)
    if (lost) break;
    cx<float> v[RB][EPT];
#pragma unroll
    for (int k = 0; k < RB; ++k) {
      const cx<float>* src = stage + (size_t)(st * RB + k) * CH;
      const bool have = RB * g + k < J;
      if constexpr (EPT == 1) {
        v[k][0] = have && c0 + threadIdx.x < len ? src[threadIdx.x] : mkc(0.f, 0.f);
      } else {
#pragma unroll
        for (int e = 0; e < EPT / 2; ++e) {
          const int o = 2 * (e * KR_THREADS + threadIdx.x);
          const float4 f = have && c0 + o < len ? *reinterpret_cast<const float4*>(src + o)
                                                : make_float4(0.f, 0.f, 0.f, 0.f);
          v[k][2 * e] = mkc(f.x, f.y);
          v[k][2 * e + 1] = mkc(f.z, f.w);
        }
      }
    }
    if (RB * g + RB <= J) {
      bd_dots<float, S, EPT, RB>(v, w, red, RB * g, lane);
    } else {
#pragma unroll
      for (int k = 0; k < RB - 1; ++k)
        if (RB * g + k < J) {
          cx<float> one[1][EPT];
#pragma unroll
          for (int e = 0; e < EPT; ++e) one[0][e] = v[k][e];
          bd_dots<float, S, EPT, 1>(one, w, red, RB * g + k, lane);
        }
    }
    if (i + KD_STAGES < total) stage_release();
    __syncthreads();  // stage st has been read by every thread: refill it
    if (threadIdx.x == 0 && i + KD_STAGES < total) issue(i + KD_STAGES);
    if (g == ngrp - 1) bd_gram<float, S, EPT>(w, red, J, lane);
  }
  if (i < total) {
    // a wait ran out: report it, drain this CTA's copies still in flight (bounded), return
    if (threadIdx.x == 0) {
      if (a.err) atomicExch(a.err, 1);
      const int issued = total < i + KD_STAGES ? total : i + KD_STAGES;
      for (int q = i; q < issued; ++q) mbar_wait(&bar[q % KD_STAGES], (uint32_t)((q / KD_STAGES) & 1));
    }
    return;
  }
  bd_store<float>(a, redf, nit, slot);
}

template <typename T, int S, int EPT, bool XU>
__global__ void __launch_bounds__(KR_THREADS) k_bupdate_bulk(const BlockArgs a, const int* __restrict__ upd,
                                                              cx<T>* __restrict__ V, long long vss, int J) {
  constexpr int KB_STAGES = KBStages<T>::value, CH = KR_THREADS * EPT;
  extern __shared__ __align__(128) unsigned char kb_stage_raw[];
  cx<T>* stage = reinterpret_cast<cx<T>*>(kb_stage_raw);  // [KB_STAGES][CH]
  __shared__ __align__(8) uint64_t bar[KB_STAGES];
  __shared__ T cf[S * S + 129 * S];
  __shared__ T yc[129 + S];
  __shared__ int lost;
  const int slot = blockIdx.y;
  const int u = upd[slot];
  if (u != (XU ? 2 : 1)) return;
  // packed box vectors: the chunks beyond the box are skipped; the last chunk works on the
  // elements after the box's end too (inside the vector's n-element slot, read by nobody)
  if ((long long)blockIdx.x * CH >= box_len(a.box, slot, a.n)) return;
  constexpr uint32_t kBytes = CH * sizeof(cx<T>);
  cx<T>* Vs = V + (size_t)slot * vss;
  const long long c0 = (long long)blockIdx.x * CH;  // this CTA's chunk: elements c0 .. c0 + CH - 1
  if (threadIdx.x == 0) {
    lost = 0;
    for (int s = 0; s < KB_STAGES; ++s) mbar_init(&bar[s], 1);
    mbar_fence_init();
    // the first KB_STAGES basis vectors of the sweep
    for (int r = 0; r < KB_STAGES && r < J; ++r) {
      // (a.tx_extra > 0 only under the test hook: that stage's phase cannot complete)
      mbar_expect_tx(&bar[r], kBytes + (r == 0 ? (uint32_t)a.tx_extra : 0u));
      bulk_g2s(stage + (size_t)r * CH, Vs + (size_t)r * a.n + c0, kBytes, &bar[r]);
    }
  }
  const double* bc = a.bcoef + (size_t)slot * (S * S + a.mp1 * S);
  for (int q = threadIdx.x; q < S * S + J * S; q += blockDim.x) cf[q] = (T)bc[q];
  if (XU)
    for (int q = threadIdx.x; q < J + S; q += blockDim.x) yc[q] = (T)a.ycoef[(size_t)slot * a.mp1 + q];
  __syncthreads();
  cx<T> acc[S][EPT];
  {
    cx<T> w[S][EPT];
#pragma unroll
    for (int k = 0; k < S; ++k)
#pragma unroll
      for (int e = 0; e < EPT; ++e) w[k][e] = ldg(Vs + (size_t)(J + k) * a.n + c0 + threadIdx.x + e * KR_THREADS);
#pragma unroll
    for (int i = 0; i < S; ++i)
#pragma unroll
      for (int e = 0; e < EPT; ++e) {
        cx<T> s = mkc((T)0, (T)0);
#pragma unroll
        for (int k = 0; k <= i; ++k) s = mkc(s.re + cf[k * S + i] * w[k][e].re, s.im + cf[k * S + i] * w[k][e].im);
        acc[i][e] = s;
      }
  }
  cx<T> dx[EPT];
#pragma unroll
  for (int e = 0; e < EPT; ++e) dx[e] = mkc((T)0, (T)0);
  int r = 0;
  for (; r < J; ++r) {
    const int st = r % KB_STAGES;
    if (!mbar_wait(&bar[st], (uint32_t)((r / KB_STAGES) & 1))) lost = 1;
    __syncthreads();  // every thread has waited (and sees `lost`)
    if (lost) break;
    const T yr = XU ? yc[r] : (T)0;
    const cx<T>* src = stage + (size_t)st * CH + threadIdx.x;
#pragma unroll
    for (int e = 0; e < EPT; ++e) {
      const cx<T> v = src[e * KR_THREADS];
#pragma unroll
      for (int i = 0; i < S; ++i) {
        const T c = cf[S * S + r * S + i];
        acc[i][e] = mkc(acc[i][e].re + c * v.re, acc[i][e].im + c * v.im);
      }
      if (XU) dx[e] = mkc(dx[e].re + yr * v.re, dx[e].im + yr * v.im);
    }
    if (r + KB_STAGES < J) stage_release();
    __syncthreads();  // stage st has been read by every thread: refill it
    if (threadIdx.x == 0 && r + KB_STAGES < J) {
      mbar_expect_tx(&bar[st], kBytes);
      bulk_g2s(stage + (size_t)st * CH, Vs + (size_t)(r + KB_STAGES) * a.n + c0, kBytes, &bar[st]);
    }
  }
  if (r < J) {
    // a wait ran out: report it, drain this CTA's copies still in flight (bounded), return
    if (threadIdx.x == 0) {
      if (a.err) atomicExch(a.err, 1);
      const int issued = J < r + KB_STAGES ? J : r + KB_STAGES;
      for (int q = r; q < issued; ++q) mbar_wait(&bar[q % KB_STAGES], (uint32_t)((q / KB_STAGES) & 1));
    }
    return;
  }
#pragma unroll
  for (int i = 0; i < S; ++i)
#pragma unroll
    for (int e = 0; e < EPT; ++e) Vs[(size_t)(J + i) * a.n + c0 + threadIdx.x + e * KR_THREADS] = acc[i][e];
  if (XU) {
#pragma unroll
    for (int e = 0; e < EPT; ++e) {
      const long long idx = c0 + threadIdx.x + e * KR_THREADS;
      cx<T> d = dx[e];
#pragma unroll
      for (int i = 0; i < S; ++i) d = mkc(d.re + yc[J + i] * acc[i][e].re, d.im + yc[J + i] * acc[i][e].im);
      if constexpr (std::is_same<T, float>::value) {
        if (a.x_dd) {
          cx<dd>* xp = reinterpret_cast<cx<dd>*>(a.X) + (size_t)slot * a.xss + idx;
          *xp = xadd(*xp, d);
          continue;
        }
      }
      cx<double>* xp = reinterpret_cast<cx<double>*>(a.X) + (size_t)slot * a.xss + idx;
      *xp = xadd(*xp, d);
    }
  }
}

}  // namespace dbar
