// Coarse-grid correction of the solve on the potential's box (box.cuh).
//
// (I + K) u = r is an integral equation of the second kind (K is compact), so its error on a grid that
// resolves E_k Q is the smooth one of a quadrature, and the classical two-grid iteration of
// Brakhage and Atkinson applies: solve (I + K_c) u_c = R r on a coarser grid (R: every 2nd or 4th
// point), and correct with  u = r - K P u_c,  P u_c the trigonometric interpolation (its modes padded
// with zeros), one application of the fine operator.  The true residual on the fine grid, the
// stopping test and the solution are those of the fine discretisation: the coarse solve only replaces
// the Krylov cycle that reduces the residual, at 1/4 or 1/16 of its work, and a slot whose cycle
// falls short of its aim moves to the next finer grid.
//
// Which grid a slot's cycle takes: the share of the residual's modes beyond the coarse grid, by one
// transform of the residual (k_box_modes).  What a coarse cycle leaves is about that share, plus the
// modes that K brings in, which the next cycle's share shows.  The correction (interpolation and
// fine application) runs in the residual's arithmetic: in FP32 its rounding, white noise at 1e-7,
// would be beyond every coarse grid, and each later cycle would gain a factor of ten at most.
#pragma once
#include "krylov.cuh"

namespace dbar {

// Sums of |r|^2 over the box, and over its points at even and at 4-divisible coordinates: FP32 squares
// of r scaled by the slot's power of two near 1/||b||, block totals in FP64.  FP64 plans: FP64.
template <typename T>
__global__ void __launch_bounds__(256) k_coarse_norms(const CoarseArgs a, const cx<T>* __restrict__ V, long long vss,
                                                      CycleState f) {
  __shared__ double sh[kLevels + 1][8];
  const int slot = blockIdx.y;
  if ((a.mask && !a.mask[slot]) || !f.active[slot]) return;
  const int4 bx = a.box[slot];
  const int W = bx.y - bx.x;
  const T sc = std::is_same<T, float>::value ? (T)f.nscale[slot] : (T)1;
  T s[kLevels + 1];
#pragma unroll
  for (int l = 0; l <= kLevels; ++l) s[l] = 0;
  const cx<T>* r = V + (size_t)slot * vss;
  for (int y = bx.z + blockIdx.x; y < bx.w; y += gridDim.x) {
    const cx<T>* row = r + (size_t)(y - bx.z) * W;
    for (int x = bx.x + threadIdx.x; x < bx.y; x += blockDim.x) {
      const cx<T> v = ldg(row + x - bx.x);
      const T re = v.re * sc, im = v.im * sc, q = re * re + im * im;
      s[0] += q;
      if (!((x | y) & 1)) s[1] += q;
      if (!((x | y) & 3)) s[2] += q;
    }
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int l = 0; l <= kLevels; ++l) {
    const T t = warp_sum_t(s[l], 32);
    if (lane == 0) sh[l][wid] = (double)t;
  }
  __syncthreads();
  if (threadIdx.x <= kLevels) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += sh[threadIdx.x][w];
    a.part[((size_t)slot * kCoarseBlocks + blockIdx.x) * (kLevels + 1) + threadIdx.x] = t;
  }
}

// The grid of a cycle: the one that gains the most decades of residual per unit of time.  A cycle on a
// coarse grid gains down to the share of the residual's modes beyond it (or down to the Krylov
// arithmetic's limit, or to what is still needed); its cost is the correction and the true residual,
// in units of one fine Krylov step (FP32 steps are cheap beside a double-float residual), and
// kStepsPerDecade steps of 1/4 or 1/16 of a fine one.  Of 0.3 and 1 times the share and overheads of 5
// to 30 (FP64: 0.5 to 4) these were the fastest over three potentials of each of the solve workloads, by
// 1-4 % in mixed precision (1024^2 x 128 k 78.6 -> 75.2 ms) and 296 -> 164 ms in FP64 (512^2 x 48 k).  One
// number each for every grid and batch: at one slot a cycle's fixed cost is launches, at many it is arithmetic,
// so away from those workloads the choice is a good one rather than the best.
constexpr double kStepsPerDecade = 4.5;
constexpr double kOverheadMixed = 12.0, kOverheadFp64 = 4.0;
// Caps below which the caller asks for so few cycles, or iterations of so few restarts, that all are the fine grid's.
constexpr int kMinCycles = 8, kMinRestarts = 4;
// A coarse cycle that leaves more than this of the residual (and more than four times its aim) sends the
// slot to the next finer grid for good.
constexpr double kCoarseLeft = 0.3;

// Per slot (one block): its level, and the first state of the level's Krylov cycle; the fine cycle's
// run flag is cleared for the slots that take a coarse one.
static __global__ void __launch_bounds__(256) k_coarse_start(const CoarseArgs a, CycleState f) {
  __shared__ double sh[2 * (kLevels + 1)][8];
  const int slot = blockIdx.x, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (a.mask && !a.mask[slot]) return;
  const bool act = f.active[slot] != 0;
  double s[kLevels + 1], h[kLevels + 1];
#pragma unroll
  for (int l = 0; l <= kLevels; ++l) {
    float t = 0.f;
    double u = 0.0;
    if (act) {
      for (int q = threadIdx.x; q < a.nrough; q += 256) t += a.rough[((size_t)slot * a.nrough + q) * (kLevels + 1) + l];
      if (threadIdx.x < kCoarseBlocks) u = a.part[((size_t)slot * kCoarseBlocks + threadIdx.x) * (kLevels + 1) + l];
    }
    t = warp_sum_t(t, 32);
    u = warp_sum(u, 32);
    if (lane == 0) {
      sh[l][wid] = u;
      sh[kLevels + 1 + l][wid] = (double)t;
    }
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
#pragma unroll
  for (int l = 0; l <= kLevels; ++l) {
    s[l] = h[l] = 0.0;
    for (int w = 0; w < 8; ++w) {
      s[l] += sh[l][w];
      h[l] += sh[kLevels + 1 + l][w];
    }
  }
  const double beta = act ? f.g[(size_t)slot * (f.m + 1)] : 0.0, bn = f.bnorm[slot];
  int lv = -1;
  double share = 0.0;
  // Cycles and iterations on coarse grids come on top of the caps, half of each at most: the fine grid has all
  // that the plan alone would have (counted together, a solve that the plan alone ends within its cap missed it,
  // 37 of 3179 solves at caps of 8 to 64 iterations or 1 to 8 cycles).  Small caps leave them out.
  const bool early = f.ncyc[slot] > 0 && f.max_outer >= kMinCycles && f.max_iter >= kMinRestarts * f.m &&
                     f.ccyc[slot] < f.max_outer / 2 && f.cit[slot] < f.max_iter / 2;
  if (act) {
    // levels still open to the slot: all at its first cycle, none coarser than one that fell short; none
    // when the shares are no numbers or the caps allow none
    int top = -1;
    if (early && h[0] > 0.0 && isfinite(h[0])) {
      top = a.nlev - 1;
      if (f.ncyc[slot] > 1) {
        top = min(a.top[slot], top);
        if (a.level[slot] >= 0 && beta > a.bprev[slot] * fmax(kCoarseLeft, 4.0 * a.eprev[slot])) top = a.level[slot] - 1;
      }
    }
    a.top[slot] = top;
    // decades to gain, and at most in one cycle; the fine grid's cycle saves the correction
    const double need = fmax(log10(beta / (0.5 * f.tol * bn)), 0.1);
    const double most = fmin(need, f.inner_tol > 0.0 ? -log10(f.inner_tol) : (double)f.m / kStepsPerDecade);
    const double over = f.inner_tol > 0.0 ? kOverheadMixed : kOverheadFp64;
    double best = most / (0.6 * over + kStepsPerDecade * most);
    for (int l = 0; l < kLevels; ++l) {
      if (l > top) break;
      const double sh_l = sqrt(h[l + 1] / h[0]), d = fmin(most, -log10(fmin(sh_l + 1e-16, 0.9)));
      const double rate = d / (over + kStepsPerDecade * d / (double)(4 << (2 * l)));
      if (rate > best) {
        best = rate;
        lv = l;
        share = sh_l;
      }
    }
  }
  double aim = 0.0, bc = 0.0;
  if (lv >= 0) {
    aim = fmax(fmax(f.inner_tol, share), 0.5 * f.tol * bn / beta);
    const double ff = (double)(1 << (2 * (lv + 1)));  // u_c = f^2 u at the coarse points (sw_c = f^2 sw)
    bc = s[0] > 0.0 ? beta * ff * sqrt(s[lv + 1] / s[0]) : 0.0;
    if (!(bc > 0.0)) lv = -1;
  }
  a.level[slot] = lv;
  a.bprev[slot] = lv >= 0 ? beta : 0.0;
  a.eprev[slot] = aim;
  if (lv >= 0) {
    f.run[slot] = 0;
    f.ccyc[slot] += 1;
  }
#pragma unroll
  for (int l = 0; l < kLevels; ++l) {
    if (l >= a.nlev) break;
    const CycleState& c = a.c[l];
    const int on = l == lv;
    c.run[slot] = c.active[slot] = on;
    c.nsteps[slot] = 0;
    if (!on) continue;
    c.itot[slot] = f.itot[slot];
    c.cit[slot] = f.itot[slot] - f.cit[slot];
    c.sigma[(size_t)slot * (c.m + 1)] = 1.0 / bc;
    c.thr[slot] = aim * bc;
    double* g = c.g + (size_t)slot * (c.m + 1);
    g[0] = bc;
    for (int i = 1; i <= c.m; ++i) g[i] = 0.0;
  }
}

// Level l: V_c0 = f^2 r at the coarse points, x_c = 0.
template <typename T, typename XS>
__global__ void __launch_bounds__(256) k_coarse_restrict(const CoarseArgs a, int l, const cx<T>* __restrict__ V,
                                                         long long vss, cx<T>* Vc, long long vcss, cx<XS>* xc) {
  const int slot = blockIdx.y;
  if ((a.mask && !a.mask[slot]) || !a.c[l].run[slot]) return;
  const int f = 2 << l, Nc = a.N / f;
  const int4 b = a.box[slot], c = a.cbox[l][slot];
  const int W = b.y - b.x, Wc = c.y - c.x;
  const T ff = (T)(f * f);
  const cx<T>* r = V + (size_t)slot * vss;
  for (int y = c.z + blockIdx.x; y < c.w; y += gridDim.x) {
    const int yf = y * f;
    const bool iny = yf >= b.z && yf < b.w;
    for (int x = c.x + threadIdx.x; x < c.y; x += blockDim.x) {
      const int xf = x * f;
      const bool in = iny && xf >= b.x && xf < b.y;
      const size_t o = (size_t)(y - c.z) * Wc + x - c.x;
      Vc[(size_t)slot * vcss + o] = cscale(ldg_if(r + (long long)(yf - b.z) * W + xf - b.x, in), ff);
      xc[(size_t)slot * Nc * Nc + o] = mkc(XS(0.f), XS(0.f));
    }
  }
}

// the coarse cycle's steps counted to the solve, and outside its cap
static __global__ void k_coarse_count(CycleState f, CycleState c, int nslots) {
  const int slot = blockIdx.x * blockDim.x + threadIdx.x;
  if (slot < nslots && c.active[slot]) {
    f.cit[slot] += c.itot[slot] - f.itot[slot];
    f.itot[slot] = c.itot[slot];
  }
}

}  // namespace dbar
