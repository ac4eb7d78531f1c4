// The solve on the potential's box.
//
// K S = i (-1)^p DFT(w) with w = sw E_k Q conj(h(S)), and b = -i (-1)^p DFT(sw E_k Q): both are
// transforms of fields that vanish wherever Q does.  So is the solution S = b - K S, and so is
// every Krylov vector that starts from b.  With
//     S = Phi(u) := i (-1)^{p1+p2} DFT(u),   u supported on the box of Q,
// the system A S = b reads  u + w(Phi(u)) = -sw E_k Q  for u on the box alone.  Phi is N times an
// isometry (Parseval), so the inner products, the Krylov space and the minimisation are those of
// GMRES on S; only the representation of the vectors changes: one value per box point instead of
// one per grid point.  On the benchmark's potential the box is 0.21 of the grid, so the basis
// sweeps move 0.21 of the bytes, and the row pass no longer writes the N^2-point vector.
//
// Passes of one application:
//   k_box_cols FWD   columns: u on the box -> column DFT -> T2        (start of a chain)
//   k_box_rows       rows: DFT, Taylor row moments, S/xi, row IDFT    T2 -> T1
//   k_coef           Taylor coefficients (passes.cuh)
//   k_box_cols STEP  columns: IDFT, h, w -> the next vector (box), and its column DFT -> T2
//   k_box_cols LAST  the same without the forward transform
// T1 and T2 hold the box's columns of every row.  The solution leaves as S = Phi(u) by one
// 2-D transform in the refinement's arithmetic (FWD, then k_box_out).
//
// A box vector is packed: point (x, y) at (y - y0) W + (x - x0), W = x1 - x0 columns.  The box
// lives in device memory, one per slot, so that captured graphs and slots with potentials of
// their own follow it; grids cover every column tile and the blocks beyond the box return.
#pragma once
#include "ddround.cuh"
#include "passes.cuh"

namespace dbar {

template <typename T, int LOGN, int RV = 0>
struct BoxRowG {
  static constexpr int N = 1 << LOGN, E = box_ept(LOGN, std::is_same<T, double>::value), TPL = N / E;
  static constexpr int LINES = box_row_lines(LOGN, E, RV), THREADS = LINES * TPL;
  static_assert(E == 16 || TPL <= 32, "seg_count: one row segment per line");
  static constexpr int P = pitch_of(N);
  static constexpr int MINB = E == 16 ? RowG<T, LOGN, RV>::MINB : 1;
};
template <typename T, int LOGN, int CV = 0>
struct BoxColG {
  static constexpr int N = 1 << LOGN, E = box_ept(LOGN, std::is_same<T, double>::value), TPL = N / E;
  static constexpr int CW = box_col_cw(LOGN, (int)sizeof(cx<T>), E, CV), TW = 32 / CW;
  static constexpr int COLS = box_col_cols(LOGN, (int)sizeof(cx<T>), E, CV), THREADS = COLS * TPL;
  static constexpr int WPG = TPL / TW;  // warps per group of CW columns
  static constexpr int P = pitch_of(N);
  static constexpr int MINB = E == 16 ? ColG<T, LOGN, CV>::MINB : 1;
};

// Column kernel: block shapes of k_pass_b (ColG).  SL slots per block (2: variant 2 of the
// FP32 pass, one potential for all slots: the table tiles are loaded once for both).  Bound by issue and
// load latency (FP32: 0.159 ms for 16 slots of 1024^2 with the whole grid as box), by FP32 issue and
// instruction fetch in double-float, by the FP64 pipe in FP64.
template <typename T, int LOGN, int MODE, int CV, int SL>
__global__ void __launch_bounds__(BoxColG<T, LOGN, CV>::THREADS, SL == 2 ? 1 : BoxColG<T, LOGN, CV>::MINB)
k_box_cols(const BoxArgs<T> a) {
  using G = BoxColG<T, LOGN, CV>;
  constexpr int N = G::N, E = G::E, TPL = G::TPL, P = G::P;
  constexpr bool F32 = std::is_same<T, float>::value;
  constexpr bool DD = std::is_same<T, dd>::value;
  constexpr bool TAB = MODE != BX_FWD;  // modes that form h and w
  extern __shared__ __align__(16) unsigned char smem[];
  // slot-major block order (k_pass_b): resident blocks share the table tiles
  const int s0 = SL * blockIdx.x;
  int slot[SL];
  bool on[SL];
  bool any = false;
#pragma unroll
  for (int i = 0; i < SL; ++i) {
    slot[i] = s0 + i < a.nslots ? s0 + i : s0;
    on[i] = (i == 0 || slot[i] != s0) && (!a.run || a.run[slot[i]]);
    any |= on[i];
  }
  if (!any) return;
  const int4 bx = a.box[s0];  // SL == 2: one potential, one box
  const int c0 = a.allcols ? 0 : bx.x, c1 = a.allcols ? N : bx.y;
  const int tile0 = c0 + blockIdx.y * G::COLS;
  if (tile0 >= c1) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = (warp / G::WPG) * G::CW + lane % G::CW;
  const int t = (warp % G::WPG) * G::TW + lane / G::CW;
  const int j1 = tile0 + c;
  const int W = bx.y - bx.x;
  const bool inx = j1 >= bx.x && j1 < bx.y;
  cx<T>* line[SL];
#pragma unroll
  for (int i = 0; i < SL; ++i) line[i] = reinterpret_cast<cx<T>*>(smem) + (i * G::COLS + c) * P;
  constexpr size_t off = ((size_t)SL * G::COLS * P * sizeof(cx<T>) + 15) & ~(size_t)15;
  cx<T>* coef = reinterpret_cast<cx<T>*>(smem + off);  // [SL][M + 2]
  const int M = a.M;

  cx<T> v[SL][E];
  if constexpr (MODE == BX_FWD) {
#pragma unroll
    for (int i = 0; i < SL; ++i) {
      const T sc = a.in_scale ? (T)a.in_scale[(size_t)slot[i] * a.in_scale_ss] : (T)1;
      const cx<T>* src = a.in + (size_t)slot[i] * a.in_ss + (j1 - bx.x);
#pragma unroll
      for (int q = 0; q < E; ++q) {
        const int y = t + q * TPL;
        v[i][q] = ldg_if(src + (long long)(y - bx.z) * W, inx && y >= bx.z && y < bx.w);
      }
      if (a.loadE) {  // iterated equation: the rolled field h(. + xi0) is Phi(E_k u)
        const cx<T> exv = ldg(a.ex + (size_t)slot[i] * N + j1);
        const cx<T>* EY = a.ey + (size_t)slot[i] * N + t;
#pragma unroll
        for (int q = 0; q < E; ++q) v[i][q] = cmul(cmul(exv, ldg(EY + q * TPL)), v[i][q]);
      }
      if (a.in_scale) {
#pragma unroll
        for (int q = 0; q < E; ++q) v[i][q] = cscale(v[i][q], sc);
      }
    }
  } else {
#pragma unroll
    for (int i = 0; i < SL; ++i) {
      const cx<T>* src = a.in + (size_t)slot[i] * a.in_ss + (size_t)t * N + j1;
#pragma unroll
      for (int q = 0; q < E; ++q) v[i][q] = ldg(src + (size_t)q * TPL * N);
    }
    if (threadIdx.x < SL * (M + 2)) {
      const int h = threadIdx.x / (M + 2), i = threadIdx.x - h * (M + 2);
      coef[threadIdx.x] = ccast<T>(a.coef[(size_t)(h ? slot[SL - 1] : s0) * (M + 2) + i]);
    }
  }
  // double-float: the inverse transform as conj(DFT(conj(x))) in a loop with the forward one,
  // one copy of the code (two inlined double-float transforms miss in the instruction cache)
  constexpr bool LOOP = DD && MODE == BX_STEP;
  // FP64: squares in FP64.  Double-float: FP32 squares of r scaled by the slot's power of two near 1/||b||.
  using NT = typename std::conditional<std::is_same<T, double>::value, double, float>::type;
  NT nrm = 0;
#pragma unroll 1
  for (int ph = 0; ph < (LOOP ? 2 : 1); ++ph) {
    if constexpr (LOOP) {
      if (ph == 0) {
#pragma unroll
        for (int q = 0; q < E; ++q) v[0][q].im = -v[0][q].im;
      }
      fft_line_compact<T, LOGN, false>(v[0], line[0], t, a.tw);
      if (ph == 1) break;
#pragma unroll
      for (int q = 0; q < E; ++q) v[0][q].im = -v[0][q].im;
    } else if constexpr (TAB) {
      if constexpr (SL == 2) fft_line2<T, LOGN, true, F32>(v[0], v[SL - 1], line[0], line[SL - 1], t, a.tw);
      else if constexpr (DD) fft_line_compact<T, LOGN, true>(v[0], line[0], t, a.tw);
      else fft_line<T, LOGN, true, F32>(v[0], line[0], t, a.tw);
    }
    if constexpr (TAB) {
      __syncthreads();  // coefficients visible
      // h = u + sum_n c_n Delta_n + d'.  Rows outside the box: w = 0 below, and their table loads
      // are predicated off
#pragma unroll
      for (int i = 0; i < SL; ++i) {
        const cx<T> fill = coef[i * (M + 2) + M + 1];
#pragma unroll
        for (int q = 0; q < E; ++q) v[i][q] = v[i][q] + fill;
      }
      for (int n = 0; n <= M; ++n) {
        cx<T> cn[SL];
#pragma unroll
        for (int i = 0; i < SL; ++i) cn[i] = coef[i * (M + 2) + n];
        const cx<T>* D = a.Delta + ((size_t)n * N + t) * N + j1;
#pragma unroll
        for (int q = 0; q < E; ++q) {
          const int y = t + q * TPL;
          const cx<T> d = ldg_if(D + (size_t)q * TPL * N, y >= bx.z && y < bx.w);
#pragma unroll
          for (int i = 0; i < SL; ++i) cacc(v[i][q], cn[i], d);
        }
      }
      if constexpr (DD) {
#pragma unroll
        for (int q = 0; q < E; ++q) v[0][q] = cnorm(v[0][q]);
      }
      // w = (2 pi L^2/N^2) E_k Q conj(h) on the box, 0 elsewhere (Q taken as 0)
#pragma unroll
      for (int i = 0; i < SL; ++i) {
        const cx<T> exv = cscale(ldg(a.ex + (size_t)slot[i] * N + j1), (T)a.sw);
        const cx<T>* EY = a.ey + (size_t)slot[i] * N + t;
        const cx<T>* QC = a.Q + (size_t)slot[i] * a.q_ss + (size_t)t * N + j1;
        // FP64 and double-float: the right-hand side b = -sw E_k Q is at hand (12 to 30 % of the pass's
        // arithmetic was the two products that form it again); RES and COR need b itself as well
        if (std::is_same<T, double>::value ? a.b != nullptr : (MODE == BX_RES || MODE == BX_COR)) {
          const cx<T>* bq = a.b + (size_t)slot[i] * a.f_ss + (j1 - bx.x);
#pragma unroll
          for (int q = 0; q < E; ++q) {
            const int y = t + q * TPL;
            const cx<T> bv = ldg_if(bq + (long long)(y - bx.z) * W, inx && y >= bx.z && y < bx.w);
            v[i][q] = cmulc(mkc(-bv.re, -bv.im), v[i][q]);
          }
        } else {
#pragma unroll
          for (int q = 0; q < E; ++q) {
            const int y = t + q * TPL;
            const cx<T> eq = cmul(cmul(exv, ldg(EY + q * TPL)),
                                  ldg_if(QC + (size_t)q * TPL * N, inx && y >= bx.z && y < bx.w));
            v[i][q] = cmulc(eq, v[i][q]);
          }
        }
        const size_t o0 = (size_t)(j1 - bx.x);
        if constexpr (MODE == BX_RES) {
          // r = b - x - w (w negated for the iterated equation), |r|^2 of the box column
          const NT nsc = DD ? (NT)a.nscale[slot[i]] : (NT)1;
          const cx<T>* bb = a.b + (size_t)slot[i] * a.f_ss + o0;
          const cx<T>* xx = a.x + (size_t)slot[i] * a.f_ss + o0;
          const size_t r0 = (size_t)slot[i] * a.r_ss + o0;
#pragma unroll
          for (int q = 0; q < E; ++q) {
            const int y = t + q * TPL;
            const bool in = inx && y >= bx.z && y < bx.w;
            const long long e = (long long)(y - bx.z) * W;
            const cx<T> w = a.neg ? mkc(-v[i][q].re, -v[i][q].im) : v[i][q];
            const cx<T> bv = ldg_if(bb + e, in), xv = ldg_if(xx + e, in);
            const cx<T> r = mkc(bv.re - xv.re - w.re, bv.im - xv.im - w.im);  // 0 outside the box
            if (in) {
              if (!DD && a.r_f64) {
                reinterpret_cast<cx<double>*>(a.r)[r0 + e] = ccast<double>(r);
              } else {
                const cx<float> hi = ccast<float>(r);
                reinterpret_cast<cx<float>*>(a.r)[r0 + e] = hi;
                if (a.rlo) a.rlo[(size_t)slot[i] * a.f_ss + o0 + e] = ccast<float>(mkc(r.re - T(hi.re), r.im - T(hi.im)));
              }
            }
            const NT fr = (NT)r.re * nsc, fi = (NT)r.im * nsc;
            nrm += fr * fr + fi * fi;
          }
        } else if constexpr (MODE == BX_COR) {
          // x += r - w on the box: the correction u = r - K u_c of a coarse-grid solve (coarse.cuh), in the
          // residual's arithmetic
          const size_t r0 = (size_t)slot[i] * a.r_ss + o0, f0 = (size_t)slot[i] * a.f_ss + o0;
#pragma unroll
          for (int q = 0; q < E; ++q) {
            const int y = t + q * TPL;
            const bool in = inx && y >= bx.z && y < bx.w;
            const long long e = (long long)(y - bx.z) * W;
            cx<T> d;
            if (!DD && a.r_f64) {
              d = ccast<T>(ldg_if(reinterpret_cast<const cx<double>*>(a.r) + r0 + e, in));
            } else {
              const cx<float> hi = ldg_if(reinterpret_cast<const cx<float>*>(a.r) + r0 + e, in);
              d = ccast<T>(hi);
              if (a.rlo) d = d + ccast<T>(ldg_if(a.rlo + f0 + e, in));
            }
            d = d - v[i][q];
            if (in) {
              cx<T>* xp = a.xw + f0 + e;
              *xp = *xp + d;
            }
          }
        } else if (a.out) {
          if (on[i]) {
            cx<T>* o = a.out + (size_t)slot[i] * a.out_ss + o0;
#pragma unroll
            for (int q = 0; q < E; ++q) {
              const int y = t + q * TPL;
              if (inx && y >= bx.z && y < bx.w)
                o[(size_t)(y - bx.z) * W] = a.neg ? mkc(-v[i][q].re, -v[i][q].im) : v[i][q];
            }
          }
        }
      }
    }
    if constexpr (!LOOP && (MODE == BX_STEP || MODE == BX_FWD)) {
      if constexpr (SL == 2) fft_line2<T, LOGN, false, F32>(v[0], v[SL - 1], line[0], line[SL - 1], t, a.tw);
      else fft_line<T, LOGN, false, F32>(v[0], line[0], t, a.tw);
    }
  }
  if constexpr (MODE == BX_STEP || MODE == BX_FWD) {
#pragma unroll
    for (int i = 0; i < SL; ++i) {
      if (!on[i]) continue;
      cx<T>* dst = a.mid + (size_t)slot[i] * a.mid_ss + (size_t)t * N + j1;
#pragma unroll
      for (int q = 0; q < E; ++q) dst[(size_t)q * TPL * N] = v[i][q];
    }
  }
  if constexpr (MODE == BX_RES) {
    // one partial per box column and warp of it: the same sums whatever the columns per block
    for (int o = G::CW; o < 32; o *= 2) nrm += __shfl_xor_sync(0xffffffffu, nrm, o);
    if (lane < G::CW) {
      const double nsc = DD ? (double)a.nscale[s0] : 1.0;
      a.part[(size_t)s0 * a.part_ss + (size_t)(j1 - c0) * G::WPG + warp % G::WPG] = (double)nrm / (nsc * nsc);
    }
  }
}

// Row moments R_a(p2) = i N (-1)^{p2} sum_x x^a T2(x, p2), a = 1..MA, of a row of T2 (ca_moments,
// passes.cuh) for the double-float and FP64 passes: the powers x_j^a from a table.
template <typename T, int LOGN, int E>
__device__ __forceinline__ void box_moments(const BoxArgs<T>& a, const cx<T> (&v)[E], cx<double>* part, int p2,
                                            int t, int seg) {
  constexpr int N = 1 << LOGN, TPL = N / E, SEGW = TPL >= 32 ? 32 : TPL;
  const int MA = a.M > 1 ? a.M : 1;
  const double sN = (p2 & 1) ? -(double)N : (double)N;
  for (int aa = 1; aa <= MA; ++aa) {
    cx<T> acc = mkc((T)0, (T)0);
    const T* X = a.xpow + (size_t)aa * N + t;
#pragma unroll
    for (int q = 0; q < E; ++q) {
      if constexpr (std::is_same<T, dd>::value) {
        const T x = X[q * TPL];
        dd_acc(acc.re, v[q].re, x);
        dd_acc(acc.im, v[q].im, x);
      } else {
        acc = acc + cscale(v[q], X[q * TPL]);
      }
    }
    acc = cnorm(acc);
    const T re = warp_sum_t(acc.re, SEGW), im = warp_sum_t(acc.im, SEGW);
    if ((t & (SEGW - 1)) == 0) part[seg * (MA + 1) + aa] = mkc(-(double)im * sN, (double)re * sN);
  }
}

// Row kernel: T2 row -> moments, DFT, S/xi, IDFT -> T1 row (box columns).  SH: the shifted
// quotient of the iterated equation (row_a, passes.cuh).  The signs (-1)^{p1+p2} of Phi and of
// F^{-1} cancel: S~ (-1)^p/(2 pi L^2) = DFT(T2) (m2 + i m1)/(2 pi L (m1^2 + m2^2)).
// Bound by issue (two transforms a row, no N^2-point vector written): FP32, 16 slots of 1024^2, 0.082 ms
// in the shape the tuner takes, where a plain pass C and pass A in turn take 0.118 ms.  FP64, 48 slots of
// 512^2: 0.47 ms a launch, the FP64 pipe's rate.
template <typename T, int LOGN, bool SH, int RV>
__global__ void __launch_bounds__(BoxRowG<T, LOGN, RV>::THREADS, BoxRowG<T, LOGN, RV>::MINB) k_box_rows(const BoxArgs<T> a) {
  using G = BoxRowG<T, LOGN, RV>;
  constexpr int N = G::N, E = G::E, TPL = G::TPL, LINES = G::LINES, P = G::P;
  constexpr bool F32 = std::is_same<T, float>::value;
  constexpr int SEGW = TPL >= 32 ? 32 : TPL, NSEG = TPL >= 32 ? TPL / 32 : 1;
  using PT = typename std::conditional<F32, float, double>::type;
  extern __shared__ __align__(16) unsigned char smem[];
  const int slot = blockIdx.y;
  if (a.run && !a.run[slot]) return;
  const int line = threadIdx.x / TPL, t = threadIdx.x - line * TPL;
  const int p2 = blockIdx.x * LINES + line;
  cx<T>* sl = reinterpret_cast<cx<T>*>(smem) + line * P;
  const int4 bx = a.box[slot];
  const int c0 = a.allcols ? 0 : bx.x, c1 = a.allcols ? N : bx.y;
  const cx<T>* src = a.in + (size_t)slot * a.in_ss + (size_t)p2 * N + t;
  cx<T> v[E];
#pragma unroll
  for (int q = 0; q < E; ++q) {
    const int x = t + q * TPL;
    v[q] = ldg_if(src + q * TPL, x >= c0 && x < c1);
  }
  const int MA = a.M > 1 ? a.M : 1;
  const int seg = TPL >= 32 ? t / 32 : 0;
  cx<PT>* part = reinterpret_cast<cx<PT>*>(a.partA) + ((size_t)slot * N + p2) * NSEG * (MA + 1);
  if constexpr (F32) {
    const float tm = (float)(t - N / 2), hx = a.hx_f;
    const float sN = (p2 & 1) ? -(float)N : (float)N;
    if (MA <= 2) {
      // orders up to 2: both moments in one sweep, no powers held in registers
      float m[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int q = 0; q < E; ++q) {
        const float x = hx * (tm + (float)(q * TPL)), xx = x * x;
        m[0] = fmaf(x, v[q].re, m[0]);
        m[1] = fmaf(x, v[q].im, m[1]);
        m[2] = fmaf(xx, v[q].re, m[2]);
        m[3] = fmaf(xx, v[q].im, m[3]);
      }
#pragma unroll
      for (int aa = 1; aa <= 2; ++aa) {
        const float re = warp_sum_t(m[2 * aa - 2], SEGW), im = warp_sum_t(m[2 * aa - 1], SEGW);
        if (aa <= MA && (t & (SEGW - 1)) == 0) part[seg * (MA + 1) + aa] = mkc(-im * sN, re * sN);
      }
    } else {
      float pw[E];  // x^a of this thread's columns
#pragma unroll
      for (int q = 0; q < E; ++q) pw[q] = hx * (tm + (float)(q * TPL));
      for (int aa = 1; aa <= MA; ++aa) {
        float re = 0.f, im = 0.f;
#pragma unroll
        for (int q = 0; q < E; ++q) {
          if (aa > 1) pw[q] *= hx * (tm + (float)(q * TPL));
          re = fmaf(pw[q], v[q].re, re);
          im = fmaf(pw[q], v[q].im, im);
        }
        re = warp_sum_t(re, SEGW);
        im = warp_sum_t(im, SEGW);
        if ((t & (SEGW - 1)) == 0) part[seg * (MA + 1) + aa] = mkc(-im * sN, re * sN);
      }
    }
  } else {
    box_moments<T, LOGN>(a, v, part, p2, t, seg);
  }
  T c2piL;
  if constexpr (F32) c2piL = a.inv2piL_f;
  else c2piL = (T)a.inv2piL;
  const float tf = (float)t;
  // one copy of the double-float transform's code for both transforms (k_box_cols)
  constexpr bool LOOP = std::is_same<T, dd>::value;
#pragma unroll 1
  for (int ph = 0; ph < (LOOP ? 2 : 1); ++ph) {
    if constexpr (LOOP) fft_line_compact<T, LOGN, false>(v, sl, t, a.tw);
    else fft_line<T, LOGN, false, F32>(v, sl, t, a.tw);
    if (LOOP && ph == 1) break;
    if (t == 0) {  // R_0 = N S(p1 = 0), S = i (-1)^p DFT(T2); its other segments are not read
      const PT s = (p2 & 1) ? -(PT)N : (PT)N;
      part[0] = mkc(-(PT)v[0].im * s, (PT)v[0].re * s);
    }
    int m2 = wavenum(p2, N), hi1 = N >> 1, lo1 = -(N >> 1) + 1;
    if constexpr (SH) {
      const int s1 = a.dshift[2 * slot], s2 = a.dshift[2 * slot + 1];
      if (m2 > (N >> 1) - s2) m2 -= N;
      else if (m2 < -(N >> 1) + 1 - s2) m2 += N;
      hi1 -= s1;
      lo1 -= s1;
    }
    // wavenumbers and their squares are exact in FP32 (|m| <= 2 N, m1^2 + m2^2 < 2^24)
    const float m2f = (float)m2, m2sq = m2f * m2f;
    const bool tab = !SH && std::is_same<T, double>::value && a.kap;
    const cx<T>* kap = a.kap + (size_t)p2 * N + t;
#pragma unroll
    for (int q = 0; q < E; ++q) {
      cx<T> k;
      if (tab) {  // FP64: the factor from a table (its division was 15 % of the pass's FP64 instructions)
        k = ldg(kap + q * TPL);
      } else {
        const int p1 = t + q * TPL;
        // m1 = p1 or p1 - N: p1 > N/2 for every t when q > E/2, for no t when q < E/2
        float m1f = tf + (float)(q <= E / 2 ? q * TPL : q * TPL - N);
        if (q == E / 2 && t > 0) m1f -= (float)N;
        if constexpr (SH) {
          const int m1 = wavenum(p1, N);
          if (m1 > hi1) m1f -= (float)N;
          else if (m1 < lo1) m1f += (float)N;
        }
        T f = kappa_scale<T>(c2piL, T(fmaf(m1f, m1f, m2sq)));
        if (q == 0 && p1 == 0 && p2 == 0) f = T(0.f);
        k = mkc(f * m2f, f * m1f);
      }
      const cx<T> y = cmul(v[q], k);
      v[q] = LOOP && !a.spec ? mkc(y.re, -y.im) : y;
    }
    if (a.spec) {
      cx<T>* dst = a.mid + (size_t)slot * a.mid_ss + (size_t)p2 * N + t;
#pragma unroll
      for (int q = 0; q < E; ++q) dst[q * TPL] = v[q];
      return;
    }
  }
  if constexpr (LOOP) {
#pragma unroll
    for (int q = 0; q < E; ++q) v[q].im = -v[q].im;
  } else {
    fft_line<T, LOGN, true, F32>(v, sl, t, a.tw);
  }
  cx<T>* dst = a.mid + (size_t)slot * a.mid_ss + (size_t)p2 * N + t;
#pragma unroll
  for (int q = 0; q < E; ++q) {
    const int x = t + q * TPL;
    if (x >= c0 && x < c1) dst[q * TPL] = v[q];
  }
}

// Rows of the prolongation: T1 row p2 = IDFT of the coarse grid's spectrum S~ (k_box_rows with spec on
// the grid of N / 2^cs points) padded with zeros to N modes; rows beyond the coarse modes are zero.  The
// coarse Nyquist modes are left out.  Latency- and HBM-bound like k_box_rows; once per coarse cycle.
template <typename T, int LOGN, int RV>
__global__ void __launch_bounds__(BoxRowG<T, LOGN, RV>::THREADS, BoxRowG<T, LOGN, RV>::MINB) k_box_embed(const BoxArgs<T> a, int cs) {
  using G = BoxRowG<T, LOGN, RV>;
  constexpr int N = G::N, E = G::E, TPL = G::TPL, LINES = G::LINES, P = G::P;
  constexpr bool F32 = std::is_same<T, float>::value;
  extern __shared__ __align__(16) unsigned char smem[];
  const int slot = blockIdx.y;
  if (a.run && !a.run[slot]) return;
  const int line = threadIdx.x / TPL, t = threadIdx.x - line * TPL;
  const int p2 = blockIdx.x * LINES + line, NC = N >> cs, m2 = wavenum(p2, N);
  cx<T>* sl = reinterpret_cast<cx<T>*>(smem) + line * P;
  const int4 bx = a.box[slot];
  const int c0 = a.allcols ? 0 : bx.x, c1 = a.allcols ? N : bx.y;
  const bool row = 2 * (m2 < 0 ? -m2 : m2) < NC;
  const cx<T>* src = a.in + (size_t)slot * a.in_ss + (size_t)(m2 & (NC - 1)) * NC;
  cx<T> v[E];
#pragma unroll
  for (int q = 0; q < E; ++q) {
    const int m1 = wavenum(t + q * TPL, N);
    v[q] = ldg_if(src + (m1 & (NC - 1)), row && 2 * (m1 < 0 ? -m1 : m1) < NC);
  }
  fft_line<T, LOGN, true, F32>(v, sl, t, a.tw);
  cx<T>* dst = a.mid + (size_t)slot * a.mid_ss + (size_t)p2 * N + t;
#pragma unroll
  for (int q = 0; q < E; ++q) {
    const int x = t + q * TPL;
    if (x >= c0 && x < c1) dst[q * TPL] = v[q];
  }
}

// Rows of the residual's spectrum, DFT of a T2 row: |.|^2 over all modes, and over the modes beyond the
// grid of N / 2^{l+1} points (|m| >= N / 2^{l+2} in either direction), per row and warp of it, in FP32.
// Values scaled by scale[slot] (a power of two near 1/||b||).  Once per cycle: 0.31 ms at 128 slots of
// 1024^2, a quarter of one FP32 step there (row and column pass 1.3 ms).
template <typename T, int LOGN, int RV>
__global__ void __launch_bounds__(BoxRowG<T, LOGN, RV>::THREADS, BoxRowG<T, LOGN, RV>::MINB) k_box_modes(const BoxArgs<T> a, const float* scale, float* rough) {
  using G = BoxRowG<T, LOGN, RV>;
  constexpr int N = G::N, E = G::E, TPL = G::TPL, LINES = G::LINES, P = G::P;
  constexpr bool F32 = std::is_same<T, float>::value;
  constexpr int SEGW = TPL >= 32 ? 32 : TPL, NSEG = TPL >= 32 ? TPL / 32 : 1;
  extern __shared__ __align__(16) unsigned char smem[];
  const int slot = blockIdx.y;
  if (a.run && !a.run[slot]) return;
  const int line = threadIdx.x / TPL, t = threadIdx.x - line * TPL;
  const int p2 = blockIdx.x * LINES + line, m2 = wavenum(p2, N);
  cx<T>* sl = reinterpret_cast<cx<T>*>(smem) + line * P;
  const int4 bx = a.box[slot];
  const int c0 = a.allcols ? 0 : bx.x, c1 = a.allcols ? N : bx.y;
  const cx<T>* src = a.in + (size_t)slot * a.in_ss + (size_t)p2 * N + t;
  const float sc = scale[slot];
  cx<T> v[E];
#pragma unroll
  for (int q = 0; q < E; ++q) {
    const int x = t + q * TPL;
    v[q] = cscale(ldg_if(src + q * TPL, x >= c0 && x < c1), (T)sc);
  }
  fft_line<T, LOGN, false, F32>(v, sl, t, a.tw);
  float s[kLevels + 1];
#pragma unroll
  for (int l = 0; l <= kLevels; ++l) s[l] = 0.f;
#pragma unroll
  for (int q = 0; q < E; ++q) {
    const int m1 = wavenum(t + q * TPL, N), mm = max(m1 < 0 ? -m1 : m1, m2 < 0 ? -m2 : m2);
    const float re = (float)v[q].re, im = (float)v[q].im, e = re * re + im * im;
    s[0] += e;
#pragma unroll
    for (int l = 0; l < kLevels; ++l)
      if (mm >= (N >> (l + 2))) s[l + 1] += e;
  }
  float* dst = rough + (((size_t)slot * N + p2) * NSEG + (TPL >= 32 ? t / 32 : 0)) * (kLevels + 1);
#pragma unroll
  for (int l = 0; l <= kLevels; ++l) {
    const float w = warp_sum_t(s[l], SEGW);
    if ((t & (SEGW - 1)) == 0) dst[l] = w;
  }
}

// Read-out: S = i (-1)^p DFT(T2 row) in FP64, straight to the caller's buffer (device, or mapped
// host memory).  The rounding of hi + lo is done in integer arithmetic (ddround.cuh).
__device__ __forceinline__ double box_to_double(double x) { return x; }
__device__ __forceinline__ double box_to_double(dd x) { return dd_sum_rn(x.hi, x.lo); }
template <typename T, int LOGN, int RV>
__global__ void __launch_bounds__(BoxRowG<T, LOGN, RV>::THREADS, BoxRowG<T, LOGN, RV>::MINB) k_box_out(const BoxArgs<T> a) {
  using G = BoxRowG<T, LOGN, RV>;
  constexpr int N = G::N, E = G::E, TPL = G::TPL, LINES = G::LINES, P = G::P;
  extern __shared__ __align__(16) unsigned char smem[];
  const int slot = blockIdx.y;
  const int line = threadIdx.x / TPL, t = threadIdx.x - line * TPL;
  const int p2 = blockIdx.x * LINES + line;
  cx<T>* sl = reinterpret_cast<cx<T>*>(smem) + line * P;
  const int4 bx = a.box[slot];
  const int c0 = a.allcols ? 0 : bx.x, c1 = a.allcols ? N : bx.y;
  const cx<T>* src = a.in + (size_t)slot * a.in_ss + (size_t)p2 * N + t;
  cx<T> v[E];
#pragma unroll
  for (int q = 0; q < E; ++q) {
    const int x = t + q * TPL;
    v[q] = ldg_if(src + q * TPL, x >= c0 && x < c1);
  }
  fft_line<T, LOGN, false, false>(v, sl, t, a.tw);
  double2* dst = reinterpret_cast<double2*>(a.S + (size_t)slot * N * N + (size_t)p2 * N + t);
#pragma unroll
  for (int q = 0; q < E; ++q) {
    const cx<T> y = ((t + q * TPL + p2) & 1) ? mkc(v[q].im, -v[q].re) : mkc(-v[q].im, v[q].re);
    dst[q * TPL] = make_double2(box_to_double(y.re), box_to_double(y.im));
  }
}

}  // namespace dbar
