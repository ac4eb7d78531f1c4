// Argument structures shared by the kernels and the host driver.
#pragma once
#include "cx.cuh"

namespace dbar {

struct Geo {
  int N, logN, tpl, lines, P;
};

template <typename T>
struct PassArgs {
  Geo g;
  int colv;  // column-pass tile variant (autotuned)
  int rowv;  // row-pass shape of the FP32 operator's row passes (autotuned; 0 elsewhere)
  int M;  // Taylor order
  // input field (T), per-slot stride in complex elements; optional per-slot scale
  const cx<T>* in;
  long long in_ss;
  const double* in_scale;
  int in_scale_ss;
  // outputs
  void* out;
  long long out_ss;
  void* out2;  // second output (pass C right-hand side / residual: Krylov start vector)
  long long out2_ss;
  // pass C residual inputs, stored in the residual's arithmetic (FP64 or
  // double-float: x and b of the mixed path never pass through FP64)
  const cx<T>* b;
  const cx<T>* x;
  long long f_ss;
  const int* run;  // per-slot flags (nullable)
  // tables
  const cx<T>* tw;       // [N]   e^{-2 pi i t/N}
  const cx<T>* Da;       // [MA+1][N]
  const cx<double>* Da64;
  const cx<T>* Delta;    // [M+1][N (y index)][N (x index)]  W_n - V_n
  const cx<T>* Q;        // [N (y index)][N (x index)], per slot at stride q_ss (0: shared)
  long long q_ss;
  const cx<T>* ex;       // [slot][N]  e^{-2 i k2 x_j}
  const cx<T>* ey;       // [slot][N]  e^{-2 i k1 y_j}
  double inv2piL;        // 1/(2 pi L)
  float inv2piL_f;       // the same, rounded once on the host (FP32 pass A)
  float hx_f;            // grid spacing 2 pi L / N, rounded once (FP32 fused row pass moments)
  double sw;             // 2 pi L^2 / N^2
  double fillscale;      // 1/(2 pi L^2), or 0 for the zero-fill reading
  cx<double>* partA;     // [slot][p2][nseg][MA+1] row-moment partials (pass A -> k_coef);
                         // stored as cx<float> by the FP32 pass A
  int nseg;              // warp segments per row: seg_count(N)
  const cx<double>* coef;  // [slot][M+2] c_0..c_M, d' (k_coef output, read by pass B)
  double* part;          // [slot][gridDim.x] squared-norm partials (pass C)
  const float* nscale;   // [slot] power-of-two ~1/||b|| (double-float residual norms)
  int neg;               // row pass C: the transform's output negated (K of the iterated equation)
  // pass A of the iterated equation's shifted quotient (eq. dbarinvShift): per slot the signed
  // grid offset (s1, s2) of xi0 by which the input was rolled, so that the divisor of rolled
  // element p is the unwrapped xi_{p + s} - xi0 (nullable: the plain divisor xi_p)
  const int* dshift;
  // the potential's box in the FP32 and double-float passes: the columns [sx0, sx1) (a multiple of every
  // column-pass tile width) outside which |Q| is below 2^-100 of its largest and w = E_k Q conj(h) is taken
  // as zero: pass A stores and pass C loads only those columns of the pass intermediates, and
  // pass B transforms only those columns.  Rows [sy0, sy1): pass B loads its tables
  // only there (the full range -- no per-row test -- unless the plan sets a band).
  int sx0, sx1, sy0, sy1;
};

// Arguments of the passes on the potential's box (box.cuh).  Packed box vectors have a stride of
// N*N elements per vector whatever the box.
template <typename T>
struct BoxArgs {
  int logN, colv, rowv;  // column tile variant, row shape
  int M;                 // Taylor order
  int nslots;
  const int* run;        // per-slot flags (nullable)
  const int4* box;       // [slot] x0, x1 (multiples of every column tile), y0, y1
  int allcols;           // 1: T1, T2 hold and the passes transform every column (support_skip = 0)
  const cx<T>* in;       // columns FWD: box vectors; STEP / LAST / RES: T1; rows: T2
  long long in_ss;
  const double* in_scale;  // FWD: per-slot scale of the input (nullable)
  int in_scale_ss;
  int loadE;             // FWD: the input multiplied by E_k
  cx<T>* mid;            // transform output: T2 (columns), T1 (rows)
  long long mid_ss;
  cx<T>* out;            // STEP / LAST: w on the box (nullable)
  long long out_ss;
  int neg;               // w negated (iterated equation)
  const cx<T>* tw;
  const cx<T>* Delta;
  const cx<T>* Q;
  long long q_ss;
  const cx<T>* ex;
  const cx<T>* ey;
  double sw;
  const cx<double>* coef;
  // RES
  const cx<T>* b;
  const cx<T>* x;
  long long f_ss;
  void* r;               // cx<float>, or cx<double> when r_f64 (FP64 Krylov basis)
  int r_f64;
  long long r_ss;
  double* part;          // [slot][box columns][warps per column] squared-norm partials
  long long part_ss;
  const float* nscale;   // (double-float)
  // RES / COR: the residual r in full: r (V[slot][0]) plus, where the Krylov basis is FP32, its low part
  cx<float>* rlo;        // [slot] at stride f_ss (nullable)
  cx<T>* xw;             // COR: x += r - w
  // rows
  int spec;              // 1: the row's spectrum S~ is stored to mid, every column (no inverse transform)
  cx<double>* partA;
  const T* xpow;         // [MA+1][N] x_j^a (double-float, FP64)
  const cx<T>* kap;      // [N][N] (m2 + i m1)/(2 pi L (m1^2 + m2^2)), 0 at xi = 0 (FP64)
  double inv2piL;
  float inv2piL_f, hx_f;
  const int* dshift;
  // read-out
  cx<double>* S;
};

constexpr int KR_THREADS = 256;
constexpr int KR_EPT = 8;  // complex elements per thread
constexpr int KR_CHUNK = KR_THREADS * KR_EPT;

struct KryArgs {
  long long n;       // complex elements per vector (N*N): their stride
  const int4* box;   // [slot] the vectors' box (nullable: all n elements), packed
  int mp1;           // basis vectors per slot (restart + 1)
  int nchunk;        // blocks per slot
  const int* run;    // per-slot flags of the current cycle
  const double* sigma;  // [slot][mp1]
  double* coef;         // [slot][mp1] update coefficients
  double* part;         // [slot][mp1][nchunk]
  double* part2;        // [slot][nchunk]
};

// s-step (block) Arnoldi sweeps (krylov.cuh)
constexpr int KB_EPT = 4;                      // complex elements per thread (block sweeps)
constexpr int KB_CHUNK = KR_THREADS * KB_EPT;  // elements per block of a block sweep
constexpr double kBlockPivot = 1e-5;           // smallest accepted Cholesky pivot of the normalised Gram
constexpr int kMaxRestart = 128;               // largest restart (basis vectors - 1) of a plan
constexpr int kBlockDotBlocks = 128;           // dot-sweep blocks per slot (fewer partials to fold in FP64)

// elements of a packed box vector
__device__ __forceinline__ long long box_len(const int4* box, int slot, long long n) {
  if (!box) return n;
  const int4 b = box[slot];
  return (long long)(b.y - b.x) * (b.w - b.z);
}

struct BlockArgs {
  long long n;          // complex elements per vector (their stride)
  const int4* box;      // [slot] the vectors' box (nullable: all n elements), packed
  int mp1;              // basis vectors per slot (restart + 1)
  int nwork;            // KB_CHUNK-element chunks per vector (update sweep: one block each)
  int chunk;            // elements per chunk (block_chunk)
  int nchunk;           // dot-sweep blocks per slot (each sums several chunks): partials per item
  int nitem;            // partial-sum items per slot (capacity): mp1 * S + S (S + 1) / 2
  const int* run;       // per-slot flags
  const double* sigma;  // [slot][mp1] scales of the stored basis vectors
  const double* bcoef;  // [slot][S*S + mp1*S]: R^{-1} / ||p|| (S x S), then -sigma_r (C R^{-1})_{r,i}
  double* part;         // [slot][nitem][nchunk]
  // solution update fused into a slot's last block: x += sum_i ycoef_i v~_i
  const double* ycoef;  // [slot][mp1] y_i sigma_i (written by the block's scalar step)
  void* X;              // [slot][n] at stride xss: cx<double>, or cx<dd> when x_dd
  long long xss;
  int x_dd;
  int* err;             // set to 1 when a bounded device wait runs out (nullable)
  int tx_extra;         // bytes the first bulk-copy stage announces beyond its copy (test hook; 0)
};

__host__ __device__ constexpr int block_items(int J, int S) { return J * S + S * (S + 1) / 2; }

struct CycleState {
  double* H;       // [slot][m][m+1]  column j holds rows 0..j+1
  double* cs;      // [slot][m]
  double* sn;      // [slot][m]
  double* g;       // [slot][m+1]
  double* sigma;   // [slot][m+1]
  double* ycoef;   // [slot][m+1]
  double* thr;     // [slot] stop threshold of the current cycle
  double* bnorm;   // [slot]
  float* nscale;   // [slot] 2^-e with 2^e ~ ||b|| (scales FP32 squared norms of residuals)
  double* resid;   // [slot] last true relative residual
  int* run;        // [slot]
  int* active;     // [slot]
  int* nsteps;     // [slot]
  int* itot;       // [slot] total inner iterations on any grid
  int* ncyc;       // [slot] cycles on any grid
  int* cit;        // [slot] of itot, those outside the cap max_iter: on coarse grids (a level's state: on the fine one)
  int* ccyc;       // [slot] of ncyc, those on coarse grids (outside max_outer)
  int m;
  int max_iter;
  int max_outer;
  double tol;
  double inner_tol;  // > 0: mixed-precision inner criterion relative to beta
};

// Coarse-grid correction (coarse.cuh): the levels of a plan, the grids of N / 2 and N / 4 points.
constexpr int kLevels = 2;
constexpr int kCoarseBlocks = 64;
struct CoarseArgs {
  int nlev;
  int N;                     // fine grid
  const int4* box;           // [slot] fine box
  const int4* cbox[kLevels];  // [slot] the level's box
  CycleState c[kLevels];     // the level's cycle state
  double* part;              // [slot][kCoarseBlocks][kLevels + 1] sums of |r|^2
  const float* rough;        // [slot][N][warps per row][kLevels + 1] |DFT r|^2: all modes, beyond each level's
  int nrough;                // N * warps per row
  int* level;                // [slot] level of the slot's cycles, -1: the fine grid
  int* top;                  // [slot] coarsest level still open to the slot
  double* bprev;             // [slot] ||r|| at the last coarse cycle, 0: none
  double* eprev;             // [slot] the reduction it aimed at
  const int* mask;           // only these slots (nullable)
};

// pass B modes: operator, right-hand side, h only, raw column DFTs, and the
// operator's first half (column IDFT, h, w = E_k Q conj(h); no column DFT)
enum { PB_MATVEC = 0, PB_RHS = 1, PB_HOUT = 2, PB_FWD = 3, PB_INV = 4, PB_WF = 5 };
// box column modes (box.cuh): forward transform, operator + forward transform, operator,
// operator + true residual
// (BX_COR: the operator's w, and the coarse correction x += r - w)
enum { BX_FWD = 0, BX_STEP = 1, BX_LAST = 2, BX_RES = 3, BX_COR = 4 };
// pass C modes: K S, right-hand side, FP64 residual, raw row DFTs
enum { PC_KS = 0, PC_RHS = 1, PC_RES = 2, PC_FWD = 3, PC_INV = 4 };

}  // namespace dbar
