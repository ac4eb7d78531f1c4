// Box of a potential, the right-hand side on it, and the solution's value at xi = 0 (box.cuh).
#include "krylov.cuh"
#include "launch.cuh"

namespace dbar {

// scan: x0, x1, y0, y1 (inclusive) of the box, high word of the largest |Re|, |Im|
__global__ void k_box_arm(int* scan, int N) {
  scan[0] = scan[2] = N;
  scan[1] = scan[3] = -1;
  scan[4] = 0;
}
cudaError_t launch_box_arm(int* scan, int N, cudaStream_t s) {
  k_box_arm<<<1, 1, 0, s>>>(scan, N);
  return cudaGetLastError();
}

// high word of |x|: orders like |x| (no FP64 instruction)
__device__ __forceinline__ int hi_abs(double x) { return __double2hiint(x) & 0x7fffffff; }

// Copies of the potential, the finiteness check and the largest magnitude in one pass (HBM-bound:
// one read, three writes; four kernels before).
__global__ void __launch_bounds__(256) k_box_load(const cx<double>* __restrict__ Q, int N, int stride, cx<double>* Q64,
                                                  cx<float>* Q32, cx<dd>* Qdd, int* flag, int* scan) {
  int hm = 0;
  const long long n = (long long)N * N;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    // stride > 1: the coarse grid's points of a grid of N stride points
    const long long y = i / N, o = stride == 1 ? i : y * stride * N * stride + (i - y * N) * stride;
    const cx<double> v = Q[o];
    Q64[i] = v;
    Q32[i] = ccast<float>(v);
    if (Qdd) Qdd[i] = ccast<dd>(v);
    hm = max(hm, max(hi_abs(v.re), hi_abs(v.im)));
  }
  hm = __reduce_max_sync(0xffffffffu, hm);
  if ((threadIdx.x & 31) == 0) {
    if (flag && hm >= 0x7ff00000) *flag = 1;
    atomicMax(scan + 4, hm);
  }
}
// Box of the entries of at least 2^-100 of the largest one.  What it leaves out is 2^-47 of one rounding
// error of the FP64 transforms (2^-52 in double-float), times at most N^2 <= 2^22 terms: the products
// with it are below the rounding of the sums they would enter.
constexpr int kBoxOctaves = 100;
__global__ void __launch_bounds__(256) k_box_scan(const cx<double>* __restrict__ Q, int N, int* scan) {
  const long long n = (long long)N * N;
  const int cut = scan[4] - (kBoxOctaves << 20);
  int x0 = N, x1 = -1, y0 = N, y1 = -1;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const cx<double> v = Q[i];
    const bool nz = (hi_abs(v.re) | hi_abs(v.im) | __double2loint(v.re) | __double2loint(v.im)) != 0;
    if (nz && max(hi_abs(v.re), hi_abs(v.im)) >= cut) {
      const int y = (int)(i / N), x = (int)(i - (long long)y * N);
      x0 = min(x0, x), x1 = max(x1, x), y0 = min(y0, y), y1 = max(y1, y);
    }
  }
  const unsigned full = 0xffffffffu;
  x0 = __reduce_min_sync(full, x0);
  y0 = __reduce_min_sync(full, y0);
  x1 = __reduce_max_sync(full, x1);
  y1 = __reduce_max_sync(full, y1);
  if ((threadIdx.x & 31) == 0 && x1 >= 0) {
    atomicMin(scan + 0, x0);
    atomicMax(scan + 1, x1);
    atomicMin(scan + 2, y0);
    atomicMax(scan + 3, y1);
  }
}
// box and qmax (a power of two near the largest magnitude) of slots [0, nset) from the scan; x0, x1
// widened to whole column tiles of `align`; the last statement re-arms the scan
__global__ void k_box_set(int* scan, int N, int align, int4* box, float* qmax, int nset) {
  __shared__ int c[5];
  if (threadIdx.x < 5) c[threadIdx.x] = scan[threadIdx.x];
  __syncthreads();
  const bool none = c[1] < 0;
  const int4 b = none ? make_int4(0, 0, 0, 0)
                      : make_int4((c[0] / align) * align, min(N, (c[1] + align) / align * align), c[2], c[3] + 1);
  const int e = min(max((c[4] >> 20) - 1023, -100), 100);
  for (int i = threadIdx.x; i < nset; i += blockDim.x) {
    box[i] = b;
    qmax[i] = __int_as_float((e + 127) << 23);
  }
  if (threadIdx.x == 0) {
    scan[0] = scan[2] = N;
    scan[1] = scan[3] = -1;
    scan[4] = 0;
  }
}
cudaError_t launch_box_load(const cx<double>* Q, int N, int stride, cx<double>* Q64, cx<float>* Q32, cx<dd>* Qdd, int* flag,
                            int* scan, int4* box, float* qmax, int nset, cudaStream_t s) {
  const long long n = (long long)N * N;
  const int blocks = (int)((n + 1023) / 1024 < 608 ? (n + 1023) / 1024 : 608);
  k_box_load<<<blocks, 256, 0, s>>>(Q, N, stride, Q64, Q32, Qdd, flag, scan);
  k_box_scan<<<blocks, 256, 0, s>>>(Q64, N, scan);
  k_box_set<<<1, 128, 0, s>>>(scan, N, col_align(N), box, qmax, nset);
  return cudaGetLastError();
}

// One row of the box per step and block.  The squared norm: FP64 squares in FP64, else FP32 squares
// scaled by a power of two near 1/(sw max|Q|), summed in FP32 over a thread's part of a row (at most 8
// values) and in FP64 beyond, unscaled once per block.
template <typename T, typename TI>
__global__ void __launch_bounds__(256) k_box_rhs(const int4* __restrict__ box, const float* __restrict__ qmax,
                                                 const int* __restrict__ mask, const cx<T>* __restrict__ Q,
                                                 long long q_ss, const cx<T>* __restrict__ ex,
                                                 const cx<T>* __restrict__ ey, int N, double sw, cx<T>* b, cx<T>* x,
                                                 long long f_ss, cx<TI>* v0, long long v_ss, cx<float>* rlo, double* part) {
  using NT = typename std::conditional<std::is_same<T, double>::value, double, float>::type;
  __shared__ double sh[8];
  const int slot = blockIdx.y;
  if (mask && !mask[slot]) return;
  const int4 bx = box[slot];
  const int W = bx.y - bx.x;
  NT sc = 1;
  if constexpr (!std::is_same<T, double>::value) {
    int e = (__float_as_int((float)sw * qmax[slot]) >> 23) & 0xff;
    e = e < 1 ? 1 : (e > 253 ? 253 : e);
    sc = __int_as_float((254 - e) << 23);
  }
  const T swd = T(sw);
  double sum = 0.0;
  for (int y = bx.z + blockIdx.x; y < bx.w; y += gridDim.x) {
    NT nrm = 0;
    const cx<T> eyv = ldg(ey + (size_t)slot * N + y);
    const size_t o = (size_t)(y - bx.z) * W;
    for (int i = threadIdx.x; i < W; i += blockDim.x) {
      const cx<T> exv = cscale(ldg(ex + (size_t)slot * N + bx.x + i), swd);
      const cx<T> eq = cmul(cmul(exv, eyv), ldg(Q + (size_t)slot * q_ss + (size_t)y * N + bx.x + i));
      const cx<T> u = mkc(-eq.re, -eq.im);
      b[(size_t)slot * f_ss + o + i] = u;
      x[(size_t)slot * f_ss + o + i] = mkc(T(0.f), T(0.f));
      const cx<TI> hi = ccast<TI>(u);
      v0[(size_t)slot * v_ss + o + i] = hi;
      if (rlo) rlo[(size_t)slot * f_ss + o + i] = ccast<float>(mkc(u.re - T(hi.re), u.im - T(hi.im)));
      const NT fr = (NT)u.re * sc, fi = (NT)u.im * sc;
      nrm += fr * fr + fi * fi;
    }
    sum += (double)nrm;
  }
  const double s = block_sum_256(sum, sh);
  if (threadIdx.x == 0) {
    const double inv = 1.0 / (double)sc;
    part[(size_t)slot * gridDim.x + blockIdx.x] = s * inv * inv;
  }
}
template <typename T, typename TI>
cudaError_t launch_box_rhs(const int4* box, const float* qmax, const int* mask, const cx<T>* Q, long long q_ss,
                           const cx<T>* ex, const cx<T>* ey, int N, double sw, cx<T>* b, cx<T>* x, long long f_ss,
                           cx<TI>* v0, long long v_ss, cx<float>* rlo, double* part, int nslots,
                           cudaStream_t s) {
  if (nslots <= 0) return cudaSuccess;
  k_box_rhs<T, TI><<<dim3(kBoxRhsBlocks, nslots), 256, 0, s>>>(box, qmax, mask, Q, q_ss, ex, ey, N, sw, b, x, f_ss, v0,
                                                               v_ss, rlo, part);
  return cudaGetLastError();
}
#define RHS_INST(T, TI)                                                                                             \
  template cudaError_t launch_box_rhs<T, TI>(const int4*, const float*, const int*, const cx<T>*, long long,       \
                                             const cx<T>*, const cx<T>*, int, double, cx<T>*, cx<T>*, long long,   \
                                             cx<TI>*, long long, cx<float>*, double*, int, cudaStream_t);
RHS_INST(dd, float)
RHS_INST(double, float)
RHS_INST(double, double)

// (m2 + i m1)/(2 pi L (m1^2 + m2^2)), 0 at xi = 0
__global__ void k_box_kappa(cx<double>* __restrict__ out, int N, double inv2piL) {
  const int n = N * N;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int m2 = wavenum(i / N, N), m1 = wavenum(i % N, N);
    const double f = i == 0 ? 0.0 : inv2piL / ((double)m1 * m1 + (double)m2 * m2);
    out[i] = mkc((double)m2 * f, (double)m1 * f);
  }
}
cudaError_t launch_box_kappa(cx<double>* out, int N, double inv2piL, cudaStream_t s) {
  k_box_kappa<<<N, 256, 0, s>>>(out, N, inv2piL);
  return cudaGetLastError();
}

// S(0) = i sum u, or h(xi0) = i sum E_k u (the field rolled by xi0 is Phi(E_k u))
template <typename T>
__global__ void __launch_bounds__(256) k_box_sum(const int4* __restrict__ box, const cx<T>* __restrict__ x,
                                                 long long f_ss, const cx<T>* __restrict__ ex,
                                                 const cx<T>* __restrict__ ey, int N, cx<double>* __restrict__ out) {
  __shared__ double sr[8], si[8];
  const int slot = blockIdx.x;
  const int4 bx = box[slot];
  const int W = bx.y - bx.x, n = W * (bx.w - bx.z);
  T re(0.f), im(0.f);
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    cx<T> v = ldg(x + (size_t)slot * f_ss + i);
    if (ex) {
      const int r = i / W;
      v = cmul(cmul(ldg(ex + (size_t)slot * N + bx.x + i - r * W), ldg(ey + (size_t)slot * N + bx.z + r)), v);
    }
    re += v.re;
    im += v.im;
  }
  re = warp_sum_t(re, 32);
  im = warp_sum_t(im, 32);
  const int w = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    sr[w] = (double)re;
    si[w] = (double)im;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0, c = 0.0;
    for (int i = 0; i < 8; ++i) {
      a += sr[i];
      c += si[i];
    }
    out[slot] = mkc(-c, a);
  }
}
template <typename T>
cudaError_t launch_box_sum(const int4* box, const cx<T>* x, long long f_ss, const cx<T>* ex, const cx<T>* ey, int N,
                           cx<double>* out, int nslots, cudaStream_t s) {
  if (nslots <= 0) return cudaSuccess;
  k_box_sum<T><<<nslots, 256, 0, s>>>(box, x, f_ss, ex, ey, N, out);
  return cudaGetLastError();
}
template cudaError_t launch_box_sum<dd>(const int4*, const cx<dd>*, long long, const cx<dd>*, const cx<dd>*, int,
                                        cx<double>*, int, cudaStream_t);
template cudaError_t launch_box_sum<double>(const int4*, const cx<double>*, long long, const cx<double>*,
                                            const cx<double>*, int, cx<double>*, int, cudaStream_t);

}  // namespace dbar
