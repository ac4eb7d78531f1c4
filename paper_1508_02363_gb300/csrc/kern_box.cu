// The passes on the potential's box for one precision (DBAR_T: float or dd) and one grid size
// (N = 2^DBAR_LOGN), compiled once per pair like kern_pass.cu.
#include "box.cuh"
#include "launch.cuh"

namespace dbar {

template <typename T, int LOGN, int MODE, int CV, int SL>
static cudaError_t launch_cols_shape(const BoxArgs<T>& a, int nslots, cudaStream_t s) {
  using G = BoxColG<T, LOGN, CV>;
  constexpr size_t lines = align16((size_t)SL * G::COLS * G::P * sizeof(cx<T>)), per = SL * sizeof(cx<T>);
  static_assert(lines + (KC_MAXM + 2) * per <= kSmemLimit, "k_box_cols' shared memory");
  const size_t sm = lines + (a.M + 2) * per;
  const cudaError_t e = allow_smem(k_box_cols<T, LOGN, MODE, CV, SL>, lines + (KC_MAXM + 2) * per);
  if (e != cudaSuccess) return e;
  k_box_cols<T, LOGN, MODE, CV, SL><<<dim3((nslots + SL - 1) / SL, G::N / G::COLS), G::THREADS, sm, s>>>(a);
  return cudaGetLastError();
}

// Launches whose ordinary blocks are fewer than this take the small shapes (one warp per row block,
// one column group per column block): about two blocks per SM.  A 64^2 FP64 solve ran each pass as one
// block, 80 us on one SM; in eight blocks it is 10-12 us.  The arithmetic per line does not change.
constexpr long long kFewBlocks = 304;

template <typename T, int LOGN, int MODE>
static cudaError_t launch_cols_mode(const BoxArgs<T>& a, int nslots, cudaStream_t s) {
  if constexpr (BoxColG<T, LOGN, kColSmall>::COLS < BoxColG<T, LOGN, 0>::COLS)
    if ((long long)nslots * (BoxColG<T, LOGN, 0>::N / BoxColG<T, LOGN, 0>::COLS) < kFewBlocks)
      return launch_cols_shape<T, LOGN, MODE, kColSmall, 1>(a, nslots, s);
  if constexpr (std::is_same<T, float>::value) {
    if (a.colv == 1) return launch_cols_shape<T, LOGN, MODE, 1, 1>(a, nslots, s);
    // two slots per block share the potential's tiles: one potential (and box) for all slots
    if (a.colv == 2 && a.q_ss == 0) return launch_cols_shape<T, LOGN, MODE, 0, 2>(a, nslots, s);
  }
  return launch_cols_shape<T, LOGN, MODE, 0, 1>(a, nslots, s);
}

template <typename T, int LOGN>
cudaError_t launch_box_cols_n(const BoxArgs<T>& a0, int mode, int nslots, cudaStream_t s) {
  BoxArgs<T> a = a0;
  a.nslots = nslots;
  switch (mode) {
    case BX_FWD: return launch_cols_mode<T, LOGN, BX_FWD>(a, nslots, s);
    case BX_STEP: return launch_cols_mode<T, LOGN, BX_STEP>(a, nslots, s);
    case BX_LAST: return launch_cols_mode<T, LOGN, BX_LAST>(a, nslots, s);
    case BX_COR:
      if constexpr (!std::is_same<T, float>::value) return launch_cols_mode<T, LOGN, BX_COR>(a, nslots, s);
      return cudaErrorInvalidValue;
    case BX_RES:
      if constexpr (!std::is_same<T, float>::value) return launch_cols_mode<T, LOGN, BX_RES>(a, nslots, s);
  }
  return cudaErrorInvalidValue;
}

template <typename T, int LOGN, bool SH, int RV>
static cudaError_t launch_rows_shape(const BoxArgs<T>& a, int nslots, cudaStream_t s) {
  using G = BoxRowG<T, LOGN, RV>;
  const size_t sm = (size_t)G::LINES * G::P * sizeof(cx<T>);
  const cudaError_t e = allow_smem(k_box_rows<T, LOGN, SH, RV>, sm);
  if (e != cudaSuccess) return e;
  k_box_rows<T, LOGN, SH, RV><<<dim3(G::N / G::LINES, nslots), G::THREADS, sm, s>>>(a);
  return cudaGetLastError();
}

template <typename T, int LOGN>
cudaError_t launch_box_rows_n(const BoxArgs<T>& a, int nslots, cudaStream_t s) {
  if constexpr (BoxRowG<T, LOGN, kRowSmall>::LINES < BoxRowG<T, LOGN, 0>::LINES)
    if ((long long)nslots * (BoxRowG<T, LOGN>::N / BoxRowG<T, LOGN>::LINES) < kFewBlocks)
      return a.dshift ? launch_rows_shape<T, LOGN, true, kRowSmall>(a, nslots, s)
                      : launch_rows_shape<T, LOGN, false, kRowSmall>(a, nslots, s);
  if (a.dshift) return launch_rows_shape<T, LOGN, true, 0>(a, nslots, s);  // shifted quotient
  if constexpr (std::is_same<T, float>::value) {
    if (a.rowv == 1) return launch_rows_shape<T, LOGN, false, 1>(a, nslots, s);
    if (a.rowv == 2) return launch_rows_shape<T, LOGN, false, 2>(a, nslots, s);
    if (a.rowv == 3) return launch_rows_shape<T, LOGN, false, 3>(a, nslots, s);
    if (a.rowv == 4) return launch_rows_shape<T, LOGN, false, 4>(a, nslots, s);
  }
  return launch_rows_shape<T, LOGN, false, 0>(a, nslots, s);
}

template <typename T, int LOGN, int RV>
static cudaError_t launch_embed_shape(const BoxArgs<T>& a, int cs, int nslots, cudaStream_t s) {
  using G = BoxRowG<T, LOGN, RV>;
  const size_t sm = (size_t)G::LINES * G::P * sizeof(cx<T>);
  const cudaError_t e = allow_smem(k_box_embed<T, LOGN, RV>, sm);
  if (e != cudaSuccess) return e;
  k_box_embed<T, LOGN, RV><<<dim3(G::N / G::LINES, nslots), G::THREADS, sm, s>>>(a, cs);
  return cudaGetLastError();
}
template <typename T, int LOGN>
cudaError_t launch_box_embed_n(const BoxArgs<T>& a, int cs, int nslots, cudaStream_t s) {
  if constexpr (BoxRowG<T, LOGN, kRowSmall>::LINES < BoxRowG<T, LOGN, 0>::LINES)
    if ((long long)nslots * (BoxRowG<T, LOGN>::N / BoxRowG<T, LOGN>::LINES) < kFewBlocks)
      return launch_embed_shape<T, LOGN, kRowSmall>(a, cs, nslots, s);
  return launch_embed_shape<T, LOGN, 0>(a, cs, nslots, s);
}

template <typename T, int LOGN, int RV>
static cudaError_t launch_modes_shape(const BoxArgs<T>& a, const float* scale, float* rough, int nslots, cudaStream_t s) {
  using G = BoxRowG<T, LOGN, RV>;
  const size_t sm = (size_t)G::LINES * G::P * sizeof(cx<T>);
  const cudaError_t e = allow_smem(k_box_modes<T, LOGN, RV>, sm);
  if (e != cudaSuccess) return e;
  k_box_modes<T, LOGN, RV><<<dim3(G::N / G::LINES, nslots), G::THREADS, sm, s>>>(a, scale, rough);
  return cudaGetLastError();
}
template <typename T, int LOGN>
cudaError_t launch_box_modes_n(const BoxArgs<T>& a, const float* scale, float* rough, int nslots, cudaStream_t s) {
  if constexpr (BoxRowG<T, LOGN, kRowSmall>::LINES < BoxRowG<T, LOGN, 0>::LINES)
    if ((long long)nslots * (BoxRowG<T, LOGN>::N / BoxRowG<T, LOGN>::LINES) < kFewBlocks)
      return launch_modes_shape<T, LOGN, kRowSmall>(a, scale, rough, nslots, s);
  return launch_modes_shape<T, LOGN, 0>(a, scale, rough, nslots, s);
}

template <typename T, int LOGN, int RV>
static cudaError_t launch_out_shape(const BoxArgs<T>& a, int nslots, cudaStream_t s) {
  using G = BoxRowG<T, LOGN, RV>;
  const size_t sm = (size_t)G::LINES * G::P * sizeof(cx<T>);
  const cudaError_t e = allow_smem(k_box_out<T, LOGN, RV>, sm);
  if (e != cudaSuccess) return e;
  k_box_out<T, LOGN, RV><<<dim3(G::N / G::LINES, nslots), G::THREADS, sm, s>>>(a);
  return cudaGetLastError();
}
template <typename T, int LOGN>
cudaError_t launch_box_out_n(const BoxArgs<T>& a, int nslots, cudaStream_t s) {
  if constexpr (BoxRowG<T, LOGN, kRowSmall>::LINES < BoxRowG<T, LOGN, 0>::LINES)
    if ((long long)nslots * (BoxRowG<T, LOGN>::N / BoxRowG<T, LOGN>::LINES) < kFewBlocks)
      return launch_out_shape<T, LOGN, kRowSmall>(a, nslots, s);
  return launch_out_shape<T, LOGN, 0>(a, nslots, s);
}

template cudaError_t launch_box_cols_n<DBAR_T, DBAR_LOGN>(const BoxArgs<DBAR_T>&, int, int, cudaStream_t);
template cudaError_t launch_box_rows_n<DBAR_T, DBAR_LOGN>(const BoxArgs<DBAR_T>&, int, cudaStream_t);
#if DBAR_KIND != 2
template cudaError_t launch_box_modes_n<DBAR_T, DBAR_LOGN>(const BoxArgs<DBAR_T>&, const float*, float*, int, cudaStream_t);
#endif
#if DBAR_KIND != 0
template cudaError_t launch_box_embed_n<DBAR_T, DBAR_LOGN>(const BoxArgs<DBAR_T>&, int, int, cudaStream_t);
template cudaError_t launch_box_out_n<DBAR_T, DBAR_LOGN>(const BoxArgs<DBAR_T>&, int, cudaStream_t);
#endif

}  // namespace dbar
