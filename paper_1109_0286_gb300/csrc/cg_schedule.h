// Default launch schedule of the power-of-two passes, shared by the plans
// (cgfill.cu) and the plan-free operator entry point (cg_static.cu), so the
// two cannot drift apart.
#pragma once
#include <algorithm>
#include <type_traits>

#include "cg_launch.h"
#include "cg_types.h"

namespace cgf {

// Row-pass CTA height.  FP32 and double-float: 8 rows (64-byte runs of the
// transposed spectrum), within 512 threads (two CTAs per SM) unless that
// would leave fewer than 4 rows, and within the shared memory of a CTA.  FP64:
// 4 rows, 2 on rows of 1024 pixels and more: the FP64 pipe bounds these
// passes, and small CTAs spread it evenly.  Measured per CG iteration:
// 1024^2 FP32, one map, 16 rows 86.6, 8 rows 76.7, 4 rows 75.8 us; 16 maps
// 364, 359, 433 us; FP64 256^2 16, 8, 4 rows 224, 152, 120 us; FP64 2048^2
// 4, 2 rows 2359, 2156 us.
template <typename T>
inline int default_rows(int log_l, int ny) {
  const int TT = (1 << log_l) >> row_le<T>(log_l);
  int rows = 8;
  if (std::is_same<T, double>::value) rows = log_l >= 9 ? 2 : 4;
  const int cap = std::min(512, Launch<T>::max_threads());
  rows = std::min(rows, std::max(cap / TT, std::min(4, Launch<T>::max_threads() / TT)));
  while (rows > 1 && Launch<T>::row_smem(log_l, rows) > 210 * 1024) rows /= 2;
  return std::min(rows, ny);
}

// Column FFTs per CTA: about 256 threads (FP64: 64, as above; 256^2, one
// map, 8 columns 269, 2 columns 203 us per iteration), within the thread and
// shared-memory limits, and in FP32 no more than leaves two CTAs per SM (1024^2,
// one map, 4 columns 70.5, 1 column 66.0 us per iteration; 16 maps 300 and 348;
// double-float relaxation of 1024^2 1174 and 1257 us, so not there).  ninst
// maps share a launch; the results do not depend on the choice.
template <typename T>
inline int default_ffts(int log_n, int nkx, int ninst) {
  const int TT = (1 << log_n) >> col_le<T>(log_n);
  int f = std::max(1, (std::is_same<T, double>::value ? 64 : 256) / TT);
  f = std::min(f, std::max(1, Launch<T>::max_threads() / TT));
  while (f > 1 && (Launch<T>::col_smem(log_n, f) > 100 * 1024 ||
                   (std::is_same<T, float>::value && (long long)nkx * ninst < 2LL * 152 * f)))
    f /= 2;
  return std::min(f, nkx);
}

// A CTA shape asked for by the options or read from a tuning cache, cut to the
// threads of a CTA: such shapes are stated for 16 elements per thread
// (L / 16 threads per row); a transform with fewer elements per thread takes
// as many rows (columns) as fit.  Shapes that are too large at 16 elements
// per thread are left as they are (and refused).
template <typename T>
inline int fit_shape(int log, int le, int count) {
  const int per16 = (1 << log) / 16, old_max = std::is_same<T, float>::value ? 1024 : 512;
  if (count < 1 || count * per16 > old_max) return count;
  while (count > 1 && (count << log >> le) > Launch<T>::max_threads()) count /= 2;
  return count;
}
template <typename T>
inline int fit_rows(int log_l, int rows) { return fit_shape<T>(log_l, row_le<T>(log_l), rows); }
template <typename T>
inline int fit_ffts(int log_n, int ffts) { return fit_shape<T>(log_n, col_le<T>(log_n), ffts); }

// Whether a (rows, ffts) schedule can be launched on an ny x nx grid.
template <typename T>
inline bool schedule_valid(int log_l, int log_n, int ny, int rows, int ffts) {
  const int TT = (1 << log_l) >> row_le<T>(log_l), TN = (1 << log_n) >> col_le<T>(log_n);
  return rows >= 1 && ffts >= 1 && rows * TT <= Launch<T>::max_threads() && ny % rows == 0 &&
         ny / rows <= kMaxPartials && Launch<T>::row_smem(log_l, rows) <= 227 * 1024 &&
         ffts * TN <= Launch<T>::max_threads() && Launch<T>::col_smem(log_n, ffts) <= 227 * 1024;
}

}  // namespace cgf
