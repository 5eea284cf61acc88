// Shared host/device data structures of the constrained-realization solver.
//
// Layout on the device, per realization ("instance"):
//   * full maps (d, y, w, out, gx): row-major ny x nx;
//   * CG vectors (r, p, q, z, u, b and the mixed-mode r32 / dlt): COMPACT, two
//     values for every pixel pair (2j, 2j + 1) with a masked pixel, in row-major
//     order, zero on its observed pixel (the masked system of Sect. 2.4 lives
//     on M only; the vectors are zero on U);
//   * half spectrum "spec": transposed, (nx/2+1) rows of ny complex values,
//     spec[kx * ny + y]; the column pass runs along contiguous rows;
//   * spectral tables [kx][ky] (same transposed layout), real, with the
//     1/n of the inverse DFT folded in;
//   * mask words: for each 32 pixels, the observed bits (1 = constraint, also
//     beyond the last pixel) and the index of the word's first value in the CG
//     vectors (the number of values of all words before it).
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define CGF_HD __host__ __device__
#else
#define CGF_HD
#endif

namespace cgf {

// Scalar state of one CG solve (Sect. 2.4), kept on the device so the
// iteration runs without host round trips.
struct CgState {
  double rho;      // r^T z of the current iterate
  double alpha;    // step length
  double beta;     // direction update
  float alpha_f, beta_f;   // alpha, beta rounded to FP32 (the FP32 passes)
  double bb;       // ||b||^2
  double rr;       // ||r||^2 after the last update
  double tol2;     // tol^2 (stop when rr <= tol2 * bb)
  double pq;       // last p^T A p
  double rrmax;    // ||r||^2 at the last true-residual update (reliable updates)
  double delta2;   // update when rr <= delta2 * rrmax (reliable updates)
  int iter;        // completed operator applications
  int max_iter;
  int done;        // 1 once converged / stopped; later passes skip the instance
  int status;      // 0 ok, 1 invalid data (non-finite), 3 not converged, 4 breakdown
  int first;       // 1 before the first z: beta = 0
  int hist_cap;
  unsigned int ticket;  // last-CTA counter for the grid reductions
  int refine;      // true-residual recomputations (mixed mode)
  int total_iter;  // inner iterations summed over refinement steps
  int upd;         // reliable updates: update (high-precision state) / reload (FP32 state) due
  int last_iter;   // mixed mode, FP32 state: iterations of the last inner solve
  CgState* peer;   // the other precision's state of the same instance (mixed mode)
  double* hist;    // ||r_k|| / ||b||, k = 0..iter
  double* coef;    // CG coefficients: alpha_j at [2j], beta_j at [2j+1], j < hist_cap
};


// Double-float number hi + lo (|lo| <= ulp(hi) / 2, about 48 significant
// bits): the high-precision type of the mixed mode, whose arithmetic runs on
// the FP32 pipes (GB300's FP64 rate is 1/58 of its FP32 rate).
struct df {
  float hi, lo;
  df() = default;
  CGF_HD constexpr df(float h, float l) : hi(h), lo(l) {}
  CGF_HD constexpr df(double x) : hi((float)x), lo((float)(x - (double)(float)x)) {}
  CGF_HD constexpr df(float x) : hi(x), lo(0.f) {}
  CGF_HD constexpr df(int x) : df((double)x) {}
  CGF_HD explicit operator float() const { return hi + lo; }
  CGF_HD explicit operator double() const { return (double)hi + (double)lo; }
};
struct alignas(16) df2 {
  df x, y;
};

// Element type of the caller's maps (d, out, dL/dx) for a pass element type.
template <typename T>
struct MapOf {
  using type = T;
};
template <>
struct MapOf<df> {
  using type = double;
};

// Per-instance pointers handed to every kernel (element type T of the pass).
template <typename T>
struct InstDesc {
  const uint2* mw;         // mask words: x = observed bits, y = CG-vector offset
  const T* t_inv;          // 1 / (n P)     [kx][ky]
  const T* t_sqrt;         // sqrt(P) / n   [kx][ky]
  T* spec;                 // interleaved complex half spectrum, transposed
  T* spec2;                // second spectrum (gradient products), or null
  T* r;
  T* p;
  T* q;
  T* z;
  T* u;
  T* y;
  T* b;
  const typename MapOf<T>::type* d;    // caller's data map
  typename MapOf<T>::type* out;        // caller's output map (dL/dd in the backward pass)
  const typename MapOf<T>::type* gx;   // caller's dL/dx (backward pass)
  T* w;                    // w = d - y on U, u on M (backward pass)
  float* dlt;              // FP32 correction (mixed mode, high-precision passes)
  float* r32;              // FP32 residual target (mixed mode, high-precision passes)
  CgState* st;
  double* partial;         // per-CTA partial sums
  double* hist;            // residual history (hist_cap entries), or null
  double* coef;            // CG coefficients (2 hist_cap entries), or null
  const T* kt;             // kernel tables [j][kx][ky] of the Sect. 6.3 solver, or null
  T* speck;                // spectra of that solver's kernels that run together, or null
  const uint8_t* cls;      // kernel class of every pixel (Sect. 6.3 solver), or null
  const double* noise;     // tables of the white-noise source
  long long nvec;          // CG-vector length: 2 per pixel pair with a masked pixel
  unsigned long long seed;
};

// Elementwise operations fused into the row passes (runtime-uniform switch).
enum RowOp : int {
  // sources (row pass without an input spectrum)
  OP_XI = 1,        // v = unit white noise (Philox4x32-10 + Box-Muller)
  OP_LOAD_R = 2,    // v = r
  OP_P_UPD_Z = 3,   // p = z + beta p; store p; v = p
  OP_P_UPD_R = 4,   // p = r + beta p; store p; v = p   (no preconditioner)
  OP_R_UPD = 5,     // r -= alpha q; u += alpha p; store; acc ||r||^2; v = r
  OP_U64_UPD = 6,   // u += dlt (FP32 correction); store; v = u  (mixed mode)
  OP_LOAD_W_MASK = 7,  // v = P_x w (full maps; operator checks)
  OP_LOAD_U = 8,    // v = u
  OP_LOAD_Y = 9,    // v = y
  OP_LOAD_D_U = 28, // v = d on U, 0 on M (maximum-likelihood right-hand side)
  OP_LOAD_D = 31,   // v = d (operator applications on the caller's map)
  OP_LOAD_D_M = 32, // v = P_x d
  // middles (input spectrum -> output spectrum)
  OP_MASK = 10,     // v = P_x v
  OP_Y_W = 11,      // store y = v; v = (d - y) on U, 0 on M
  // sinks (input spectrum, no output spectrum)
  OP_STORE_Y = 20,  // store y = v
  OP_STORE_Y_MASK = 27,  // store y = P_x v (full maps; operator checks)
  OP_Q = 21,        // q = P_x v; store; acc p^T q
  OP_Z = 22,        // z = P_x v; store; acc r^T z
  OP_B = 23,        // b = -P_x v; store r = b (and b); acc ||b||^2
  OP_RES = 24,      // r = b - P_x v; store; acc ||r||^2; r32 = (float) r
  OP_GRAD = 25,     // v = C^-1 lam: out = (g - v) on U, 0 on M; y = h = g on M, v on U
  OP_RELAX = 29,    // v = C^-1 w: w -= alpha v on M (alpha = 1/a, Sect. 5 relaxation);
                    // acc ||v_M||^2
  OP_KSEL = 30,     // v = kernel j * w: y = v on the masked pixels of class j (Sect. 6.3)
  OP_LOAD_W = 26,   // (source) v = w
  OP_STORE_OUT = 33,       // out = v (the caller's map)
  OP_STORE_OUT_MASK = 34,  // out = P_x v
};

// Scalar updates run by the last CTA of a reducing pass.
enum ScalarOp : int {
  SC_NONE = 0,
  SC_BB = 1,          // bb = sum; rr = bb; done if bb == 0
  SC_BB_RHO = 2,      // as SC_BB, plus rho = bb, beta = 0 (no preconditioner)
  SC_ALPHA = 3,       // pq = sum; alpha = rho / pq (breakdown if pq <= 0)
  SC_RCHECK = 4,      // rr = sum; iter++; convergence / iteration limit
  SC_RCHECK_BETA = 5, // SC_RCHECK, then beta = rr / rho; rho = rr
  SC_BETA = 6,        // rz = sum; beta = rz / rho (0 on the first); rho = rz
  SC_RES = 7,         // rr = sum (true residual); refine++; done if rr <= tol2 bb
  SC_RCHECK_UPD = 8,  // reliable updates, FP32 state: rr = sum; iter++; request an
                      // update when rr <= delta2 rrmax or rr <= tol2 bb or at max_iter
  SC_RES_UPD = 9,     // reliable updates, high-precision state: true residual; converged -> both
                      // done; else FP32 residual replaced, reload of its spectrum due
  SC_CLEAR_UPD = 10,  // upd = 0 (after the reload)
};

// Instance skipping of a pass: 0 never; 1 once the state is done;
// 2 unless an update is due (and the state is not done).
enum SkipMode : int { SKIP_NEVER = 0, SKIP_DONE = 1, SKIP_UNLESS_UPD = 2 };

enum VecOp : int {
  VOP_UPDATE = 1,     // r -= alpha q; u += alpha p; acc ||r||^2
  VOP_ASSEMBLE = 2,   // out = d on U, y + u on M
  VOP_COPY_D = 3,     // out = d
  VOP_MAKE_W = 5,     // w = d - y on U, u on M
  VOP_LOAD_G = 6,     // r = b = P_x g (r32 = (float) r if set); acc ||r||^2
  VOP_ZERO_UP = 7,    // u = 0, p = 0
  VOP_W_FROM_D = 10,  // w = d on U, 0 on M
  VOP_W_TO_OUT = 11,  // out = w (pass element type -> caller's map)
  VOP_ANNULUS = 12,   // w = 1 where r_in^2 < |offset|^2 <= r_out^2 (offset from pixel 0), else 0
  VOP_Y_TO_W_M = 13,  // w = y on M; acc ||y - w||^2 over M
  VOP_NORM_R = 14,    // acc ||r||^2
};

// Launch arguments of the pass kernels.
struct RowArgs {
  int ny, nx;       // grid (nx = 2 L)
  int rows;         // rows per CTA (power of two)
  int log_rows;     // log2(rows)
  int op;           // RowOp
  int sop;          // ScalarOp (SC_NONE: no reduction)
  int check_done;   // skip instances whose CG state is done
  int spec_sel;     // 0: spec, 1: spec2, 2: speck (grid z: one kernel's spectrum each)
  int param;        // op parameter (OP_KSEL: the kernel class, plus grid z)
  int pdl;          // launch as a programmatic dependent of the previous kernel
  int nz;           // grid z (spec_sel = 2), else 0
};

struct ColArgs {
  int ny;           // column length (FFT size)
  int nkx;          // nx/2 + 1 spectrum rows
  int ffts;         // column FFTs per CTA
  int table;        // 0: 1/(nP), 1: sqrt(P)/n; j + 2: kernel table j; -1: forward only
  int check_done;
  int spec_sel;     // 0: spec, 1: spec2
  int pre;          // 1: the input is spec, already column-transformed (table >= 2; the
                    // forward FFT is skipped; grid z takes table + z into speck's z-th spectrum)
  int* err;         // device error flag (set to 1 when a bounded wait gave up), or null
  int variant;      // FP32 table passes: 0 register-fed kernel, 1 persistent bulk-copy-fed
                    // kernel (chosen per grid by the autotuner)
  int pdl;          // as RowArgs::pdl
  int nz;           // grid z (pre), else 0
};

// Band-binned spectral products for the band-power gradient.
struct DotArgs {
  long long nmodes;     // (nx/2+1) * ny half-plane modes per instance
  int nbands;
  const int* band;      // [kx][ky] band of every mode
  const void* coef;     // [kx][ky] weight (element type of the pass)
  double* part;         // [inst][cta][nbands] partial sums
};

struct VecArgs {
  long long npix;   // pixels per instance
  int op;           // VecOp
  int sop;
  int check_done;
  double p0, p1;    // op parameters (VOP_ANNULUS: r_in^2, r_out^2)
  int nx;           // row length (VOP_ANNULUS)
  int pdl;          // as RowArgs::pdl
};

constexpr int kLmax = 8192;        // twiddle master table: W_8192^m

// Elements per thread of the register-resident FFTs (cg_fft.cuh), as log2:
// the row transform of length 2^log (nx / 2) and the column transform of
// length 2^log (ny), per element type.  They depend on the grid and the type
// only (not on the batch), so a map's results do not depend on what it is
// batched with.  Fewer elements per thread shorten the chain of instructions
// that a small grid's pass consists of (one wave of CTAs); more save
// exchanges once the chip is full.  Measured with 16, 8 and 4 elements:
//   FP32, us per CG iteration: 64^2 62, 44, 38; 256^2 65, 53, 46 (16 maps 71,
//   66, 71; rows 8 and columns 4: 49 and 67); 512^2 69, 55, 56 (16 maps 128,
//   137, 186); 1024^2 76, 72, 78 (16 maps 359, 477, 424); 2048^2 149, 183, -.
//   (256^2 with rows of 8: columns of 4 or 8, one map 2.26, 2.33 ms a call, a
//   group of 24 maps 4.34, 4.06; 128 x 256^2 + 96 x 512^2 + 32 x 1024^2 in one group
//   133.8, 131.3, in mixed precision 280.3, 275.8: 8.  That group with 16 everywhere
//   117, 251, but single maps of 256^2 2.84, of 512^2 3.92 against 3.24: not taken.)
//   FP64: 64^2 264, -, 82; 512^2 586, -, 165; 1024^2 966, -, 606.  An FP64
//   instruction holds its scheduler's pipe for 64 cycles, so a short chain
//   counts most; from 2048 pixels on, 8 and 16 keep the rows of a CTA.
//   Double-float (20 relaxation sweeps): 256^2 1641, 979, 661; 512^2 1877,
//   1028, 767 (8 maps 2178, 2047, 2151); 1024^2 2127, 1352, -; 2048^2 x 8
//   37176, 29635, -; 4096^2 21013, 17847, - us.
template <typename T>
CGF_HD constexpr int row_le(int log) { return log <= 6 ? 2 : log <= 8 ? 3 : 4; }
template <typename T>
CGF_HD constexpr int col_le(int log) { return log <= 7 ? 2 : log <= 9 ? 3 : 4; }
struct df;
template <>
CGF_HD constexpr int row_le<df>(int log) { return log <= 8 ? 2 : log <= 11 ? 3 : 4; }
template <>
CGF_HD constexpr int col_le<df>(int log) { return log <= 9 ? 2 : log <= 12 ? 3 : 4; }
template <>
CGF_HD constexpr int row_le<double>(int log) { return log <= 9 ? 2 : log <= 11 ? 3 : 4; }
template <>
CGF_HD constexpr int col_le<double>(int log) { return log <= 10 ? 2 : log <= 12 ? 3 : 4; }

// Per-stage twiddle tables of the register-resident FFT (cg_fft.cuh), stored
// after the master table.  With 2^le elements per thread (le = 2, 3, 4) a
// transform of length 2^log (4 <= log <= 13) has one leading stage of radix
// 2^(log mod le) (if nonzero) and log/le stages of radix R = 2^le; the
// radix-R stage s runs on sub-transforms of size ns = 2^(log mod le) R^s and
// needs W_{R ns}^(jm r), jm < ns, r = 1..R-1 (none for the very first stage,
// ns = 1).  Its table holds them as [r - 1][jm], so that the threads of a warp
// (consecutive jm) read consecutive entries.
CGF_HD constexpr int stw_first(int le, int log) { return (log % le) ? 0 : 1; }   // first twiddled stage
CGF_HD constexpr int stw_ns(int le, int log, int s) {
  return ((log % le) ? (1 << (log % le)) : 1) << (le * s);
}
// entries of the stages before s of length 2^log
CGF_HD constexpr int stw_stage_off(int le, int log, int s) {
  int o = 0;
  for (int t = stw_first(le, log); t < s; ++t) o += ((1 << le) - 1) * stw_ns(le, log, t);
  return o;
}
CGF_HD constexpr int stw_size(int le, int log) { return stw_stage_off(le, log, log / le); }
// entries of the smaller le and, within le, of the lengths 2^4 .. 2^(log-1)
CGF_HD constexpr int stw_base(int le, int log) {
  int o = 0;
  for (int e = 2; e <= le; ++e)
    for (int l = 4; l < (e < le ? 14 : log); ++l) o += stw_size(e, l);
  return o;
}
constexpr int kStwEntries = stw_base(4, 14);   // all lengths 2^4 .. 2^13, le = 2, 3, 4
constexpr int kTwEntries = kLmax + kStwEntries;   // complex entries of a twiddle buffer

// Tables of the white-noise source (normal_pair in cg_common.cuh), doubles:
// 256 pairs (-2/c, 2 log(1/c)), c the centre of [1 + i/256, 1 + (i+1)/256), halved
// from 3/2 on, 1 for the intervals next to 1; 256 times cos, sin of 2 pi i/256 and
// their low parts; 2 k log 2, k < 54.
constexpr int kNoiseLog = 0, kNoiseArc = 512, kNoiseExp = 1536, kNoiseEntries = 1536 + 54;
constexpr int kMaxPartials = 4096; // CTAs per instance per reducing pass
constexpr int kMaxBands = 64;      // band-power gradient bins
constexpr int kDotCtas = 256;      // CTAs per instance of the band-binned product

}  // namespace cgf
