// Device building blocks: complex arithmetic, the Philox4x32-10 counter-based
// generator with Box-Muller normals, and reductions whose result is accurate
// to FP64 level.
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

#include "cg_types.h"

namespace cgf {

template <typename T>
struct cx {
  T r, i;
};

template <typename T>
__device__ __forceinline__ cx<T> operator+(cx<T> a, cx<T> b) { return {a.r + b.r, a.i + b.i}; }
template <typename T>
__device__ __forceinline__ cx<T> operator-(cx<T> a, cx<T> b) { return {a.r - b.r, a.i - b.i}; }
template <typename T>
__device__ __forceinline__ cx<T> cmul(cx<T> a, cx<T> b) {
  return {a.r * b.r - a.i * b.i, a.r * b.i + a.i * b.r};
}
// a * conj(b)
template <typename T>
__device__ __forceinline__ cx<T> cmulc(cx<T> a, cx<T> b) {
  return {a.r * b.r + a.i * b.i, a.i * b.r - a.r * b.i};
}
template <typename T>
__device__ __forceinline__ cx<T> conjx(cx<T> a) { return {a.r, -a.i}; }
template <typename T>
__device__ __forceinline__ cx<T> scal(cx<T> a, T s) { return {a.r * s, a.i * s}; }

// a * s rounded on its own (not contracted into the additions that follow), so
// that two kernels that spell the same steps agree bit for bit.
template <typename T>
__device__ __forceinline__ cx<T> scal_rn(cx<T> a, T s) { return {a.r * s, a.i * s}; }
template <>
__device__ __forceinline__ cx<float> scal_rn<float>(cx<float> a, float s) {
  return {__fmul_rn(a.r, s), __fmul_rn(a.i, s)};
}

// Double-float arithmetic (error-free transformations: Knuth's TwoSum for
// the high parts, FMA-exact products; Dekker's renormalisation).  Relative
// error of an operation about 2^-46 of the operands' magnitude.
__device__ __forceinline__ df operator+(df a, df b) {
  const float s = a.hi + b.hi;
  const float v = s - a.hi;
  const float e = ((a.hi - (s - v)) + (b.hi - v)) + (a.lo + b.lo);
  const float h = s + e;
  return df(h, e - (h - s));
}
__device__ __forceinline__ df operator-(df a) { return df(-a.hi, -a.lo); }
__device__ __forceinline__ df operator-(df a, df b) { return a + (-b); }
__device__ __forceinline__ df operator*(df a, df b) {
  const float p = a.hi * b.hi;
  const float e = fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, fmaf(a.hi, b.hi, -p)));
  const float h = p + e;
  return df(h, e - (h - p));
}

// Programmatic dependent launch: a pass launched with the attribute
// (RowArgs::pdl and so on) starts while the pass before it in the stream still
// runs, does what does not depend on it (descriptor, mask words, twiddles),
// and waits here for its end (all its writes visible).  Without the attribute
// both are no-ops.  The trigger, before a CTA's last stores and sums, lets the
// next pass start in turn.  (Triggered right after the wait, the CTAs of the
// next pass crowd onto the SMs that hold none of this one: 512^2 FP64 186
// against 162 us per iteration, 256^2 x 16 70 against 63.)
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// a b + c d with one renormalisation: both high products exact (FMA), their
// TwoSum, and all low-order terms in one FP32 sum (20 FP32 instructions against
// 25 for two products and an addition, and one rounding to a pair instead of
// three).
__device__ __forceinline__ df dot2(df a, df b, df c, df d) {
  const float p = a.hi * b.hi, q = c.hi * d.hi;
  const float ep = fmaf(a.hi, b.hi, -p), eq = fmaf(c.hi, d.hi, -q);
  const float s = p + q, v = s - p;
  const float e = ((p - (s - v)) + (q - v)) + (ep + eq);
  const float l = e + fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, fmaf(c.hi, d.lo, c.lo * d.hi)));
  const float h = s + l;
  return df(h, l - (h - s));
}
template <>
__device__ __forceinline__ cx<df> cmul(cx<df> a, cx<df> b) {
  return {dot2(a.r, b.r, -a.i, b.i), dot2(a.r, b.i, a.i, b.r)};
}
template <>
__device__ __forceinline__ cx<df> cmulc(cx<df> a, cx<df> b) {
  return {dot2(a.r, b.r, a.i, b.i), dot2(a.i, b.r, -a.r, b.i)};
}

// Vector types for 8- / 16-byte global accesses.
template <typename T> struct V2;
template <> struct V2<float> { using t = float2; };
template <> struct V2<double> { using t = double2; };
template <> struct V2<df> { using t = df2; };

template <typename T>
__device__ __forceinline__ cx<T> ldg_cx(const T* p) {
  typename V2<T>::t v = __ldg(reinterpret_cast<const typename V2<T>::t*>(p));
  return {v.x, v.y};
}
// Read-only scalar load.
template <typename T>
__device__ __forceinline__ T ldg1(const T* p) { return __ldg(p); }
template <>
__device__ __forceinline__ df ldg1<df>(const df* p) {
  const float2 v = __ldg(reinterpret_cast<const float2*>(p));
  return df(v.x, v.y);
}
template <>
__device__ __forceinline__ cx<df> ldg_cx<df>(const df* p) {
  const float4 v = __ldg(reinterpret_cast<const float4*>(p));
  return {df(v.x, v.y), df(v.z, v.w)};
}
template <typename T>
__device__ __forceinline__ cx<T> ld_cx(const T* p) {
  typename V2<T>::t v = *reinterpret_cast<const typename V2<T>::t*>(p);
  return {v.x, v.y};
}
template <typename T>
__device__ __forceinline__ void st_cx(T* p, cx<T> a) {
  typename V2<T>::t v;
  v.x = a.r;
  v.y = a.i;
  *reinterpret_cast<typename V2<T>::t*>(p) = v;
}
// Real pixel pairs (2j, 2j+1) as one vector access.
template <typename T>
__device__ __forceinline__ void ld_pair(const T* p, T& a, T& b) {
  typename V2<T>::t v = *reinterpret_cast<const typename V2<T>::t*>(p);
  a = v.x;
  b = v.y;
}
template <typename T>
__device__ __forceinline__ void st_pair(T* p, T a, T b) {
  typename V2<T>::t v;
  v.x = a;
  v.y = b;
  *reinterpret_cast<typename V2<T>::t*>(p) = v;
}

// Complex load of data read once by this kernel: no allocation in L1, so the
// twiddle table cached there stays resident (coherent path: the kernel may
// write the same address after reading it).
template <typename T>
__device__ __forceinline__ cx<T> ld_stream_cx(const T* p);
template <>
__device__ __forceinline__ cx<float> ld_stream_cx<float>(const float* p) {
  float x, y;
  asm volatile("ld.global.L1::no_allocate.v2.f32 {%0, %1}, [%2];" : "=f"(x), "=f"(y) : "l"(p));
  return {x, y};
}
template <>
__device__ __forceinline__ cx<double> ld_stream_cx<double>(const double* p) {
  double x, y;
  asm volatile("ld.global.L1::no_allocate.v2.f64 {%0, %1}, [%2];" : "=d"(x), "=d"(y) : "l"(p));
  return {x, y};
}
template <>
__device__ __forceinline__ cx<df> ld_stream_cx<df>(const df* p) {
  float a, b, c, d;
  asm volatile("ld.global.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(a), "=f"(b), "=f"(c), "=f"(d)
               : "l"(p));
  return {df(a, b), df(c, d)};
}

// Loads from L2 of values that other CTAs of the same kernel, or the kernel
// before, wrote (volatile: kept behind the waits and barriers they follow).
__device__ __forceinline__ double ld_l2(const double* p) {
  double v;
  asm volatile("ld.global.cg.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ unsigned long long ld_l2(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.global.cg.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

// Asks the copy engine to bring elements [c0, c1) of a vector into L2 (one
// instruction for the whole range; rounded out to 16-byte boundaries, which
// stay inside the vector's allocation since its length is padded to a
// multiple of 64 elements).
template <typename S>
__device__ __forceinline__ void prefetch_l2(const S* v, long long c0, long long c1) {
  if (!v || c1 <= c0) return;
  const uintptr_t b = reinterpret_cast<uintptr_t>(v + c0) & ~uintptr_t(15);
  const uintptr_t e = (reinterpret_cast<uintptr_t>(v + c1) + 15) & ~uintptr_t(15);
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(b), "r"((uint32_t)(e - b))
               : "memory");
}

// Pixel pairs of the caller's maps, converted to / from the pass element type.
template <typename T>
__device__ __forceinline__ void ld_map_pair(const typename MapOf<T>::type* p, T& a, T& b) {
  using M = typename MapOf<T>::type;
  typename V2<M>::t v = *reinterpret_cast<const typename V2<M>::t*>(p);
  a = (T)v.x;
  b = (T)v.y;
}
template <typename T>
__device__ __forceinline__ void st_map_pair(typename MapOf<T>::type* p, T a, T b) {
  using M = typename MapOf<T>::type;
  typename V2<M>::t v;
  v.x = static_cast<M>(a);
  v.y = static_cast<M>(b);
  *reinterpret_cast<typename V2<M>::t*>(p) = v;
}

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): 10 rounds of the
// multiply/xor bijection on a 128-bit counter under a 64-bit key.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
  const uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u;
  const uint32_t W0 = 0x9E3779B9u, W1 = 0xBB67AE85u;
#pragma unroll
  for (int rnd = 0; rnd < 10; ++rnd) {
    if (rnd > 0) {
      k.x += W0;
      k.y += W1;
    }
    uint32_t hi0 = __umulhi(M0, c.x), lo0 = M0 * c.x;
    uint32_t hi1 = __umulhi(M1, c.z), lo1 = M1 * c.z;
    c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
  }
  return c;
}

// Unit normals for pixels 2j and 2j+1 of the instance (row-major), counter
// (j, 0, 0, 0), key (seed lo, seed hi); Box-Muller in FP64 on the uniforms
// u = ((a>>6) 2^26 + (b>>6) + 1/2) 2^-52 of two pairs of words:
// sqrt(-2 log u1) (cos, sin)(2 pi u2).
//
// The FP64 pipe bounds the draws (64 cycles per warp instruction and
// scheduler), so everything that is exact runs on integers and the logarithm
// and the angle start from tables (noise_* in cg_types.h):
//   u1 = z 2^-k with z in [3/4, 3/2) from the leading bits; the interval of z
//   (of 256) gives -2/c and 2 log(1/c) for its centre c, r = 2 - 2z/c, and
//   -2 log u1 = 2k log 2 + 2 log(1/c) + sum_n r^n / (n 2^(n-1)), |r| <= 2^-7,
//   n <= 7 (c = 1 next to 1, where the logarithm vanishes);
//   2 pi u2 = 2 pi (i/256 + rho 2^-53), |rho| <= 2^44: the table's cos, sin turned
//   by the small angle's series.
// 38 FP64 instructions per pair; the library's log and sincospi with the
// conversions to double took about 100 (2048^2 x 4, double-float: draw 2040 ->
// 1421 us; 2048^2 x 2 FP32 915 -> 530 us).  Error of the noise against 64-bit
// arithmetic as before (with the transforms, 2048^2 FP64: 5.35e-16, now 5.30e-16).
__device__ __forceinline__ void normals_of(const double* __restrict__ tab, uint4 w, double& x0,
                                           double& x1) {
  // u1 = m 2^-53 (m odd), and z, k
  const unsigned long long m =
      ((((unsigned long long)(w.x >> 6) << 26) | (w.y >> 6)) << 1) | 1ull;
  const int lead = 63 - __clzll((long long)m);
  const unsigned long long mant = (m << (52 - lead)) & 0xfffffffffffffull;
  const int i1 = (int)(mant >> 44), half = i1 >> 7;
  const double z =
      __longlong_as_double((long long)(mant | ((unsigned long long)(1023 - half) << 52)));
  const double2 lt = __ldg(reinterpret_cast<const double2*>(tab + kNoiseLog) + i1);
  const double k2 = __ldg(tab + kNoiseExp + (53 - lead - half));
  const double r = fma(z, lt.x, 2.0);
  double p = fma(1.0 / 448.0, r, 1.0 / 192.0);
  p = fma(p, r, 1.0 / 80.0);
  p = fma(p, r, 1.0 / 32.0);
  p = fma(p, r, 1.0 / 12.0);
  p = fma(p, r, 0.25);
  const double rad = sqrt((k2 + lt.y) + fma(r * r, p, r));
  // u2 = n 2^-53: sector and remainder (as a double: 1.5 2^52 + rho has rho's bits
  // at the end of its mantissa)
  const unsigned long long n =
      ((((unsigned long long)(w.z >> 6) << 26) | (w.w >> 6)) << 1) | 1ull;
  const unsigned long long sec = (n + (1ull << 44)) >> 45;
  const double rho =
      __longlong_as_double((long long)(0x4338000000000000ull + (n - (sec << 45)))) -
      6755399441055744.0;
  const double th = rho * (6.283185307179586476925 / 9007199254740992.0);
  const double2* arc = reinterpret_cast<const double2*>(tab + kNoiseArc) + 2 * (sec & 255ull);
  const double2 cs = __ldg(arc), lo = __ldg(arc + 1);   // and what rounding took from them
  const double q = th * th;
  const double sn = fma(th * q, fma(fma(-1.0 / 5040.0, q, 1.0 / 120.0), q, -1.0 / 6.0), th);
  const double cm = q * fma(fma(-1.0 / 720.0, q, 1.0 / 24.0), q, -0.5);   // cos - 1
  x0 = rad * (cs.x + fma(cs.x, cm, fma(-cs.y, sn, lo.x)));
  x1 = rad * (cs.y + fma(cs.y, cm, fma(cs.x, sn, lo.y)));
}
__device__ __forceinline__ void normal_pair(const double* __restrict__ tab,
                                            unsigned long long seed, uint32_t j, double& x0,
                                            double& x1) {
  normals_of(tab,
             philox4x32_10(make_uint4(j, 0u, 0u, 0u),
                           make_uint2((uint32_t)seed, (uint32_t)(seed >> 32))),
             x0, x1);
}

// ---------------------------------------------------------------------------
// Inner-product accumulators.  FP32 data: each product is split exactly into
// hi + lo (fma), and the running sum is a compensated FP32 pair, so that a
// thread's partial carries ~44 bits; partials then combine in FP64.  This
// keeps the reductions FP64-accurate without one FP64 instruction per
// element.  FP64 data: plain FP64 accumulation.
// ---------------------------------------------------------------------------
template <typename T> struct Acc;

// A sum in three FP32 parts.  The additions are exact but for the last parts'
// (2^-24 of what the first two, 48 bits, leave): closer than FP64.
struct Sum3 {
  float h, m, l;
};
__device__ __forceinline__ float two_sum(float a, float b, float& e) {
  const float s = a + b, v = s - a;
  e = (a - (s - v)) + (b - v);
  return s;
}
__device__ __forceinline__ Sum3 operator+(Sum3 a, Sum3 b) {
  float e, f, g;
  const float h = two_sum(a.h, b.h, e);
  const float t = two_sum(a.m, b.m, f);
  const float m = two_sum(e, t, g);
  return {h, m, (a.l + b.l) + (f + g)};
}

template <>
struct Acc<float> {
  using total_t = Sum3;
  float hi = 0.f, lo = 0.f;
  __device__ __forceinline__ void add_prod(float a, float b) {
    float p = a * b;
    float e = fmaf(a, b, -p);
    float t = hi + p;
    float bp = t - hi;
    float e2 = (hi - (t - bp)) + (p - bp);
    lo += e + e2;
    hi = t;
  }
  __device__ __forceinline__ Sum3 total() const { return {hi, lo, 0.f}; }
};

template <>
struct Acc<df> {
  using total_t = Sum3;
  df s = df(0.f, 0.f);
  __device__ __forceinline__ void add_prod(df a, df b) { s = s + a * b; }
  __device__ __forceinline__ Sum3 total() const { return {s.hi, s.lo, 0.f}; }
};

template <>
struct Acc<double> {
  using total_t = double;
  double s = 0.0;
  __device__ __forceinline__ void add_prod(double a, double b) { s = fma(a, b, s); }
  __device__ __forceinline__ double total() const { return s; }
};

// Partial sums in transit between threads: FP32 and double-float passes carry
// three FP32 parts, FP64 passes doubles.
__device__ __forceinline__ Sum3 shfl_down_sum(unsigned mask, Sum3 v, int o) {
  return {__shfl_down_sync(mask, v.h, o), __shfl_down_sync(mask, v.m, o),
          __shfl_down_sync(mask, v.l, o)};
}
__device__ __forceinline__ double shfl_down_sum(unsigned mask, double v, int o) {
  return __shfl_down_sync(mask, v, o);
}
__device__ __forceinline__ double sum_value(Sum3 v) {
  return (double)v.h + ((double)v.m + (double)v.l);
}
__device__ __forceinline__ double sum_value(double v) { return v; }
// A sum whose first part is this large could overflow FP32 in the sum of a
// CTA (at most 1024 threads); such sums go through FP64.
__device__ __forceinline__ bool sum_large(Sum3 v) { return !(fabsf(v.h) < 1e34f); }
__device__ __forceinline__ bool sum_large(double) { return false; }
// Beyond FP32 altogether.
__device__ __forceinline__ bool sum_lost(Sum3 v) { return !(fabsf(v.h) < 3.4e38f); }
__device__ __forceinline__ bool sum_lost(double) { return false; }

// Sum over the segments of `len` consecutive lanes of a warp (len <= 32, any
// value; nl lanes present): the first lane of each segment gets its segment's
// sum, added pairwise in a fixed order.
template <typename V>
__device__ __forceinline__ V segment_sum(V v, unsigned mask, int lane, int nl, int len) {
  const int in = lane % len;
  for (int o = 16; o > 0; o >>= 1) {
    if (o >= len) continue;
    const V t = shfl_down_sum(mask, v, o);
    if (in + o < len && lane + o < nl) v = v + t;
  }
  return v;
}

// CG coefficient record for the Lanczos estimate (Sect. 6.4): alpha_j when
// computed (j = iterations completed so far), beta_j after iteration j.
__device__ __forceinline__ void record_alpha(const CgState& c, double alpha) {
  if (c.coef && c.iter < c.hist_cap) c.coef[2 * c.iter] = alpha;
}
__device__ __forceinline__ void set_beta(CgState* st, const CgState& c, int iter, double sum) {
  const double beta = sum / c.rho;
  st->beta = beta;
  st->beta_f = (float)beta;
  st->rho = sum;
  if (c.coef && iter >= 1 && iter - 1 < c.hist_cap) c.coef[2 * (iter - 1) + 1] = beta;
}
__device__ __forceinline__ void zero_beta(CgState* st, double rho) {
  st->rho = rho;
  st->beta = 0.0;
  st->beta_f = 0.f;
  st->first = 0;
}
__device__ __forceinline__ void stop(CgState* st, int status) {
  if (status) st->status = status;
  st->done = 1;
}
__device__ __forceinline__ void record_hist(const CgState& c, int k, double sum) {
  if (c.hist && k < c.hist_cap) c.hist[k] = sqrt(sum / c.bb);
}

// Scalar update executed once per instance by the last CTA of a pass, with
// the sum of all CTA partials (fixed order, so results are reproducible).
// c: the state as it was when the pass began, in shared memory (grid_reduce
// brings it there with one load per lane while the sums are formed; reading
// the fields one after another from L2 took about 1.5 us of each reducing
// pass); st: where the new values go.
__device__ __forceinline__ void scalar_update(int sop, CgState* st, const CgState& c, double sum) {
  switch (sop) {
    case SC_BB:
    case SC_BB_RHO:
      st->bb = sum;
      st->rr = sum;
      st->rrmax = sum;
      if (c.hist && c.hist_cap > 0) c.hist[0] = sum > 0.0 ? 1.0 : 0.0;
      if (!isfinite(sum)) {
        stop(st, 1);    // FILL_EINVAL: NaN / Inf in the data (P is validated on the host)
      } else if (sum == 0.0) {
        stop(st, 0);    // nothing to solve: u = 0
      }
      if (sop == SC_BB_RHO) zero_beta(st, sum);   // plain CG: z = r, rho = ||r||^2, p = r
      break;
    case SC_ALPHA:
      st->pq = sum;
      if (!(sum > 0.0) || !isfinite(sum)) {
        stop(st, 4);
      } else {
        const double alpha = c.rho / sum;
        st->alpha = alpha;
        st->alpha_f = (float)alpha;
        record_alpha(c, alpha);
      }
      break;
    case SC_RCHECK:
    case SC_RCHECK_BETA: {
      const int iter = c.iter + 1;
      st->rr = sum;
      st->iter = iter;
      record_hist(c, iter, sum);
      if (!isfinite(sum))
        stop(st, 4);
      else if (sum <= c.tol2 * c.bb)
        stop(st, 0);
      else if (iter >= c.max_iter)
        stop(st, 3);
      else if (sop == SC_RCHECK_BETA)
        set_beta(st, c, iter, sum);
      break;
    }
    case SC_BETA:
      if (!(sum > 0.0) || !isfinite(sum))
        stop(st, 4);
      else if (c.first)
        zero_beta(st, sum);
      else
        set_beta(st, c, c.iter, sum);
      break;
    case SC_RCHECK_UPD: {
      const int iter = c.iter + 1;
      st->rr = sum;
      st->iter = iter;
      record_hist(c, iter, sum);
      // at the end of the iterations, too: fold what was gained and report the
      // true residual (which may have converged)
      const bool fails = !isfinite(sum), end = iter >= c.max_iter;
      if (fails || end) stop(st, fails ? 4 : 3);
      if (fails || end || sum <= c.delta2 * c.rrmax || sum <= c.tol2 * c.bb) c.peer->upd = 1;
      break;
    }
    case SC_RES_UPD: {
      CgState* f = c.peer;
      st->rr = sum;
      st->upd = 0;
      st->refine = c.refine + 1;
      record_hist(c, c.refine + 1, sum);
      if (!isfinite(sum)) {
        stop(st, 4);
        f->done = 1;
      } else if (sum <= c.tol2 * c.bb) {
        stop(st, 0);
        f->done = 1;
      } else if (!f->done) {
        f->rr = sum;
        f->rrmax = sum;
        f->upd = 1;
      }
      break;
    }
    case SC_CLEAR_UPD:
      st->upd = 0;
      break;
    case SC_RES:
      st->rr = sum;
      st->refine = c.refine + 1;
      record_hist(c, c.refine + 1, sum);
      if (!isfinite(sum))
        stop(st, 4);
      else if (sum <= c.tol2 * c.bb)
        stop(st, 0);
      break;
    default:
      break;
  }
}

// Whether a pass skips this instance (SkipMode).
__device__ __forceinline__ bool skip_instance(int mode, const CgState* st) {
  if (mode == SKIP_NEVER) return false;
  const int done = *(volatile const int*)&st->done;
  if (mode == SKIP_DONE) return done != 0;
  return done != 0 || *(volatile const int*)&st->upd == 0;
}

// CG scalars in a pass's element type.  The FP32 copies are kept in the state:
// a double -> float conversion runs on the FP64 pipe, where one warp
// instruction takes 64 cycles (19 per SM with every scheduler queueing), and
// every warp of a source pass needs one before its arithmetic.
template <typename T>
__device__ __forceinline__ T cg_alpha(const CgState* st) { return (T)st->alpha; }
template <>
__device__ __forceinline__ float cg_alpha<float>(const CgState* st) { return st->alpha_f; }
template <typename T>
__device__ __forceinline__ T cg_beta(const CgState* st) { return (T)st->beta; }
template <>
__device__ __forceinline__ float cg_beta<float>(const CgState* st) { return st->beta_f; }

// Partial sums of a CTA: one of every `seg` consecutive threads' v (seg divides
// the CTA; fewer than 32 threads or whole warps).  A segment of several warps
// is added warp on warp by its first one, lane by lane, then across the lanes:
// the other warps only store their values (buf: one per thread of the CTA, free to
// write), where shuffles in every warp took five additions of each.  K: the
// segment's warps hold K shares of what B = seg / (32 K) warps would hold, share
// by share; the shares are added first.
template <typename V>
__device__ __forceinline__ void segment_partials(V v, V* buf, double* out, int seg, int K = 1) {
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (seg <= 32) {
    const int nl = min(32, (int)blockDim.x - (wid << 5));   // lanes of this warp
    const unsigned mask = nl == 32 ? 0xffffffffu : ((1u << nl) - 1u);
    const V w = segment_sum(v, mask, lane, nl, seg);
    double s = sum_value(w);
    if (__any_sync(mask, sum_large(w))) {   // out of the FP32 range: in FP64
      const double d = segment_sum(sum_value(v), mask, lane, nl, seg);
      if (sum_large(w)) s = d;
    }
    if (lane % seg == 0) out[tid / seg] = s;
    return;
  }
  const int wps = seg >> 5, sg = wid / wps;
  if (wid != sg * wps) buf[tid] = v;
  __syncthreads();
  if (wid != sg * wps) return;
  const V* b = buf + tid;
  const int B = wps / K;
  auto warp = [&](int w) {
    V x = w ? b[32 * w] : v;
    for (int k = 1; k < K; ++k) x = x + b[32 * (k * B + w)];
    return x;
  };
  V t = warp(0);
  int w = 1;
  for (; w + 4 <= B; w += 4) t = t + ((warp(w) + warp(w + 1)) + (warp(w + 2) + warp(w + 3)));
  for (; w < B; ++w) t = t + warp(w);
  t = segment_sum(t, ~0u, lane, 32, 32);
  double s = sum_value(t);
  if (__any_sync(~0u, lane == 0 && sum_large(t))) {   // out of the FP32 range: in FP64
    s = 0.0;
    for (w = 0; w < B; ++w) {
      const V x = warp(w);
      double d = sum_value(x);
      if (sum_lost(x)) {
        d = w ? sum_value(b[32 * w]) : sum_value(v);
        for (int k = 1; k < K; ++k) d += sum_value(b[32 * (k * B + w)]);
      }
      s += d;
    }
    s = segment_sum(s, ~0u, lane, 32, 32);
  }
  if (lane == 0) out[sg] = s;
}

// Reduction of a pass: every `seg` consecutive threads of a CTA give one
// partial sum, and the last CTA of the instance adds all partials and runs the
// scalar update.  Called by all threads of the CTA.  partials(out) writes the
// CTA's nseg partial sums (before the barrier that follows it).
//
// Every order is fixed and, for a given seg, independent of how many segments
// a CTA holds, so results are reproducible and the same for every CTA height of
// at least kRedRows rows (cg_kernels.cuh).
// What bounds it is the FP64 pipe (64 cycles per dependent instruction): the
// sums inside a CTA are carried in three FP32 parts (Sum3: no further from
// the exact sum than FP64 additions; in two parts, 2^-47 per addition, sums
// with cancellation came out 1.8 times as far), only a segment's total becomes
// a double, and the last CTA adds the partials in FP64 on 32 lanes in parallel.
// Measured against shuffles and sums in FP64 with one thread adding the partials
// (1024 of them at 4096^2, 32 us): 4096^2, one map, sink 104 -> 59 us, r-update
// 124 -> 76 us; an iteration of 1024^2 94.5 -> 84 us; 600 x 7000 x 4, r-update
// 106 -> 93 us.  Two parts and three with shuffles in every warp, three with the
// warps added first (segment_partials): 8 x 4096^2 FP32 679, 686 and 677 ms a call,
// 16 x 1024^2 28.2, 28.8 and 28.7, one map 6.0, 6.1 and 6.1.
template <typename F>
__device__ __forceinline__ void grid_reduce(double* sh, double* partial, CgState* st, int sop,
                                            int ncta, int cta, int nseg, F partials) {
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int nthr = blockDim.x;
  const int nl = min(32, nthr - (wid << 5));   // lanes of this warp
  const unsigned mask = nl == 32 ? 0xffffffffu : ((1u << nl) - 1u);
  __shared__ bool last;
  __shared__ alignas(8) unsigned char shst[sizeof(CgState)];   // for scalar_update
  static_assert(sizeof(CgState) % 8 == 0, "copied in 8-byte words");
  if (wid == 0) {
    const unsigned long long* src = reinterpret_cast<const unsigned long long*>(st);
    for (int i = lane; i < (int)(sizeof(CgState) / 8); i += nl)
      reinterpret_cast<unsigned long long*>(shst)[i] = ld_l2(src + i);
  }
  partials(partial + (long long)cta * nseg);
  __syncthreads();
  if (tid == 0) {
    // releases the CTA's partials (ordered before it by the barrier); the last
    // CTA alone acquires the others'.  (Full fences around a relaxed atomic:
    // 64^2 32.1 instead of 31.1 us per iteration, 1024^2 x 16 sink 41.4 / 40.7 us;
    // letting the other warps exit before the atomic, or not inlining this
    // function, was slower on large grids: r update at 4096^2 67.5 -> 71 us.)
    unsigned int t;
    asm volatile("atom.global.add.release.gpu.u32 %0, [%1], 1;"
                 : "=r"(t)
                 : "l"(&st->ticket)
                 : "memory");
    last = (t == (unsigned int)(ncta - 1));
  }
  __syncthreads();
  if (!last || wid > 0) return;
  asm volatile("fence.acq_rel.gpu;" ::: "memory");
  __syncwarp(mask);
  // 32 fixed lanes (a CTA may have fewer threads), then their pairwise sum
  const int np = ncta * nseg, nt = min(nthr, 32);
  if (nt == 32) {
    double a = 0.0;
#pragma unroll 8
    for (int c = lane; c < np; c += 32) a += ld_l2(partial + c);
    a = segment_sum(a, mask, lane, 32, 32);
    if (lane == 0) sh[0] = a;
  } else {
    for (int l = lane; l < 32; l += nt) {
      double a = 0.0;
      for (int c = l; c < np; c += 32) a += ld_l2(partial + c);
      sh[l] = a;
    }
    __syncwarp(mask);
    for (int o = 16; o > 0; o >>= 1) {
      for (int l = lane; l < o; l += nt) sh[l] += sh[l + o];
      __syncwarp(mask);
    }
  }
  if (tid == 0) {
    st->ticket = 0u;
    scalar_update(sop, st, *reinterpret_cast<const CgState*>(shst), sh[0]);
  }
}

}  // namespace cgf
