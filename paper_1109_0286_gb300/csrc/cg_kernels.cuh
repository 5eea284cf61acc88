// Fused FFT passes of the masked operator (Sect. 2.4, eq. ModEq):
//
//   C^s v = F^-1 diag(P^s) F v on the periodic grid (exact unitarity, Sect. 4)
//
// is split into a ROW pass (real row <-> half-spectrum row, R2C / C2R by a
// half-length complex FFT), a COLUMN pass (forward column FFT, multiply by the
// real table, inverse column FFT, all in registers), and the inverse ROW pass.
// The row passes write / read the half spectrum transposed (kx-major), so the
// column pass streams contiguous rows.  Everything elementwise -- the mask
// projections P_x, the white-noise draw, the CG vector updates and the inner
// products -- is fused into the row passes.
#pragma once
#include <type_traits>

#include "cg_async.cuh"
#include "cg_fft.cuh"

namespace cgf {
// Pixel pairs whose loads a source / sink issues together: with 16 elements per
// thread, a register budget of 64 (two 512-thread CTAs per SM); the smaller
// kernels have the registers for all their loads at once.
template <int E> CGF_HD constexpr int src_chunk() { return 4; }
template <int E> CGF_HD constexpr int src_chunk_wide() { return E == 16 ? 2 : 4; }
template <int E> CGF_HD constexpr int sink_chunk() { return 4; }

// Rows per partial sum of a row pass, so that the sums do not depend on the CTA
// height.  A CTA of fewer rows (two by default in FP64 on rows of 1024 pixels
// and more) sums what it holds: there the partials follow the height.
constexpr int kRedRows = 4;

template <typename T> struct KCfg;
template <> struct KCfg<float> { static constexpr int kMaxThreads = 1024; };
template <> struct KCfg<double> { static constexpr int kMaxThreads = 512; };
template <> struct KCfg<df> { static constexpr int kMaxThreads = 512; };

// Masked flags and CG-vector index of the pixel pair (pix, pix+1), pix even,
// from the pair's mask word.  The CG vectors hold two values for every pair with
// a masked pixel, zero on an observed one, so a pair is one aligned vector
// access, at the word's offset plus two values for every such pair below it in
// the word.  (32 values for every word with a masked pixel save the popcount,
// but make the vectors of scattered single pixels up to 32 times as long: 5% of
// 2048^2 x 2, FP32, plan 298 -> 166 MB, PCG 28.2 -> 25.2 ms; band-and-disc masks
// of 256^2 to 2048^2 0 to 2% faster with them, 8 x 4096^2 the same.)
struct PairIdx {
  bool m0, m1;   // pixel masked (to fill)
  int i;         // index of the pair's first value (valid where any())
  __device__ __forceinline__ bool any() const { return m0 || m1; }
};

// Bit 2k is set where pair k of a mask word has a masked pixel.
__device__ __forceinline__ uint32_t masked_pairs(uint32_t observed) {
  const uint32_t m = ~observed;
  return (m | (m >> 1)) & 0x55555555u;
}

__device__ __forceinline__ PairIdx pair_from_word(uint2 w, int pix) {
  const int b = pix & 31;
  const uint32_t t = ~w.x >> b;
  PairIdx q;
  q.m0 = t & 1u;
  q.m1 = t & 2u;
  q.i = (int)w.y + 2 * __popc(masked_pairs(w.x) & ((1u << b) - 1u));
  return q;
}

__device__ __forceinline__ PairIdx pair_index(const uint2* __restrict__ mw, int pix) {
  return pair_from_word(__ldg(mw + (pix >> 5)), pix);
}

// In-row pixel pair j (pixels 2j, 2j+1) from the row's mask words staged in
// shared memory.
__device__ __forceinline__ PairIdx pair_at(const uint2* mwr, int j) {
  return pair_from_word(mwr[j >> 4], 2 * j);
}
__device__ __forceinline__ void observed_at(const uint2* mwr, int j, bool& o0, bool& o1) {
  const uint32_t ob = mwr[j >> 4].x;
  const int b = (2 * j) & 31;
  o0 = (ob >> b) & 1u;
  o1 = (ob >> (b + 1)) & 1u;
}

// CG-vector loads / stores of a pixel pair (nothing for a pair without a
// masked pixel, whose values are zero).  stc expects zeros on observed
// pixels.
template <typename T, typename S>
__device__ __forceinline__ void ldc(const S* v, const PairIdx& q, T& a0, T& a1) {
  a0 = (T)0;
  a1 = (T)0;
  if (q.any()) {
    S s0, s1;
    ld_pair(v + q.i, s0, s1);
    a0 = (T)s0;
    a1 = (T)s1;
  }
}
template <typename T, typename S>
__device__ __forceinline__ void stc(S* v, const PairIdx& q, T a0, T a1) {
  if (q.any()) st_pair(v + q.i, (S)a0, (S)a1);
}

// The CG-vector elements of a CTA's rows form one contiguous range [c0, c1)
// (the pairs with masked pixels in row-major order): its first word's offset,
// and the last word's offset plus its values.
// One thread asks the copy engine to bring the ranges the op will read into
// L2, so that the per-pixel-pair gathers later in the pass hit L2 instead of
// waiting on HBM one chunk after another.
template <typename T>
__device__ __forceinline__ void prefetch_compact(const InstDesc<T>& I, int op, const uint2* mws,
                                                 int nwords) {
  const uint2 w0 = mws[0], w1 = mws[nwords - 1];
  const long long c0 = w0.y, c1 = (long long)w1.y + 2 * __popc(masked_pairs(w1.x));
  switch (op) {
    case OP_R_UPD:
      prefetch_l2(I.r, c0, c1);
      prefetch_l2(I.q, c0, c1);
      prefetch_l2(I.u, c0, c1);
      prefetch_l2(I.p, c0, c1);
      break;
    // (not for the p updates: measured 8% slower with it at 4096^2 x 8,
    // against 4% faster for the r update and 1% for the sinks)
    case OP_LOAD_R: prefetch_l2(I.r, c0, c1); break;
    case OP_LOAD_U: prefetch_l2(I.u, c0, c1); break;
    case OP_U64_UPD:
      prefetch_l2(I.u, c0, c1);
      prefetch_l2(I.dlt, c0, c1);
      break;
    case OP_Q: prefetch_l2(I.p, c0, c1); break;
    case OP_Z: prefetch_l2(I.r, c0, c1); break;
    case OP_RES: prefetch_l2(I.b, c0, c1); break;
    default: break;
  }
}

// ----------------------------------------------------------------- sources
// A source fills v[e] = (x[2j], x[2j+1]), j = tid + e TT, with the real row
// values fed to the forward transform.  One instantiation per op: a chunk of
// CK pixel pairs issues all its loads (indices come from shared memory, so
// they do not wait on a global load) before its arithmetic and stores.  The r
// update skips the pairs of a warp (64 pixels of a row) without a masked pixel
// by a branch that the whole warp takes: on the 4096^2 wide cut (a band and
// 2000 discs) that is 63% of them (8 maps: 497 -> 453 us with it; the p
// update, with half the work per pair, 331 -> 352, so it has none).
template <typename T, int TT, int E, int OP>
__device__ __forceinline__ void src_fill(const InstDesc<T>& I, const uint2* mwr, int rowpix,
                                         int tid, T alpha, T beta, cx<T> (&v)[E], Acc<T>& acc) {
  constexpr int CK = (OP == OP_R_UPD || OP == OP_U64_UPD) ? src_chunk_wide<E>() : src_chunk<E>();
  constexpr bool C = OP == OP_R_UPD || OP == OP_P_UPD_Z || OP == OP_P_UPD_R || OP == OP_LOAD_R ||
                     OP == OP_LOAD_U || OP == OP_U64_UPD;
  constexpr bool SKIP = OP == OP_R_UPD || OP == OP_U64_UPD;
  const unsigned warp = __activemask();
#pragma unroll
  for (int h = 0; h < E; h += CK) {
    PairIdx q[CK];
    bool on[CK];
    T x0[CK], x1[CK], y0[CK], y1[CK], z0[CK], z1[CK], w0[CK], w1[CK];
#pragma unroll
    for (int e = 0; e < CK; ++e) {
      const int j = tid + (h + e) * TT;
      on[e] = true;
      if constexpr (OP == OP_LOAD_W || OP == OP_LOAD_W_MASK || OP == OP_LOAD_Y) {
        ld_pair((OP == OP_LOAD_Y ? I.y : I.w) + rowpix + 2 * j, x0[e], x1[e]);
        if constexpr (OP == OP_LOAD_W_MASK) q[e] = pair_at(mwr, j);
      } else {
        q[e] = pair_at(mwr, j);
        if constexpr (OP == OP_LOAD_D_U || OP == OP_LOAD_D || OP == OP_LOAD_D_M)
          ld_map_pair<T>(I.d + rowpix + 2 * j, x0[e], x1[e]);
        if constexpr (SKIP) on[e] = __any_sync(warp, q[e].any());
        if (C && on[e]) {
          if constexpr (OP == OP_LOAD_R) ldc(I.r, q[e], x0[e], x1[e]);
          if constexpr (OP == OP_LOAD_U) ldc(I.u, q[e], x0[e], x1[e]);
          if constexpr (OP == OP_P_UPD_Z || OP == OP_P_UPD_R) {
            ldc(OP == OP_P_UPD_Z ? I.z : I.r, q[e], x0[e], x1[e]);
            ldc(I.p, q[e], y0[e], y1[e]);
          }
          if constexpr (OP == OP_R_UPD) {
            ldc(I.r, q[e], x0[e], x1[e]);
            ldc(I.q, q[e], y0[e], y1[e]);
            ldc(I.u, q[e], z0[e], z1[e]);
            ldc(I.p, q[e], w0[e], w1[e]);
          }
          if constexpr (OP == OP_U64_UPD) {
            ldc(I.u, q[e], x0[e], x1[e]);
            ldc(I.dlt, q[e], y0[e], y1[e]);
          }
        }
      }
    }
#pragma unroll
    for (int e = 0; e < CK; ++e) {
      T a0 = (T)0, a1 = (T)0;
      if constexpr (OP == OP_LOAD_W_MASK || OP == OP_LOAD_D_M) {
        a0 = q[e].m0 ? x0[e] : (T)0;
        a1 = q[e].m1 ? x1[e] : (T)0;
      } else if constexpr (OP == OP_LOAD_D_U) {
        a0 = q[e].m0 ? (T)0 : x0[e];
        a1 = q[e].m1 ? (T)0 : x1[e];
      } else if constexpr (!C) {
        a0 = x0[e];
        a1 = x1[e];
      } else if (on[e]) {
        if constexpr (OP == OP_P_UPD_Z || OP == OP_P_UPD_R) {
          a0 = x0[e] + beta * y0[e];
          a1 = x1[e] + beta * y1[e];
          stc(I.p, q[e], a0, a1);
        } else if constexpr (OP == OP_R_UPD) {
          a0 = x0[e] - alpha * y0[e];
          a1 = x1[e] - alpha * y1[e];
          stc(I.r, q[e], a0, a1);
          stc(I.u, q[e], z0[e] + alpha * w0[e], z1[e] + alpha * w1[e]);
          acc.add_prod(a0, a0);
          acc.add_prod(a1, a1);
        } else if constexpr (OP == OP_U64_UPD) {
          a0 = x0[e] + y0[e];
          a1 = x1[e] + y1[e];
          stc(I.u, q[e], a0, a1);
          stc(I.dlt, q[e], 0.f, 0.f);   // folded
        } else {
          a0 = x0[e];
          a1 = x1[e];
          if constexpr (OP == OP_LOAD_R) {
            acc.add_prod(a0, a0);
            acc.add_prod(a1, a1);
          }
        }
      }
      v[h + e] = cx<T>{a0, a1};
    }
  }
}

// ----------------------------------------------------------------- sinks
// A sink consumes the inverse transform's row values v[e] (pairs j = tid + e
// TT): projection, stores and the inner product of its op.
template <typename T, int TT, int E, int OP>
__device__ __forceinline__ void sink_fill(const InstDesc<T>& I, const uint2* mwr, int rowpix,
                                          int tid, const cx<T> (&v)[E], Acc<T>& acc,
                                          int param = 0) {
  constexpr int CK = sink_chunk<E>();
#pragma unroll
  for (int h = 0; h < E; h += CK) {
    PairIdx q[CK];
    T x0[CK], x1[CK];
#pragma unroll
    for (int e = 0; e < CK; ++e) {
      const int j = tid + (h + e) * TT;
      q[e] = pair_at(mwr, j);
      if constexpr (OP == OP_Q) ldc(I.p, q[e], x0[e], x1[e]);
      if constexpr (OP == OP_Z) ldc(I.r, q[e], x0[e], x1[e]);
      if constexpr (OP == OP_RES) ldc(I.b, q[e], x0[e], x1[e]);
      if constexpr (OP == OP_GRAD) ld_map_pair<T>(I.gx + rowpix + 2 * j, x0[e], x1[e]);
      if constexpr (OP == OP_RELAX) ld_pair(I.w + rowpix + 2 * j, x0[e], x1[e]);
    }
#pragma unroll
    for (int e = 0; e < CK; ++e) {
      const int j = tid + (h + e) * TT;
      const bool m0 = q[e].m0, m1 = q[e].m1;   // masked = not observed
      // CG-vector ops: nothing to store or add (exactly) for a pair without a
      // masked pixel
      constexpr bool C = OP == OP_Q || OP == OP_Z || OP == OP_B || OP == OP_RES || OP == OP_KSEL;
      if (C && !q[e].any()) continue;
      T a0 = v[h + e].r, a1 = v[h + e].i;
      if constexpr (OP == OP_Q || OP == OP_Z) {
        a0 = m0 ? a0 : (T)0;
        a1 = m1 ? a1 : (T)0;
        stc(OP == OP_Q ? I.q : I.z, q[e], a0, a1);
        acc.add_prod(x0[e], a0);
        acc.add_prod(x1[e], a1);
      } else if constexpr (OP == OP_B) {
        a0 = m0 ? -a0 : (T)0;
        a1 = m1 ? -a1 : (T)0;
        stc(I.r, q[e], a0, a1);
        if (I.b) stc(I.b, q[e], a0, a1);
        if (I.r32) stc(I.r32, q[e], a0, a1);
        acc.add_prod(a0, a0);
        acc.add_prod(a1, a1);
      } else if constexpr (OP == OP_RES) {
        a0 = x0[e] - (m0 ? a0 : (T)0);
        a1 = x1[e] - (m1 ? a1 : (T)0);
        stc(I.r, q[e], a0, a1);
        if (I.r32) stc(I.r32, q[e], a0, a1);
        acc.add_prod(a0, a0);
        acc.add_prod(a1, a1);
      } else if constexpr (OP == OP_GRAD) {
        // v = C^-1 lam.  dL/dd_U = g_U - (C^-1 lam)_U, dL/dd_M = 0;
        // dL/dy = h = g on M, (C^-1 lam)_U on U (kept in y).
        st_map_pair<T>(I.out + rowpix + 2 * j, m0 ? (T)0 : x0[e] - a0, m1 ? (T)0 : x1[e] - a1);
        st_pair(I.y + rowpix + 2 * j, m0 ? x0[e] : a0, m1 ? x1[e] : a1);
      } else if constexpr (OP == OP_RELAX) {
        const T step = cg_alpha<T>(I.st);
        a0 = m0 ? a0 : (T)0;
        a1 = m1 ? a1 : (T)0;
        st_pair(I.w + rowpix + 2 * j, x0[e] - step * a0, x1[e] - step * a1);
        acc.add_prod(a0, a0);
        acc.add_prod(a1, a1);
      } else if constexpr (OP == OP_KSEL) {
        const uchar2 c = *reinterpret_cast<const uchar2*>(I.cls + rowpix + 2 * j);
        if (m0 && c.x == param) I.y[rowpix + 2 * j] = a0;
        if (m1 && c.y == param) I.y[rowpix + 2 * j + 1] = a1;
      } else if constexpr (OP == OP_STORE_Y) {
        st_pair(I.y + rowpix + 2 * j, a0, a1);
      } else if constexpr (OP == OP_STORE_Y_MASK) {
        st_pair(I.y + rowpix + 2 * j, m0 ? a0 : (T)0, m1 ? a1 : (T)0);
      } else if constexpr (OP == OP_STORE_OUT) {
        st_map_pair<T>(I.out + rowpix + 2 * j, a0, a1);
      } else if constexpr (OP == OP_STORE_OUT_MASK) {
        st_map_pair<T>(I.out + rowpix + 2 * j, m0 ? a0 : (T)0, m1 ? a1 : (T)0);
      }
    }
  }
}

// Middle of a chain (between the inverse and the forward row transform):
// P_x (OP_MASK), or y = v and v = (d - y) on U, 0 on M (OP_Y_W).
template <typename T, int TT, int E, int OP>
__device__ __forceinline__ void mid_fill(const InstDesc<T>& I, const uint2* mwr, int rowpix,
                                         int tid, cx<T> (&v)[E]) {
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int j = tid + e * TT;
    bool o0, o1;
    observed_at(mwr, j, o0, o1);
    if constexpr (OP == OP_Y_W) {
      T d0, d1;
      ld_map_pair<T>(I.d + rowpix + 2 * j, d0, d1);
      st_pair(I.y + rowpix + 2 * j, v[e].r, v[e].i);
      v[e].r = o0 ? d0 - v[e].r : (T)0;
      v[e].i = o1 ? d1 - v[e].i : (T)0;
    } else {
      v[e].r = o0 ? (T)0 : v[e].r;
      v[e].i = o1 ? (T)0 : v[e].i;
    }
  }
}

// ----------------------------------------------------------------- row pass
// CTA = `rows` consecutive grid rows, L/E threads per row; blockIdx.y is the
// instance.  Shared memory: per-row FFT exchange areas, which also hand the
// row between its FFT threads (row, tid) and the threads (kk, rr) that load
// and store the transposed half spectrum, then the rows' mask words (nx/32 =
// L/16 per row).
//
// Half spectrum <-> half-length transform: thread (kk, rr) takes k = kk + i TT
// (i < E/2, so k < L/2) together with L - k of row rr.  Z[k] and Z[L-k], and X[k]
// and X[L-k], follow from one another, so each step is one write and one read
// of the exchange area and one complex product per pair (two rows per thread
// in 16-byte accesses measured 3% slower):
//   s = X[k] + conj X[L-k], d = e^{+2 pi i k/nx} (X[k] - conj X[L-k]):
//     Z[k] = s + i d, Z[L-k] = conj(s) + i conj(d);
//   ev = (Z[k] + conj Z[L-k]) / 2, od = e^{-2 pi i k/nx} (-i/2)(Z[k] - conj Z[L-k]):
//     X[k] = ev + od, X[L-k] = conj(ev - od);
// k = 0 pairs with the Nyquist row L (Z[L] = Z[0]); k = L/2 is its own partner.
// The passes are bound by the L1 data pipe (shared-memory and global
// wavefronts; at 4096^2 77% of its peak in the middle pass, 72% in the p
// update) and by the barriers.  Against a tile in shared memory, written once
// and read twice with a CTA barrier on either side: FP32 passes at 8 x 4096^2
// sink 377 -> 349, middle 511 -> 451, r update 454 -> 447 us; 1024^2 x 16 middle
// 52 -> 47; 512^2 FP64 164 -> 152 us per iteration.
// AUX: the source is the seed's white noise, or the sink selects the pixels of
// one kernel's class (Sect. 6.3; grid z = kernel), skipping the rows without
// one.  Both are kept out of the other kernels, whose registers and barriers
// they would burden (the row check in every sink: 349 -> 384 us at 8 x 4096^2).

// Exchange area of one row, in 8-byte words: XBuf's L + L/16 + 1 complex
// elements, padded so that the areas of a CTA's rows start 16 / rows words
// apart modulo the banks: 16 lanes of (kk, rr) -- 16 / rows consecutive k of
// every row -- then touch 16 different 8-byte banks.
template <typename T>
__host__ __device__ __forceinline__ int row_area_words(int log_l, int rows) {
  const int L = 1 << log_l, padl = L + L / 16 + 1;
  const int words = sizeof(T) == 4 ? padl : 2 * padl;
  const int want = rows < 16 ? 16 / rows : 1;
  return words + ((want - words) & 15);
}
template <typename T>
__host__ __device__ __forceinline__ size_t row_main_bytes(int log_l, int rows) {
  return (size_t(rows) * row_area_words<T>(log_l, rows) * 8 + 15) & ~size_t(15);
}

template <typename T, int LOG_L, bool IN_SPEC, bool OUT_SPEC, bool AUX = false>
__global__ void __launch_bounds__(KCfg<T>::kMaxThreads)
k_row(const InstDesc<T>* __restrict__ insts, RowArgs a, const T* __restrict__ tw) {
  constexpr int LE = row_le<T>(LOG_L), E = 1 << LE;
  constexpr int L = 1 << LOG_L, TT = L / E, NW = L / 16, PADL = L + L / 16 + 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* sm = reinterpret_cast<T*>(smem_raw);
  __shared__ double red[32];
  const InstDesc<T>& I = insts[blockIdx.y];
  CgState* const st = I.st;

  const int rows = a.rows, lr = a.log_rows;
  const int row = threadIdx.x / TT, tid = threadIdx.x - row * TT;
  const int y0 = blockIdx.x * rows, y = y0 + row;
  const int ny = a.ny;
  constexpr int W8 = 8 / sizeof(T);             // T values per 8-byte word
  const int area = row_area_words<T>(LOG_L, rows) * W8;
  const XBuf<T> xb(sm + row * area, PADL);      // this thread's row
  uint2* mws = reinterpret_cast<uint2*>(smem_raw + row_main_bytes<T>(LOG_L, rows));
  const uint2* mwr = mws + row * NW;            // this row's mask words
  constexpr int TWS = kLmax / (2 * L);          // W_{nx}^k = table[k * TWS]
  const int rowpix = y * a.nx;
  // half-spectrum side: pairs (k, L - k), k = kk + i TT, of row rr
  const int rr = threadIdx.x & (rows - 1), kk = threadIdx.x >> lr;
  const size_t tstep = 2 * (size_t)TT * ny;
  const XBar rbar = XBar::make(TT, rows, row);   // this row's barrier
  cx<T> v[E];
  Acc<T> acc;

  constexpr bool XI = AUX && !IN_SPEC, KS = AUX && IN_SPEC;
  if constexpr (!XI) {
    if (E == 16 || threadIdx.x < rows * NW)
      mws[threadIdx.x] = __ldg(I.mw + (size_t)y0 * NW + threadIdx.x);
  }
  T* const specp = KS ? I.speck + 2 * (size_t)blockIdx.z * (L + 1) * ny
                   : a.spec_sel ? I.spec2 : I.spec;
  cx<T> wk{};   // W_nx^kk
  if constexpr (IN_SPEC || OUT_SPEC) wk = twiddle<T>(tw, kk * TWS);
  pdl_wait();
  if (skip_instance(a.check_done, st)) return;

  if constexpr (KS) {
    const int param = a.param + blockIdx.z;
    __syncthreads();   // mask words
    bool any = false;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const PairIdx q = pair_at(mwr, tid + e * TT);
      if (!q.any()) continue;
      const uchar2 c = *reinterpret_cast<const uchar2*>(I.cls + rowpix + 2 * (tid + e * TT));
      any = any || (q.m0 && c.x == param) || (q.m1 && c.y == param);
    }
    if (!__syncthreads_or(any)) return;
  }

  if constexpr (IN_SPEC) {
    // rows kk and L - kk of the half spectrum, stepping up and down by TT rows
    const T* speck = specp + 2 * ((size_t)kk * ny + y0 + rr);
    const T* specm = specp + 2 * ((size_t)(L - kk) * ny + y0 + rr);
    const XBuf<T> xs(sm + rr * area, PADL);
    cx<T> xk[E / 2], xm[E / 2], xh{};
#pragma unroll
    for (int i = 0; i < E / 2; ++i) {
      xk[i] = ld_stream_cx<T>(speck + i * tstep);
      xm[i] = ld_stream_cx<T>(specm - i * tstep);
    }
    if (kk == 0) {
      xh = ld_stream_cx<T>(specp + 2 * ((size_t)(L / 2) * ny + y0 + rr));
      xk[0].i = (T)0;   // X[0] and X[L] are real
      xm[0].i = (T)0;
    }
#pragma unroll
    for (int i = 0; i < E / 2; ++i) {
      const int k = kk + i * TT;
      const cx<T> w = cmul(wk, w32<T>(i * (16 / E)));   // W_nx^k
      const cx<T> xc = conjx(xm[i]);
      const cx<T> s = xk[i] + xc, d = cmulc(xk[i] - xc, w);
      xs.st(k, cx<T>{s.r - d.i, s.i + d.r});
      xs.st(L - k, cx<T>{s.r + d.i, d.r - s.i});   // (k = 0: the unused slot L)
    }
    if (kk == 0) xs.st(L / 2, cx<T>{xh.r + xh.r, -(xh.i + xh.i)});
    __syncthreads();
    if (threadIdx.x == 0 && !OUT_SPEC && !AUX) prefetch_compact(I, a.op, mws, rows * NW);
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = xb.ld(tid + e * TT);
    fft_regs<T, LOG_L, LE, true>(v, xb, tid, tw, rbar, rbar);
    // v[e] = x[2j] + i x[2j+1], j = tid + e TT
    if constexpr (OUT_SPEC) {
      if (a.op == OP_Y_W)
        mid_fill<T, TT, E, OP_Y_W>(I, mwr, rowpix, tid, v);
      else
        mid_fill<T, TT, E, OP_MASK>(I, mwr, rowpix, tid, v);
    } else if constexpr (KS) {
      sink_fill<T, TT, E, OP_KSEL>(I, mwr, rowpix, tid, v, acc, a.param + blockIdx.z);
    } else {
      switch (a.op) {
        case OP_Q: sink_fill<T, TT, E, OP_Q>(I, mwr, rowpix, tid, v, acc); break;
        case OP_Z: sink_fill<T, TT, E, OP_Z>(I, mwr, rowpix, tid, v, acc); break;
        case OP_B: sink_fill<T, TT, E, OP_B>(I, mwr, rowpix, tid, v, acc); break;
        case OP_RES: sink_fill<T, TT, E, OP_RES>(I, mwr, rowpix, tid, v, acc); break;
        case OP_GRAD: sink_fill<T, TT, E, OP_GRAD>(I, mwr, rowpix, tid, v, acc); break;
        case OP_RELAX: sink_fill<T, TT, E, OP_RELAX>(I, mwr, rowpix, tid, v, acc); break;
        case OP_STORE_Y: sink_fill<T, TT, E, OP_STORE_Y>(I, mwr, rowpix, tid, v, acc); break;
        case OP_STORE_Y_MASK:
          sink_fill<T, TT, E, OP_STORE_Y_MASK>(I, mwr, rowpix, tid, v, acc);
          break;
        case OP_STORE_OUT: sink_fill<T, TT, E, OP_STORE_OUT>(I, mwr, rowpix, tid, v, acc); break;
        case OP_STORE_OUT_MASK:
          sink_fill<T, TT, E, OP_STORE_OUT_MASK>(I, mwr, rowpix, tid, v, acc);
          break;
        default: break;
      }
    }
  } else if constexpr (XI) {
#pragma unroll
    for (int e = 0; e < E; ++e) {
      double x0, x1;
      normal_pair(I.noise, I.seed, (uint32_t)((rowpix >> 1) + tid + e * TT), x0, x1);
      v[e] = cx<T>{(T)x0, (T)x1};
    }
  } else {
    __syncthreads();   // mask words
    if (threadIdx.x == 0) prefetch_compact(I, a.op, mws, rows * NW);
    const T alpha = a.op == OP_R_UPD ? cg_alpha<T>(st) : (T)0;
    const T beta = a.op == OP_P_UPD_Z || a.op == OP_P_UPD_R ? cg_beta<T>(st) : (T)0;
    switch (a.op) {
      case OP_R_UPD: src_fill<T, TT, E, OP_R_UPD>(I, mwr, rowpix, tid, alpha, beta, v, acc); break;
      case OP_P_UPD_Z:
        src_fill<T, TT, E, OP_P_UPD_Z>(I, mwr, rowpix, tid, alpha, beta, v, acc);
        break;
      case OP_P_UPD_R:
        src_fill<T, TT, E, OP_P_UPD_R>(I, mwr, rowpix, tid, alpha, beta, v, acc);
        break;
      case OP_LOAD_R: src_fill<T, TT, E, OP_LOAD_R>(I, mwr, rowpix, tid, alpha, beta, v, acc); break;
      case OP_LOAD_U: src_fill<T, TT, E, OP_LOAD_U>(I, mwr, rowpix, tid, alpha, beta, v, acc); break;
      case OP_LOAD_Y: src_fill<T, TT, E, OP_LOAD_Y>(I, mwr, rowpix, tid, alpha, beta, v, acc); break;
      case OP_LOAD_W: src_fill<T, TT, E, OP_LOAD_W>(I, mwr, rowpix, tid, alpha, beta, v, acc); break;
      case OP_LOAD_W_MASK:
        src_fill<T, TT, E, OP_LOAD_W_MASK>(I, mwr, rowpix, tid, alpha, beta, v, acc);
        break;
      case OP_LOAD_D_U:
        src_fill<T, TT, E, OP_LOAD_D_U>(I, mwr, rowpix, tid, alpha, beta, v, acc);
        break;
      case OP_LOAD_D: src_fill<T, TT, E, OP_LOAD_D>(I, mwr, rowpix, tid, alpha, beta, v, acc); break;
      case OP_LOAD_D_M:
        src_fill<T, TT, E, OP_LOAD_D_M>(I, mwr, rowpix, tid, alpha, beta, v, acc);
        break;
      case OP_U64_UPD:
        src_fill<T, TT, E, OP_U64_UPD>(I, mwr, rowpix, tid, alpha, beta, v, acc);
        break;
      default:
#pragma unroll
        for (int e = 0; e < E; ++e) v[e] = cx<T>{(T)0, (T)0};
        break;
    }
  }

  if constexpr (OUT_SPEC) {
    fft_regs<T, LOG_L, LE, false>(v, xb, tid, tw, rbar, rbar);
    rbar.sync();   // the row's last exchange has been read
#pragma unroll
    for (int e = 0; e < E; ++e) xb.st(tid + e * TT, v[e]);
    __syncthreads();
    pdl_trigger();
    // (the middle pass recomputes what it would otherwise keep in registers
    // through both transforms)
    unsigned t2 = threadIdx.x;
    const T* tw2 = tw;
    if constexpr (IN_SPEC) {
      asm volatile("" : "+r"(t2));
      asm volatile("" : "+l"(tw2));
    }
    const int rr2 = t2 & (rows - 1), kk2 = t2 >> lr;
    const XBuf<T> xs(sm + rr2 * area, PADL);
    if constexpr (IN_SPEC) wk = twiddle<T>(tw2, kk2 * TWS);
    T* speck = specp + 2 * ((size_t)kk2 * ny + y0 + rr2);
    T* specm = specp + 2 * ((size_t)(L - kk2) * ny + y0 + rr2);
#pragma unroll
    for (int i = 0; i < E / 2; ++i) {
      const int k = kk2 + i * TT;
      const cx<T> zk = xs.ld(k);
      const cx<T> zc = conjx(xs.ld(i == 0 && kk2 == 0 ? 0 : L - k));
      const cx<T> w = cmul(wk, w32<T>(i * (16 / E)));   // W_nx^k
      const cx<T> ev = scal(zk + zc, (T)0.5);
      const cx<T> od = cmul(scal(mul_mi<T, false>(zk - zc), (T)0.5), w);
      st_cx<T>(speck + i * tstep, ev + od);
      st_cx<T>(specm - i * tstep, conjx(ev - od));
    }
    if (kk2 == 0)
      st_cx<T>(specp + 2 * ((size_t)(L / 2) * ny + y0 + rr2), conjx(xs.ld(L / 2)));
  }

  if constexpr (!OUT_SPEC) pdl_trigger();
  if constexpr (!AUX) {
    if (a.sop != SC_NONE)
      grid_reduce(red, I.partial, st, a.sop, gridDim.x, blockIdx.x,
                  rows > kRedRows ? rows / kRedRows : 1, [&](double* out) {
                    using V = typename Acc<T>::total_t;
                    const int seg = min(rows, kRedRows) * TT;
                    if (seg > 32) __syncthreads();   // the exchange areas have been read
                    segment_partials(acc.total(), reinterpret_cast<V*>(smem_raw), out, seg);
                  });
  }
}

// ----------------------------------------------------------------- column pass
// CTA = `ffts` spectrum rows (one kx each), N/E threads per row; forward
// column FFT, multiply by the real table, inverse column FFT, in place
// (table < 0: forward transform only; PRE, Sect. 6.3: start from the forward
// transform held in spec, times kernel table (table - 2 + grid z), into speck's
// z-th spectrum).  blockIdx.x is the instance, so the
// CTAs of all instances for the same kx run together and share the table
// row through L2.
template <typename T, int LOG_N, bool PRE = false>
__global__ void __launch_bounds__(KCfg<T>::kMaxThreads)
k_col(const InstDesc<T>* __restrict__ insts, ColArgs a, const T* __restrict__ tw) {
  constexpr int LE = col_le<T>(LOG_N), E = 1 << LE;
  constexpr int N = 1 << LOG_N, TT = N / E, PADN = N + N / 16 + 1;
  constexpr bool TAB = LE < 4 || !std::is_same<T, float>::value;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* sm = reinterpret_cast<T*>(smem_raw);
  const InstDesc<T>& I = insts[blockIdx.x];
  CgState* const st = I.st;
  const int f = threadIdx.x / TT, tid = threadIdx.x - f * TT;
  const int kx = blockIdx.y * a.ffts + f;
  const bool act = kx < a.nkx;
  const XBuf<T> xb(sm + f * 2 * PADN, PADN);
  const XBar bar = XBar::make(TT, a.ffts, f);
  const int kz = PRE ? blockIdx.z : 0;
  T* col = (PRE ? I.speck + 2 * (long long)kz * a.nkx * N : a.spec_sel ? I.spec2 : I.spec) +
           2 * (long long)(act ? kx : 0) * N;
  const T* src = PRE ? I.spec + 2 * (long long)(act ? kx : 0) * N : col;
  const T* tab = nullptr;
  if (a.table >= 0)
    tab = (PRE ? I.kt + (long long)(a.table - 2 + kz) * a.nkx * N : a.table ? I.t_sqrt : I.t_inv) +
          (long long)(act ? kx : 0) * N;
  // fewer elements per thread: the table's values are fetched before the wait
  constexpr bool PT = E < 16;
  T tv[PT ? E : 1];
  if constexpr (PT) {
#pragma unroll
    for (int e = 0; e < E; ++e) tv[e] = act && tab ? ldg1(tab + tid + e * TT) : (T)0;
  }
  pdl_wait();
  if (skip_instance(a.check_done, st)) return;
  cx<T> v[E];
#pragma unroll
  for (int e = 0; e < E; ++e) v[e] = act ? ld_stream_cx<T>(src + 2 * (tid + e * TT)) : cx<T>{(T)0, (T)0};
  if constexpr (!PRE) fft_regs<T, LOG_N, LE, false, TAB>(v, xb, tid, tw, bar, bar);
  if (a.table >= 0) {
#pragma unroll
    for (int e = 0; e < E; ++e) {
      if constexpr (PT)
        v[e] = scal_rn(v[e], tv[e]);
      else
        v[e] = scal(v[e], act ? ldg1(tab + tid + e * TT) : (T)0);
    }
    // the inverse transform reloads its twiddles through an opaque copy of
    // the table pointer: sharing the forward transform's loads would keep
    // them live across the table multiply and spill registers
    const T* tw_inv;
    asm("mov.b64 %0, %1;" : "=l"(tw_inv) : "l"(tw));
    fft_regs<T, LOG_N, LE, true, TAB>(v, xb, tid, tw_inv, bar, bar);
  }
  pdl_trigger();
  if (act) {
#pragma unroll
    for (int e = 0; e < E; ++e) st_cx<T>(col + 2 * (tid + e * TT), v[e]);
  }
}

// ----------------------------------------------------------------- column pass (TMA)
// FP32 column pass of the CG loops (forward column FFT, x 1/(nP) or x sqrt(P)/n,
// inverse FFT) as a persistent kernel fed by bulk copies.  A work item is a
// block of F consecutive spectrum rows (kx .. kx+F-1) of one instance: F N
// contiguous complex values and the matching F N table values.  CTA c takes
// a contiguous run of items (kx-major, instance-minor, so an item's table
// rows were usually just read by the previous item and come from L2).  While
// item j is transformed, one thread has the copy engine bring item j+1 into
// the other of two shared-memory slots (cp.async.bulk, completion on the
// slot's mbarrier), so no thread waits on global loads.  The landing area of
// each column is then its exchange area (XBufSw, unpadded), and the results
// go to global memory straight from registers.  Items of instances that are
// done are skipped.  Every wait is bounded: on a timeout the CTA sets
// *a.err, waits (bounded) for the copies it issued, and returns.
constexpr int kColTmaSlots = 2;
// Columns per item: 256 threads' worth (F N = 256 E complex values), one
// 8192-point column above that.
CGF_HD constexpr int col_tma_ffts(int log_n) {
  const int f = (256 << col_le<float>(log_n)) >> log_n;
  return f > 0 ? f : 1;
}
CGF_HD constexpr int col_tma_threads(int log_n) {
  return (col_tma_ffts(log_n) << log_n) >> col_le<float>(log_n);
}

__host__ __device__ __forceinline__ size_t col_tma_smem(int log_n, int ffts) {
  const size_t fn = size_t(ffts) << log_n;
  return kColTmaSlots * fn * (sizeof(float2) + sizeof(float)) + 2 * kColTmaSlots * sizeof(uint64_t);
}

template <int LOG_N>
__global__ void __launch_bounds__(col_tma_threads(LOG_N), LOG_N >= 13 ? 1 : 2)
k_col_tma(const InstDesc<float>* __restrict__ insts, ColArgs a, const float* __restrict__ tw,
          int ninst) {
  constexpr int LE = col_le<float>(LOG_N), E = 1 << LE;
  constexpr int N = 1 << LOG_N, TT = N / E;
  constexpr bool TAB = LE < 4;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int F = a.ffts;
  const size_t fn = size_t(F) * N;
  float2* slot0 = reinterpret_cast<float2*>(smem_raw);
  float* tab0 = reinterpret_cast<float*>(smem_raw + kColTmaSlots * fn * sizeof(float2));
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw + kColTmaSlots * fn * (sizeof(float2) + sizeof(float)));
  const int f = threadIdx.x / TT, tid = threadIdx.x - f * TT;
  const XBar fbar = XBar::make(TT, F, f);
  const int nkb = (a.nkx + F - 1) / F;
  const long long total = (long long)nkb * ninst;
  const long long per = (total + gridDim.x - 1) / gridDim.x;
  const long long first = (long long)blockIdx.x * per;
  const long long end = first + per < total ? first + per : total;

  auto next_item = [&](long long i) {
    while (i < end && skip_instance(a.check_done, insts[i % ninst].st)) ++i;
    return i;
  };
  auto issue = [&](long long i, int sl) {   // one thread
    const InstDesc<float>& I = insts[i % ninst];
    const int kx0 = (int)(i / ninst) * F;
    const int nc = a.nkx - kx0 < F ? a.nkx - kx0 : F;
    const uint32_t bs = (uint32_t)nc * N * sizeof(float2), bt = (uint32_t)nc * N * sizeof(float);
    mbar_arrive_expect(&bar[sl], bs + bt);
    bulk_g2s(slot0 + sl * fn, I.spec + 2 * (long long)kx0 * N, bs, &bar[sl]);
    bulk_g2s(tab0 + sl * fn, (a.table ? I.t_sqrt : I.t_inv) + (long long)kx0 * N, bt, &bar[sl]);
  };

  if (threadIdx.x == 0) {
    for (int sl = 0; sl < kColTmaSlots; ++sl) mbar_init(&bar[sl], 1);
    fence_mbar_init();
  }
  __syncthreads();
  long long it = next_item(first);
  if (threadIdx.x == 0 && it < end) issue(it, 0);
  uint32_t phase = 0u;                   // bit sl: parity of slot sl's next completion
  uint32_t pending = it < end ? 1u : 0u;  // bit sl: a copy into slot sl is in flight
  int sl = 0;
  while (it < end) {
    const long long nxt = next_item(it + 1);
    if (nxt < end) {
      // the other slot's previous item is finished (CTA barrier at the end of
      // the last iteration): hand it to the copy engine
      if (threadIdx.x == 0) {
        fence_proxy_async();
        issue(nxt, sl ^ 1);
      }
      pending |= 1u << (sl ^ 1);
    }
    const bool ok = mbar_wait(&bar[sl], (phase >> sl) & 1u);
    if (__syncthreads_or(!ok)) {
      if (threadIdx.x == 0) {
        if (a.err) atomicExch(a.err, 1);
        for (int q = 0; q < kColTmaSlots; ++q)   // let the copies in flight land (bounded)
          if (((pending >> q) & 1u) && !(q == sl && ok)) mbar_wait(&bar[q], (phase >> q) & 1u);
      }
      __syncthreads();
      return;
    }
    pending &= ~(1u << sl);
    phase ^= 1u << sl;

    const InstDesc<float>& I = insts[it % ninst];
    const int kx = (int)(it / ninst) * F + f;
    const bool act = kx < a.nkx;
    float2* buf = slot0 + sl * fn + size_t(f) * N;
    const float* tb = tab0 + sl * fn + size_t(f) * N;
    cx<float> v[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const float2 t = act ? buf[tid + e * TT] : make_float2(0.f, 0.f);
      v[e] = cx<float>{t.x, t.y};
    }
    const XBufSw xb(buf);
    fft_regs<float, LOG_N, LE, false, TAB>(v, xb, tid, tw, fbar, fbar);
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const float t = act ? tb[tid + e * TT] : 0.f;
      v[e] = E < 16 ? scal_rn(v[e], t) : scal(v[e], t);
    }
    // the inverse transform reloads its twiddles (an opaque copy of the table
    // pointer): keeping the forward transform's alive across the table
    // multiply would cost some 60 registers and spills
    const float* tw_inv;
    asm("mov.b64 %0, %1;" : "=l"(tw_inv) : "l"(tw));
    fft_regs<float, LOG_N, LE, true, TAB>(v, xb, tid, tw_inv, fbar, fbar);
    if (act) {
      float* col = I.spec + 2 * (long long)kx * N;
#pragma unroll
      for (int e = 0; e < E; ++e) st_cx<float>(col + 2 * (tid + e * TT), v[e]);
    }
    __syncthreads();   // slot sl is free again
    it = nxt;
    sl ^= 1;
  }
}

// ----------------------------------------------------------------- elementwise
template <typename T>
__global__ void __launch_bounds__(256)
k_vec(const InstDesc<T>* __restrict__ insts, VecArgs a) {
  __shared__ double red[32];
  const InstDesc<T>& I = insts[blockIdx.y];
  pdl_wait();
  if (skip_instance(a.check_done, I.st)) return;
  Acc<T> acc;
  const long long gid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const long long gstride = (long long)gridDim.x * blockDim.x;
  if (a.op == VOP_UPDATE || a.op == VOP_ZERO_UP || a.op == VOP_NORM_R) {
    // the CG vectors, elementwise (zero on observed pixels)
    const T alpha = cg_alpha<T>(I.st);
    for (long long i = gid; i < I.nvec; i += gstride) {
      if (a.op == VOP_ZERO_UP) {
        I.u[i] = (T)0;
        I.p[i] = (T)0;
      } else if (a.op == VOP_NORM_R) {
        const T r = I.r[i];
        acc.add_prod(r, r);
      } else {
        const T r = I.r[i] - alpha * I.q[i];
        I.r[i] = r;
        I.u[i] = I.u[i] + alpha * I.p[i];
        acc.add_prod(r, r);
      }
    }
  } else {
    // pixel pairs of the full maps
    for (long long j = gid; j < (a.npix >> 1); j += gstride) {
      const int pix = 2 * j;
      const PairIdx q = pair_index(I.mw, pix);
      switch (a.op) {
        case VOP_ASSEMBLE: {   // observed pixels: the caller's values, bit for bit
          using M = typename MapOf<T>::type;
          M d0, d1;
          T y0, y1, u0, u1;
          ld_pair(I.d + pix, d0, d1);
          ld_pair(I.y + pix, y0, y1);
          ldc(I.u, q, u0, u1);
          st_pair(I.out + pix, q.m0 ? static_cast<M>(y0 + u0) : d0,
                  q.m1 ? static_cast<M>(y1 + u1) : d1);
          break;
        }
        case VOP_COPY_D: {
          typename MapOf<T>::type d0, d1;
          ld_pair(I.d + pix, d0, d1);
          st_pair(I.out + pix, d0, d1);
          break;
        }
        case VOP_MAKE_W: {
          T d0, d1, y0, y1, u0, u1;
          ld_map_pair<T>(I.d + pix, d0, d1);
          ld_pair(I.y + pix, y0, y1);
          ldc(I.u, q, u0, u1);
          st_pair(I.w + pix, q.m0 ? u0 : d0 - y0, q.m1 ? u1 : d1 - y1);
          break;
        }
        case VOP_ANNULUS: {   // offsets by minimum image from pixel 0
          const long long nx = a.nx, ny = a.npix / a.nx;
          T av[2];
          for (int t = 0; t < 2; ++t) {
            const long long pp = pix + t, yy = pp / nx, xx = pp % nx;
            const double dy = (double)(yy <= ny / 2 ? yy : yy - ny);
            const double dx = (double)(xx <= nx / 2 ? xx : xx - nx);
            const double r2 = dy * dy + dx * dx;
            av[t] = (r2 > a.p0 && r2 <= a.p1 && r2 > 0.0) ? (T)1 : (T)0;
          }
          st_pair(I.w + pix, av[0], av[1]);
          break;
        }
        case VOP_Y_TO_W_M: {
          T w0, w1, y0, y1;
          ld_pair(I.w + pix, w0, w1);
          ld_pair(I.y + pix, y0, y1);
          const T d0 = q.m0 ? y0 - w0 : (T)0, d1 = q.m1 ? y1 - w1 : (T)0;
          st_pair(I.w + pix, q.m0 ? y0 : w0, q.m1 ? y1 : w1);
          acc.add_prod(d0, d0);
          acc.add_prod(d1, d1);
          break;
        }
        case VOP_W_FROM_D: {
          T a0, a1;
          ld_map_pair<T>(I.d + pix, a0, a1);
          st_pair(I.w + pix, q.m0 ? (T)0 : a0, q.m1 ? (T)0 : a1);
          break;
        }
        case VOP_W_TO_OUT: {   // observed pixels: the caller's values, bit for bit
          using M = typename MapOf<T>::type;
          M d0, d1;
          T a0, a1;
          ld_pair(I.d + pix, d0, d1);
          ld_pair(I.w + pix, a0, a1);
          st_pair(I.out + pix, q.m0 ? static_cast<M>(a0) : d0, q.m1 ? static_cast<M>(a1) : d1);
          break;
        }
        case VOP_LOAD_G: {
          T g0, g1;
          ld_map_pair<T>(I.gx + pix, g0, g1);
          g0 = q.m0 ? g0 : (T)0;
          g1 = q.m1 ? g1 : (T)0;
          stc(I.r, q, g0, g1);
          stc(I.b, q, g0, g1);
          if (I.r32) stc(I.r32, q, g0, g1);
          acc.add_prod(g0, g0);
          acc.add_prod(g1, g1);
          break;
        }
        default:
          break;
      }
    }
  }
  pdl_trigger();
  if (a.sop != SC_NONE)
    grid_reduce(red, I.partial, I.st, a.sop, gridDim.x, blockIdx.x, 1, [&](double* out) {
      __shared__ typename Acc<T>::total_t buf[256];
      segment_partials(acc.total(), buf, out, blockDim.x);
    });
}

// ----------------------------------------------------------------- band products
// part[inst][cta][b] = sum over the CTA's half-plane modes k with band(k) = b
// of coef(k) Re(conj(spec(k)) spec2(k)); both spectra are full 2D transforms
// in the transposed layout, coef carries the Hermitian weight (1 on the two
// self-conjugate columns, 2 elsewhere).  The sums are reproducible bit for
// bit: each warp takes fixed runs of 32 modes, the lanes of one band are
// added in lane order by the band's lowest lane into the warp's own row of
// partial sums, and the rows are added in warp order at the end.
constexpr int kDotThreads = 256;

template <typename T>
__global__ void __launch_bounds__(kDotThreads)
k_band_dot(const InstDesc<T>* __restrict__ insts, DotArgs a) {
  constexpr int NW = kDotThreads / 32;
  __shared__ double hist[NW][kMaxBands];
  __shared__ double vals[NW][32];
  const InstDesc<T>& I = insts[blockIdx.y];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int b = lane; b < a.nbands; b += 32) hist[warp][b] = 0.0;
  __syncwarp();
  const T* coef = reinterpret_cast<const T*>(a.coef);
  const long long stride = (long long)gridDim.x * NW * 32;
  for (long long base = ((long long)blockIdx.x * NW + warp) * 32; base < a.nmodes; base += stride) {
    const long long m = base + lane;
    const bool valid = m < a.nmodes;
    double v = 0.0;
    int b = -1;
    if (valid) {
      const cx<T> x = ld_cx<T>(I.spec + 2 * m), z = ld_cx<T>(I.spec2 + 2 * m);
      v = (double)((x.r * z.r + x.i * z.i) * ldg1(coef + m));
      b = __ldg(a.band + m);
    }
    vals[warp][lane] = v;
    const unsigned g = __match_any_sync(0xffffffffu, b);
    __syncwarp();
    if (valid && lane == __ffs(g) - 1) {
      double sum = 0.0;
      for (unsigned r = g; r; r &= r - 1) sum += vals[warp][__ffs(r) - 1];
      hist[warp][b] += sum;
    }
    __syncwarp();
  }
  __syncthreads();
  double* out = a.part + ((long long)blockIdx.y * gridDim.x + blockIdx.x) * a.nbands;
  for (int b = threadIdx.x; b < a.nbands; b += blockDim.x) {
    double sum = 0.0;
    for (int w = 0; w < NW; ++w) sum += hist[w][b];
    out[b] = sum;
  }
}

}  // namespace cgf
