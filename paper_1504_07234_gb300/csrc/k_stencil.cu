// k_stencil.cu — PSF stencils of the blurring operator (Section 2), their
// residual / PCG epilogues, and the elementwise kernels of the Krylov
// preconditioner (Section 4.2).
//
// Blur A (Eq. modeld, Table 1, Eq. Arect): (A f)(i,j) = sum_{dy,dx}
// h(dy,dx) f_ext(i-dy, j-dx), f_ext being f padded by the boundary condition
// (index math only) or, for the rectangular operator, the m x m unknown whose
// field of view is offset by c = (p-1)/2.
// Adjoint: the full correlation V(a,b) = sum h(dy,dx) t0(a-c+dy, b-c+dx) on
// the (n+p-1)^2 extended domain (t zero outside), which is A^T t for the
// rectangular operator; for a boundary condition the fold of V by the
// transpose of the padding gives A^T t (done where u is consumed).
// Antireflective BCs (Section 2.2) pad by 2 F(edge) - F(mirror) instead of a
// copy, and A^T is replaced by the reblurring matrix A': the correlation of
// the antireflectively padded t on the n x n domain.
#include "mlba_internal.cuh"
#include "mlba_launch.h"

namespace mlba {

// stop rule and iteration bookkeeping after ||r^n||^2 is known
// (Eq. discrpr; Algorithm 4-NS and Eq. Alg4_rev_12)
static __device__ void finalize_residual(const Prob& pd, State& st, double sumsq) {
  const int it = st.iter;
  const double rn = sqrt(sumsq);
  st.resnorm = rn;
  if (st.nres < pd.max_iter + 2) pd.hist_res[st.nres] = rn;
  st.nres++;
  if (!isfinite(rn)) { st.status = -5; st.stopped = 1; return; }
  const bool crossed = pd.ns ? (rn <= pd.tau * pd.delta) : (it > 0 && rn <= pd.gamma * pd.delta);
  if (crossed && st.stop_iter < 0) st.stop_iter = it;
  if ((crossed && pd.stop) || it >= pd.max_iter) { st.stopped = 1; return; }
  if (pd.ns) {
    if (!crossed) {
      // q_n = max{q, 2 rho + (1 + rho)/tau_n}, tau_n = ||r^n|| / delta
      const double qn = fmax(pd.q, 2.0 * pd.rho + (1.0 + pd.rho) * pd.delta / rn);
      st.qn = qn;
      st.ns_active = 1;
      st.nconv = 0;
      st.npass = 0;
      st.nphase = 0;
      st.nb_lo = -INFINITY;
      st.nb_hi = INFINITY;
    } else {
      st.ns_active = 0;   // past the discrepancy point alpha_n is kept
      if (it < pd.max_iter + 2) pd.hist_alpha[it] = st.alpha_n;
    }
  }
  st.iter = it + 1;
}

__device__ __forceinline__ bool skip(const State& st, int pcg) {
  return st.stopped || (pcg && st.pdone);
}

// asynchronous global -> shared copy of a B-byte chunk (B = 8 or 16, both
// addresses B-aligned) of which the first nbytes come from global memory and
// the rest are zero-filled
template <int B>
__device__ __forceinline__ void cp_async_bytes(void* smem, const void* gmem, int nbytes) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  if (B == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(sa), "l"(gmem), "r"(nbytes) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(sa), "l"(gmem), "r"(nbytes) : "memory");
}

// asynchronous global -> shared copy of one 4- or 8-byte element; !valid
// writes zeros (0 source bytes)
template <int B>
__device__ __forceinline__ void cp_async_zfill(void* smem, const void* gmem, bool valid) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  const int src_bytes = valid ? B : 0;
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;\n" ::"r"(sa), "l"(gmem), "n"(B),
               "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.wait_all;\n" ::: "memory");
}

// Table 1 map for an extended index within one period of the image (the
// common case), else the general map
__device__ __forceinline__ int bc_map_near(int e, int n, int bc) {
  if (e >= 0 && e < n) return e;
  if (e >= -n && e < 2 * n) {
    if (bc == BC_ZERO) return -1;
    if (bc == BC_PERIODIC) return e < 0 ? e + n : e - n;
    return e < 0 ? -1 - e : 2 * n - 1 - e;
  }
  return bc_map(e, n, bc);
}

// Pairs of values: the paired FP32 instructions of sm_100+ do two
// multiply-adds in one (the weight is kept twice in shared memory, so a pair
// is one load); FP64 falls back to two scalar ones.
template <typename T> struct Pair;
template <> struct Pair<float> {
  using type = float2;
  using weight = float2;
  static __device__ __forceinline__ float2 w(float v) { return make_float2(v, v); }
  static __device__ __forceinline__ float2 fma(float2 a, float2 w, float2 acc) { return __ffma2_rn(a, w, acc); }
};
template <> struct Pair<double> {
  using type = double2;
  using weight = double;
  static __device__ __forceinline__ double w(double v) { return v; }
  static __device__ __forceinline__ double2 fma(double2 a, double w, double2 acc) {
    return make_double2(::fma(a.x, w, acc.x), ::fma(a.y, w, acc.y));
  }
};

// single values with the same weights (the row pass of the row-first order)
template <typename T> struct One {
  using type = T;
  using weight = typename Pair<T>::weight;
  static __device__ __forceinline__ float fma(float a, float2 w, float acc) { return fmaf(a, w.x, acc); }
  static __device__ __forceinline__ double fma(double a, double w, double acc) { return ::fma(a, w, acc); }
};

// B taps t .. t + B - 1 of a run for R outputs: acc[j] += w[t + u] v[t + u + j].
// The window is a ring: slot (ROT + j) % R holds v[t + j] on entry, slot
// (ROT + B + j) % R holds v[t + B + j] on exit, so every register index is static
// and no value moves (copying the window cost 400 of 2700 instructions per warp
// at 31 taps).  The value past the last tap's reach is not loaded.
template <typename P, int R, int B, int ROT, typename LD>
__device__ __forceinline__ void window_taps(typename P::type (&acc)[R], typename P::type (&win)[R],
                                            const typename P::weight* __restrict__ w, int t, int len,
                                            LD ld) {
#pragma unroll
  for (int u = 0; u < B; ++u) {
    const typename P::weight wt = w[t + u];
#pragma unroll
    for (int j = 0; j < R; ++j) acc[j] = P::fma(win[(ROT + u + j) % R], wt, acc[j]);
    if (u + 1 < B || t + B < len) win[(ROT + u) % R] = ld(t + u + R);
  }
}
template <typename P, int R, int ROT, typename LD>
__device__ __forceinline__ void window_tail3(typename P::type (&acc)[R], typename P::type (&win)[R],
                                             const typename P::weight* __restrict__ w, int t, int len,
                                             LD ld) {
  if (t + 2 <= len) {
    window_taps<P, R, 2, ROT>(acc, win, w, t, len, ld);
    if (t + 2 < len) window_taps<P, R, 1, ROT + 2>(acc, win, w, t + 2, len, ld);
  } else if (t < len) {
    window_taps<P, R, 1, ROT>(acc, win, w, t, len, ld);
  }
}

// acc[j] += sum_t w[t] v[t + j], j < R, over a run of len taps, v[i] = ld(i)
// (P: pairs of values, or single ones): blocks of 8 (R = 8) or 4 taps, then the
// rest by halves.
template <typename P, int R, typename LD>
__device__ __forceinline__ void window_run(typename P::type (&acc)[R],
                                           const typename P::weight* __restrict__ w, int len, LD ld) {
  constexpr int B0 = R >= 8 ? 8 : 4;       // a multiple of R: the ring is aligned after a block
  typename P::type win[R];
#pragma unroll
  for (int j = 0; j < R; ++j) win[j] = ld(j);
  int t = 0;
#pragma unroll 1
  for (; t + B0 <= len; t += B0) window_taps<P, R, B0, 0>(acc, win, w, t, len, ld);
  if constexpr (B0 == 8) {
    if (t + 4 <= len) {
      window_taps<P, R, 4, 0>(acc, win, w, t, len, ld);
      window_tail3<P, R, 4>(acc, win, w, t + 4, len, ld);
      return;
    }
  }
  window_tail3<P, R, 0>(acc, win, w, t, len, ld);
}

// Stencil tile geometry: 64 x 4 R outputs per CTA of 128 threads; a thread
// owns two neighbouring columns over R rows.  The input tile (4 R + p - 1) x
// (64 + p - 1) lives in shared memory with an even row pitch (pairs of columns
// are one 8-byte word when the column is even).  R = 8 reuses each loaded value
// most; small images take fewer rows per thread (the host's stencil_variant).
constexpr int ST_TX = 64;
// row pitch of the input tile: a multiple of 16 bytes with room for the
// shift (< 16 bytes) that aligns a row's source to 16 bytes
__host__ __device__ constexpr int st_pitch(int RX, int elem) {
  return (RX + 16 / elem - 1 + 16 / elem - 1) / (16 / elem) * (16 / elem);
}
// rank-one PSF: pitch in pairs of the column-pass result (row pairs x columns),
// odd so that the lanes of the row pass (one row pair each) hit different banks
__host__ __device__ constexpr int st_tpitch(int RX, int elem) { return (st_pitch(RX, elem) + 2) | 1; }
// rank-one PSF, row pass first: pitch of its result, and whether that needs a
// tile of its own (else the rows fit the threads' registers and overwrite the input)
constexpr int ST_RP = ST_TX + 2;
__host__ __device__ constexpr bool st_rows_tile(int RY) { return 8 * RY > 4 * STENCIL_THREADS; }
// shared memory of a tile: weights, runs (general PSF), the source rows
// and columns of the tile, input tile (which the
// column-pass result and the output tile of a rank-one PSF overwrite)
__host__ __device__ constexpr size_t st_smem(int variant, int p, int sep, int nrw, int nruns, int elem) {
  const int R = st_rows_of(variant), RY = 4 * R + p - 1, RX = ST_TX + p - 1;
  const int nw = sep ? 2 * p : nrw, we = elem == 4 ? 2 : 1;
  size_t in = (size_t)RY * st_pitch(RX, elem);
  const size_t tmp = sep ? (size_t)4 * R * st_tpitch(RX, elem) : 0;
  if (sep && (variant & ST_ROW_FIRST)) in += st_rows_tile(RY) ? (size_t)RY * ST_RP : 0;
  else if (tmp > in) in = tmp;
  return (((size_t)nw * we + 3) / 4 * 4 + in) * elem + (sep ? 0 : (size_t)nruns * 16) +
         (size_t)((2 * (RY + RX) + 3) / 4 * 4) * 4;
}

#ifndef MLBA_BODIES_ONLY
int stencil_tiles(int outN, int variant) {
  const int ty = 4 * st_rows_of(variant);
  return ((outN + ST_TX - 1) / ST_TX) * ((outN + ty - 1) / ty);
}
size_t stencil_smem(int variant, int p, int sep, int nrw, int nruns, int elem) {
  return st_smem(variant, p, sep, nrw, nruns, elem);
}
#endif

// Blur A (Eq. 2 with the Table 1 boundary conditions, or the valid part for
// rectangular A) and the full correlation that A^T is built from, as
// register-window stencils:
//  - general PSF: the taps are grouped by PSF column b into dense runs
//    [lo_b, hi_b] of rows; a thread slides an R-row window of two input
//    columns down the run, so each tap costs one (or two) shared loads, one
//    broadcast weight and R paired FMAs for 2 R outputs;
//  - rank-one PSF (h = hy hx^T): a column pass first (pairs of columns, R-row
//    windows, over the tile's 64 + p - 1 columns), kept in registers and written
//    over the input tile as pairs of rows, then the row pass on the row pairs
//    (R-column windows): both passes are paired FMAs on conflict-free loads.
//    Row pass first (ROWF; 32 + p - 1 rows for 32, single values, four-way
//    conflicting loads: 4096^2, p = 33, residual and correlation 147 + 131 us): z in
//    BF16 (the host's stencil_variant).
// Forward (A f)(y, x) = sum_{a,b} H[a][b] f_ext(y + c - a, x + c - b); the
// correlation (ne x ne) is sum_{a,b} H[a][b] t(y - 2c + a, x - 2c + b).
// (FP32: 8 CTAs per SM, 64 registers; the tile of the largest PSF of a batch
// decides how many fit in shared memory)
// One stencil item (tile) on the thread group `blk` of STENCIL_THREADS threads,
// with its shared memory at smraw, 32 doubles of reduction space and one int.
template <typename T, int MODE, int R, bool ROWF, typename BLK>
__device__ __forceinline__ void stencil_body(const int2 item, const Prob* __restrict__ probs,
                                             State* __restrict__ states, int src_slot, int dst_slot,
                                             int aux_slot, int pcg, unsigned char* smraw,
                                             double* red, int* flag, BLK blk) {
  using T2 = typename Pair<T>::type;
  using TW = typename Pair<T>::weight;
  constexpr int ST_TY = 4 * R;
  const int tid = blk.tid();
  const Prob& pd = probs[item.x];
  State& st = states[item.x];
  if (skip(st, pcg)) return;

  // CORR: correlation weights and run offsets (the full correlation and the
  // reblurring A' of antireflective BCs); ZPAD: the full correlation of the
  // zero-padded t on the (n+p-1)^2 domain
  constexpr bool CORR = (MODE == ST_CORR || MODE == ST_REBLUR);
  constexpr bool ZPAD = (MODE == ST_CORR);
  constexpr int NT = STENCIL_THREADS;
  const int n = pd.n, p = pd.p, c = pd.c;
  const int outN = ZPAD ? pd.ne : n;
  const int tilesX = (outN + ST_TX - 1) / ST_TX;
  const int ty0 = (item.y / tilesX) * ST_TY, tx0 = (item.y % tilesX) * ST_TX;
  const int RY = ST_TY + p - 1, RX = ST_TX + p - 1;
  const int RP = st_pitch(RX, (int)sizeof(T));
  const bool sep = pd.sep != 0;

  // shared memory: weights, column runs (general PSF), tables of source rows
  // and columns, input tile (and a row-pass tile: ROWF, tall tiles)
  const int nw = sep ? 2 * p : pd.nrw;
  TW* s_w = reinterpret_cast<TW*>(smraw);
  constexpr int WE = (int)(sizeof(TW) / sizeof(T));
  int4* s_runs = reinterpret_cast<int4*>(reinterpret_cast<T*>(smraw) + ((nw * WE + 3) & ~3));
  int* s_map = reinterpret_cast<int*>(s_runs + (sep ? 0 : pd.nruns));     // 2 (RY + RX) entries
  T* s_in = reinterpret_cast<T*>(s_map + ((2 * (RY + RX) + 3) & ~3));

  // src_slot < 0: the per-problem default operand (t, or r for P = I, in the
  // correlation; A^T p for the PCG product: V for rectangular A, U otherwise)
  if (src_slot < 0)
    src_slot = CORR ? (pd.precond == P_NONE ? SL_R : SL_T) : (pd.bc == BC_RECT ? SL_V : SL_U);
  if (MODE == ST_REBLUR && dst_slot < 0) dst_slot = SL_U;
  const T* src = static_cast<const T*>(pd.buf[src_slot]);
  // weights in the order the windows consume them: the forward stencil runs
  // over the reversed PSF
  if (sep) {
    const T* hy = static_cast<const T*>(pd.hy);
    const T* hx = static_cast<const T*>(pd.hx);
    for (int k = tid; k < p; k += NT) {
      s_w[k] = Pair<T>::w(CORR ? hx[k] : hx[p - 1 - k]);
      s_w[p + k] = Pair<T>::w(CORR ? hy[k] : hy[p - 1 - k]);
    }
  } else {
    // the weights are stored in both orders: one flat, coalesced copy
    const T* tw = static_cast<const T*>(pd.tap_w) + (CORR ? 0 : pd.nrw);
    for (int k = tid; k < pd.nruns; k += NT) s_runs[k] = pd.tap_runs[k];
    for (int k = tid; k < pd.nrw; k += NT) s_w[k] = Pair<T>::w(tw[k]);
  }
  // input region
  const int oy0 = ZPAD ? ty0 - 2 * c : ty0 - c;
  const int ox0 = ZPAD ? tx0 - 2 * c : tx0 - c;
  // asynchronous copies straight into shared memory (no registers held, all
  // of a thread's copies in flight together); positions outside the source
  // are zero-filled by a copy of 0 source bytes.  The source row (and, where
  // copied by elements, column) of every tile row (column) is mapped once, into a
  // table: mapping every copy was a third of the kernel's instructions.
  // When the tile's columns lie inside the source, every tile row is one
  // contiguous source run: it is copied in 16-byte (or 8-byte) chunks from a
  // chunk-aligned start, the tile sitting xs elements into its shared-memory
  // row (xs = the start's offset from the chunk boundary; the same for every
  // row when the source pitch is a multiple of the chunk), a thread keeping its
  // chunk column and stepping down the rows; bytes past the source row are
  // zero-filled.  Other tiles are walked flat, element by element.
  int xs = 0;
  {
    const int pitch = (!ZPAD && pd.bc == BC_RECT) ? pd.nf : n;
    const int sx0 = (!ZPAD && pd.bc == BC_RECT) ? ox0 + c : ox0;
    const bool colin = sx0 >= 0 && sx0 + RX <= pitch;
    // antireflective BCs: outside the image a value is a combination of up to
    // four pixels (Section 2.2), so tiles that reach outside take the
    // per-element path below
    const bool ar = !ZPAD && pd.bc == BC_AR;
    const bool ar_out = ar && !(colin && oy0 >= 0 && oy0 + RY <= n);
    // chunk in elements: 16 bytes when the pitch keeps the rows aligned alike,
    // 8 bytes (FP32) for an even pitch, 0: element by element
    const int c16 = 16 / (int)sizeof(T);
    const int ce = !colin ? 0 : (pitch % c16 == 0 ? c16 : (sizeof(T) == 4 && pitch % 2 == 0 ? 2 : 0));
    if (ar_out) {
      // 1-D antireflection of an extended index: the pixel itself, or 2 x the
      // edge minus the mirror pixel; nothing past the reach of any output of the
      // image.  Tables of (first, second or -1) pixel per tile row and column.
      auto terms = [&](int e, int* first, int* second) {
        *first = e; *second = -1;
        if (e >= 0 && e < n) return;
        const int k = e < 0 ? -e : e - (n - 1);          // distance outside the edge
        *first = k > n - 1 ? -1 : (e < 0 ? 0 : n - 1);
        *second = k > n - 1 ? -1 : (e < 0 ? k : n - 1 - k);
      };
      int *r0 = s_map, *q0 = s_map + RY, *r1 = s_map + RY + RX, *q1 = r1 + RY;
      for (int k = tid; k < RY; k += NT) terms(oy0 + k, r0 + k, r1 + k);
      for (int k = tid; k < RX; k += NT) terms(ox0 + k, q0 + k, q1 + k);
      blk.sync();
      const FastDiv frx(RX);
      for (int idx = tid; idx < RY * RX; idx += NT) {
        const int ry = frx.div(idx), rx = idx - ry * RX;
        const int i0 = r0[ry], i1 = r1[ry], j0 = q0[rx], j1 = q1[rx];
        T* d = s_in + ry * RP + rx;
        const bool ok = (i0 | j0) >= 0;
        const T* g = src + (ok ? (size_t)i0 * n + j0 : 0);
        if (i1 < 0 && j1 < 0) {
          cp_async_zfill<sizeof(T)>(d, g, ok);           // one pixel (or none)
        } else if (!ok) {
          *d = T(0);
        } else {
          // up to four pixels, loaded together
          const T wy = i1 < 0 ? T(1) : T(2), wx = j1 < 0 ? T(1) : T(2);
          const T v00 = g[0], v01 = j1 < 0 ? T(0) : src[(size_t)i0 * n + j1];
          const T v10 = i1 < 0 ? T(0) : src[(size_t)i1 * n + j0];
          const T v11 = (i1 < 0 || j1 < 0) ? T(0) : src[(size_t)i1 * n + j1];
          T v = wy * wx * v00;
          if (j1 >= 0) v -= wy * v01;
          if (i1 >= 0) v -= wx * v10;
          if (i1 >= 0 && j1 >= 0) v += v11;
          *d = v;
        }
      }
    } else {
      const bool rect = !ZPAD && pd.bc == BC_RECT;
      // source index of an extended index (-1: zero)
      auto mapped = [&](int e) -> int {
        if (ZPAD || rect) { const int q = e + (rect ? c : 0); return (q >= 0 && q < pitch) ? q : -1; }
        return bc_map_near(e, n, pd.bc);
      };
      for (int k = tid; k < RY; k += NT) s_map[k] = mapped(oy0 + k);
      if (ce == 0)
        for (int k = tid; k < RX; k += NT) s_map[RY + k] = mapped(ox0 + k);
      blk.sync();
      if (ce > 0) {
        xs = sx0 % ce;
        const int gs = sx0 - xs;
        const int nch = (xs + RX + ce - 1) / ce;       // <= 65 (8-byte chunks of <= 129 values)
        const int lw = nch <= 32 ? 5 : nch <= 64 ? 6 : 7;   // threads per row: 32, 64 or 128
        const int ch = tid & ((1 << lw) - 1), x = ch * ce;
        int nv = pitch - gs - x;
        nv = (nv < 0 ? 0 : (nv > ce ? ce : nv)) * (int)sizeof(T);
        const T* g0 = src + (nv > 0 ? gs + x : 0);
        if (ch < nch) {
          const int dr = NT >> lw;
          T* d = s_in + (tid >> lw) * RP + x;
#pragma unroll 4
          for (int ry = tid >> lw; ry < RY; ry += dr, d += dr * RP) {
            const int sy = s_map[ry];
            const T* g = g0 + (size_t)(sy < 0 ? 0 : sy) * pitch;
            const int nb = sy < 0 ? 0 : nv;
            if (ce * (int)sizeof(T) == 16) cp_async_bytes<16>(d, g, nb);
            else cp_async_bytes<8>(d, g, nb);
          }
        }
      } else {
        const FastDiv frx(RX);
        for (int idx = tid; idx < RY * RX; idx += NT) {
          const int ry = frx.div(idx), rx = idx - ry * RX;
          const int sy = s_map[ry], sx = s_map[RY + rx];
          const bool ok = (sy | sx) >= 0;
          cp_async_zfill<sizeof(T)>(s_in + ry * RP + rx, src + (ok ? (size_t)sy * pitch + sx : 0), ok);
        }
      }
    }
    cp_async_wait_all();
  }
  blk.sync();
  // this thread's outputs: columns x2, x2 + 1, rows y8 .. y8 + R - 1 of the tile
  const int x2 = 2 * (tid & 31), y8 = (tid >> 5) * R;
  T2 acc[R];
#pragma unroll
  for (int j = 0; j < R; ++j) { acc[j].x = T(0); acc[j].y = T(0); }
  if (ROWF && sep) {
    // row pass: h(y, x) = sum_t wx[t] in(y, x + t), an item being 8 columns of a
    // row; written over the input tile (row y at the start of its row) once every
    // thread holds its items, or into a tile of its own.  (Two rows at a time as
    // pairs: 4096^2, p = 33, 226 + 215 us for the residual and the correlation.)
    static_assert(!ROWF || R == 8, "row pass first: 8 rows per thread");
    constexpr int RND = 4;
    auto row = [&](int it, T (&h)[8]) {
      const T* base = s_in + (it >> 3) * RP + xs + (it & 7) * 8;
#pragma unroll
      for (int j = 0; j < 8; ++j) h[j] = T(0);
      window_run<One<T>, 8>(h, s_w, p, [&](int q) { return base[q]; });
    };
    auto put = [&](int it, const T (&h)[8], T* to, int pitch) {
      T* d = to + (it >> 3) * pitch + (it & 7) * 8;
#pragma unroll
      for (int j = 0; j < 8; ++j) d[j] = h[j];
    };
    T* hb = s_in;
    int hp = RP;
    if (!st_rows_tile(RY)) {
      T h[RND][8];
#pragma unroll
      for (int i = 0; i < RND; ++i)
        if (tid + i * NT < 8 * RY) row(tid + i * NT, h[i]);
      blk.sync();
#pragma unroll
      for (int i = 0; i < RND; ++i)
        if (tid + i * NT < 8 * RY) put(tid + i * NT, h[i], hb, hp);
    } else {
      hb = s_in + RY * RP;
      hp = ST_RP;
      for (int it = tid; it < 8 * RY; it += NT) {
        T h[8];
        row(it, h);
        put(it, h, hb, hp);
      }
    }
    blk.sync();
    // column pass: out(y, x) = sum_t wy[t] h(y + t, x)
    hb += y8 * hp + x2;
    window_run<Pair<T>, R>(acc, s_w + p, p, [&](int q) { return *reinterpret_cast<const T2*>(hb + q * hp); });
  } else if (sep) {
    // column pass: tmp(y, c) = sum_t wy[t] in(y + t, c) for the tile's columns
    // in pairs, an item being R rows of a pair.  Pairs are aligned in shared
    // memory where the tile's shifted columns fit 64 pairs (else they start at
    // the tile's first column); columns outside the tile give values nobody reads.
    constexpr int RND = 2;                       // items per thread: 4 groups x 64 pairs = 2 x 128
    const bool al = xs + RX <= 128;
    const int c0 = al ? 0 : xs;                  // shared column of pair 0
    const int np = al ? (xs + RX + 1) / 2 : (RX + 1) / 2;
    const FastDiv fnp(np);
    T2 tv[RND][R];
#pragma unroll
    for (int i = 0; i < RND; ++i) {
      const int it = tid + i * NT;
#pragma unroll
      for (int j = 0; j < R; ++j) { tv[i][j].x = T(0); tv[i][j].y = T(0); }
      if (it < 4 * np) {
        const int gr = fnp.div(it), cp = it - gr * np;
        const T* base = s_in + (gr * R) * RP + c0 + 2 * cp;
        if (al)
          window_run<Pair<T>, R>(tv[i], s_w + p, p, [&](int q) { return *reinterpret_cast<const T2*>(base + q * RP); });
        else
          window_run<Pair<T>, R>(tv[i], s_w + p, p, [&](int q) { T2 v; v.x = base[q * RP]; v.y = base[q * RP + 1]; return v; });
      }
    }
    blk.sync();
    // as row pairs over the input tile: element (y / 2, c) = (tmp(y, c), tmp(y + 1, c))
    T2* tmp = reinterpret_cast<T2*>(s_in);
    const int TP = st_tpitch(RX, (int)sizeof(T));
#pragma unroll
    for (int i = 0; i < RND; ++i) {
      const int it = tid + i * NT;
      if (it < 4 * np) {
        const int gr = fnp.div(it), cp = it - gr * np;
        T2* d = tmp + (gr * (R / 2)) * TP + 2 * cp;
#pragma unroll
        for (int j = 0; j < R; j += 2) {
          T2 lo, hi;
          lo.x = tv[i][j].x; lo.y = tv[i][j + 1].x;
          hi.x = tv[i][j].y; hi.y = tv[i][j + 1].y;
          d[(j / 2) * TP] = lo;
          d[(j / 2) * TP + 1] = hi;
        }
      }
    }
    blk.sync();
    // row pass: a thread does R columns of one row pair, out(y, x) = sum_t wx[t] tmp(y, x + t)
    constexpr int NRP = ST_TY / 2;               // row pairs of the tile; 64 / R column groups
    const int rp = tid % NRP, xg = (tid / NRP) * R;
    const T2* hb = tmp + rp * TP + (xs - c0) + xg;
    window_run<Pair<T>, R>(acc, s_w, p, [&](int q) { return hb[q]; });
    blk.sync();
    // to the epilogue's layout (two columns x R rows) through shared memory
    constexpr int OP = ST_TX + 2;
    T* ot = s_in;
#pragma unroll
    for (int j = 0; j < R; ++j) {
      ot[(2 * rp) * OP + xg + j] = acc[j].x;
      ot[(2 * rp + 1) * OP + xg + j] = acc[j].y;
    }
    blk.sync();
#pragma unroll
    for (int j = 0; j < R; ++j) acc[j] = *reinterpret_cast<const T2*>(ot + (y8 + j) * OP + x2);
  } else {
    // runs of PSF column b over rows lo..hi: input columns x + (CORR ? b : 2c - b),
    // window rows from y8 + (CORR ? lo : 2c - hi)
    for (int k = 0; k < pd.nruns; ++k) {
      const int4 rn = s_runs[k];
      const int len = rn.z - rn.y + 1;
      const int col = CORR ? x2 + rn.x : x2 + 2 * c - rn.x;
      const int r0 = CORR ? y8 + rn.y : y8 + 2 * c - rn.z;
      const T* base = s_in + r0 * RP + xs + col;
      const bool aligned = ((xs + col) & 1) == 0;
      window_run<Pair<T>, R>(acc, s_w + rn.w, len, [&](int q) -> T2 {
        const T* v = base + q * RP;
        if (aligned) return *reinterpret_cast<const T2*>(v);
        T2 o; o.x = v[0]; o.y = v[1]; return o;
      });
    }
  }
  T* dst = static_cast<T*>(pd.buf[dst_slot]);
  const T* aux = static_cast<const T*>(pd.buf[aux_slot]);
  T lacc = T(0);
  const int gx = tx0 + x2;
  auto emit = [&](size_t o, T a, T xv) {
    if (MODE == ST_FWD_RESID) {
      const T r = xv - a;
      dst[o] = r;
      lacc += r * r;
    } else if (MODE == ST_FWD_PCGQ) {
      const T pv = xv;
      const T qv = a + T(pd.alpha) * pv;
      dst[o] = qv;
      lacc += pv * qv;
    } else {
      dst[o] = a;
    }
  };
  // the second operand (g or p) for all outputs first, then the stores
  T2 av[R];
  if (MODE == ST_FWD_RESID || MODE == ST_FWD_PCGQ) {
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const int gy = ty0 + y8 + j;
      const size_t o = (size_t)gy * outN + gx;
      av[j].x = (gy < outN && gx < outN) ? aux[o] : T(0);
      av[j].y = (gy < outN && gx + 1 < outN) ? aux[o + 1] : T(0);
    }
  }
#pragma unroll
  for (int j = 0; j < R; ++j) {
    const int gy = ty0 + y8 + j;
    if (gy < outN) {
      const size_t o = (size_t)gy * outN + gx;
      if (gx < outN) emit(o, acc[j].x, av[j].x);
      if (gx + 1 < outN) emit(o + 1, acc[j].y, av[j].y);
    }
  }
  if (MODE == ST_FWD_RESID || MODE == ST_FWD_PCGQ) {
    // each thread's 2 R terms in T; from the warp sum on, FP64 (an FP32
    // partial of 16 squares is within 16 u = 1e-6 of its exact value)
    double dl = (double)lacc;
    for (int o = 16; o > 0; o >>= 1) dl += __shfl_xor_sync(0xffffffffu, dl, o);
    if ((tid & 31) == 0) red[tid >> 5] = dl;
    blk.sync();
    double vals[1] = {0.0};
    if (tid == 0)
      for (int w = 0; w < NT / 32; ++w) vals[0] += red[w];
    blk.sync();
    double tot[1];
    if (last_block_reduce_b<NT, 1>(pd, st, item.y, pd.nblk_blur, vals, tot, red, flag, blk)) {
      if (tid == 0) {
        if (MODE == ST_FWD_RESID) {
          finalize_residual(pd, st, tot[0]);
        } else {
          st.pa = (tot[0] != 0.0) ? st.prho / tot[0] : 0.0;
        }
      }
    }
  }
}

template <typename T, int MODE, int R, bool ROWF = false>
__global__ void __launch_bounds__(STENCIL_THREADS, sizeof(T) == 4 ? 8 : 4)
k_stencil(const Prob* __restrict__ probs, State* __restrict__ states, const int2* __restrict__ items,
          int src_slot, int dst_slot, int aux_slot, int pcg) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ double red[32];
  __shared__ int flag;
  stencil_body<T, MODE, R, ROWF>(items[blockIdx.x], probs, states, src_slot, dst_slot, aux_slot, pcg, smraw,
                                 red, &flag, BlkFull{});
}

template <typename T, int MODE>
__global__ void __launch_bounds__(VEC_THREADS)
k_vec(const Prob* __restrict__ probs, State* __restrict__ states, const int2* __restrict__ items,
      int pcg) {
  const int2 item = items[blockIdx.x];
  const Prob& pd = probs[item.x];
  State& st = states[item.x];
  if (st.stopped) return;
  // RHO0 starts a solve; FINISH always copies the solution out
  constexpr bool DOT = MODE == VEC_PCG_RHO0 || MODE == VEC_PCG_RHO;
  if (pcg && st.pdone && MODE != VEC_PCG_RHO0 && MODE != VEC_PCG_FINISH) return;
  const int n = pd.n;
  const size_t nn = (size_t)n * n;
  const size_t chunk = (size_t)VEC_THREADS * VEC_PER_THREAD;
  const size_t beg = (size_t)item.y * chunk;
  const size_t end = beg + chunk < nn ? beg + chunk : nn;
  // (distinct buffers: a thread's loads go out together)
  T* __restrict__ U = static_cast<T*>(pd.buf[SL_U]);
  T* __restrict__ PP = static_cast<T*>(pd.buf[SL_PP]);
  T* __restrict__ TT = static_cast<T*>(pd.buf[SL_T]);
  const T* __restrict__ V = static_cast<const T*>(pd.buf[SL_V]);
  const T* __restrict__ PX = static_cast<const T*>(pd.buf[SL_PX]);
  const T* __restrict__ PZ = static_cast<const T*>(pd.buf[SL_PZ]);
  const T* __restrict__ RES = static_cast<const T*>(pd.buf[MODE == VEC_PCG_RHO0 ? SL_R : SL_PRES]);
  T dot = T(0);
  const T beta = MODE == VEC_PCG_PUPD ? T(st.pbeta) : T(0);
  const bool any = MODE == VEC_PCG_FINISH && st.psteps > 0;
#pragma unroll
  for (int k = 0; k < VEC_PER_THREAD; ++k) {
    const size_t i = beg + threadIdx.x + (size_t)k * VEC_THREADS;
    if (i >= end) break;
    if (MODE == VEC_FOLD) {
      const int a = (int)((unsigned)i / (unsigned)n), b = (int)i - a * n;      // n^2 < 2^31
      U[i] = fold_fetch<T>(pd, V, a, b);
    } else if (MODE == VEC_PCG_PUPD) {
      PP[i] = PZ[i] + beta * PP[i];
    } else if (DOT) {
      const T z = PZ[i];
      dot += RES[i] * z;
      if (MODE == VEC_PCG_RHO0) PP[i] = z;
    } else if (MODE == VEC_PCG_FINISH) {
      TT[i] = any ? PX[i] : T(0);
    }
  }
  if (DOT) {
    __shared__ double red[32];
    double tot[1];
    const double vals[1] = {block_sum<VEC_THREADS>((double)dot, red)};
    if (last_block_reduce<VEC_THREADS, 1>(pd, st, item.y, pd.nblk_vec, vals, tot, red) && threadIdx.x == 0)
      pcg_scalars(pd, st, tot[0], MODE == VEC_PCG_RHO0);
  }
  if (MODE == VEC_PCG_FINISH && item.y == 0 && threadIdx.x == 0) {
    const int it = st.iter - 1;
    st.beta_last = st.psteps;
    if (it >= 0 && it < pd.max_iter + 2) pd.hist_beta[it] = st.psteps;
  }
}


// ---------------------------------------------------------------------------
// Blur by FFT convolution (Section 2.1 and 2.2: A and A^T applied with FFTs
// after padding).  Each problem on this path has two convolution entries in
// the problem table, forward and adjoint, of size M >= m = n + p - 1 (their
// `sidx` is the problem), whose spectra are conj(H^) and H^ (H^ = DFT of the
// PSF centred at the origin) with |lambda|^2 = 0, so that the spectral
// column pass with alpha = 1 and the Algorithm-4 weight conj(lambda)/M^2
// multiplies by H^/M^2 (convolution) or conj(H^)/M^2 (correlation).
// Circular convolution of size M >= m has no wrap-around on the samples used:
//   forward:  X = f extended by the BCs (m x m, zero beyond), Y = X (*) h,
//             (A f)(i, j) = Y(i + c, j + c);
//   adjoint:  X = t at offset (c, c), Y = X (x) h, V(a, b) = Y(a, b), a, b < m
//             (antireflective BCs: X = t extended antireflectively,
//             (A' t)(i, j) = Y(i + c, j + c)).

// 1-D antireflection of an extended index into up to two (index, weight) terms
template <typename T>
__device__ __forceinline__ int fc_ar_terms(int e, int n, int (&ix)[2], T (&wt)[2]) {
  if (e >= 0 && e < n) { ix[0] = e; wt[0] = T(1); return 1; }
  const int k = e < 0 ? -e : e - (n - 1);
  if (k > n - 1) return 0;
  ix[0] = e < 0 ? 0 : n - 1;
  ix[1] = e < 0 ? k : n - 1 - k;
  wt[0] = T(2); wt[1] = T(-1);
  return 2;
}

// X of a convolution entry (item.x) from its problem's image: src_slot < 0
// takes f (forward) or t (r for P = I) (adjoint)
template <typename T>
__global__ void __launch_bounds__(VEC_THREADS)
k_fc_pad(const Prob* __restrict__ probs, const State* __restrict__ states,
         const int2* __restrict__ items, int adj, int src_slot) {
  const int2 item = items[blockIdx.x];
  const Prob& sh = probs[item.x];
  const Prob& pd = probs[sh.sidx];
  if (states[sh.sidx].stopped) return;
  const int M = sh.n, n = pd.n, c = pd.c, m = pd.ne;
  const size_t MM = (size_t)M * M;
  if (src_slot < 0) src_slot = adj ? (pd.precond == P_NONE ? SL_R : SL_T) : SL_F;
  const T* src = static_cast<const T*>(pd.buf[src_slot]);
  T* X = static_cast<T*>(sh.buf[SL_R]);
  const bool ext = !adj || pd.bc == BC_AR;          // BC-extended input on [0, m)^2
  const size_t beg = (size_t)item.y * VEC_THREADS * VEC_PER_THREAD;
  for (size_t e = beg + threadIdx.x; e < beg + VEC_THREADS * VEC_PER_THREAD && e < MM; e += VEC_THREADS) {
    const int y = (int)(e / M), x = (int)(e - (size_t)y * M);
    T v = T(0);
    if (ext) {
      if (y < m && x < m) {
        if (pd.bc == BC_RECT) {
          v = src[(size_t)y * m + x];
        } else if (pd.bc == BC_AR) {
          int iy[2], ix[2];
          T wy[2], wx[2];
          const int ny = fc_ar_terms<T>(y - c, n, iy, wy), nx = fc_ar_terms<T>(x - c, n, ix, wx);
          for (int a = 0; a < ny; ++a)
            for (int b = 0; b < nx; ++b) v += wy[a] * wx[b] * src[(size_t)iy[a] * n + ix[b]];
        } else {
          const int sy = bc_map(y - c, n, pd.bc), sx = bc_map(x - c, n, pd.bc);
          if (sy >= 0 && sx >= 0) v = src[(size_t)sy * n + sx];
        }
      }
    } else if (y >= c && y < c + n && x >= c && x < c + n) {
      v = src[(size_t)(y - c) * n + (x - c)];
    }
    X[e] = v;
  }
}

// from the convolution entry's Y to the problem (item.x = problem):
//   FC_RESID: r = g - Y(i + c, j + c), ||r||^2 and the stop rule (as the
//             residual stencil), FC_STORE: dst = Y(i + c, j + c) (n x n),
//   FC_CORR: V = Y on [0, m)^2
enum { FC_RESID = 0, FC_STORE = 1, FC_CORR = 2 };
template <typename T, int MODE>
__global__ void __launch_bounds__(VEC_THREADS)
k_fc_out(const Prob* __restrict__ probs, State* __restrict__ states, const int2* __restrict__ items,
         int adj, int dst_slot) {
  __shared__ double red[32];
  const int2 item = items[blockIdx.x];
  const Prob& pd = probs[item.x];
  State& st = states[item.x];
  if (st.stopped) return;
  const Prob& sh = probs[pd.fc_sh[adj]];
  const int M = sh.n, n = pd.n, c = pd.c, m = pd.ne;
  const T* Y = static_cast<const T*>(sh.buf[SL_T]);
  const int w = (MODE == FC_CORR) ? m : n;
  const size_t tot = (size_t)w * w;
  const int off = (MODE == FC_CORR) ? 0 : c;
  T* dst = static_cast<T*>(pd.buf[dst_slot]);
  const T* g = static_cast<const T*>(pd.buf[SL_G]);
  const size_t beg = (size_t)item.y * VEC_THREADS * VEC_PER_THREAD;
  T lacc = T(0);
  for (size_t e = beg + threadIdx.x; e < beg + VEC_THREADS * VEC_PER_THREAD && e < tot; e += VEC_THREADS) {
    const int y = (int)(e / w), x = (int)(e - (size_t)y * w);
    const T yv = Y[(size_t)(y + off) * M + (x + off)];
    if (MODE == FC_RESID) {
      const T r = g[e] - yv;
      dst[e] = r;
      lacc += r * r;
    } else {
      dst[e] = yv;
    }
  }
  if (MODE == FC_RESID) {
    // (each thread's terms in T, FP64 from the block sum on, fixed order)
    const double bs = block_sum<VEC_THREADS>((double)lacc, red);
    const double vals[1] = {bs};
    double tot1[1];
    if (last_block_reduce<VEC_THREADS, 1>(pd, st, item.y, pd.nblk_vec, vals, tot1, red) &&
        threadIdx.x == 0)
      finalize_residual(pd, st, tot1[0]);
  }
}

// Balanced formulation: the framelet step's input becomes f + u, with u as
// the step left it: the BC fold of V (written to U), V (rectangular A, in
// place), U (A' t of antireflective BCs, in place) or t (Algorithm 4 forms,
// in place).  item.y: block of the N_f^2 plane.
template <typename T>
__device__ __forceinline__ void balance_body(const int2 item, const Prob* __restrict__ probs,
                                             const State* __restrict__ states) {
  const Prob& pd = probs[item.x];
  if (states[item.x].stopped) return;
  const int nf = pd.nf;
  const size_t tot = (size_t)nf * nf;
  const T* F = static_cast<const T*>(pd.buf[SL_F]);
  const bool fold = pd.use_adj && pd.bc != BC_RECT && pd.bc != BC_AR;
  T* dst = static_cast<T*>(pd.buf[!pd.use_adj ? SL_T : (pd.bc == BC_RECT ? SL_V : SL_U)]);
  const T* V = static_cast<const T*>(pd.buf[SL_V]);
  const size_t beg = (size_t)item.y * VEC_THREADS * VEC_PER_THREAD;
  for (size_t e = beg + threadIdx.x; e < beg + VEC_THREADS * VEC_PER_THREAD && e < tot; e += VEC_THREADS) {
    const int a = (int)(e / nf), b = (int)(e - (size_t)a * nf);
    const T u = fold ? fold_fetch<T>(pd, V, a, b) : dst[e];
    dst[e] = F[e] + u;
  }
}
template <typename T>
__global__ void __launch_bounds__(VEC_THREADS)
k_balance(const Prob* __restrict__ probs, const State* __restrict__ states,
          const int2* __restrict__ items) {
  balance_body<T>(items[blockIdx.x], probs, states);
}

#ifndef MLBA_BODIES_ONLY  // launchers: not in the persistent kernel's unit
template <typename T>
void launch_balance(const Prob* probs, State* states, const int2* items, int nitems, cudaStream_t s) {
  if (nitems > 0) k_balance<T><<<nitems, VEC_THREADS, 0, s>>>(probs, states, items);
}

template <typename T>
void launch_fc_pad(const Prob* probs, State* states, const int2* items, int nitems, int adj,
                   int src_slot, cudaStream_t s) {
  if (nitems > 0) k_fc_pad<T><<<nitems, VEC_THREADS, 0, s>>>(probs, states, items, adj, src_slot);
}
template <typename T>
void launch_fc_out(const Prob* probs, State* states, const int2* items, int nitems, int mode,
                   int adj, int dst_slot, cudaStream_t s) {
  if (nitems <= 0) return;
  if (mode == FC_RESID) k_fc_out<T, FC_RESID><<<nitems, VEC_THREADS, 0, s>>>(probs, states, items, adj, dst_slot);
  else if (mode == FC_STORE) k_fc_out<T, FC_STORE><<<nitems, VEC_THREADS, 0, s>>>(probs, states, items, adj, dst_slot);
  else k_fc_out<T, FC_CORR><<<nitems, VEC_THREADS, 0, s>>>(probs, states, items, adj, dst_slot);
}

// ---------------------------------------------------------------------------
// the stencil kernel of a mode and a variant (st_variant)
template <typename T, int R, bool ROWF = false>
auto stencil_kernel_r(int mode) {
  switch (mode) {
    case ST_FWD_RESID: return k_stencil<T, ST_FWD_RESID, R, ROWF>;
    case ST_FWD_STORE: return k_stencil<T, ST_FWD_STORE, R, ROWF>;
    case ST_FWD_PCGQ: return k_stencil<T, ST_FWD_PCGQ, R, ROWF>;
    case ST_REBLUR: return k_stencil<T, ST_REBLUR, R, ROWF>;
    default: return k_stencil<T, ST_CORR, R, ROWF>;
  }
}
template <typename T>
auto stencil_kernel(int mode, int variant) {
  if constexpr (sizeof(T) == 4)
    if (variant & ST_ROW_FIRST) return stencil_kernel_r<T, 8, true>(mode);
  const int R = st_rows_of(variant);
  return R == 2 ? stencil_kernel_r<T, 2>(mode) : R == 4 ? stencil_kernel_r<T, 4>(mode) : stencil_kernel_r<T, 8>(mode);
}

template <typename T>
void launch_stencil(int mode, const Prob* probs, State* states, const int2* items, int nitems,
                    int src, int dst, int aux, int pcg, int variant, size_t smem, cudaStream_t s) {
  if (nitems <= 0) return;
  stencil_kernel<T>(mode, variant)<<<nitems, STENCIL_THREADS, smem, s>>>(probs, states, items, src, dst, aux, pcg);
}

template <typename T>
cudaError_t stencil_set_smem(int variant) {
  for (int mode : {(int)ST_FWD_RESID, (int)ST_FWD_STORE, (int)ST_FWD_PCGQ, (int)ST_REBLUR, (int)ST_CORR}) {
    const cudaError_t e = cudaFuncSetAttribute((const void*)stencil_kernel<T>(mode, variant),
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_LIMIT);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <typename T>
void launch_vec(int mode, const Prob* probs, State* states, const int2* items, int nitems,
                int pcg, cudaStream_t s) {
  if (nitems <= 0) return;
  dim3 g(nitems), b(VEC_THREADS);
  switch (mode) {
    case VEC_FOLD: k_vec<T, VEC_FOLD><<<g, b, 0, s>>>(probs, states, items, pcg); break;
    case VEC_PCG_RHO0: k_vec<T, VEC_PCG_RHO0><<<g, b, 0, s>>>(probs, states, items, pcg); break;
    case VEC_PCG_RHO: k_vec<T, VEC_PCG_RHO><<<g, b, 0, s>>>(probs, states, items, pcg); break;
    case VEC_PCG_PUPD: k_vec<T, VEC_PCG_PUPD><<<g, b, 0, s>>>(probs, states, items, pcg); break;
    default: k_vec<T, VEC_PCG_FINISH><<<g, b, 0, s>>>(probs, states, items, pcg); break;
  }
}

template void launch_stencil<float>(int, const Prob*, State*, const int2*, int, int, int, int, int, int, size_t, cudaStream_t);
template void launch_stencil<double>(int, const Prob*, State*, const int2*, int, int, int, int, int, int, size_t, cudaStream_t);
template cudaError_t stencil_set_smem<float>(int);
template cudaError_t stencil_set_smem<double>(int);
template void launch_balance<float>(const Prob*, State*, const int2*, int, cudaStream_t);
template void launch_balance<double>(const Prob*, State*, const int2*, int, cudaStream_t);
template void launch_fc_pad<float>(const Prob*, State*, const int2*, int, int, int, cudaStream_t);
template void launch_fc_pad<double>(const Prob*, State*, const int2*, int, int, int, cudaStream_t);
template void launch_fc_out<float>(const Prob*, State*, const int2*, int, int, int, int, cudaStream_t);
template void launch_fc_out<double>(const Prob*, State*, const int2*, int, int, int, int, cudaStream_t);
template void launch_vec<float>(int, const Prob*, State*, const int2*, int, int, cudaStream_t);
template void launch_vec<double>(int, const Prob*, State*, const int2*, int, int, cudaStream_t);

#endif  // MLBA_BODIES_ONLY

}  // namespace mlba
