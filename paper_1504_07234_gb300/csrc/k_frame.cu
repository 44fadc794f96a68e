// k_frame.cu — fused undecimated B-spline framelet step of Eq. MLBA2:
//
//     z_out = z_in + W u,   x = S_mu(z_out),   f = W^T x
//
// W is the L-level undecimated transform of Section 6.1 (masks b0, b1, b2,
// dilated by 2^(l-1) at level l, half-sample reflective boundary).  All
// values are computed on the reflectively extended domain around a tile: z
// outside the image is its mirror image with the sign of the band's symmetry
// (b1 is antisymmetric).  The extension of W u under the same mirroring
// equals W of the extended u, and S_mu is odd, so every value on a halo is
// exact and W^T reduces to plain (dilated) convolutions there.  z is read from
// one ping-pong buffer and written to the other (no in-place race between
// neighbouring tiles), once per owned coefficient.
//
// Two kernel families: for L <= 2 one fused row sweep per tile (k_frame3);
// for L >= 3 a low-pass chain and one row-sweep kernel per level, which works
// in the polyphase order of its dilation so that its halo is one position
// (k_lowpass, k_frame_lev).
//
// u comes from (per problem): the full correlation V folded by the BC
// transpose (A^T t for imposed boundary conditions), V itself (rectangular
// A), or t (Algorithm 4 forms, where C^T is already applied).
#include <algorithm>
#include <type_traits>
#include "mlba_internal.cuh"
#include "mlba_launch.h"

namespace mlba {

// ---------------------------------------------------------------------------
// asynchronous global -> shared copies (one thread, 4 or 8 bytes) and their groups
__device__ __forceinline__ void cp_async_4(void* smem, const void* gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_8(void* smem, const void* gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }
__device__ __forceinline__ void cp_async_16(void* smem, const void* gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}

// ---------------------------------------------------------------------------
// Bulk asynchronous copies (cp.async.bulk, completion counted in bytes on an
// mbarrier) for the z rows of the ring variant of the framelet sweep.  Every
// wait on an mbarrier is bounded: after about one second (global timer) or
// Z_SPIN_LIMIT polls it gives up and the caller reports MLBA_E_TIMEOUT
// instead of hanging.
constexpr unsigned Z_SPIN_LIMIT = 1u << 26;
constexpr unsigned long long Z_WAIT_NS = 1000000000ull;
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ unsigned smem_u32(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(unsigned long long* b, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_init_fence() {
  asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long* b, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(b)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, unsigned bytes,
                                         unsigned long long* b) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(b))
      : "memory");
}
__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
}
// true once the phase with the given parity has completed; false after the
// spin limit
__device__ __forceinline__ bool mbar_wait(unsigned long long* b, unsigned parity) {
  const unsigned a = smem_u32(b);
  unsigned long long t0 = 0;
  for (unsigned it = 0; it < Z_SPIN_LIMIT; ++it) {
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(a), "r"(parity)
        : "memory");
    if (ok) return true;
    if (it == 0) t0 = global_ns();
    else if ((it & 255) == 0 && global_ns() - t0 > Z_WAIT_NS) return false;
  }
  return false;
}

// ---------------------------------------------------------------------------
// Warp row-sweep variant for L <= 2 (the measured workloads).
//
// A CTA owns an F3_TX x (SEG F3_NWR) tile of f and of every z band; warp w
// owns the SEG-row segment w of it (32 rows; fewer in launches with few warps,
// whose time is one warp's chain of rows: the host's frame_segment has the
// rule and its measurements).  In each level a lane owns one column of
// the band region (coefficients at columns tx0 - X .. tx0 - X + 31) and the
// warp sweeps down the rows:
//   analysis   h_j(y, x) = sum_t b_j[t] c(y, x + (t-1)D)     (shared memory)
//              a_ij(y, x) = sum_s b_i[s] h_j(y + (s-1)D, x)  (register ring)
//   update     z' = z + a, x_ij = S_mu(z')                   (z in registers,
//              loaded PF rows ahead straight from global memory)
//   synthesis  P_j(y + (s-1)D) += b_i[s] x_ij                (register ring)
//              out(y, x) = A(x + D) + B(x) + C(x - D)         (warp shuffles)
//              with A, B, C = sum_j b_j[0], b_j[1], b_j[2] P_j
// Every lane computes a coefficient column, but only lanes whose +-D
// neighbours are in the warp produce output: level 2 (D = 2) lanes 2..29,
// level 1 lanes 1..26.  Neighbouring warps and tiles recompute the
// overlapping coefficients (from the same z_in) and only the owner writes
// z_out.  Shared memory carries only the input u (c_1 = (b0 x b0) u is formed
// on the fly by the level-2 sweep) and the level-2 part of f, so there are no
// shared-memory atomics; the only CTA-wide barrier follows the u tile.
constexpr int F3_TX = 26;      // tile columns: level-2 output lanes 3..28 after the +-1 low-pass
// rows past the register queue whose z lines are prefetched into L2: the
// queue holds PF rows in registers, the prefetch reaches further without
// holding any (measured on the 64-problem batch and on L = 4: 0.61 -> 0.51 ms
// per framelet launch; distances 1..10 tried)
constexpr int Z_L2_AHEAD = 2;   // k_frame3
constexpr int LV_L2_AHEAD = 1;  // k_frame_lev
// k_frame_lev: rows of the register queue and resident CTAs per SM (FP32) by
// segment height.  Long segments run with the SM full of warps, where a row
// takes longer than an L2 access: one queued row and 64 registers (4096^2,
// L = 4, a step: 2.04 ms with 3 rows at 96 registers, 1.98 with 3 rows in 80,
// 1.97 with 1 row in 64).  Short ones run in idle SMs: 3 rows (226^2: 2 %
// faster per step than 1).
__host__ __device__ constexpr int lv_pf(int seg) { return seg >= 16 ? 1 : 3; }
__host__ __device__ constexpr int lv_minb(int seg, int elem_bytes) { return seg >= 16 && elem_bytes == 4 ? 32 : 1; }
constexpr int F3_SEG = 32;     // rows per warp of the tile shapes below
constexpr int F3_SEG_NWR = 2;   // warps per CTA of the sweeps with shorter segments (16, 8, 4 rows)
// Tile shapes the autotuner chooses from: warps (32-row segments) per CTA and
// the z prefetch distance in rows.  Every shape computes the same values in
// the same order (a warp's sweep does not depend on its CTA), so the choice
// changes the time only.  Shape 0 is the default; FP64 always uses it.  Its
// queue of one row (the L2 prefetch hides the rest) lets the sweep keep its
// rings in place (f3_level): a launch of 4096^2, L = 2 went from 419 to 411 us
// together with the sum / difference form of the masks (f3_row).
// Shapes with ring > 0 stream each warp's z rows through a ring of `ring`
// row slots in shared memory, filled by bulk asynchronous copies (one 1 KB
// copy per row for FP32 z, 512 B for BF16) so that many rows are in flight
// without holding registers; warps whose 32 columns cross the left or right
// image edge (mirrored columns) fill the same ring with per-lane 16-byte
// asynchronous copies.
struct F3Shape { int nwr, pf, ring; };
constexpr F3Shape F3_SHAPES[FRAME_SHAPES] = {{2, 1, 0}, {1, 2, 0}, {4, 2, 0}, {2, 3, 0}, {1, 3, 0},
                                             {2, 2, 6}, {2, 2, 10}, {1, 2, 12}};

template <int L, int NWR, int SEG = F3_SEG>
struct F3 {
  static constexpr int TY = SEG * NWR;
  static constexpr int C0 = (L == 2) ? 6 : 2;         // radius of the u tile
  static constexpr int UW = F3_TX + 2 * C0, UH = TY + 2 * C0;
  static constexpr size_t elems = (size_t)UW * UH + (L == 2 ? (size_t)F3_TX * TY : 0);
};
// bytes of one ring slot: 32 pixels' groups of 8 z values
template <typename TZ>
__host__ __device__ constexpr size_t f3_slot_bytes() { return 32 * 8 * sizeof(TZ); }
// shared memory: u tile and level-2 part of f (T), then per warp `ring` slots
// and `ring` mbarriers
template <typename T, typename TZ, int L, int NWR, int RING, int SEG = F3_SEG>
__host__ __device__ constexpr size_t frame3_ring_offset() {
  return (F3<L, NWR, SEG>::elems * sizeof(T) + 15) / 16 * 16;
}
template <typename T, typename TZ, int L, int NWR, int RING, int SEG = F3_SEG>
__host__ __device__ constexpr size_t frame3_smem_bytes() {
  return frame3_ring_offset<T, TZ, L, NWR, RING, SEG>() + (size_t)NWR * RING * (f3_slot_bytes<TZ>() + 8);
}

// half-sample reflection of an index with the parity of the mirroring; the
// common cases (inside, or one mirror away) avoid the division
__device__ __forceinline__ int f3_refl(int e, int n, bool* par) {
  if (e >= 0 && e < n) { *par = false; return e; }
  if (e < 0 && e >= -n) { *par = true; return -1 - e; }
  if (e >= n && e < 2 * n) { *par = true; return 2 * n - 1 - e; }
  int o;
  const int r = refl_half(e, n, &o);
  *par = o != 0;
  return r;
}

// Grouped z layout (L <= 2): the 8 high-pass bands of level l of pixel q are
// contiguous, at (l - 1) 8 nf^2 + 8 q + (3 i + j - 1); the final low-pass band
// keeps its plane at 8 L nf^2 + q.  A lane then moves one pixel's bands of a
// level with one to four 16-byte accesses and one address.
template <typename TZ>
union ZGroup {
  uint4 v[8 * sizeof(TZ) / 16];
  TZ e[8];
};
__device__ __forceinline__ float to_z(float v, float*) { return v; }
__device__ __forceinline__ double to_z(double v, double*) { return v; }
__device__ __forceinline__ __nv_bfloat16 to_z(float v, __nv_bfloat16*) { return __float2bfloat16_rn(v); }

// S_mu(v) = v - clamp(v, -mu, mu).  FP64: the comparison on the bits of |v|
// (for mu >= 0 the same values, NaN and infinities included), because a
// comparison in FP64 costs as much as an addition there and the FP64 pipe is
// what bounds the sweep.
__device__ __forceinline__ float f3_soft(float v, float mu) { return v - fminf(fmaxf(v, -mu), mu); }
__device__ __forceinline__ double f3_soft(double v, double mu) {
  const long long m = __double_as_longlong(v) & 0x7fffffffffffffffll;
  const double c = m > __double_as_longlong(mu) ? copysign(mu, v) : v;
  return v - c;
}
// v with its sign flipped when the (sign-bit) mask is set
__device__ __forceinline__ float f3_flip(float v, int m) { return __int_as_float(__float_as_int(v) ^ m); }
__device__ __forceinline__ double f3_flip(double v, int m) {
  return __hiloint2double(__double2hiint(v) ^ m, __double2loint(v));
}

// One row of coefficients of a level: rows ha, hb, hc of the horizontal
// analysis at y - D, y, y + D (h[j], mask j), the row's z (group and, with
// LOW, the low-pass value zl), the threshold, and the vertical synthesis
// into pa += (row y - D), pb += (row y), pc = (row y + D, its first
// contribution).  mrow, mcol, m11: sign masks of mirrored rows / columns for
// the antisymmetric bands.  The masks are applied through their sums and
// differences: with s = h_a + h_c, d = h_a - h_c,
//   z0 += s / 4 + h_b / 2,  z1 += (sqrt 2 / 4) d,  z2 += h_b / 2 - s / 4,
// and the transpose the same way: 15 operations per horizontal mask instead
// of 19 (FP32: an issue-bound sweep; FP64: the pipe is full).  A correction is
// complete before z is added, so z is rounded once per update at its own
// magnitude (z inside the chain of multiply-adds: 14 operations, 406 us for a
// launch of 4096^2, L = 2 instead of 411, two roundings).
// BF16 z: the masks tap by tap, in one fixed order (the rounding of z to 8 bits
// makes the last bit of these sums matter, see the host's stencil_variant).
// PARTS: a row's three shares are summed by themselves and then added to its
// rows (k_frame_lev); else every tap is added to them directly (k_frame3).
template <bool LOW, bool PARTS, typename T, typename TZ>
__device__ __forceinline__ void f3_row(const T (&ha)[3], const T (&hb)[3], const T (&hc)[3],
                                       const ZGroup<TZ>& zi, TZ zl, int mrow, int mcol, T mu,
                                       ZGroup<TZ>& zo, TZ& zlo, T (&pa)[3], T (&pb)[3], T (&pc)[3]) {
  const T s2q = T(0.35355339059327376220);               // sqrt(2) / 4
  const int m11 = mrow ^ mcol;
  constexpr bool TAPS = sizeof(TZ) == 2;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    auto in = [&](int i) {                               // z of band (i, j), mirrored sign applied
      T v = T(ld_z(&zi.e[3 * i + j - 1]));
      if (i == 1 && j == 1) v = f3_flip(v, m11);
      else if (i == 1) v = f3_flip(v, mrow);
      else if (j == 1) v = f3_flip(v, mcol);
      return v;
    };
    if constexpr (TAPS) {
      // (a quarter of a sum is exactly the sum of the quarters)
      const T q = T(0.25) * (ha[j] + hc[j]);
      T a0 = PARTS ? T(0) : pa[j], a1 = PARTS ? T(0) : pb[j], a2 = T(0);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        if (i == 0 && j == 0 && !LOW) continue;
        const T b0 = i == 0 ? T(0.25) : i == 1 ? s2q : T(-0.25), b2 = i == 1 ? -s2q : b0;
        const T a = i == 1 ? b0 * ha[j] + b2 * hc[j] : fma(T(0.5), hb[j], i == 0 ? q : -q);
        const T zn = (i == 0 && j == 0 ? T(ld_z(&zl)) : in(i)) + a;
        if (i == 0 && j == 0) zlo = to_z(zn, (TZ*)nullptr);
        else zo.e[3 * i + j - 1] = to_z(zn, (TZ*)nullptr);
        const T x = f3_soft(zn, mu);
        a0 += b0 * x;
        if (i != 1) a1 += T(0.5) * x;
        a2 += b2 * x;
      }
      pa[j] = PARTS ? pa[j] + a0 : a0;
      pb[j] = PARTS ? pb[j] + a1 : a1;
      pc[j] = a2;
      continue;
    }
    const T q = T(0.25) * (ha[j] + hc[j]), d = ha[j] - hc[j];
    T x0 = T(0);
    if (j > 0 || LOW) {
      const T v = j == 0 ? T(ld_z(&zl)) : in(0);
      const T zn = v + fma(T(0.5), hb[j], q);
      if (j == 0) zlo = to_z(zn, (TZ*)nullptr);
      else zo.e[j - 1] = to_z(zn, (TZ*)nullptr);
      x0 = f3_soft(zn, mu);
    }
    const T z1 = fma(s2q, d, in(1));
    const T z2 = in(2) + fma(T(0.5), hb[j], -q);
    zo.e[3 + j - 1] = to_z(z1, (TZ*)nullptr);
    zo.e[6 + j - 1] = to_z(z2, (TZ*)nullptr);
    const T x1 = f3_soft(z1, mu), x2 = f3_soft(z2, mu);
    const T D = (j > 0 || LOW) ? x0 - x2 : -x2;
    const T S = (j > 0 || LOW) ? x0 + x2 : x2;
    pa[j] = fma(s2q, x1, fma(T(0.25), D, pa[j]));
    pb[j] = fma(T(0.5), S, pb[j]);
    pc[j] = fma(-s2q, x1, T(0.25) * D);
  }
}
// horizontal analysis of one position (values at x - D, x, x + D)
template <typename T>
__device__ __forceinline__ void f3_hrow(T cm, T c0, T cp, T (&h)[3]) {
  const T t = T(0.25) * (cm + cp);
  h[0] = fma(T(0.5), c0, t);
  h[1] = T(0.35355339059327376220) * (cm - cp);
  h[2] = fma(T(0.5), c0, -t);
}
// horizontal synthesis parts of a completed row: A(x + D) + B(x) + C(x - D)
// (TZ: BF16 z term by term, as f3_row)
template <typename TZ, typename T>
__device__ __forceinline__ void f3_abc(const T (&P)[3], T& A, T& B, T& C) {
  if (sizeof(TZ) == 2) {
    const T s2q = T(0.35355339059327376220);
    A = T(0.25) * P[0] + s2q * P[1] - T(0.25) * P[2];
    B = T(0.5) * (P[0] + P[2]);
    C = T(0.25) * P[0] - s2q * P[1] - T(0.25) * P[2];
    return;
  }
  const T e = T(0.25) * (P[0] - P[2]), s2q = T(0.35355339059327376220);
  A = fma(s2q, P[1], e);
  B = T(0.5) * (P[0] + P[2]);
  C = fma(-s2q, P[1], e);
}

// A warp's ring of z rows (RING > 0): slot k holds one row's 32 groups at
// buf + k * 256 values and completes on bar[k]; seq counts the rows that went
// through the bulk path (every bulk row advances one slot and, every RING rows,
// the expected parity); bad is set when a bounded wait gave up.
template <typename TZ>
struct F3Ring {
  TZ* buf;
  unsigned long long* bar;
  int seq;
  bool bad;
};

template <typename T, typename TZ, int LEV, int L, int F3_PF, int RING>
__device__ __forceinline__ void f3_level(const Prob& pd, const T* __restrict__ cin, int cpitch,
                                         int cy0, int cx0, const TZ* __restrict__ zin,
                                         TZ* __restrict__ zout, bool fresh, int ty0, int tx0,
                                         int seg_lo, int seg_hi, T mu, T* __restrict__ f2s,
                                         T* __restrict__ fout, F3Ring<TZ>& rg) {
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int D = 1 << (LEV - 1);
  constexpr bool TOP = (LEV == L);
  constexpr int XO = (LEV == 2) ? 3 : 1;                 // first coefficient column tx0 - XO
  constexpr int NL = (LEV == 2) ? 32 : F3_TX + 2;        // lanes with a coefficient column
  const int lane = threadIdx.x & 31;
  const int x = tx0 - XO + lane;
  const bool act = lane < NL;
  const int nf = pd.nf;
  const int plane = nf * nf;     // nbands nf^2 < 2^31 is checked at set-up
  // rows: outputs [yo0, yo1), coefficients [yc0, yc1)
  const int yo0 = (LEV == 2) ? seg_lo - 1 : seg_lo;
  const int yo1 = (LEV == 2) ? seg_hi + 1 : seg_hi;
  const int yc0 = yo0 - D, yc1 = yo1 + D;
  // column part of the z offsets and its mirroring parity
  bool pcx;
  const int zc = f3_refl(x, nf, &pcx);
  const int mcol = pcx ? (int)0x80000000 : 0;
  const bool own_c = act && x >= tx0 && x < tx0 + F3_TX && x < nf;
  // owned rows [seg_lo, own_hi): one unsigned compare per row
  const unsigned own_rows = (unsigned)max(min(seg_hi, nf) - seg_lo, 0);
  const T* ccol = cin + (act ? x - cx0 : D);   // idle lanes read a valid column
  // level 2 reads c_1 = (b0 x b0) u, formed here from the u tile: lane l keeps
  // c_1 at columns x - 2 and x + 2 (a sliding ring of the horizontally
  // filtered u rows, g), and gets c_1 at x from lane l - 2 (or l + 2)
  const T* ua = cin + (x - 2 - cx0);
  T gr[3][2];
  auto grow = [&](int y, T (&g)[2]) {
    const T* r = ua + (y - cy0) * cpitch;
    g[0] = T(0.25) * (r[-1] + r[1]) + T(0.5) * r[0];
    g[1] = T(0.25) * (r[3] + r[5]) + T(0.5) * r[4];
  };
  // this level's band group and (top level) the low-pass plane
  constexpr int NV = 8 * (int)sizeof(TZ) / 16;
  const int gbase = (LEV - 1) * 8 * plane, lbase = 8 * L * plane;
  // h ring: rows y - D .. y + D of the current coefficient row y
  T hr[2 * D + 1][3];
  auto hrow = [&](int y, T (&h)[3]) {
    T cm, c0, cp;
    if constexpr (LEV == 2) {
      // rows are requested in order: g holds rows y - 1, y and gets y + 1
      grow(y + 1, gr[2]);
      cm = T(0.25) * (gr[0][0] + gr[2][0]) + T(0.5) * gr[1][0];
      cp = T(0.25) * (gr[0][1] + gr[2][1]) + T(0.5) * gr[1][1];
      const T up = __shfl_up_sync(FULL, cp, 2), dn = __shfl_down_sync(FULL, cm, 2);
      c0 = lane >= 2 ? up : dn;
#pragma unroll
      for (int q = 0; q < 2; ++q) { gr[0][q] = gr[1][q]; gr[1][q] = gr[2][q]; }
    } else {
      const T* r = ccol + (y - cy0) * cpitch;
      cm = r[-D]; c0 = r[0]; cp = r[D];
    }
    f3_hrow(cm, c0, cp, h);
  };
  if constexpr (LEV == 2) {
    grow(yc0 - D - 1, gr[0]);
    grow(yc0 - D, gr[1]);
  }
  // Ring slots.  A queue of one row: the sweep is unrolled by the ring length
  // and the rows keep their slots (row y of phase ph has slot ph + D, modulo
  // the length): nothing moves.  Deeper queues are unrolled by the queue's
  // length and shift the rings by one row per step (phase 0 always).
  constexpr int RL = 2 * D + 1;
  constexpr int RINGD = RING > 0 ? RING : 1;
  constexpr bool STATIC_RING = F3_PF == 1 && RING == 0;
  constexpr int UNR = STATIC_RING ? RL : F3_PF;
#pragma unroll
  for (int k = 0; k < 2 * D; ++k) hrow(yc0 - D + k, hr[k]);
  // z queue: rows y .. y + PF - 1 (group and low-pass value per row; with a
  // ring, the low-pass value only)
  ZGroup<TZ> zq[RING > 0 ? 1 : F3_PF];
  TZ zl[F3_PF];
  // each queued row's mirrored offset and mirroring parity, mapped once when
  // the row is queued and used again when it is swept
  int zqo[F3_PF];
  int zqm[F3_PF];              // (the parity as a sign mask)
  // (idle lanes load a valid mirrored column too; their values are unused.
  // Offsets stay in 32 bits: nbands nf^2 < 2^31.)
  auto zload = [&](int y, int k) {
    bool par;
    const int q = f3_refl(y, nf, &par) * nf + zc;
    zqo[k] = q;
    zqm[k] = par ? (int)0x80000000 : 0;
    if (fresh) return;                 // z_in = 0: the queue keeps its zeros
    if constexpr (RING == 0) {
      const uint4* src = reinterpret_cast<const uint4*>(zin + (gbase + 8 * q));
#pragma unroll
      for (int v = 0; v < NV; ++v) zq[k].v[v] = src[v];
    }
    if (TOP) zl[k] = zin[lbase + q];
  };
#pragma unroll
  for (int k = 0; k < F3_PF; ++k) {
#pragma unroll
    for (int v = 0; v < NV; ++v) zq[RING > 0 ? 0 : k].v[v] = make_uint4(0, 0, 0, 0);
    zl[k] = TZ(0.0f);
    zload(yc0 + k, k);
  }
  // ring: rows are issued RING ahead of the sweep.  Bulk path when the warp's
  // 32 columns lie inside the image (one contiguous run of 32 groups per row),
  // else per-lane 16-byte asynchronous copies of the mirrored columns.
  const int x0 = tx0 - XO;
  const bool bulk = RING > 0 && x0 >= 0 && x0 + 32 <= nf;
  const int nrows = yc1 - yc0;
  const int seq0 = rg.seq;
  int n_issued = 0, first_bad = nrows;      // bulk rows issued; first row whose wait gave up
  auto issue = [&](int i) {                 // row yc0 + i into its slot
    if constexpr (RING > 0) {
      bool par;
      const int yr = f3_refl(yc0 + i, nf, &par);
      if (bulk) {
        const int slot = (seq0 + i) % RING;
        ++n_issued;
        if (lane == 0) {
          // (the slot's previous row was only read, by this warp, before the
          // __syncwarp that precedes this copy: no proxy fence is needed)
          mbar_expect_tx(rg.bar + slot, (unsigned)f3_slot_bytes<TZ>());
          bulk_g2s(rg.buf + slot * 256, zin + (gbase + 8 * (yr * nf + x0)),
                   (unsigned)f3_slot_bytes<TZ>(), rg.bar + slot);
        }
      } else {
        const int slot = i % RING;
        const TZ* src = zin + (gbase + 8 * (yr * nf + zc));
        TZ* dst = rg.buf + slot * 256 + 8 * lane;
#pragma unroll
        for (int v = 0; v < NV; ++v) cp_async_16(dst + v * (16 / (int)sizeof(TZ)), src + v * (16 / (int)sizeof(TZ)));
        cp_commit();
      }
    }
  };
  if constexpr (RING > 0) {
    // the ring may hold rows an earlier level wrote with per-lane copies:
    // order those writes before this level's bulk copies
    if (bulk && lane == 0) fence_proxy_async();
    for (int i = 0; i < RING && !fresh; ++i) {
      if (i < nrows) issue(i);
      else if (!bulk) cp_commit();          // empty group: one group per row slot
    }
  }
  // synthesis ring: rows y - D .. y + D
  T pr[2 * D + 1][3];
#pragma unroll
  for (int k = 0; k <= 2 * D; ++k) pr[k][0] = pr[k][1] = pr[k][2] = T(0);
  // level-2 low-pass ring of the horizontally filtered s_1 rows r-2, r-1, r
  T gq[3] = {T(0), T(0), T(0)};
  // one coefficient row; queue slot kq holds its z and is refilled with row
  // y + PF.  The queue is indexed statically (the sweep is unrolled by PF) so
  // that no register receiving an outstanding load is copied before it is used.
  auto step = [&](int y, int k) {
    const int kq = STATIC_RING ? 0 : k, ph = STATIC_RING ? k : 0;
    const int ia = ph, ib = (ph + D) % RL, ic = (ph + 2 * D) % RL;   // rows y - D, y, y + D
    if (RING > 0 && !fresh) {
      // this row's groups from the ring, then the slot is refilled with row y + RING
      const int i = y - yc0;
      if (bulk) {
        const int g = seq0 + i;
        if (!rg.bad && !mbar_wait(rg.bar + g % RINGD, (unsigned)(g / RINGD) & 1u)) {
          rg.bad = true;
          first_bad = i;
        }
        const uint4* sv = reinterpret_cast<const uint4*>(rg.buf + (g % RINGD) * 256 + 8 * lane);
#pragma unroll
        for (int v = 0; v < NV; ++v) zq[0].v[v] = sv[v];
      } else {
        cp_wait<RINGD - 1>();
        const uint4* sv = reinterpret_cast<const uint4*>(rg.buf + (i % RINGD) * 256 + 8 * lane);
#pragma unroll
        for (int v = 0; v < NV; ++v) zq[0].v[v] = sv[v];
      }
      __syncwarp();
      if (i + RING < nrows && !rg.bad) issue(i + RING);
      else if (!bulk) cp_commit();
    }
    hrow(y + D, hr[ic]);
    // z outside the image is its mirror image; antisymmetric (b1) bands
    // change sign under an odd number of mirrorings
    const bool own = own_c && (unsigned)(y - seg_lo) < own_rows;
    const int zwo = zqo[kq];
    ZGroup<TZ> zo;
    TZ zlo = TZ(0.0f);
    f3_row<TOP, false, T, TZ>(hr[ia], hr[ib], hr[ic], zq[RING > 0 ? 0 : kq], zl[kq], zqm[kq], mcol, mu, zo, zlo,
                       pr[ia], pr[ib], pr[ic]);
    if (own) {
      uint4* dstz = reinterpret_cast<uint4*>(zout + (gbase + 8 * zwo));
#pragma unroll
      for (int v = 0; v < NV; ++v) dstz[v] = zo.v[v];
      if (TOP) zout[lbase + zwo] = zlo;
    }
    if (y + F3_PF < yc1) zload(y + F3_PF, kq);
    if (RING == 0 && !fresh) {
      // the z lines of a row further ahead into L2 (no registers held): the
      // register queue then finds them there
      const int ya = y + F3_PF + Z_L2_AHEAD;
      if (ya < yc1) {
        // (ya >= 0; past the bottom edge the row is clamped rather than
        // mirrored: a prefetch of a neighbouring line only costs an L2 miss)
        const int qa = min(ya, nf - 1) * nf + zc;
        prefetch_l2(zin + (gbase + 8 * qa));
        if (TOP) prefetch_l2(zin + (lbase + qa));
      }
    }
    // row y - D has all its contributions: horizontal synthesis
    const int r = y - D;
    if (r >= yo0) {
      T A, B, C;
      f3_abc<TZ>(pr[ia], A, B, C);
      const T out = B + __shfl_down_sync(FULL, A, D) + __shfl_up_sync(FULL, C, D);
      if (LEV == 2 && L == 2) {
        // s_1 row r (lanes 2..29) -> (b0 x b0)^T s_1 row r - 1 (lanes 3..28)
        const T g = T(0.5) * out +
                    T(0.25) * (__shfl_up_sync(FULL, out, 1) + __shfl_down_sync(FULL, out, 1));
        gq[0] = gq[1]; gq[1] = gq[2]; gq[2] = g;
        if (r - 1 >= seg_lo && lane >= 3 && lane < 3 + F3_TX)
          f2s[(r - 1 - ty0) * F3_TX + (lane - 3)] = T(0.25) * (gq[0] + gq[2]) + T(0.5) * gq[1];
      } else {
        // level 1: f row r (lanes 1..26) = out + level-2 part
        if (lane >= 1 && lane < 1 + F3_TX) {
          T fv = out;
          if (L == 2) fv += f2s[(r - ty0) * F3_TX + (lane - 1)];
          if (r < nf && x < nf) fout[(size_t)r * nf + x] = fv;
        }
      }
    }
    if constexpr (!STATIC_RING) {
#pragma unroll
      for (int q = 0; q < 2 * D; ++q)
#pragma unroll
        for (int j = 0; j < 3; ++j) { hr[q][j] = hr[q + 1][j]; pr[q][j] = pr[q + 1][j]; }
    }
  };
#pragma unroll 1
  for (int y = yc0; y < yc1; y += UNR) {
#pragma unroll
    for (int k = 0; k < UNR; ++k)
      if (y + k < yc1) step(y + k, k);
  }
  if (RING > 0 && !fresh) {
    if (bulk) {
      if (rg.bad) {
        // a wait gave up: wait (bounded) for the copies this level issued
        // from that row on, so none lands after the CTA has gone
        for (int i = first_bad; i < n_issued; ++i) {
          const int g = seq0 + i;
          mbar_wait(rg.bar + g % RINGD, (unsigned)(g / RINGD) & 1u);
        }
      }
      rg.seq = seq0 + nrows;
    } else {
      cp_wait<0>();
    }
    __syncwarp();
  }
}

// No z to read: the first update after a reset (z^0 = 0), and every step of the
// balanced formulation.  (Storing the zeros cost a memset of all of z per
// reset and their read in the first step: 4096^2, L = 2: 181 + 190 us.)
__device__ __forceinline__ bool frame_fresh(const Prob& pd, const State& st, const void* zin_op) {
  return !zin_op && (pd.balanced || (st.zfresh && st.iter == 1));
}

// One framelet tile on the thread group `blk` of 32 F3_NWR threads with its
// shared memory at smraw.
template <typename T, typename TZ, int L, int F3_NWR, int F3_PF, int RING, int SEG, typename BLK>
__device__ __forceinline__ void frame3_body(const int2 item, const Prob* __restrict__ probs,
                                            State* __restrict__ states, int u_slot, int f_slot,
                                            const void* zin_op, void* zout_op, double op_mu,
                                            unsigned char* smraw, BLK blk) {
  const int tid = blk.tid();
  using Gm = F3<L, F3_NWR, SEG>;
  constexpr int F3_TY = Gm::TY;
  const Prob& pd = probs[item.x];
  const State& st = states[item.x];
  if (st.stopped) return;
  const int nf = pd.nf;
  const int tilesX = (nf + F3_TX - 1) / F3_TX;
  const int ty0 = (item.y / tilesX) * F3_TY, tx0 = (item.y % tilesX) * F3_TX;
  const T mu = T(zin_op ? op_mu : pd.mu);
  const TZ* zin;
  TZ* zout;
  if (zin_op) {
    zin = static_cast<const TZ*>(zin_op);
    zout = static_cast<TZ*>(zout_op);
  } else {
    zin = static_cast<const TZ*>(pd.z[(st.iter - 1) & 1]);
    zout = static_cast<TZ*>(pd.z[st.iter & 1]);
  }
  const bool fresh = frame_fresh(pd, st, zin_op);
  T* su = reinterpret_cast<T*>(smraw);            // u on rows ty0 - C0.., cols tx0 - C0..
  T* sf2 = su + Gm::UW * Gm::UH;                  // level-2 part of f on the tile (L = 2)
  constexpr int C0 = Gm::C0;
  {
    int mode;
    const T* src;
    if (u_slot >= 0) { src = static_cast<const T*>(pd.buf[u_slot]); mode = 1; }
    else if (!pd.use_adj) { src = static_cast<const T*>(pd.buf[SL_T]); mode = 1; }
    else if (pd.bc == BC_RECT) { src = static_cast<const T*>(pd.buf[SL_V]); mode = 1; }
    else if (pd.bc == BC_AR || pd.balanced) { src = static_cast<const T*>(pd.buf[SL_U]); mode = 1; }   // A' t; f + u
    else { src = static_cast<const T*>(pd.buf[SL_V]); mode = 0; }
    const bool interior = ty0 - C0 >= 0 && tx0 - C0 >= 0 && ty0 + F3_TY + C0 <= nf &&
                          tx0 + F3_TX + C0 <= nf;
    constexpr int NT = 32 * F3_NWR;
    constexpr int UN = Gm::UW * Gm::UH;
    // the BC fold of V has a single term wherever the tile keeps c pixels
    // from the image edges (or for zero BCs): u(a, b) = V(a + c, b + c)
    const int cc = pd.c;
    const bool single = mode == 0 && interior &&
                        (pd.bc == BC_ZERO || (ty0 - C0 >= cc && tx0 - C0 >= cc &&
                                              ty0 + F3_TY + C0 <= nf - cc && tx0 + F3_TX + C0 <= nf - cc));
    if (mode || single) {
      // plain copies of the (reflected) source: asynchronous, all of a
      // thread's copies in flight together, no registers held
      const int pitch = mode ? nf : pd.ne, off = mode ? 0 : cc;
      for (int idx = tid; idx < UN; idx += NT) {
        const int ry = idx / Gm::UW, rx = idx - ry * Gm::UW;
        bool par;
        const int ay = interior ? ty0 - C0 + ry : f3_refl(ty0 - C0 + ry, nf, &par);
        const int ax = interior ? tx0 - C0 + rx : f3_refl(tx0 - C0 + rx, nf, &par);
        const T* g = src + ((size_t)(ay + off) * pitch + (ax + off));
        if (sizeof(T) == 8) cp_async_8(su + idx, g); else cp_async_4(su + idx, g);
      }
      cp_commit();
      cp_wait<0>();
    } else {
      // the BC fold of V sums up to four entries per element
      for (int idx = tid; idx < UN; idx += NT) {
        const int ry = idx / Gm::UW, rx = idx - ry * Gm::UW;
        const int gy = ty0 - C0 + ry, gx = tx0 - C0 + rx;
        int o;
        const int ay = interior ? gy : refl_half(gy, nf, &o);
        const int ax = interior ? gx : refl_half(gx, nf, &o);
        su[idx] = fold_fetch<T>(pd, src, ay, ax);
      }
    }
  }
  blk.sync();
  const int w = tid >> 5;
  const int seg_lo = ty0 + w * SEG, seg_hi = seg_lo + SEG;
  if (seg_lo >= nf) return;        // no barrier follows
  T* f = static_cast<T*>(pd.buf[f_slot]);
  // this warp's ring of z rows and its mbarriers (RING > 0)
  F3Ring<TZ> rg;
  rg.seq = 0;
  rg.bad = false;
  rg.buf = nullptr;
  rg.bar = nullptr;
  if constexpr (RING > 0) {
    unsigned char* rb = smraw + frame3_ring_offset<T, TZ, L, F3_NWR, RING, SEG>();
    rg.buf = reinterpret_cast<TZ*>(rb + (size_t)w * RING * f3_slot_bytes<TZ>());
    rg.bar = reinterpret_cast<unsigned long long*>(rb + (size_t)F3_NWR * RING * f3_slot_bytes<TZ>()) +
             w * RING;
    if ((tid & 31) == 0) {
      for (int k = 0; k < RING; ++k) mbar_init(rg.bar + k, 1);
      mbar_init_fence();
    }
    __syncwarp();
  }
  if (L == 2) {
    f3_level<T, TZ, 2, L, F3_PF, RING>(pd, su, Gm::UW, ty0 - C0, tx0 - C0, zin, zout, fresh, ty0, tx0,
                                       seg_lo, seg_hi, mu, sf2, f, rg);
    __syncwarp();
  }
  if (!rg.bad)
    f3_level<T, TZ, 1, L, F3_PF, RING>(pd, su, Gm::UW, ty0 - C0, tx0 - C0, zin, zout, fresh, ty0, tx0,
                                       seg_lo, seg_hi, mu, sf2, f, rg);
  if (rg.bad && (tid & 31) == 0) {
    // a bounded wait gave up: the problem stops with a timeout status
    volatile State* vs = &states[item.x];
    vs->status = -4;
    vs->stopped = 1;
  }
}
template <typename T, typename TZ, int L, int F3_NWR, int F3_PF, int RING, int SEG = F3_SEG>
__global__ void __launch_bounds__(32 * F3_NWR)
k_frame3(const Prob* __restrict__ probs, State* __restrict__ states, const int2* __restrict__ items,
         int u_slot, int f_slot, const void* zin_op, void* zout_op, double op_mu) {
  extern __shared__ __align__(16) unsigned char smraw[];
  frame3_body<T, TZ, L, F3_NWR, F3_PF, RING, SEG>(items[blockIdx.x], probs, states, u_slot, f_slot, zin_op,
                                             zout_op, op_mu, smraw, BlkFull{});
}


// ---------------------------------------------------------------------------
// L >= 3: the step level by level (the paper's experiments use L = 4).
//
//   c_0 = u,  c_l = (b0 x b0)_{2^(l-1)} c_{l-1}         (k_lowpass, kept in HBM)
//   level l = L, L-1, ..., 1 (k_frame_lev, dilation D = 2^(l-1)):
//     z_l <- z_l + W_l c_{l-1},  x = S_mu(z_l),
//     s_{l-1} = sum over the level's bands of B_ij^T x_ij  +  (b0 x b0)^T s_l
//   (the top level's nine bands include the final low-pass and it has no
//   s_L term), f = s_0.  s_1 .. s_{L-1} live in HBM too, so each kernel needs
//   a halo of its own dilation only (the fused single-pass form needs
//   2 (2^L - 1) = 30 pixels per side at L = 4), and in the polyphase order of
//   that dilation (Poly) the halo is one position: c_{l-1}, s_l and the
//   level's z are kept in the order of 2^(l-1), s_{l-1} in that of 2^(l-2).

// u as the level-1 kernel and the first low-pass read it: the op entry
// point's slot, t (Algorithm 4 forms), V (rectangular A), or U: the BC fold
// of V materialised before the sweep, or A' t for antireflective BCs
template <typename T>
__device__ __forceinline__ const T* frame_u(const Prob& pd, int u_slot) {
  if (u_slot >= 0) return static_cast<const T*>(pd.buf[u_slot]);
  if (!pd.use_adj) return static_cast<const T*>(pd.buf[SL_T]);
  if (pd.bc == BC_RECT) return static_cast<const T*>(pd.buf[SL_V]);
  return static_cast<const T*>(pd.buf[SL_U]);     // (also f + u of the balanced form)
}

// c_lev = (b0 x b0) with dilation d = 2^(lev-1) applied to c_{lev-1}, half-
// sample mirror at the border.  c_{lev-1} is read in the polyphase order of d
// (u, lev = 1: plain) and c_lev is written in that of 2d, the order of the
// kernels that read it.  The launch walks the input order: item.y = (row
// sub-lattice b of d, chunk of RB of its rows, which are neighbouring input
// rows); for each column sub-lattice a of d the threads stride along it, its taps
// d apart being its neighbouring positions (contiguous reads), and its even and
// odd positions land in the output sub-lattices a and a + d (two contiguous runs
// of writes).  A thread walks down the chunk's rows with the horizontally
// filtered rows y - d, y, y + d in registers: 3 (RB + 2) / RB loads per output
// instead of 9.  The kernel is bound by those loads (4126^2, 0.136 GB: 55 us a
// launch with one row per CTA, 40 with 8); small images keep one row per CTA
// (lowpass_rows).
template <typename T, int RB>
__global__ void __launch_bounds__(LP_THREADS)
k_lowpass(const Prob* __restrict__ probs, const State* __restrict__ states,
          const int2* __restrict__ items, int lev, int u_slot) {
  const int2 item = items[blockIdx.x];
  const Prob& pd = probs[item.x];
  if (states[item.x].stopped) return;
  const int nf = pd.nf;
  const size_t plane = (size_t)nf * nf;
  const int d = 1 << (lev - 1);
  const Poly pin(nf, d), pout(nf, 2 * d);
  const int sb = item.y & (d - 1), m0 = (item.y >> (lev - 1)) * RB;
  const int nr = min(RB, pin.count(sb) - m0);    // rows of this chunk
  if (nr <= 0) return;
  const T* in = (lev == 1) ? frame_u<T>(pd, u_slot)
                           : static_cast<const T*>(pd.lp) + (size_t)(lev - 2) * plane;
  T* out = static_cast<T*>(pd.lp) + (size_t)(lev - 1) * plane;
  bool par;
  // rows m0 - 1 .. m0 + RB of the sub-lattice (mirrored into the image; past the
  // chunk's end the last row again) and the output rows
  const T* row[RB + 2];
  T* orow[RB];
#pragma unroll
  for (int k = 0; k < RB + 2; ++k)
    row[k] = in + (size_t)pin.pos(f3_refl(sb + d * (m0 + min(k, nr + 1) - 1), nf, &par)) * nf;
#pragma unroll
  for (int k = 0; k < RB; ++k) orow[k] = out + (size_t)pout.pos(sb + d * (m0 + min(k, nr - 1))) * nf;
  for (int a = 0; a < d; ++a) {
    const int ma = pin.count(a), sa = pin.start(a);
    // output run starts of the even and odd positions of sub-lattice a
    const int oe = a < nf ? pout.pos(a) : 0, oo = (a + d < nf) ? pout.pos(a + d) : 0;
    for (int m = threadIdx.x; m < ma; m += LP_THREADS) {
      const int ic = sa + m;
      int im = ic - 1, ip = ic + 1;             // neighbours inside the sub-lattice
      if (m == 0) im = pin.pos(f3_refl(a - d, nf, &par));
      if (m == ma - 1) ip = pin.pos(f3_refl(a + d * (m + 1), nf, &par));
      const int o = (m & 1) ? oo + (m >> 1) : oe + (m >> 1);
      T h[RB + 2];
#pragma unroll
      for (int k = 0; k < RB + 2; ++k) h[k] = T(0.25) * (row[k][im] + row[k][ip]) + T(0.5) * row[k][ic];
#pragma unroll
      for (int k = 0; k < RB; ++k)
        if (k < nr) orow[k][o] = T(0.25) * (h[k] + h[k + 2]) + T(0.5) * h[k + 1];
    }
  }
}

// Level kernel geometry.  A level of dilation dp works in the polyphase
// order of dp (Poly): the taps dp apart join neighbouring positions m - 1, m,
// m + 1 of one sub-lattice, so the kernel runs the dilation-1 sweep on each
// of the dp^2 sub-lattices (a, b) (columns x = a + dp m, rows y = b + dp m).
// A CTA (one warp) owns OUTW positions of a column sub-lattice x SEG
// positions of a row sub-lattice; lane k owns the coefficient column
// m = tx0 - 1 + k (every lane computes coefficients, lanes 1 .. 30 produce
// output).  The halo is one position whatever dp is.
template <int SEG>
struct LV {
  static constexpr int OUTW = 30;                 // output columns of a tile
  static constexpr int TY = SEG;
  static constexpr int CW = 34, CH = TY + 4;      // c tile: positions tx0 - 2.., ty0 - 2..
};
// tiles of one sub-lattice pair and of the whole level
__host__ __device__ inline void lev_tile_grid(int nf, int dp, int seg, int* tx, int* ty) {
  const int m = Poly(nf, dp).count_max();
  *tx = (m + LV<32>::OUTW - 1) / LV<32>::OUTW;
  *ty = (m + seg - 1) / seg;
}

// One level of the step.  The warp sweeps down its rows (one row
// sub-lattice): the horizontal analysis of row m + 1 of c_{l-1} (shared-memory
// tile, polyphase order of dp) joins rows m - 1 and m in a register ring, then
// the vertical masks, the update of z (register queue, PF rows ahead; z of the
// level in the same order), the threshold, and the vertical synthesis into a
// register ring of three rows (f3_row); row m - 1 then has all its
// contributions and is combined horizontally by warp shuffles at +-1 and, for
// l < L, with (b0 x b0)^T s_l: each lane loads s_l at its own column with the
// z rows and keeps the horizontally filtered rows m - 2 .. m in registers
// (shuffles at +-1).  The sweep is unrolled by the ring length, so every ring
// and queue index is static and nothing moves.  s_{l-1} is written in the
// polyphase order of dp / 2 (f, and s_1, plainly).  Coefficients outside the
// image are mirrored with the sign of the band's symmetry, as in k_frame3.
template <typename T, typename TZ, bool TOP, int SEG>
__global__ void __launch_bounds__(32, lv_minb(SEG, sizeof(T)))
k_frame_lev(const Prob* __restrict__ probs, State* __restrict__ states,
            const int2* __restrict__ items, int lev, int u_slot, int f_slot, const void* zin_op,
            void* zout_op, double op_mu) {
  using G = LV<SEG>;
  constexpr int PF = lv_pf(SEG);
  static_assert(PF == 1 || PF == 3, "queue index static under the unrolling by 3");
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int NV = 8 * (int)sizeof(TZ) / 16;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int2 item = items[blockIdx.x];
  const Prob& pd = probs[item.x];
  const State& st = states[item.x];
  if (st.stopped) return;
  const int nf = pd.nf, L = pd.levels;
  const int plane = nf * nf;                 // nbands nf^2 < 2^31 is checked at set-up
  const int dp = 1 << (lev - 1);
  const Poly P(nf, dp), PO(nf, dp > 1 ? dp / 2 : 1);
  int tX, tY;
  lev_tile_grid(nf, dp, SEG, &tX, &tY);
  int t = item.y;
  const int tx = t % tX;
  t /= tX;
  const int ty = t % tY;
  t /= tY;
  const int sa = t % dp, sb = t / dp;        // column and row sub-lattices
  const int Ma = P.count(sa), Mb = P.count(sb);
  const int tx0 = tx * G::OUTW, ty0 = ty * G::TY;
  if (tx0 >= Ma || ty0 >= Mb) return;        // an empty tile (uniform over the CTA)
  const T mu = T(zin_op ? op_mu : pd.mu);
  const TZ* zin;
  TZ* zout;
  if (zin_op) {
    zin = static_cast<const TZ*>(zin_op);
    zout = static_cast<TZ*>(zout_op);
  } else {
    zin = static_cast<const TZ*>(pd.z[(st.iter - 1) & 1]);
    zout = static_cast<TZ*>(pd.z[st.iter & 1]);
  }
  const bool fresh = frame_fresh(pd, st, zin_op);
  // position of the local coordinate m of a sub-lattice in the level's order
  // (mirrored into the image first)
  auto cpos = [&](int m, int off, bool* par) { return P.pos(f3_refl(off + dp * m, nf, par)); };
  T* sc = reinterpret_cast<T*>(smraw);       // c_{l-1} on rows ty0 - 2.., cols tx0 - 2..
  const int lane = threadIdx.x;
  {
    const T* cin = (lev == 1) ? frame_u<T>(pd, u_slot)
                              : static_cast<const T*>(pd.lp) + (size_t)(lev - 2) * plane;
    // lanes along the row (columns lane and lane + 32, mapped once per lane),
    // each row's position mapped once
    static_assert(G::CW <= 64, "two columns per lane");
    bool par;
    const int ax0 = cpos(tx0 - 2 + lane, sa, &par);
    const bool two = lane + 32 < G::CW;
    const int ax1 = two ? cpos(tx0 - 2 + lane + 32, sa, &par) : 0;
    for (int ry = 0; ry < G::CH; ++ry) {
      const T* row = cin + (size_t)cpos(ty0 - 2 + ry, sb, &par) * nf;
      T* d = sc + ry * G::CW + lane;
      if (sizeof(T) == 8) cp_async_8(d, row + ax0); else cp_async_4(d, row + ax0);
      if (two) {
        if (sizeof(T) == 8) cp_async_8(d + 32, row + ax1); else cp_async_4(d + 32, row + ax1);
      }
    }
    cp_commit();
  }
  const int seg_lo = ty0, seg_hi = ty0 + SEG;
  const int mx = tx0 - 1 + lane;             // this lane's coefficient column (local)
  bool pcx;
  const int zc = cpos(mx, sa, &pcx);
  const int mcol = pcx ? (int)0x80000000 : 0;
  const bool own_c = lane >= 1 && lane < 31 && mx < Ma;
  const unsigned own_rows = (unsigned)(min(seg_hi, Mb) - seg_lo);   // owned rows [seg_lo, seg_lo + own_rows)
  const int yc0 = seg_lo - 1, yc1 = seg_lo + (int)own_rows + 1;
  const T* ccol = sc + (lane + 1);                  // c tile column of mx, row ty0 - 2
  const int gbase = (lev - 1) * 8 * plane, lbase = 8 * L * plane;
  T* dst = (lev == 1) ? static_cast<T*>(pd.buf[f_slot])
                      : static_cast<T*>(pd.sy) + (size_t)(lev - 2) * plane;
  const int dcol = (own_c) ? PO.pos(sa + dp * mx) : 0;   // output column in dst's order
  const T* sin = TOP ? nullptr : static_cast<const T*>(pd.sy) + (size_t)(lev - 1) * plane;
  ZGroup<TZ> zq[PF];
  TZ zl[PF];
  T sq[PF];
  int zqo[PF];                               // queued rows' offsets and mirroring masks
  int zqm[PF];
  auto zload = [&](int y, int k) {
    bool par;
    const int q = cpos(y, sb, &par) * nf + zc;
    zqo[k] = q;
    zqm[k] = par ? (int)0x80000000 : 0;
    if (!TOP) sq[k] = sin[q];                // s_l at (y, mx), mirrored like z
    if (fresh) return;                       // z_in = 0: the queue keeps its zeros
    const uint4* src = reinterpret_cast<const uint4*>(zin + (gbase + 8 * q));
#pragma unroll
    for (int v = 0; v < NV; ++v) zq[k].v[v] = src[v];
    if (TOP) zl[k] = zin[lbase + q];
  };
#pragma unroll
  for (int k = 0; k < PF; ++k) {
#pragma unroll
    for (int v = 0; v < NV; ++v) zq[k].v[v] = make_uint4(0, 0, 0, 0);
    zl[k] = TZ(0.0f);
    zload(yc0 + k, k);
  }
  cp_wait<0>();
  __syncwarp();
  auto hrow = [&](int y, T (&h)[3]) {
    const T* r = ccol + (y - (ty0 - 2)) * G::CW;
    f3_hrow(r[-1], r[0], r[1], h);
  };
  // register rings: slot of row y - 1 is the step's phase, of y the next, of
  // y + 1 the one after
  T hr[3][3], pr[3][3];
  T hs[3] = {T(0), T(0), T(0)};              // horizontally filtered s_l rows
  hrow(yc0 - 1, hr[0]);
  hrow(yc0, hr[1]);
#pragma unroll
  for (int j = 0; j < 3; ++j) pr[0][j] = pr[1][j] = pr[2][j] = T(0);
  auto step = [&](int y, int ph) {
    const int ia = ph, ib = (ph + 1) % 3, ic = (ph + 2) % 3, kq = ph % PF;
    hrow(y + 1, hr[ic]);
    const bool own = own_c && (unsigned)(y - seg_lo) < own_rows;
    const int zwo = zqo[kq];
    ZGroup<TZ> zo;
    TZ zlo = TZ(0.0f);
    f3_row<TOP, true, T, TZ>(hr[ia], hr[ib], hr[ic], zq[kq], zl[kq], zqm[kq], mcol, mu, zo, zlo, pr[ia],
                       pr[ib], pr[ic]);
    if (own) {
      uint4* dz = reinterpret_cast<uint4*>(zout + (gbase + 8 * zwo));
#pragma unroll
      for (int v = 0; v < NV; ++v) dz[v] = zo.v[v];
      if (TOP) zout[lbase + zwo] = zlo;
    }
    if (!TOP) {
      const T sv = sq[kq];
      hs[ic] = T(0.25) * (__shfl_up_sync(FULL, sv, 1) + __shfl_down_sync(FULL, sv, 1)) + T(0.5) * sv;
    }
    if (y + PF < yc1) zload(y + PF, kq);
    {
      const int ya = y + PF + LV_L2_AHEAD;     // z (and s_l) lines further ahead into L2
      if (ya < yc1) {
        bool par;
        const int qa = cpos(ya, sb, &par) * nf + zc;
        if (!fresh) {
          prefetch_l2(zin + (gbase + 8 * qa));
          if (TOP) prefetch_l2(zin + (lbase + qa));
        }
        if (!TOP) prefetch_l2(sin + qa);
      }
    }
    // row y - 1 is complete
    const int r = y - 1;
    T A, B, C;
    f3_abc<TZ>(pr[ia], A, B, C);
    T out = B + __shfl_down_sync(FULL, A, 1) + __shfl_up_sync(FULL, C, 1);
    if (r >= seg_lo && own_c) {
      // (b0 x b0)^T s_l at (r, mx): rows r - 1, r, r + 1 = y
      if (!TOP) out += T(0.25) * (hs[ia] + hs[ic]) + T(0.5) * hs[ib];
      dst[(size_t)PO.pos(sb + dp * r) * nf + dcol] = out;
    }
  };
#pragma unroll 1
  for (int y = yc0; y < yc1; y += 3) {
#pragma unroll
    for (int k = 0; k < 3; ++k)
      if (y + k < yc1) step(y + k, k);
  }
}

#ifndef MLBA_BODIES_ONLY  // launchers: not in the persistent kernel's unit
int lev_tiles(int nf, int lev, int seg) {
  const int dp = 1 << (lev - 1);
  int tx, ty;
  lev_tile_grid(nf, dp, seg, &tx, &ty);
  return dp * dp * tx * ty;
}
// rows per CTA of the low-pass chain: 8 where one row per CTA gives more CTAs than
// fit the chip (8 of 256 threads per SM)
int lowpass_rows(int nf) { return nf > 152 * 8 ? 8 : 1; }
int lowpass_blocks(int nf, int levels) {
  int most = 0;
  for (int l = 1; l < levels; ++l) {
    const int d = 1 << (l - 1), m = Poly(nf, d).count_max(), rb = lowpass_rows(nf);
    most = std::max(most, d * ((m + rb - 1) / rb));
  }
  return most;
}

// level kernel of a segment height (32 rows: FP64 only)
template <typename T, typename TZ, bool TOP>
const void* lev_kernel(int seg) {
  if (seg == 4) return (const void*)k_frame_lev<T, TZ, TOP, 4>;
  if (seg == 8) return (const void*)k_frame_lev<T, TZ, TOP, 8>;
  if constexpr (sizeof(T) == 8)
    if (seg == 32) return (const void*)k_frame_lev<T, TZ, TOP, 32>;
  return (const void*)k_frame_lev<T, TZ, TOP, 16>;
}

template <typename T, typename TZ>
void launch_frame_levels(const Prob* probs, State* states, const int2* items, const int* sec,
                         int levels, int seg, int u_slot, int f_slot, const void* zin, void* zout,
                         double op_mu, cudaStream_t s) {
  // sec: (offset, count) of the fold, low-pass and level-L .. level-1 sections
  if (u_slot < 0 && sec[1] > 0) launch_vec<T>(VEC_FOLD, probs, states, items + sec[0], sec[1], 0, s);
  // low-pass chain: the problems with one row per CTA, then those with 8
  for (int l = 1; l < levels; ++l) {
    if (sec[3] > 0) k_lowpass<T, 1><<<sec[3], LP_THREADS, 0, s>>>(probs, states, items + sec[2], l, u_slot);
    const int o8 = sec[2 * (FRAME_SECTIONS - 1)], n8 = sec[2 * (FRAME_SECTIONS - 1) + 1];
    if (n8 > 0) k_lowpass<T, 8><<<n8, LP_THREADS, 0, s>>>(probs, states, items + o8, l, u_slot);
  }
  for (int k = 0; k < levels; ++k) {
    int lev = levels - k;
    const int off = sec[4 + 2 * k], cnt = sec[5 + 2 * k];
    if (cnt <= 0) continue;
    const int2* it = items + off;
    void* args[] = {&probs, &states, &it, &lev, &u_slot, &f_slot, &zin, &zout, &op_mu};
    const size_t sm = (size_t)LV<32>::CW * (seg + 4) * sizeof(T);
    cudaLaunchKernel(lev == levels ? lev_kernel<T, TZ, true>(seg) : lev_kernel<T, TZ, false>(seg), dim3(cnt),
                     dim3(32), args, sm, s);
  }
}

int frame_tiles(int nf, int levels, int shape, int seg) {
  const int ty = seg < F3_SEG ? seg * F3_SEG_NWR : F3_SEG * F3_SHAPES[shape].nwr;
  (void)levels;
  return ((nf + F3_TX - 1) / F3_TX) * ((nf + ty - 1) / ty);
}

void frame_shape(int shape, int seg, int* tile_x, int* tile_y, int* prefetch) {
  *tile_x = F3_TX;
  *tile_y = seg < F3_SEG ? seg * F3_SEG_NWR : F3_SEG * F3_SHAPES[shape].nwr;
  *prefetch = F3_SHAPES[shape].ring > 0 ? F3_SHAPES[shape].ring : F3_SHAPES[shape].pf;
}

// raise when the sweep changes so that shapes may rank differently
constexpr unsigned F3_SWEEP_VERSION = 2;
unsigned frame_shapes_id() {
  unsigned h = 2166136261u ^ F3_SWEEP_VERSION;
  for (const F3Shape& s : F3_SHAPES)
    for (int v : {s.nwr, s.pf, s.ring}) h = (h ^ (unsigned)v) * 16777619u;
  return h;
}

// Planar (band-major) <-> internal z layout (z_index), elements E of 2, 4 or 8
// bytes.  A thread moves one pixel's 8 bands of a level: its accesses to the
// planes are consecutive along the warp, its group is one or more 16-byte
// words (a whole sector or more for 4- and 8-byte elements wherever the
// polyphase order puts it); then the low-pass plane.  HBM-bound: 751^2, L = 2,
// FP32 (2 x 38 MB): 15 us in, 12 us out; element by element it took 42 each.
template <typename E, bool TO_INTERNAL>
__global__ void __launch_bounds__(256)
k_zlayout(E* __restrict__ dst, const E* __restrict__ src, int levels, int nf) {
  union Group {
    uint4 v[8 * sizeof(E) / 16];
    E e[8];
  };
  const int plane = nf * nf;                       // nbands nf^2 < 2^31
  const int tot = (levels + 1) * plane;
  for (int i = blockIdx.x * 256 + threadIdx.x; i < tot; i += gridDim.x * 256) {
    const int l = i / plane, q = i - l * plane;    // level l + 1; l = levels: the low-pass plane
    const int y = q / nf, x = q - y * nf;
    const int lev = l < levels ? l : levels - 1;
    const Poly P(nf, levels >= 3 ? 1 << lev : 1);
    const int p = P.pos(y) * nf + P.pos(x);
    if (l == levels) {
      const int o = 8 * levels * plane;
      if (TO_INTERNAL) dst[o + p] = src[o + q]; else dst[o + q] = src[o + p];
      continue;
    }
    const int pb = 8 * l * plane + q, gb = 8 * l * plane + 8 * p;
    Group g;
    if (TO_INTERNAL) {
#pragma unroll
      for (int b = 0; b < 8; ++b) g.e[b] = src[pb + b * plane];
#pragma unroll
      for (int v = 0; v < (int)(8 * sizeof(E) / 16); ++v) reinterpret_cast<uint4*>(dst + gb)[v] = g.v[v];
    } else {
#pragma unroll
      for (int v = 0; v < (int)(8 * sizeof(E) / 16); ++v) g.v[v] = reinterpret_cast<const uint4*>(src + gb)[v];
#pragma unroll
      for (int b = 0; b < 8; ++b) dst[pb + b * plane] = g.e[b];
    }
  }
}

void launch_z_layout(void* dst, const void* src, int levels, int nf, int elem_bytes,
                     int to_grouped, cudaStream_t s) {
  const size_t tot = (size_t)(levels + 1) * nf * nf;
  const int blocks = (int)std::min<size_t>((tot + 255) / 256, 152 * 16);
  auto go = [&](auto e) {
    using E = decltype(e);
    if (to_grouped)
      k_zlayout<E, true><<<blocks, 256, 0, s>>>(static_cast<E*>(dst), static_cast<const E*>(src), levels, nf);
    else
      k_zlayout<E, false><<<blocks, 256, 0, s>>>(static_cast<E*>(dst), static_cast<const E*>(src), levels, nf);
  };
  if (elem_bytes == 8) go((unsigned long long)0);
  else if (elem_bytes == 4) go((unsigned int)0);
  else go((unsigned short)0);
}

// the kernel of one tile shape, its shared memory and its launch (FP64 has
// only shape 0); the cases follow F3_SHAPES
#define F3_SHAPE_CASES(X) \
  X(1, 1, 2, 0) X(2, 4, 2, 0) X(3, 2, 3, 0) X(4, 1, 3, 0) X(5, 2, 2, 6) X(6, 2, 2, 10) X(7, 1, 2, 12)

template <typename T, typename TZ, int L>
const void* frame3_kernel(int shape) {
  if constexpr (sizeof(T) == 8) {
    return (const void*)k_frame3<T, TZ, L, 2, 1, 0>;
  } else {
    switch (shape) {
#define X(S, NWR, PF, RING) case S: return (const void*)k_frame3<T, TZ, L, NWR, PF, RING>;
      F3_SHAPE_CASES(X)
#undef X
      default: return (const void*)k_frame3<T, TZ, L, 2, 1, 0>;
    }
  }
}
template <typename T, typename TZ, int L>
size_t frame3_smem(int shape) {
  if constexpr (sizeof(T) == 8) {
    return frame3_smem_bytes<T, TZ, L, 2, 0>();
  } else {
    switch (shape) {
#define X(S, NWR, PF, RING) case S: return frame3_smem_bytes<T, TZ, L, NWR, RING>();
      F3_SHAPE_CASES(X)
#undef X
      default: return frame3_smem_bytes<T, TZ, L, 2, 0>();
    }
  }
}
template <typename T, typename TZ, int L>
void launch_frame3_shape(int shape, int seg, const Prob* probs, State* states, const int2* items, int nitems,
                         int u_slot, int f_slot, const void* zin, void* zout, double op_mu,
                         cudaStream_t s) {
  if (seg < F3_SEG) {
    auto go = [&](auto sg) {
      constexpr int SG = decltype(sg)::value;
      k_frame3<T, TZ, L, F3_SEG_NWR, 1, 0, SG>
          <<<nitems, 32 * F3_SEG_NWR, frame3_smem_bytes<T, TZ, L, F3_SEG_NWR, 0, SG>(), s>>>(
              probs, states, items, u_slot, f_slot, zin, zout, op_mu);
    };
    if (seg == 16) go(std::integral_constant<int, 16>{});
    else if (seg == 8) go(std::integral_constant<int, 8>{});
    else go(std::integral_constant<int, 4>{});
    return;
  }
  if constexpr (sizeof(T) == 8) {
    k_frame3<T, TZ, L, 2, 1, 0><<<nitems, 64, frame3_smem_bytes<T, TZ, L, 2, 0>(), s>>>(
        probs, states, items, u_slot, f_slot, zin, zout, op_mu);
  } else {
    switch (shape) {
#define X(S, NWR, PF, RING)                                                                     \
  case S:                                                                                       \
    k_frame3<T, TZ, L, NWR, PF, RING><<<nitems, 32 * NWR, frame3_smem_bytes<T, TZ, L, NWR, RING>(), s>>>( \
        probs, states, items, u_slot, f_slot, zin, zout, op_mu);                               \
    break;
      F3_SHAPE_CASES(X)
#undef X
      default:
        k_frame3<T, TZ, L, 2, 1, 0><<<nitems, 64, frame3_smem_bytes<T, TZ, L, 2, 0>(), s>>>(
            probs, states, items, u_slot, f_slot, zin, zout, op_mu);
    }
  }
}

template <typename T, typename TZ>
void launch_frame(const Prob* probs, State* states, const int2* items, int nitems, const int* sec,
                  int u_slot, int f_slot, const void* zin, void* zout, double op_mu, int levels,
                  int shape, int seg, cudaStream_t s) {
  if (nitems <= 0) return;
  if (levels == 1)
    launch_frame3_shape<T, TZ, 1>(shape, seg, probs, states, items, nitems, u_slot, f_slot, zin, zout, op_mu, s);
  else if (levels == 2)
    launch_frame3_shape<T, TZ, 2>(shape, seg, probs, states, items, nitems, u_slot, f_slot, zin, zout, op_mu, s);
  else
    launch_frame_levels<T, TZ>(probs, states, items, sec, levels, seg, u_slot, f_slot, zin, zout, op_mu, s);
}

template <typename T, typename TZ>
cudaError_t frame_set_smem() {
  for (int sh = 0; sh < FRAME_SHAPES; ++sh) {
    cudaError_t e = cudaFuncSetAttribute(frame3_kernel<T, TZ, 1>(sh),
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)frame3_smem<T, TZ, 1>(sh));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(frame3_kernel<T, TZ, 2>(sh), cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)frame3_smem<T, TZ, 2>(sh));
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <typename T, typename TZ, int L, int SG>
const void* frame3_seg_kernel() { return (const void*)k_frame3<T, TZ, L, F3_SEG_NWR, 1, 0, SG>; }

bool is_frame_kernel(const void* func) {
  for (int sh = 0; sh < FRAME_SHAPES; ++sh) {
    const void* k[] = {frame3_kernel<float, float, 1>(sh), frame3_kernel<float, float, 2>(sh),
                       frame3_kernel<float, __nv_bfloat16, 1>(sh), frame3_kernel<float, __nv_bfloat16, 2>(sh),
                       frame3_kernel<double, double, 1>(sh), frame3_kernel<double, double, 2>(sh)};
    for (const void* f : k)
      if (f == func) return true;
  }
#define X(SG)                                                                                     \
  for (const void* f : {frame3_seg_kernel<float, float, 1, SG>(), frame3_seg_kernel<float, float, 2, SG>(), \
                        frame3_seg_kernel<float, __nv_bfloat16, 1, SG>(),                         \
                        frame3_seg_kernel<float, __nv_bfloat16, 2, SG>(),                         \
                        frame3_seg_kernel<double, double, 1, SG>(), frame3_seg_kernel<double, double, 2, SG>()}) \
    if (f == func) return true;
  X(16) X(8) X(4)
#undef X
  for (int sg = 4; sg <= 32; sg *= 2)
    for (const void* f : {lev_kernel<float, float, false>(sg), lev_kernel<float, float, true>(sg),
                          lev_kernel<float, __nv_bfloat16, false>(sg),
                          lev_kernel<float, __nv_bfloat16, true>(sg),
                          lev_kernel<double, double, false>(sg), lev_kernel<double, double, true>(sg)})
      if (f == func) return true;
  for (const void* f : {(const void*)k_lowpass<float, 1>, (const void*)k_lowpass<float, 8>,
                        (const void*)k_lowpass<double, 1>, (const void*)k_lowpass<double, 8>})
    if (f == func) return true;
  return false;
}

#define INST(T, TZ)                                                                          \
  template void launch_frame<T, TZ>(const Prob*, State*, const int2*, int, const int*, int,   \
                                    int, const void*, void*, double, int, int, int, cudaStream_t); \
  template cudaError_t frame_set_smem<T, TZ>();
INST(float, float)
INST(float, __nv_bfloat16)
INST(double, double)
#undef INST

#endif  // MLBA_BODIES_ONLY

}  // namespace mlba
