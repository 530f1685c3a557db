// pair.cu -- the product y = H x by coset arithmetic on the two halves of a configuration.
//
// Sublattice coding (Sec. III of arXiv:1804.05028) with two sublattices: when the blocks of
// the split fall into two halves A and B that every group element carries onto themselves or
// onto each other (the checkerboard halves of the four-block square clusters, the even and
// odd blocks of a chain, or simply the two blocks of a two-block split), a configuration is
// the pair (a, b) of its half patterns, and the orbit of a half pattern a is given by
//     g_a a = R(class(a))          (class representative, placed on half A)
// with g_a in H, the elements that keep the halves, and for b with g_b in the elements that
// carry half B onto half A.  Both come from one table per half, 2^m entries of 32 bits
// (m = N/2), small enough to stay in L2.
//
// Let the classes be ordered.  If class(a) <= class(b), h = g_a brings (a, b) to
//     (R(class a), k R(class b)),   k = g_a g_b^-1,
// and otherwise h = g_b to (R(class b), k R(class a)), k = g_b g_a^-1.  So the orbit is named
// by (lower class, upper class, k): no candidate scan, no comparison of images, and no search
// of the basis.  k is one lookup in the group's multiplication table (at most 2 |H|^2 bytes,
// shared memory), and the triple has the position
//     slot = off[lower] + K * upper + k
// in a vector xs that holds x in slot order, K the number of elements between the halves.
// The product first expands x into xs (one streaming pass over the slots: xs = chi(h2)
// sqrt(|Stab_j|) x_j, j the basis index and h2 the element that carry the slot's
// configuration to its representative, tabulated once per basis), then every row sums
// chi(h) xs[slot] over its antiparallel bonds.  Where that pass would outweigh the rows
// (pair_rules.h), a term reads the slot's index, its weight and x instead.
//
// Several slots may hold the same orbit: a lower class with a nontrivial stabiliser lists
// every image of the upper pattern, an upper class with one lists the same pattern under
// several k, and equal classes list both orders.  All of them receive the orbit's value, so
// any of the equivalent choices of h gives the right term and no case is treated apart.
// Slots whose configuration has another S^z or a vanishing projection hold 0.
//
// What a term costs: two half-table entries, one byte and one word from shared memory and one
// gather of xs, 70 thread instructions in all on the 6x6 sector; the two-level search executed
// 596 and 10 dependent loads.  One lane owns one row: without data-dependent searches the lanes
// of a warp differ only in their number of antiparallel bonds.  Every y_i is written once, no
// atomics, fixed summation order.
//
// Measured (GB300, per product, against the search kernels): 6x6 sector, 3.2e7 rows, fp32
// 62.8 -> 8.05 ms, fp64 64.1 -> 9.6 ms; 40 sites, 8.6e8 rows, fp32 841 -> 179 ms; 2.6e6 complex
// fp64 rows 9.8 -> 1.27 ms.  pair_rows_kernel is held by several limits at once: of their peaks
// the L1 data pipe 65 to 70%, instruction issue 44 to 60%, the requests to L2 36% (66% where
// every term crosses the halves), DRAM 7 to 11%;
// every term across the halves is one 32-byte sector from L2.
#include "sced_internal.cuh"
#include "dfloat.cuh"
#include "character.h"
#include "pair_rules.h"
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <type_traits>
#include <vector>

namespace {

template <typename V> struct Pv;
template <> struct Pv<double> { using A = double; static constexpr bool cplx = false; };
template <> struct Pv<float> { using A = float; static constexpr bool cplx = false; };
template <> struct Pv<double2> { using A = double; static constexpr bool cplx = true; };
template <> struct Pv<float2> { using A = float; static constexpr bool cplx = true; };

// half-table entry: class << 11 | special << 10 | sign << 9 | flip << 8 | element
//   special: the class has a nontrivial stabiliser; sign: chi = -1 (real sectors);
//   flip: the element also reverses every spin; element: its number in H (times the fixed
//   swap for half B)
constexpr uint32_t kClassShift = 11;
constexpr uint32_t kSpecial = 1u << 10;
constexpr uint32_t kSignBit = 9;
constexpr uint32_t kFlip = 1u << 8;
constexpr uint32_t kElem = 255u;
constexpr int kPosShift = 27;          // pair_rows_kernel's tables: a bit of B above 16 class bits

struct PairParams {
  int n_classes;
  int cls_word[ED_MAXCLS + 1];
  int nb_cls[ED_MAXCLS];
  double jh[ED_MAXCLS], jzq[ED_MAXCLS];
  // halves of a state: (((s >> sh[0]) & bmask_hi) << n) | ((s >> sh[1]) & bmask)
  int n;
  int shA0, shA1, shB0, shB1;
  bool blocks;                   // else by nibbles, half_x[half][n_nib][16]
  const uint32_t *half_x;
  uint32_t off_hx;
  uint32_t bmask_hi, bmask;
  const uint32_t *ta, *tb;       // half tables
  const uint32_t *off;           // [n_cls] slot offset of the lower class
  uint32_t n_cls, K, h0, sel_off;
  const uint8_t *mult;           // k of (lower element, upper element)
  uint32_t mult_bytes;
  const uint2 *bond;             // per padded bond: bits flipped in A and in B
  const uint32_t *nib;
  uint32_t n_nib;
  const double *rsqrt_tab;
  uint32_t n_sq;
  const double *chi;             // complex sectors: (cos, sin) of chi per half and element
  const uint64_t *basis;
  const uint16_t *stab;
  const void *x, *xs;
  const float *xslo;             // fp32 real vectors: remainders of xs
  const uint32_t *slot_idx;      // what xs is made of: basis index and weight number of a slot,
  const uint16_t *slot_meta;     // and the weights chi sqrt(t) (fp32 vectors: pairs of words)
  const double2 *w;
  const float4 *wf;
  uint32_t lo_special, lo_same;  // which slots may have one (both 0: none)
  uint32_t n_slots;              // xs[n_slots] = 0
  void *y;
  void *ylo;
  int64_t r0, r1;
  double *partial;
  double *chunk_part;            // pair_rows_kernel: the sums of every chunk, [value][n_sums]
  uint32_t n_chunks, n_sums;
  uint32_t off_off, off_mult, off_bond, off_nib, off_rs, off_chi, off_mask, smem_bytes;
  // rows in slot order: pair_rows_kernel
  const uint32_t *low;           // [n_cls] representative of the lower class
  const uint32_t *up;            // representatives of the upper classes, from class ubase on
  const uint32_t *t_up;          // half table of the half the upper representatives lie on
  uint32_t ubase;
  const uint32_t *row0;          // [n_cls + 1] first row of the class
  const uint32_t *slice0;        // [n_cls + 1] first 32-row slice of the class
  const uint32_t *chunk_cls;     // class of every (kRowThreads / 32)th slice
  uint32_t n_slices;
  const uint32_t *row_b;         // pattern of the other half
  const uint32_t *row_i;         // basis index
  const uint16_t *row_m;         // weight of the row's configuration (meta of its slot)
  const double2 *rw;             // conj(chi) / sqrt(t) per weight
  const uint32_t *rt;            // tables of the row order, staged as they are
  uint32_t rt_words;
  int kw[ED_MAXCLS][5];          // words of class c: across [0], [1); within A [1], [2); within up [3], [4)
  uint32_t n_w, n_wa, n_hnib, m; // words, those across or within A (the first ones)
  uint32_t n_tab, n_ucls;        // upper classes tabulated per slice, upper classes in all
  int n_up;
  bool no_swap, by_popcount;
  uint32_t rt_f, rt_pos, rt_nibA, rt_nibB, rt_img, rt_left;   // offsets (words) in rt
  uint32_t off_rt, off_et, et_words;
  uint32_t *next;                // work counter, zeroed by expand_kernel
};

constexpr int kThreads = 512;          // pair_kernel
constexpr int kMinBlocks = 2;
constexpr size_t kPairMaxSmem = 110 * 1024;   // a block's tables, two blocks per SM
constexpr size_t kRowsMaxSmem = 200 * 1024;   // pair_rows_kernel, one block per SM
// pair_rows_kernel: one block of 32 warps per SM, so that the shared tables are staged once and
// all warps of the SM work on neighbouring rows (6x6 fp32 in ms, before the last steps: 9.5;
// 2 x 512 threads 10.8, 2 x 640 10.4, 3 x 512 18.3).  Terms per round, two rounds in flight, by
// the size of a vector entry (4 bytes: 1 / 2 / 3 / 4 terms 9.9 / 9.1 / 9.3 / 9.8 ms; 8 bytes: fp64
// 1 / 2 terms 9.6 / 9.9 ms; 16 bytes in one round: 2 / 3 terms 40 / 43 ms on 6.4e7 rows)
constexpr int kRowThreads = 1024;
constexpr int kSumWarps = 4;           // warps that sum a chunk's <x, y>
constexpr int kRowBlocks = 1;
constexpr int kRowU = 2;
constexpr int kRowU8 = 1;
constexpr int kRowU16 = 2;
// and rows: below 2^21 a product is a few waves of blocks, and the row tables (10 bytes per row)
// are not made
constexpr int64_t kRowOrderMinDim = 1 << 21;
// xs from which the row order pays: early where bonds within a half gather from one cluster (6x6
// sector of 4.4e6 rows, fp32, 24 MB: 1.06 ms against 1.23 in basis order), else when xs
// outgrows the L2 (30- and 32-site chains, 42 to 87 MB: 0.40 and 0.90 ms in basis order
// against 0.55 and 1.16; 40-site cluster, 122 MB: 3.39 against 2.61)
constexpr size_t kRowOrderMinBytes = (size_t)16 << 20;
constexpr size_t kRowOrderMinBytesAcross = (size_t)96 << 20;

template <typename T>
__device__ __forceinline__ void cpy(unsigned char *sm, uint32_t off, const T *g, uint32_t n) {
  T *d = reinterpret_cast<T *>(sm + off);
  for (uint32_t k = threadIdx.x; k < n; k += blockDim.x) d[k] = g[k];
}

// one row's running sum over a coupling class: fp64, or a double-float pair for fp32
// vectors (the fp64 pipe of this GPU issues at a small fraction of the fp32 rate); signs come
// in the top bit of w
__device__ __forceinline__ float with_sign(float v, uint32_t w) {
  return __uint_as_float(__float_as_uint(v) ^ (w & 0x80000000u));
}
__device__ __forceinline__ double with_sign(double v, uint32_t w) {
  return __hiloint2double(__double2hiint(v) ^ (int)(w & 0x80000000u), __double2loint(v));
}
template <typename V> struct Acc;
template <> struct Acc<double> {
  double s = 0, s2 = 0;   // two chains: fp64 results are slow to come back
  __device__ __forceinline__ void add(double v, uint32_t w) {
    const double t = s2;
    s2 = s + with_sign(v, w);
    s = t;
  }
  __device__ __forceinline__ double re() const { return s + s2; }
  __device__ __forceinline__ double im() const { return 0; }
};
template <> struct Acc<float> {
  float h = 0, l = 0;
  __device__ __forceinline__ void add(float v, uint32_t w) { df_add(h, l, with_sign(v, w)); }
  __device__ __forceinline__ void add_lo(float v, uint32_t w) { l = __fadd_rn(l, with_sign(v, w)); }
  __device__ __forceinline__ double re() const { return df_value(h, l); }
  __device__ __forceinline__ double im() const { return 0; }
};
template <> struct Acc<double2> {
  double r = 0, i = 0, r2 = 0, i2 = 0;   // two chains
  __device__ __forceinline__ void add(double2 v, uint32_t w) {
    r += with_sign(v.x, w);
    i += with_sign(v.y, w);
  }
  __device__ __forceinline__ void add(double2 v, double2 c) {
    r = fma(c.x, v.x, r);
    r2 = fma(-c.y, v.y, r2);
    i = fma(c.x, v.y, i);
    i2 = fma(c.y, v.x, i2);
  }
  __device__ __forceinline__ double re() const { return r + r2; }
  __device__ __forceinline__ double im() const { return i + i2; }
};
template <> struct Acc<float2> {
  float rh = 0, rl = 0, ih = 0, il = 0;
  __device__ __forceinline__ void add(float2 v, uint32_t w) {
    df_add(rh, rl, with_sign(v.x, w));
    df_add(ih, il, with_sign(v.y, w));
  }
  // chi v with chi given as (cos, remainder, sin, remainder): exact products
  __device__ __forceinline__ void add(float2 v, float4 c) {
    df_add_prod(rh, rl, c.x, v.x);
    df_add_prod(rh, rl, -c.z, v.y);
    rl = __fmaf_rn(c.y, v.x, __fmaf_rn(-c.w, v.y, rl));
    df_add_prod(ih, il, c.x, v.y);
    df_add_prod(ih, il, c.z, v.x);
    il = __fmaf_rn(c.y, v.y, __fmaf_rn(c.w, v.x, il));
  }
  __device__ __forceinline__ double re() const { return df_value(rh, rl); }
  __device__ __forceinline__ double im() const { return df_value(ih, il); }
};

struct PairSm {
  const uint32_t *off;
  const uint8_t *mult;
  const uint32_t *fa, *fb;   // bits flipped in A and in B, per padded bond
};

// U terms in flight: the gathered values and what their sum needs (sign or chi index)
template <typename V, int U>
struct Terms {
  V v[U];
  float vl[U];
  uint32_t w[U];
  int n;   // how many hold a term; the rest are zeros
};

// What a term gathers: its slot, what its sum needs (Terms::w), and whether the slot may hold
// an orbit with |Stab| > 1 (fp32 real vectors then add the remainder xslo)
struct Slot {
  uint32_t slot, w;
  bool lo;
};

template <bool kChi>
__device__ __forceinline__ uint32_t lower_sign(uint32_t e, bool a_low) {
  return kChi ? (e & (kElem | kFlip)) + (a_low ? 0u : 512u) : e << (31 - kSignBit);
}

// The slot of an exchanged configuration from its half-table entries.  |Stab| > 1 needs a
// stabiliser on both halves, or halves that can be exchanged (one class; the difference also
// lets a few neighbouring classes pass, whose xslo is 0).
template <bool kChi, bool kFlips>
__device__ __forceinline__ Slot slot_of(const PairParams &P, const PairSm &S, uint32_t ea, uint32_t eb) {
  const uint32_t lo = min(ea, eb), hi = max(ea, eb);
  const bool a_low = ea <= eb;
  const uint32_t mi = (lo & kElem) * P.h0 + (hi & kElem) + (a_low ? 0u : P.sel_off);
  Slot r;
  r.slot = S.off[lo >> kClassShift] + P.K * (hi >> kClassShift) + S.mult[mi];
  if (kFlips) r.slot += ((lo ^ hi) & kFlip) ? P.h0 : 0u;
  r.w = lower_sign<kChi>(lo, a_low);
  r.lo = (lo & hi & P.lo_special) || hi - lo < P.lo_same;
  return r;
}

template <typename V, bool kChi, int U>
__device__ __forceinline__ void pair_sum(const Terms<V, U> &t, const unsigned char *chi_sm, Acc<V> &acc) {
#pragma unroll
  for (int u = 0; u < U; u++) {
    // adding zeros is harmless, but not free where it goes to the fp64 pipe
    if (sizeof(typename Pv<V>::A) == 8 && u >= t.n) continue;
    if constexpr (kChi) {
      if constexpr (sizeof(typename Pv<V>::A) == 4)
        acc.add(t.v[u], reinterpret_cast<const float4 *>(chi_sm)[t.w[u]]);
      else
        acc.add(t.v[u], reinterpret_cast<const double2 *>(chi_sm)[t.w[u]]);
    } else {
      acc.add(t.v[u], t.w[u]);
      if constexpr (std::is_same<V, float>::value) acc.add_lo(t.vl[u], t.w[u]);
    }
  }
}

template <typename V>
__device__ __forceinline__ V no_value() {
  if constexpr (Pv<V>::cplx) { V z; z.x = 0; z.y = 0; return z; } else { return V(0); }
}

template <typename V, int U>
__device__ __forceinline__ void no_terms(Terms<V, U> &t) {
  t.n = 0;
#pragma unroll
  for (int u = 0; u < U; u++) {
    t.v[u] = no_value<V>();
    t.vl[u] = 0.f;
    t.w[u] = 0u;
  }
}

// What xs holds of v = x_j: w(mt) v with w = chi sqrt(t), mt 0 being w = 1.  fp32 vectors take the
// weights as pairs of fp32 words, (re, its remainder, im, its remainder): in fp64 the products
// and conversions kept the fp64 pipe 85% busy (expansion of the 6x6 sector's 4.8e7 slots: 0.54
// ms).  Real ones give the rounding's remainder in lo, so that a weight sqrt(t) costs no precision.
template <typename V>
__device__ __forceinline__ V weighted(V v, uint32_t mt, const double2 *w, const float4 *wf, float &lo) {
  constexpr bool kF = sizeof(typename Pv<V>::A) == 4;
  lo = 0.f;
  if (!mt) return v;
  if constexpr (kF && Pv<V>::cplx) {
    const float4 c = __ldg(wf + mt);
    const V u = v;
    float h = 0.f, l = 0.f;
    df_sub_scaled(h, l, -c.x, -c.y, u.x);
    df_sub_scaled(h, l, c.z, c.w, u.y);
    v.x = df_round(h, l);
    h = l = 0.f;
    df_sub_scaled(h, l, -c.x, -c.y, u.y);
    df_sub_scaled(h, l, -c.z, -c.w, u.x);
    v.y = df_round(h, l);
  } else if constexpr (kF) {
    const float2 c = __ldg(reinterpret_cast<const float2 *>(wf + mt));
    const float u = v;
    v = __fmul_rn(c.x, u);
    lo = __fmaf_rn(c.y, u, __fmaf_rn(c.x, u, -v));
  } else if constexpr (Pv<V>::cplx) {
    const double2 c = __ldg(w + mt);
    const double a = c.x * v.x - c.y * v.y, b = c.x * v.y + c.y * v.x;
    v.x = a;
    v.y = b;
  } else {
    v *= __ldg(w + mt).x;
  }
  return v;
}

// Sums n terms, U at a time; gen(slots, nu) gives the next nu.  The gathers of one round are
// in flight while the round before is summed: two sets of registers taken in turn, as a copy
// from one to the other would wait for the loads.  t0 holds terms still to be summed, on
// entry and on exit, so that the gathers of one loop overlap the start of the next.
template <typename V, bool kChi, int U, bool kDirect, typename G>
__device__ __forceinline__ void pair_loop(const PairParams &P, int n, G gen, const V *xs,
                                          const unsigned char *chi_sm, Acc<V> &acc, Terms<V, U> &t0) {
  auto step = [&](Terms<V, U> &t) {
    Slot g[U];
    gen(g, n);
    t.n = n;
    if constexpr (kDirect) {
      uint32_t j[U], mt[U];
#pragma unroll
      for (int u = 0; u < U; u++) {
        const bool in = u == 0 || u < n;
        j[u] = in ? __ldg(P.slot_idx + g[u].slot) : 0xFFFFFFFFu;
        mt[u] = in ? __ldg(P.slot_meta + g[u].slot) : 0u;
        t.w[u] = g[u].w;
      }
#pragma unroll
      for (int u = 0; u < U; u++) {
        t.v[u] = no_value<V>();
        float lo = 0.f;
        if (j[u] != 0xFFFFFFFFu) t.v[u] = weighted<V>(__ldg(xs + j[u]), mt[u], P.w, P.wf, lo);
        t.vl[u] = g[u].lo ? lo : 0.f;
      }
    } else {
#pragma unroll
      for (int u = 0; u < U; u++) {
        const uint32_t slot = u == 0 || u < n ? g[u].slot : P.n_slots;   // xs[n_slots] = 0
        t.w[u] = g[u].w;
        t.v[u] = __ldg(xs + slot);
        t.vl[u] = 0.f;
        if constexpr (std::is_same<V, float>::value) {
          if (g[u].lo) t.vl[u] = __ldg(P.xslo + slot);
        }
      }
    }
    n -= U;
  };
  if constexpr (sizeof(V) == 16 || kDirect) {
    // 16-byte values leave no registers for a second set, and the fp64 pipe is the bound
    // (pair_kernel on 2.6e6 complex rows: 1.32 ms, with two sets 1.41); direct terms need
    // their index and weight in registers and wait for them in any case
    while (n > 0) {
      Terms<V, U> t1;
      step(t1);
      pair_sum<V, kChi, U>(t1, chi_sm, acc);
    }
  } else {
    while (n > 0) {
      Terms<V, U> t1;
      step(t1);
      pair_sum<V, kChi, U>(t0, chi_sm, acc);
      if (n > 0) step(t0); else no_terms(t0);
      pair_sum<V, kChi, U>(t1, chi_sm, acc);
    }
  }
}

// The tables of the product in shared memory (not the masks and, in pair_rows_kernel, the
// per-warp tables).
template <typename V, bool kChi>
__device__ __forceinline__ PairSm pair_stage(const PairParams &P, unsigned char *sm) {
  cpy(sm, P.off_off, P.off, P.n_cls);
  cpy(sm, P.off_mult, reinterpret_cast<const uint32_t *>(P.mult), P.mult_bytes / 4);
  const int n_words = P.cls_word[P.n_classes];
  uint32_t *fa = reinterpret_cast<uint32_t *>(sm + P.off_bond), *fb = fa + n_words * 32;
  for (int k = threadIdx.x; k < n_words * 32; k += blockDim.x) {
    const uint2 f = P.bond[k];
    fa[k] = f.x;
    fb[k] = f.y;
  }
  cpy(sm, P.off_rs, P.rsqrt_tab, P.n_sq);
  if constexpr (kChi) {
    // the elements there are: h0 numbers, with and without the flip bit, for either half
    for (uint32_t q = threadIdx.x; q < 4 * P.h0; q += blockDim.x) {
      const uint32_t k = q / P.h0 * 256 + q % P.h0;
      const double c = P.chi[2 * k], s = P.chi[2 * k + 1];
      if constexpr (sizeof(typename Pv<V>::A) == 4) {
        const float ch = (float)c, sh = (float)s;
        reinterpret_cast<float4 *>(sm + P.off_chi)[k] = make_float4(ch, (float)(c - (double)ch), sh, (float)(s - (double)sh));
      } else {
        reinterpret_cast<double2 *>(sm + P.off_chi)[k] = make_double2(c, s);
      }
    }
  }
  PairSm S;
  S.off = reinterpret_cast<const uint32_t *>(sm + P.off_off);
  S.mult = sm + P.off_mult;
  S.fa = fa;
  S.fb = fb;
  return S;
}

// y_i in fp64, rounded once to the vector type; for fp32 vectors the rounding's remainder
// goes to ylo when asked, and <x, y> then uses the unrounded value
template <typename V>
__device__ __forceinline__ void pair_store(const PairParams &P, const V *x, V *y, int64_t i, double diag,
                                           double rs, double row_re, double row_im, double &dot_re,
                                           double &dot_im) {
  using A_ = typename Pv<V>::A;
  constexpr bool kF = sizeof(A_) == 4;
  if constexpr (!Pv<V>::cplx) {
    const double xi = (double)__ldcs(x + i);   // read once: keep it from pushing xs out of L2
    const double yd = diag * xi + row_re * rs;
    const A_ yi = (A_)yd;
    __stcs(y + (i - P.r0), yi);
    if (kF && P.ylo) reinterpret_cast<float *>(P.ylo)[i - P.r0] = (float)(yd - (double)yi);
    if (P.partial) dot_re += xi * (kF && P.ylo ? yd : (double)yi);
  } else {
    const V xv = __ldcs(x + i);
    const double yr = diag * (double)xv.x + row_re * rs;
    const double yim = diag * (double)xv.y + row_im * rs;
    V yv;
    yv.x = (A_)yr;
    yv.y = (A_)yim;
    y[i - P.r0] = yv;
    double ur = (double)yv.x, ui = (double)yv.y;
    if (kF && P.ylo) {
      float2 l;
      l.x = (float)(yr - ur);
      l.y = (float)(yim - ui);
      reinterpret_cast<float2 *>(P.ylo)[i - P.r0] = l;
      ur = yr;
      ui = yim;
    }
    if (P.partial) {
      dot_re += (double)xv.x * ur + (double)xv.y * ui;
      dot_im += (double)xv.x * ui - (double)xv.y * ur;
    }
  }
}

__device__ __forceinline__ double warp_sum(double d) {
  for (int o = 16; o > 0; o >>= 1) d += __shfl_down_sync(0xFFFFFFFFu, d, o);
  return d;
}

// per-block sums of n values per thread (kMode 0: <x, y>, real and imaginary part; kMode 1: the
// classes) in a fixed order
template <int kT>
__device__ __forceinline__ void pair_dot(const PairParams &P, const double *v, int n) {
  if (!P.partial) return;
  __shared__ double red[kT / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int part = 0; part < n; part++) {
    double d = warp_sum(v[part]);
    __syncthreads();
    if (lane == 0) red[wid] = d;
    __syncthreads();
    if (wid == 0) {
      d = warp_sum(lane < kT / 32 ? red[lane] : 0.0);
      if (lane == 0) P.partial[part * gridDim.x + blockIdx.x] = d;
    }
  }
}

// Re conj(x_i) (H_c x)_i with unit exchange: the row's share of <x|H_c|x>; w is the weight
// conj(chi) / sqrt(t) that takes the row's sum to the basis state
template <typename V>
__device__ __forceinline__ double class_share(const V *x, int64_t i, double diag, double jh, double2 w, double re,
                                              double im) {
  if constexpr (!Pv<V>::cplx) {
    const double xi = (double)x[i];
    return xi * (diag * xi + jh * w.x * re);
  } else {
    const V xv = x[i];
    const double xr = (double)xv.x, xi = (double)xv.y;
    return diag * (xr * xr + xi * xi) + jh * (xr * (w.x * re - w.y * im) + xi * (w.x * im + w.y * re));
  }
}

// the next antiparallel bond of a row whose masks of the words of one class lie at mask_s
template <int kT>
__device__ __forceinline__ int next_bond(uint32_t &m, int &wd, int w0, const uint32_t *mask_s) {
  while (m == 0) m = mask_s[(++wd - w0) * kT];
  const int k = wd * 32 + __ffs(m) - 1;
  m &= m - 1;
  return k;
}

// Rows in basis order: any range of rows, and sectors whose xs stays in L2.  kDirect: no xs; a term
// reads its slot's index, its weight and x one after the other (see pair_rules.h for when).
template <typename V, bool kChi, bool kFlips, int kMode, bool kDirect>
__global__ void __launch_bounds__(kThreads, kMinBlocks) pair_kernel(const __grid_constant__ PairParams P) {
  constexpr bool kC = Pv<V>::cplx;
  constexpr int U = kDirect ? 4 : 2;
  extern __shared__ __align__(16) unsigned char sm[];
  const PairSm S = pair_stage<V, kChi>(P, sm);
  cpy(sm, P.off_nib, P.nib, (uint32_t)P.cls_word[P.n_classes] * P.n_nib * 16);
  if (!P.blocks) cpy(sm, P.off_hx, P.half_x, P.n_nib * 32);
  __syncthreads();
  const uint32_t *hx = reinterpret_cast<const uint32_t *>(sm + P.off_hx);
  const uint32_t *nibs = reinterpret_cast<const uint32_t *>(sm + P.off_nib);
  const double *rsd = reinterpret_cast<const double *>(sm + P.off_rs);
  uint32_t *mask_s = reinterpret_cast<uint32_t *>(sm + P.off_mask) + threadIdx.x;
  const V *xs = reinterpret_cast<const V *>(kDirect ? P.x : P.xs);
  double dot[kMode == 1 ? ED_MAXCLS : 2] = {};
  const int64_t stride = (int64_t)gridDim.x * kThreads;
  for (int64_t i = P.r0 + (int64_t)blockIdx.x * kThreads + threadIdx.x; i < P.r1; i += stride) {
    const uint64_t s = __ldcs(reinterpret_cast<const unsigned long long *>(P.basis) + i);
    uint32_t A = 0, B = 0;
    if (P.blocks) {
      A = (((uint32_t)(s >> P.shA0) & P.bmask_hi) << P.n) | ((uint32_t)(s >> P.shA1) & P.bmask);
      B = (((uint32_t)(s >> P.shB0) & P.bmask_hi) << P.n) | ((uint32_t)(s >> P.shB1) & P.bmask);
    } else {
      for (uint32_t q = 0; q < P.n_nib; q++) {
        const uint32_t v = (uint32_t)(s >> (4 * q)) & 15u;
        A |= hx[q * 16 + v];
        B |= hx[(P.n_nib + q) * 16 + v];
      }
    }
    double diag = 0.0, row_re = 0.0, row_im = 0.0;
    for (int c = 0; c < P.n_classes; c++) {
      const int w0 = P.cls_word[c], w1 = P.cls_word[c + 1];
      int nanti = 0;
      for (int wd = w0; wd < w1; wd++) {
        uint32_t m = 0;
        const uint32_t *nw = nibs + (uint32_t)wd * P.n_nib * 16;
        for (uint32_t q = 0; q < P.n_nib; q++) m ^= nw[q * 16 + (uint32_t)((s >> (4 * q)) & 15u)];
        nanti += __popc(m);
        mask_s[(wd - w0) * kThreads] = m;
      }
      Acc<V> acc;
      Terms<V, U> pend;
      no_terms(pend);
      int wd = w0;
      uint32_t m = w0 < w1 ? mask_s[0] : 0u;
      auto gen = [&](Slot (&g)[U], int nu) {
        int kb = 0;
        uint32_t ea[U], eb[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
          if (u == 0 || u < nu) kb = next_bond<kThreads>(m, wd, w0, mask_s);
          ea[u] = __ldg(P.ta + (A ^ S.fa[kb]));
          eb[u] = __ldg(P.tb + (B ^ S.fb[kb]));
        }
#pragma unroll
        for (int u = 0; u < U; u++) g[u] = slot_of<kChi, kFlips>(P, S, ea[u], eb[u]);
      };
      pair_loop<V, kChi, U, kDirect>(P, nanti, gen, xs, sm + P.off_chi, acc, pend);
      pair_sum<V, kChi, U>(pend, sm + P.off_chi, acc);
      const double dg = P.jzq[c] * (double)(P.nb_cls[c] - 2 * nanti);
      if constexpr (kMode == 1) {
        dot[c] += class_share(reinterpret_cast<const V *>(P.x), i, dg, P.jh[c],
                              make_double2(rsd[__ldg(P.stab + i)], 0.0), acc.re(), acc.im());
      } else {
        row_re += P.jh[c] * acc.re();
        if constexpr (kC) row_im += P.jh[c] * acc.im();
        diag += dg;
      }
    }
    if constexpr (kMode == 0)
      pair_store<V>(P, reinterpret_cast<const V *>(P.x), reinterpret_cast<V *>(P.y), i, diag,
                    rsd[__ldcs(P.stab + i)], row_re, row_im, dot[0], dot[1]);
  }
  pair_dot<kThreads>(P, dot, kMode == 1 ? P.n_classes : kC ? 2 : 1);
}

// Rows in slot order, for products whose xs is larger than the L2 keeps.  In basis order the
// gathers of xs are random over the whole vector: on the 6x6 sector 59 bytes of DRAM traffic
// per gathered fp32 value and 77% of the DRAM's peak (23.8 ms).  Rows that share the lower half
// A reach few places: the exchanged half A' takes at most one value per bond, and while
// class(A') stays the lower one the gather falls into that class's block of slots.  The GPU
// works on one or two lower classes at a time, whose blocks (10 to 20 MB on that sector) stay
// in L2.  That needs all SMs at the same place: blocks take slices from a counter (with a fixed
// stride the SMs drift apart by dozens of classes: 120 GB of DRAM reads per product, now 4).
//
// In slot order the rows of one upper class c lie together: b = k R(c), all k.  Terms within a
// half keep the other class: within A the 32 rows of a warp gather from one cluster of K slots
// (c(A'), c), and within the upper half, with the bonds taken in the frame of R(c) (the
// bonds are invariant under the group), from one cluster (c_A, c') -- half the terms of a
// J1-J2 row, a few cache lines instead of 32 sectors.  The half table is read at R(c) with
// one or two bits flipped, the same few entries for all rows of the cluster:
//     g_B b = R(c),  u' = R(c) with g_B's image of the flipped bits,  g_u u' = R(c')
// makes g_u g_B the element that carries the exchanged half to R(c'), its number from the
// left multiplication table of H.
template <typename V, bool kChi, bool kFlips, int kMode>
__global__ void __launch_bounds__(kRowThreads, kRowBlocks) pair_rows_kernel(const __grid_constant__ PairParams P) {
  constexpr bool kC = Pv<V>::cplx;
  constexpr int U = sizeof(V) == 16 ? kRowU16 : sizeof(V) == 8 ? kRowU8 : kRowU;
  extern __shared__ __align__(16) unsigned char sm[];
  const PairSm S = pair_stage<V, kChi>(P, sm);
  cpy(sm, P.off_rt, P.rt, P.rt_words);
  __syncthreads();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint32_t *rt = reinterpret_cast<const uint32_t *>(sm + P.off_rt);
  const uint32_t *nibA = rt + P.rt_nibA, *nibB = rt + P.rt_nibB;
  const uint32_t *fw = rt + P.rt_f;                                        // bits of A, or of R(c)
  const uint8_t *pos = reinterpret_cast<const uint8_t *>(rt + P.rt_pos);   // bit of B (across)
  const uint8_t *img = reinterpret_cast<const uint8_t *>(rt + P.rt_img);   // its image under g_B
  const uint8_t *left = reinterpret_cast<const uint8_t *>(rt + P.rt_left);
  uint32_t *mask_s = reinterpret_cast<uint32_t *>(sm + P.off_mask) + threadIdx.x;
  // tables of the warp: per bond across the halves or within A, the entry of A' and the slot
  // offset of its class; masks of A by word; for the slice's first upper classes c (n_tab of
  // them), per bit of R(c) the entry with it flipped, and per bond within the upper half that
  // with its two bits flipped
  uint32_t *et = reinterpret_cast<uint32_t *>(sm + P.off_et) + wid * P.et_words, *eo = et + P.n_wa * 32;
  uint32_t *ma = eo + P.n_wa * 32, *eup = ma + P.n_wa;
  const uint32_t n_up2 = (P.n_w - P.n_wa) * 32, n_eup = P.m + n_up2;
  const V *xs = reinterpret_cast<const V *>(P.xs);
  double dot[kMode == 1 ? ED_MAXCLS : 2] = {};
  uint32_t cur = 0xFFFFFFFFu, e_low = 0, off_low = 0;
  bool st_in = false, st_across = false;
  __shared__ uint32_t chunk_s;
  constexpr int kDots = kC ? 2 : 1;
  __shared__ double red[kMode == 1 ? ED_MAXCLS : 1][kRowThreads / 32];
  uint32_t chunk = 0xFFFFFFFFu;
  for (;;) {
    // which block works on a chunk differs from call to call, so <x, y> is summed by chunk:
    // the same bits every time.  The lanes' shares go through the masks' words to kSumWarps
    // warps: fp64 additions are what this costs (6x6 sector, fp32, product with <x, y>: 8.36 ms;
    // 8.24 with one sum per thread over whatever chunks it gets, 8.57 with every warp's 32 lanes
    // summed by shuffles)
    const bool sums = P.partial && chunk != 0xFFFFFFFFu;
    if (sums) {
      if constexpr (kMode == 1) {
#pragma unroll
        for (int part = 0; part < ED_MAXCLS; part++) {
          if (part >= P.n_classes) break;
          const double d = warp_sum(dot[part]);
          if (lane == 0) red[part][wid] = d;
          dot[part] = 0.0;
        }
      } else {
#pragma unroll
        for (int part = 0; part < kDots; part++) {
          mask_s[2 * part * kRowThreads] = (uint32_t)__double2loint(dot[part]);
          mask_s[(2 * part + 1) * kRowThreads] = (uint32_t)__double2hiint(dot[part]);
          dot[part] = 0.0;
        }
      }
    }
    // taken when it is worked on: a chunk taken ahead spreads the blocks over more classes
    // (fp64 on the 6x6 sector 10.5 -> 11.0 ms)
    __syncthreads();
    if (threadIdx.x == 0) chunk_s = atomicAdd(P.next, 1u);
    if constexpr (kMode == 1) {
      if (sums && wid == 1) {
        for (int part = 0; part < P.n_classes; part++) {
          const double d = warp_sum(red[part][lane]);
          if (lane == 0) P.chunk_part[(size_t)part * P.n_sums + chunk] = d;
        }
      }
    } else if (sums && wid >= 1 && wid <= kSumWarps) {
      constexpr int kRows = kRowThreads / kSumWarps;
      const uint32_t *w = reinterpret_cast<const uint32_t *>(sm + P.off_mask) + (wid - 1) * kRows + lane;
#pragma unroll
      for (int part = 0; part < kDots; part++, w += 2 * kRowThreads) {
        double d = 0.0;
#pragma unroll
        for (int q = 0; q < kRows; q += 32) d += __hiloint2double((int)w[kRowThreads + q], (int)w[q]);
        d = warp_sum(d);
        if (lane == 0) P.chunk_part[(size_t)part * P.n_sums + chunk * kSumWarps + wid - 1] = d;
      }
    }
    __syncthreads();
    chunk = chunk_s;
    if (chunk >= P.n_chunks) break;
    const uint32_t sl = chunk * (kRowThreads / 32) + wid;
    if (sl >= P.n_slices) continue;
    uint32_t lo = __ldg(P.chunk_cls + chunk);   // the class of the chunk's first slice
    while (__ldg(P.slice0 + lo + 1) <= sl) lo++;
    if (lo != cur) {
      cur = lo;
      const uint32_t A = __ldg(P.low + lo);
      e_low = __ldg(P.ta + A);
      off_low = S.off[lo];
      // where the lower class is known beforehand: classes are ordered by their number of up
      // spins (the smaller of up and down spins with spin flips, where nothing is known); an
      // exchange across the halves moves one spin.  Halves that nothing exchanges: always A.
      const int na = __popc(A), nb = P.n_up - na;
      st_in = P.no_swap || (P.by_popcount && na < nb);
      st_across = P.no_swap || (P.by_popcount && na + 1 < nb - 1);
      __syncwarp();
      for (uint32_t k = lane; k < P.n_wa * 32; k += 32) {
        const uint32_t e = __ldg(P.ta + (A ^ fw[k]));
        et[k] = e | (uint32_t)pos[k] << kPosShift;
        eo[k] = S.off[e >> kClassShift];
      }
      for (uint32_t wd = lane; wd < P.n_wa; wd += 32) {
        uint32_t m = 0;
        for (uint32_t q = 0; q < P.n_hnib; q++) m ^= nibA[(wd * P.n_hnib + q) * 16 + ((A >> (4 * q)) & 15u)];
        ma[wd] = m;
      }
      __syncwarp();
    }
    const uint32_t rw0 = __ldg(P.row0 + lo) + (sl - __ldg(P.slice0 + lo)) * 32;
    const int n_row = (int)min(32u, __ldg(P.row0 + lo + 1) - rw0);
    const uint32_t r = rw0 + min(lane, n_row - 1);   // lanes past the end repeat the last row
    const uint32_t B = __ldcs(P.row_b + r);
    const uint32_t e_up = __ldg(P.tb + B);
    const uint32_t c_up = (e_up >> kClassShift) - P.ubase, c0 = __shfl_sync(0xFFFFFFFFu, c_up, 0);
    const uint32_t R = __ldg(P.up + c_up);
    __syncwarp();
    for (uint32_t t = 0; t < P.n_tab; t++) {
      const uint32_t Rt = __ldg(P.up + min(c0 + t, P.n_ucls - 1));
      uint32_t *e = eup + t * n_eup;
      for (uint32_t q = lane; q < P.m; q += 32) e[q] = __ldg(P.t_up + (Rt ^ (1u << q)));
      for (uint32_t k = lane; k < n_up2; k += 32) e[P.m + k] = __ldg(P.t_up + (Rt ^ fw[P.n_wa * 32 + k]));
    }
    __syncwarp();
    // more classes than that occur where classes have stabilisers, and so fewer rows
    const bool all_tab = __all_sync(0xFFFFFFFFu, c_up - c0 < P.n_tab);
    if (lane >= n_row) continue;
    const uint32_t *eup_r = eup + (c_up - c0) * n_eup, *eu_r = eup_r + P.m;
    const uint32_t yB = e_up & kElem;
    const uint8_t *img_r = img + yB * P.m, *left_y = left + yB;
    const uint32_t slot_up = P.K * (e_up >> kClassShift);
    double diag = 0.0, row_re = 0.0, row_im = 0.0;
    // the entry of the exchanged upper half from that of u' = R(c) with its bits flipped
    auto carried = [&](uint32_t eu) {
      return ((eu ^ (e_up & (kFlip | 1u << kSignBit))) & ~kElem) | left_y[(eu & kElem) * P.h0];
    };
    for (int c = 0; c < P.n_classes; c++) {
      int nanti = 0;
      Acc<V> acc;
      Terms<V, U> pend;
      no_terms(pend);
      {   // bonds across the halves
        const int w0 = P.kw[c][0], w1 = P.kw[c][1];
        int n = 0;
        for (int wd = w0; wd < w1; wd++) {
          uint32_t m = ma[wd];
          const uint32_t *nw = nibB + (uint32_t)wd * P.n_hnib * 16;
          for (uint32_t q = 0; q < P.n_hnib; q++) m ^= nw[q * 16 + ((B >> (4 * q)) & 15u)];
          n += __popc(m);
          mask_s[(wd - w0) * kRowThreads] = m;
        }
        nanti += n;
        int wd = w0;
        uint32_t m = w0 < w1 ? mask_s[0] : 0u;
        auto across = [&](auto entry, auto is_static) {
          auto gen = [&](Slot (&g)[U], int nu) {
            int kb = 0;
            uint32_t e[U], off_a[U], eu[U];
#pragma unroll
            for (int u = 0; u < U; u++) {
              if (u == 0 || u < nu) kb = next_bond<kRowThreads>(m, wd, w0, mask_s);
              e[u] = et[kb];
              if constexpr (decltype(is_static)::value) off_a[u] = eo[kb];
              eu[u] = entry(img_r[e[u] >> kPosShift]);
            }
#pragma unroll
            for (int u = 0; u < U; u++) {
              if constexpr (decltype(is_static)::value) {   // class(A') is the lower one
                const uint32_t k = left_y[(eu[u] & kElem) * P.h0];
                g[u].slot = off_a[u] + P.K * (eu[u] >> kClassShift) + S.mult[(e[u] & kElem) * P.h0 + k];
                g[u].w = lower_sign<kChi>(e[u], true);
                g[u].lo = e[u] & eu[u] & P.lo_special;
              } else {
                g[u] = slot_of<kChi, kFlips>(P, S, e[u] & ((1u << kPosShift) - 1u), carried(eu[u]));
              }
            }
          };
          pair_loop<V, kChi, U, false>(P, n, gen, xs, sm + P.off_chi, acc, pend);
        };
        auto from_table = [&](uint32_t q) { return eup_r[q]; };
        auto from_memory = [&](uint32_t q) { return __ldg(P.t_up + (R ^ (1u << q))); };
        if (!all_tab) across(from_memory, std::false_type());
        else if (!kFlips && st_across) across(from_table, std::true_type());
        else across(from_table, std::false_type());
      }
      // bonds within A
      for (int wd = P.kw[c][1]; wd < P.kw[c][2]; wd++) {
        uint32_t m = ma[wd];
        const int n = __popc(m);
        nanti += n;
        auto within = [&](auto is_static) {
          auto gen = [&](Slot (&g)[U], int nu) {
            int kb = 0;
#pragma unroll
            for (int u = 0; u < U; u++) {
              if (u == 0 || u < nu) {
                kb = wd * 32 + __ffs(m) - 1;
                m &= m - 1;
              }
              const uint32_t e = et[kb];
              if constexpr (decltype(is_static)::value) {
                g[u].slot = eo[kb] + slot_up + S.mult[(e & kElem) * P.h0 + yB];
                g[u].w = lower_sign<kChi>(e, true);
                g[u].lo = e & e_up & P.lo_special;
              } else {
                g[u] = slot_of<kChi, kFlips>(P, S, e & ((1u << kPosShift) - 1u), e_up);
              }
            }
          };
          pair_loop<V, kChi, U, false>(P, n, gen, xs, sm + P.off_chi, acc, pend);
        };
        if (!kFlips && st_in) within(std::true_type()); else within(std::false_type());
      }
      // bonds within the upper half, in the frame of R(c)
      for (int wd = P.kw[c][3]; wd < P.kw[c][4]; wd++) {
        uint32_t m = 0;
        const uint32_t *nw = nibB + (uint32_t)wd * P.n_hnib * 16;
        for (uint32_t q = 0; q < P.n_hnib; q++) m ^= nw[q * 16 + ((R >> (4 * q)) & 15u)];
        const int n = __popc(m);
        nanti += n;
        const uint32_t *eu_w = eu_r + (wd - (int)P.n_wa) * 32, *fw_w = fw + wd * 32;
        auto within = [&](auto is_static) {
          // with A unchanged and lower, k g_u^-1 for the row's own k
          const uint8_t *mk = S.mult + P.sel_off + (uint32_t)S.mult[(e_low & kElem) * P.h0 + yB] * P.h0;
          auto gen = [&](Slot (&g)[U], int nu) {
            int kb = 0;
#pragma unroll
            for (int u = 0; u < U; u++) {
              if (u == 0 || u < nu) {
                kb = __ffs(m) - 1;
                m &= m - 1;
              }
              const uint32_t eu = all_tab ? eu_w[kb] : __ldg(P.t_up + (R ^ fw_w[kb]));
              if constexpr (decltype(is_static)::value) {
                g[u].slot = off_low + P.K * (eu >> kClassShift) + mk[eu & kElem];
                g[u].w = lower_sign<kChi>(e_low, true);
                g[u].lo = e_low & eu & P.lo_special;
              } else {
                g[u] = slot_of<kChi, kFlips>(P, S, e_low, carried(eu));
              }
            }
          };
          pair_loop<V, kChi, U, false>(P, n, gen, xs, sm + P.off_chi, acc, pend);
        };
        if (!kFlips && st_in) within(std::true_type()); else within(std::false_type());
      }
      pair_sum<V, kChi, U>(pend, sm + P.off_chi, acc);
      const double dg = P.jzq[c] * (double)(P.nb_cls[c] - 2 * nanti);
      if constexpr (kMode == 1) {
        dot[c] += class_share(reinterpret_cast<const V *>(P.x), (int64_t)__ldg(P.row_i + r), dg, P.jh[c],
                              __ldg(P.rw + __ldg(P.row_m + r)), acc.re(), acc.im());
      } else {
        row_re += P.jh[c] * acc.re();
        if constexpr (kC) row_im += P.jh[c] * acc.im();
        diag += dg;
      }
    }
    if constexpr (kMode == 1) continue;
    // the sums belong to the configuration (R(lower), upper): conj(chi(h2)) takes them to the
    // representative h2 carries it to
    const double2 rw = __ldg(P.rw + __ldcs(P.row_m + r));
    if constexpr (kChi) {
      const double t = row_re * rw.x - row_im * rw.y;
      row_im = row_re * rw.y + row_im * rw.x;
      row_re = t;
    }
    pair_store<V>(P, reinterpret_cast<const V *>(P.x), reinterpret_cast<V *>(P.y), (int64_t)__ldcs(P.row_i + r), diag,
                  kChi ? 1.0 : rw.x, row_re, row_im, dot[0], dot[1]);
  }
}

// partial[value][block] from pair_rows_kernel's sums by chunk
__global__ void __launch_bounds__(256) chunk_sum_kernel(const __grid_constant__ PairParams P, int n) {
  double v[ED_MAXCLS] = {};
#pragma unroll
  for (int part = 0; part < ED_MAXCLS; part++) {
    if (part >= n) break;
    for (uint32_t c = blockIdx.x * 256 + threadIdx.x; c < P.n_sums; c += gridDim.x * 256)
      v[part] += P.chunk_part[(size_t)part * P.n_sums + c];
  }
  pair_dot<256>(P, v, n);
}

// xs[p] = w(meta[p]) x[idx[p]]
template <typename V>
__global__ void __launch_bounds__(pair_rules::kExpandThreads) expand_kernel(const V *x, const uint32_t *idx, const uint16_t *meta,
                                                     const double2 *w, const float4 *wf, uint32_t n, V *xs,
                                                     float *xslo, uint32_t *next) {
  constexpr uint32_t kT = pair_rules::kExpandThreads;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *next = 0;
    xs[n] = no_value<V>();
    if (sizeof(V) == 4 && xslo) xslo[n] = 0.f;
  }
  for (uint32_t p = blockIdx.x * kT + threadIdx.x; p < n; p += gridDim.x * kT) {
    const uint32_t j = __ldcs(idx + p);
    const uint32_t mt = __ldcs(meta + p);
    V v = no_value<V>();
    float lo = 0.f;
    if (j != 0xFFFFFFFFu) v = weighted<V>(__ldg(x + j), mt, w, wf, lo);
    xs[p] = v;
    if (sizeof(V) == 4 && xslo) xslo[p] = lo;
  }
}

// ------------------------------- tables (once per basis) -----------------------------
// Images of half patterns under listed elements, eight bits at a time: img[j][chunk][value],
// from the images of the single bits (pos[j][bit]) and, for elements that also reverse every
// spin, the complement put into chunk 0.
__global__ void chunk_images(const uint8_t *pos, const uint8_t *flip, int n_list, int m, uint32_t *img) {
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n_list * 768; t += gridDim.x * blockDim.x) {
    const int j = t / 768, ch = (t / 256) % 3, v = t & 255;
    uint32_t r = flip[j] && ch == 0 ? (1u << m) - 1u : 0u;
    for (int b = 0; b < 8 && ch * 8 + b < m; b++)
      if ((v >> b) & 1) r ^= 1u << pos[j * m + ch * 8 + b];
    img[t] = r;
  }
}

__device__ __forceinline__ uint32_t half_image(const uint32_t *img, uint32_t u, uint32_t j) {
  const uint32_t *t = img + j * 768;
  return __ldg(t + (u & 255u)) ^ __ldg(t + 256 + ((u >> 8) & 255u)) ^ __ldg(t + 512 + (u >> 16));
}

// For every half pattern u the smallest image under the listed elements, the number of the
// first of them in the list, and whether several reach it.
__global__ void half_reps(const uint32_t *img, uint32_t n_list, uint32_t total, uint32_t *rep, uint32_t *first) {
  for (uint32_t u = blockIdx.x * blockDim.x + threadIdx.x; u < total; u += gridDim.x * blockDim.x) {
    uint32_t best = 0xFFFFFFFFu, at = 0, cnt = 0;
    for (uint32_t j = 0; j < n_list; j++) {
      const uint32_t v = half_image(img, u, j);
      if (v < best) { best = v; at = j; cnt = 1; }
      else if (v == best) cnt++;
    }
    rep[u] = best;
    first[u] = at | (cnt > 1 ? 0x80000000u : 0u);
  }
}

// ed_launch_pair_slots for halves that are not blocks of the split, and for splits without
// the two-level search: Alg. 2 as printed (or the whole table of a one-sublattice split).
// img: images of the upper representatives; spread[half][chunk][value]: a half's bits in place.
__global__ void __launch_bounds__(256) pair_slots_any(const DevTables T, const DevIndex I, const PairSlots Q, int n_up,
                                                      const uint32_t *img, const uint64_t *spread) {
  for (uint64_t p = (uint64_t)blockIdx.x * 256 + threadIdx.x; p < Q.n_slots; p += (uint64_t)gridDim.x * 256) {
    uint32_t lo = 0, hi = Q.n_low - 1;
    while (lo < hi) {   // the last class that starts at or before p (empty ones share a start)
      const uint32_t mid = (lo + hi + 1) >> 1;
      if (__ldg(Q.start + mid) <= (uint32_t)p) lo = mid; else hi = mid - 1;
    }
    const uint32_t r = (uint32_t)p - __ldg(Q.start + lo);
    const uint32_t a = __ldg(Q.low + lo);
    const uint32_t b = half_image(img, __ldg(Q.up + __ldg(Q.first_up + lo) + r / Q.K), r % Q.K);
    uint32_t idx = 0xFFFFFFFFu;
    uint16_t meta = 0;
    if (__popc(a) + __popc(b) == n_up) {
      uint64_t s = 0;
#pragma unroll
      for (int c = 0; c < 3; c++)
        s |= __ldg(spread + c * 256 + ((a >> (8 * c)) & 255u)) | __ldg(spread + 768 + c * 256 + ((b >> (8 * c)) & 255u));
      const RepOut R = find_rep(T, T.rep, T.sym_off, T.sym_list, T.dest, T.phase, s);
      const int64_t j = R.mixed ? -1 : lookup_index(I, R.rep);
      if (j >= 0) {
        idx = (uint32_t)j;
        meta = (uint16_t)(T.phase[R.g] + T.denom * (int)__ldg(Q.tcode + R.t));
        if (R.t > 1) *Q.any_weight = 1u;   // every writer stores the same value
      }
    }
    Q.idx[p] = idx;
    Q.meta[p] = meta;
    if (Q.pat) Q.pat[p] = b;
  }
}

__global__ void class_ids(const uint32_t *reps, uint32_t n, uint32_t base, uint32_t *id) {
  for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x)
    id[reps[c]] = base + c;
}

// code[j]: sign, flip and element number of list entry j
__global__ void half_entries(const uint32_t *rep, const uint32_t *first, const uint32_t *id,
                             const uint16_t *code, uint32_t total, uint32_t *t) {
  for (uint32_t u = blockIdx.x * blockDim.x + threadIdx.x; u < total; u += gridDim.x * blockDim.x)
    t[u] = (id[rep[u]] << kClassShift) | ((first[u] >> 31) ? kSpecial : 0u) |
           code[first[u] & 0x7FFFFFFFu];
}

// The rows in slot order: one slot for every basis state.  A warp owns a chunk of 1024 slots
// of one lower class.  A state has several slots when a class has a stabiliser or both halves
// belong to one class; those slots claim it with their position, the lowest wins.
struct RowEnum {
  const uint32_t *ta, *tb, *low, *start, *chunk0, *idx, *pat;
  uint32_t n_cls, n_chunks;
  uint32_t *first;       // [D] lowest claiming slot
  uint32_t *bits;        // [n_chunks][32] which slots are rows
  uint32_t *count;       // [n_chunks]
  const uint64_t *at;    // [n_chunks] first row of the chunk
  const uint16_t *meta;
  uint32_t *row_b, *row_i;
  uint16_t *row_m;
};

enum RowPass { kClaim, kCount, kFill };

template <RowPass kPass>
__global__ void __launch_bounds__(256) enum_rows(const RowEnum Q) {
  const int lane = threadIdx.x & 31;
  const uint32_t nw = gridDim.x * (blockDim.x / 32);
  for (uint32_t ch = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32; ch < Q.n_chunks; ch += nw) {
    uint32_t lo = 0, hi = Q.n_cls - 1;
    while (lo < hi) {
      const uint32_t mid = (lo + hi + 1) >> 1;
      if (__ldg(Q.chunk0 + mid) <= ch) lo = mid; else hi = mid - 1;
    }
    const uint32_t ea = __ldg(Q.ta + __ldg(Q.low + lo));
    const uint32_t p0 = __ldg(Q.start + lo) + (ch - __ldg(Q.chunk0 + lo)) * 1024, end = __ldg(Q.start + lo + 1);
    uint32_t total = 0;
    uint64_t w = kPass == kFill ? Q.at[ch] : 0;
    for (int step = 0; step < 32; step++) {
      const uint32_t p = p0 + step * 32 + lane;
      uint32_t bits = 0;
      bool row = p < end;
      if (kPass == kFill) {
        bits = Q.bits[ch * 32 + step];
        row = (bits >> lane) & 1u;
      }
      if (row) {
        const uint32_t i = __ldg(Q.idx + p);
        if (kPass == kFill) {
          const uint64_t at = w + __popc(bits & ((1u << lane) - 1u));
          Q.row_b[at] = __ldg(Q.pat + p);
          Q.row_i[at] = i;
          Q.row_m[at] = __ldg(Q.meta + p);
        } else {
          row = i != 0xFFFFFFFFu;
          if (row) {
            const uint32_t eb = __ldg(Q.tb + __ldg(Q.pat + p));
            if (((ea | eb) & kSpecial) || ((ea ^ eb) >> kClassShift) == 0) {
              if (kPass == kClaim) atomicMin(Q.first + i, p);
              else row = Q.first[i] == p;
            }
          }
        }
      }
      if (kPass == kCount) {
        const uint32_t m = __ballot_sync(0xFFFFFFFFu, row);
        if (lane == 0) Q.bits[ch * 32 + step] = m;
        total += __popc(m);
      }
      if (kPass == kFill) w += __popc(bits);
    }
    if (kPass == kCount && lane == 0) Q.count[ch] = total;
  }
}

__global__ void chunk_classes(const uint32_t *slice0, uint32_t n_cls, uint32_t n_chunks, uint32_t per_chunk,
                              uint32_t *cls) {
  for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < n_chunks; k += gridDim.x * blockDim.x) {
    uint32_t lo = 0, hi = n_cls - 1;
    while (lo < hi) {   // the last class that starts at or before the slice
      const uint32_t mid = (lo + hi + 1) >> 1;
      if (__ldg(slice0 + mid) <= k * per_chunk) lo = mid; else hi = mid - 1;
    }
    cls[k] = lo;
  }
}

__global__ void class_rows(const uint64_t *at, const uint32_t *chunk0, uint32_t n_cls, uint32_t n_chunks,
                           uint32_t total, uint32_t *row0) {
  for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c <= n_cls; c += gridDim.x * blockDim.x)
    row0[c] = c == n_cls || chunk0[c] >= n_chunks ? total : (uint32_t)at[chunk0[c]];
}

}  // namespace

struct PairPlan {
  int n = 0, m = 0;
  int shA0 = 0, shA1 = 0, shB0 = 0, shB1 = 0;
  bool blocks = true;
  uint32_t *half_x = nullptr;
  uint32_t bmask_hi = 0, bmask = 0;
  uint32_t n_cls = 0, K = 0, h0 = 0, sel_off = 0, mult_bytes = 0, n_slots = 0;
  uint32_t n_slices = 0, ubase = 0, n_ucls = 0;
  // tables of the row order
  int kw[ED_MAXCLS][5] = {};
  bool no_swap = false, any_flip = false;
  uint32_t rt_words = 0, rt_w = 0, rt_wa = 0, n_hnib = 0, rt_f = 0, rt_pos = 0, rt_nibA = 0, rt_nibB = 0, rt_img = 0, rt_left = 0;
  uint32_t rt_across = 0;         // most words of bonds across the halves in a class
  bool flips = false, weights = false;
  // device: the half tables, the small tables, the slots' indices and weights, the rows
  void *d_half = nullptr, *d_small = nullptr, *d_slots = nullptr, *d_rows = nullptr;
  uint32_t *ta = nullptr, *tb = nullptr, *off = nullptr, *idx = nullptr, *low = nullptr, *up = nullptr, *t_up = nullptr, *rt = nullptr;
  uint32_t *row0 = nullptr, *slice0 = nullptr, *chunk_cls = nullptr, *row_b = nullptr, *row_i = nullptr;
  uint16_t *row_m = nullptr;
  uint8_t *mult = nullptr;
  uint2 *bond = nullptr;
  double *chi = nullptr, *w = nullptr, *rw = nullptr;
  float4 *wf = nullptr;
  uint16_t *meta = nullptr;
  cudaMemPool_t pool = nullptr;   // xs of the calls in flight, stream-ordered
  bool own_pool = false;
  size_t bytes = 0;
};

void ed_free_pair(ed_basis *B) {
  PairPlan *p = B->pair;
  B->pair = nullptr;
  if (!p) return;
  for (void *q : {p->d_half, p->d_small, p->d_slots, p->d_rows})
    if (q) cudaFree(q);
  if (p->pool && p->own_pool) cudaMemPoolDestroy(p->pool);
  delete p;
}

void ed_trim_pair(const ed_basis *B) {
  if (B->pair && B->pair->pool && B->pair->own_pool) cudaMemPoolTrimTo(B->pair->pool, 0);
}

namespace {

// host tables gathered into one upload; at(k) is table k's place in it
struct Blob {
  std::vector<unsigned char> bytes;
  template <typename T> size_t add(const T *v, size_t n) {
    const size_t o = (bytes.size() + 15) / 16 * 16;
    bytes.resize(o + sizeof(T) * n);
    if (n) memcpy(bytes.data() + o, v, sizeof(T) * n);
    return o;
  }
  template <typename T> size_t add(const std::vector<T> &v) { return add(v.data(), v.size()); }
};

// xs of fp64 vectors that a pool shared with other bases serves: one of its own costs a build 0.1
// ms, 5% of that of the 28-site chain (1.4e6 states, 11 MB)
constexpr size_t kSharedPoolMax = (size_t)16 << 20;

// Row order for large sectors (see pair_rows_kernel); p->n_slices stays 0 when it is not made.
// pat: the pattern of the other half of every slot.
int build_rows(ed_basis *B, PairPlan *p, const std::vector<uint32_t> &start, const uint32_t *d_start,
               const uint32_t *pat, cudaStream_t st) {
  const uint32_t nA = p->n_cls;
  std::vector<uint32_t> chunk0(nA);
  uint64_t chunks = 0;
  for (uint32_t c = 0; c < nA; c++) {
    chunk0[c] = (uint32_t)chunks;
    chunks += ((uint64_t)start[c + 1] - start[c] + 1023) / 1024;
  }
  if (chunks >= 0xFFFFFFFFull || chunks == 0) return ED_OK;
  Blob blob;
  const size_t o_c0 = blob.add(chunk0);
  Scratch sc(st);
  unsigned char *d = (unsigned char *)sc.get(blob.bytes.size());
  uint32_t *d_first = (uint32_t *)sc.get(4 * (size_t)B->D), *d_bits = (uint32_t *)sc.get(128 * chunks);
  uint32_t *d_count = (uint32_t *)sc.get(4 * chunks);
  uint64_t *d_at = (uint64_t *)sc.get(8 * chunks);
  if (!d || !d_first || !d_bits || !d_count || !d_at) return ED_OK;
  const uint64_t max_chunks = (B->D / 32 + nA) / (kRowThreads / 32) + 1;
  const size_t rows_bytes = 10 * (size_t)B->D + 8 * ((size_t)nA + 1) + 4 * max_chunks;
  if (ed_malloc(&p->d_rows, rows_bytes) != cudaSuccess) { cudaGetLastError(); p->d_rows = nullptr; return ED_OK; }
  p->row_b = (uint32_t *)p->d_rows;
  p->row_i = p->row_b + B->D;
  p->row0 = p->row_i + B->D;
  p->slice0 = p->row0 + nA + 1;
  p->chunk_cls = p->slice0 + nA + 1;
  p->row_m = (uint16_t *)(p->chunk_cls + max_chunks);
  ED_CK(cudaMemcpyAsync(d, blob.bytes.data(), blob.bytes.size(), cudaMemcpyHostToDevice, st));
  ED_CK(cudaMemsetAsync(d_first, 0xFF, 4 * (size_t)B->D, st));
  RowEnum Q{};
  Q.ta = p->ta; Q.tb = p->tb; Q.low = p->low; Q.idx = p->idx; Q.pat = pat; Q.start = d_start;
  Q.chunk0 = (const uint32_t *)(d + o_c0);
  Q.n_cls = nA; Q.n_chunks = (uint32_t)chunks;
  Q.first = d_first; Q.bits = d_bits; Q.count = d_count; Q.at = d_at; Q.meta = p->meta;
  Q.row_b = p->row_b; Q.row_i = p->row_i; Q.row_m = p->row_m;
  const int grid = (int)std::min<uint64_t>((chunks + 7) / 8, (uint64_t)B->sm_count * 8);
  enum_rows<kClaim><<<grid, 256, 0, st>>>(Q);
  ED_CK(cudaGetLastError());
  enum_rows<kCount><<<grid, 256, 0, st>>>(Q);
  ED_CK(cudaGetLastError());
  uint64_t found = 0;
  int rc = ed_exclusive_scan(d_count, chunks, d_at, &found, st);
  if (rc) return rc;
  if (found != (uint64_t)B->D) return ed_fail(ED_ERR_CUDA, "row order does not cover the basis");
  enum_rows<kFill><<<grid, 256, 0, st>>>(Q);
  ED_CK(cudaGetLastError());
  class_rows<<<16, 256, 0, st>>>(d_at, Q.chunk0, nA, Q.n_chunks, (uint32_t)B->D, p->row0);
  ED_CK(cudaGetLastError());
  std::vector<uint32_t> row0(nA + 1), slice0(nA + 1);
  ED_CK(cudaMemcpyAsync(row0.data(), p->row0, 4 * ((size_t)nA + 1), cudaMemcpyDeviceToHost, st));
  ED_CK(cudaStreamSynchronize(st));
  uint64_t sl = 0;
  for (uint32_t c = 0; c < nA; c++) {
    slice0[c] = (uint32_t)sl;
    sl += (row0[c + 1] - row0[c] + 31) / 32;
  }
  slice0[nA] = (uint32_t)sl;
  ED_CK(cudaMemcpyAsync(p->slice0, slice0.data(), 4 * ((size_t)nA + 1), cudaMemcpyHostToDevice, st));
  const uint32_t n_ch = (uint32_t)((sl + kRowThreads / 32 - 1) / (kRowThreads / 32));
  chunk_classes<<<(int)std::min<uint32_t>((n_ch + 255) / 256, 1024), 256, 0, st>>>(p->slice0, nA, n_ch, kRowThreads / 32, p->chunk_cls);
  ED_CK(cudaGetLastError());
  ED_CK(cudaStreamSynchronize(st));
  p->n_slices = (uint32_t)sl;
  p->bytes += rows_bytes;
  return ED_OK;
}

}  // namespace

// Builds B->pair when the sector admits it; leaves it null (the search kernels serve the
// sector) when the split has no two stable halves, the tables would be too large, or device
// memory is short.  Only CUDA failures other than out-of-memory are errors.
int ed_build_pair(ed_basis *B, cudaStream_t st) {
  const int nsub = B->nsub, n = B->n, ns = B->nsym, N = B->N;
  if (B->D == 0 || ns > 1000 || N > 44 || N % 2) return ED_OK;
  const int m = N / 2;
  // The half and the bit in it of every site.  First choice: blocks {hb[0], hb[1]} and
  // {hb[2], hb[3]} of the split (one block each when it has two), whose patterns are two
  // shifts of the state.
  std::vector<int> half(N, -1), pos(N, 0);
  static const int kSplit[3][4] = {{0, 1, 2, 3}, {0, 2, 1, 3}, {0, 3, 1, 2}};
  int hb[4] = {0, -1, 1, -1};
  std::vector<uint8_t> swaps(ns, 0);
  auto stable = [&]() {   // every element keeps the halves or exchanges them
    int in_a = 0;
    for (int q = 0; q < N; q++) in_a += half[q] == 0;
    if (in_a != m) return false;
    for (int g = 0; g < ns; g++) {
      const int32_t *q = B->perm.data() + (size_t)g * N;
      const int to = half[q[0]] ^ half[0];
      for (int l = 1; l < N; l++)
        if ((half[q[l]] ^ half[l]) != to) return false;
      swaps[g] = (uint8_t)to;
    }
    return true;
  };
  bool blocks = false;
  if (B->two_level && (nsub == 2 || nsub == 4))
    for (int t = 0; t < (nsub == 4 ? 3 : 1) && !blocks; t++) {
      if (nsub == 4) for (int q = 0; q < 4; q++) hb[q] = kSplit[t][q];
      for (int l = 0; l < N; l++) {
        const int X = l / n;
        half[l] = X == hb[0] || X == hb[1] ? 0 : 1;
        pos[l] = n - 1 - l % n + (nsub == 4 && (X == hb[0] || X == hb[2]) ? n : 0);
      }
      blocks = stable();
    }
  // Else the two colours of a coupling class whose bonds form a connected bipartite graph on all
  // sites: symmetries keep the class's bonds, so they keep its colouring.
  bool found = blocks;
  for (int c = 0; c < B->n_classes && !found; c++) {
    std::fill(half.begin(), half.end(), -1);
    std::vector<int> order{0};
    half[0] = 0;
    bool ok = true;
    for (size_t q = 0; q < order.size() && ok; q++)
      for (int b = B->cls_off[c]; b < B->cls_off[c + 1] && ok; b++) {
        const int e0 = N - 1 - B->bond_pos[2 * b], e1 = N - 1 - B->bond_pos[2 * b + 1];
        if (e0 != order[q] && e1 != order[q]) continue;
        const int o = e0 == order[q] ? e1 : e0;
        if (half[o] < 0) { half[o] = 1 - half[order[q]]; order.push_back(o); }
        else if (half[o] == half[order[q]]) ok = false;
      }
    if (!ok || (int)order.size() != N) continue;
    int next[2] = {m - 1, m - 1};
    for (int l = 0; l < N; l++) pos[l] = next[half[l]]--;
    found = stable();
  }
  if (!found) return ED_OK;
  // the group as G0 x {1, F} when it holds the pure spin flip F (its elements then carry a
  // flip bit next to their number in G0), else all of it as it is
  // Elements are told apart by their flip and the images of at most three sites (enough for
  // affine lattice symmetries); products are then looked up without comparing permutations.
  const int32_t *pm = B->perm.data();
  int base[3] = {0, 0, 0}, nb = 0;
  std::vector<int16_t> at;
  auto key = [&](int i0, int i1, int i2, int f) { return ((size_t)(i0 * N + i1) * N + i2) * 2 + f; };
  for (nb = 1; nb <= 3; nb++) {
    // the next base site: the one that tells the most elements apart
    int best = 0, most = -1;
    for (int q = 0; q < N; q++) {
      base[nb - 1] = q;
      for (int r = nb; r < 3; r++) base[r] = base[0];
      std::vector<size_t> ks(ns);
      for (int g = 0; g < ns; g++) ks[g] = key(pm[g * N + base[0]], pm[g * N + base[1]], pm[g * N + base[2]], B->flip[g] ? 1 : 0);
      std::sort(ks.begin(), ks.end());
      const int d = (int)(std::unique(ks.begin(), ks.end()) - ks.begin());
      if (d > most) { most = d; best = q; }
      if (d == ns) break;
    }
    base[nb - 1] = best;
    for (int r = nb; r < 3; r++) base[r] = base[0];
    if (most == ns) break;
  }
  if (nb > 3) return ED_OK;
  at.assign((size_t)N * N * N * 2, -1);
  bool any_flip = false, pure = false;
  for (int g = 0; g < ns; g++) {
    const int f = B->flip[g] ? 1 : 0;
    at[key(pm[g * N + base[0]], pm[g * N + base[1]], pm[g * N + base[2]], f)] = (int16_t)g;
    any_flip = any_flip || f;
    bool id = f == 1;
    for (int q = 0; q < N && id; q++) id = pm[g * N + q] == q;
    pure = pure || id;
  }
  auto mul = [&](int a, int b) -> int {   // (a b)[p] = a[b[p]]
    const int32_t *pa = pm + (size_t)a * N, *pb = pm + (size_t)b * N;
    return at[key(pa[pb[base[0]]], pa[pb[base[1]]], pa[pb[base[2]]], (B->flip[a] ? 1 : 0) ^ (B->flip[b] ? 1 : 0))];
  };
  std::vector<int> inverse(ns, -1);
  {
    std::vector<int32_t> q(N);
    for (int g = 0; g < ns; g++) {
      for (int p = 0; p < N; p++) q[pm[(size_t)g * N + p]] = p;
      inverse[g] = at[key(q[base[0]], q[base[1]], q[base[2]], B->flip[g] ? 1 : 0)];
      if (inverse[g] < 0) return ED_OK;
    }
  }
  auto inv = [&](int a) { return inverse[a]; };
  std::vector<int> H0, S0;   // elements keeping / exchanging the halves (without F)
  for (int g = 0; g < ns; g++)
    if (!(pure && B->flip[g])) (swaps[g] ? S0 : H0).push_back(g);
  const uint32_t h0 = (uint32_t)H0.size();
  if (h0 > 256) return ED_OK;
  const bool has_swap = !S0.empty();
  int tau = -1;
  bool involution = false;
  for (int s : S0) {
    if (tau < 0) tau = s;
    if (mul(s, s) == B->id_g) { tau = s; involution = true; break; }
  }
  const int nf = pure ? 2 : 1;
  std::vector<int> num(ns, -1);                 // number of an element of H0
  for (uint32_t q = 0; q < h0; q++) num[H0[q]] = (int)q;
  // lists: half A by H; half B by H tau (or H when nothing exchanges the halves); K elements
  // between the halves, numbered like the list of half B
  auto with_flip = [&](int g, int f) -> int {
    if (!f) return g;
    const int32_t *q = pm + (size_t)g * N;
    return at[key(q[base[0]], q[base[1]], q[base[2]], 1)];
  };
  std::vector<uint16_t> listA, listB, codeA, codeB;
  std::vector<int> numK(ns, -1);
  for (int f = 0; f < nf; f++)
    for (uint32_t q = 0; q < h0; q++) {
      const int ga = with_flip(H0[q], f), gb0 = has_swap ? mul(H0[q], tau) : H0[q], gb = with_flip(gb0, f);
      if (ga < 0 || gb0 < 0 || gb < 0) return ED_OK;
      if (!f) numK[gb0] = (int)q;
      listA.push_back((uint16_t)ga);
      listB.push_back((uint16_t)gb);
      const uint32_t base = q | (f ? kFlip : 0u);
      codeA.push_back((uint16_t)(base | (B->is_real && B->phase[ga] ? 1u << kSignBit : 0u)));
      codeB.push_back((uint16_t)(base | (B->is_real && B->phase[gb] ? 1u << kSignBit : 0u)));
    }
  const uint32_t K = h0 * nf;
  // k of (lower, upper): x tau^-1 y^-1 when half A is the lower one, x tau y^-1 when half B
  // is (the same table when tau is an involution); x y^-1 when nothing exchanges the halves
  const int itau = has_swap ? inv(tau) : -1;
  const uint32_t n_tab = has_swap && !involution ? 2 : 1;
  std::vector<uint8_t> mult(((size_t)n_tab * h0 * h0 + 3) / 4 * 4, 0);
  for (uint32_t y = 0; y < h0; y++) {
    const int iy = inv(H0[y]);
    for (uint32_t t = 0; t < n_tab; t++) {
      const int r = has_swap ? mul(t ? tau : itau, iy) : iy;
      for (uint32_t x = 0; x < h0; x++) {
        const int e = mul(H0[x], r);
        const int k = e < 0 ? -1 : numK[e];
        if (k < 0) return ED_OK;
        mult[((size_t)t * h0 + x) * h0 + y] = (uint8_t)k;
      }
    }
  }
  PairPlan *p = new (std::nothrow) PairPlan();
  if (!p) return ED_OK;
  B->pair = p;
  p->n = n; p->m = m;
  p->h0 = h0; p->K = K;
  p->flips = pure;
  p->sel_off = n_tab == 2 ? h0 * h0 : 0u;
  p->mult_bytes = (uint32_t)mult.size();
  p->blocks = blocks;
  const int sh = N - n;   // block X sits at bit N - (X + 1) n
  if (!blocks) {
  } else if (nsub == 4) {
    p->shA0 = sh - hb[0] * n; p->shA1 = sh - hb[1] * n;
    p->shB0 = sh - hb[2] * n; p->shB1 = sh - hb[3] * n;
    p->bmask = p->bmask_hi = (1u << n) - 1u;
  } else {
    p->shA0 = p->shB0 = 0;
    p->shA1 = n; p->shB1 = 0;
    p->bmask = (1u << n) - 1u;
    p->bmask_hi = 0;
  }
  Scratch sc(st);
  auto keep = [&](size_t bytes) -> void * {
    void *q = nullptr;
    if (ed_malloc(&q, bytes) != cudaSuccess) { cudaGetLastError(); return nullptr; }
    p->bytes += bytes;
    return q;
  };
  const uint32_t total = 1u << m;
  const size_t nl = listA.size();
  std::vector<int> site[2] = {std::vector<int>(m), std::vector<int>(m)};   // of a half's bits
  for (int l = 0; l < N; l++) site[half[l]][pos[l]] = l;
  // images of half A's bits under list A, of half B's under list B, and of the upper
  // representatives' half under list B
  const int up_half = has_swap ? 0 : 1;
  auto images = [&](const std::vector<uint16_t> &list, int h) {
    std::vector<uint8_t> v(nl * m);
    for (size_t j = 0; j < nl; j++)
      for (int q = 0; q < m; q++) v[j * m + q] = (uint8_t)pos[pm[(size_t)list[j] * N + site[h][q]]];
    return v;
  };
  const std::vector<uint8_t> imA = images(listA, 0), imB = images(listB, 1), imK = images(listB, up_half);
  std::vector<uint8_t> flA(nl), flB(nl);
  for (size_t j = 0; j < nl; j++) { flA[j] = B->flip[listA[j]]; flB[j] = B->flip[listB[j]]; }
  Blob lists;
  lists.add(listB); lists.add(codeA); lists.add(codeB);
  const size_t lstep = (nl * 2 + 15) / 16 * 8;   // elements from one list to the next
  const size_t o_im[3] = {lists.add(imA), lists.add(imB), lists.add(imK)}, o_fl[2] = {lists.add(flA), lists.add(flB)};
  const size_t o_img = (lists.bytes.size() + 15) / 16 * 16;
  uint32_t *d_rep = (uint32_t *)sc.get(16 * (size_t)total + o_img + 3 * 3072 * nl);
  p->d_half = keep(8 * (size_t)total);
  if (!d_rep || !p->d_half) { ed_free_pair(B); return ED_OK; }
  uint32_t *d_first = d_rep + total, *d_id = d_first + total, *d_reps = d_id + total;
  unsigned char *d_lists = (unsigned char *)(d_reps + total);
  uint16_t *d_list = (uint16_t *)d_lists;
  uint32_t *d_img = (uint32_t *)(d_lists + o_img);   // [3][nl][768]
  p->ta = (uint32_t *)p->d_half;
  p->tb = p->ta + total;
  ED_CK(cudaMemcpyAsync(d_list, lists.bytes.data(), lists.bytes.size(), cudaMemcpyHostToDevice, st));
  for (int q = 0; q < 3; q++) {
    chunk_images<<<(int)(3 * nl), 256, 0, st>>>(d_lists + o_im[q], d_lists + o_fl[q ? 1 : 0], (int)nl, m, d_img + q * 768 * nl);
    ED_CK(cudaGetLastError());
  }
  const int gt = (int)std::min<uint32_t>((total + 255) / 256, (uint32_t)B->sm_count * 8);
  std::vector<uint32_t> rep(total);
  std::vector<std::vector<uint32_t>> cls(2);      // representatives of half A's (and B's) classes
  std::vector<uint32_t> bucket0[2];               // first class of each popcount
  for (int h = 0; h < 2; h++) {
    half_reps<<<gt, 256, 0, st>>>(d_img + h * 768 * nl, (uint32_t)nl, total, d_rep, d_first);
    ED_CK(cudaGetLastError());
    if (h == 0 || !has_swap) {
      ED_CK(cudaMemcpyAsync(rep.data(), d_rep, (size_t)total * 4, cudaMemcpyDeviceToHost, st));
      ED_CK(cudaStreamSynchronize(st));
      // classes in order of (popcount of the representative, value); with spin flips the
      // smaller of the popcounts of a pattern and its reverse
      std::vector<std::vector<uint32_t>> by(m + 1);
      for (uint32_t u = 0; u < total; u++)
        if (rep[u] == u) {
          const int pc = __builtin_popcount(u);
          by[any_flip ? std::min(pc, m - pc) : pc].push_back(u);
        }
      bucket0[h].assign(m + 2, 0);
      for (int q = 0; q <= m; q++) {
        bucket0[h][q] = (uint32_t)cls[h].size();
        cls[h].insert(cls[h].end(), by[q].begin(), by[q].end());
      }
      bucket0[h][m + 1] = (uint32_t)cls[h].size();
      const uint32_t nc = (uint32_t)cls[h].size();
      ED_CK(cudaMemcpyAsync(d_reps, cls[h].data(), (size_t)nc * 4, cudaMemcpyHostToDevice, st));
      class_ids<<<gt, 256, 0, st>>>(d_reps, nc, h ? (uint32_t)cls[0].size() : 0u, d_id);
      ED_CK(cudaGetLastError());
    }
    half_entries<<<gt, 256, 0, st>>>(d_rep, d_first, d_id, d_list + (1 + h) * lstep, total, h ? p->tb : p->ta);
    ED_CK(cudaGetLastError());
  }
  const uint32_t nA = (uint32_t)cls[0].size();
  const std::vector<uint32_t> &up = has_swap ? cls[0] : cls[1];
  const std::vector<uint32_t> &ub = has_swap ? bucket0[0] : bucket0[1];
  const uint32_t ubase = has_swap ? 0u : nA;      // class number of the first upper class
  p->n_cls = nA;
  if (nA > 16384 || ubase + up.size() >= (1u << 21)) { ed_free_pair(B); return ED_OK; }
  // slots of every lower class: the upper classes [lo, hi) that can share a configuration
  // of the sector with it
  std::vector<uint32_t> off(nA), start(nA + 1), first_up(nA);
  uint64_t acc = 0;
  for (uint32_t c = 0; c < nA; c++) {
    int pc = __builtin_popcount(cls[0][c]);
    if (any_flip) pc = std::min(pc, m - pc);
    const int want = any_flip ? pc : B->n_up - pc;
    uint32_t lo = 0, hi = 0;
    if (want >= 0 && want <= m) { lo = ub[want]; hi = ub[want + 1]; }
    if (has_swap) lo = std::max(lo, c);
    if (lo >= hi) lo = hi = 0;
    start[c] = (uint32_t)acc;
    first_up[c] = lo;
    off[c] = (uint32_t)acc - K * (ubase + lo);    // modulo 2^32: slot = off + K upper + k
    acc += (uint64_t)K * (hi - lo);
    if (acc > pair_rules::kMaxSlots) { ed_free_pair(B); return ED_OK; }
  }
  start[nA] = (uint32_t)acc;
  const uint64_t cap = std::max<uint64_t>(4 * (uint64_t)B->D, 1u << 22);
  if (acc == 0 || acc > cap) { ed_free_pair(B); return ED_OK; }
  p->n_slots = (uint32_t)acc;
  pair_rules::Plan room{true, true};
  if (!pair_rules::always_fits((uint64_t)B->D, acc)) {
    size_t free_bytes = 0, all = 0;
    ED_CK(cudaMemGetInfo(&free_bytes, &all));
    room = pair_rules::fits(free_bytes, (uint64_t)B->D, acc, B->is_real);
    if (!room.pair) { ed_free_pair(B); return ED_OK; }
  }
  // weights chi sqrt(t): index phase + denom * (number of t among the divisors of |G|)
  std::vector<uint8_t> tcode(ns + 1, 0);
  std::vector<int> divs;
  for (int t = 1; t <= ns; t++) if (ns % t == 0) { tcode[t] = (uint8_t)divs.size(); divs.push_back(t); }
  const size_t n_w = (size_t)B->denom * divs.size();
  if (n_w > 65535 || divs.size() > 255) { ed_free_pair(B); return ED_OK; }
  std::vector<double> wt(2 * n_w), rwt(2 * n_w);   // and conj(chi) / sqrt(t)
  std::vector<float4> wtf(n_w);                    // and as pairs of fp32 words
  for (size_t t = 0; t < divs.size(); t++)
    for (int q = 0; q < B->denom; q++) {
      const double r = std::sqrt((double)divs[t]);
      double c, s;
      ed_character(q, B->denom, &c, &s);
      if (B->is_real) { c = q ? -1.0 : 1.0; s = 0.0; }
      wt[2 * (t * B->denom + q)] = r * c;
      wt[2 * (t * B->denom + q) + 1] = r * s;
      rwt[2 * (t * B->denom + q)] = c / r;
      rwt[2 * (t * B->denom + q) + 1] = -s / r;
      const float ch = (float)(r * c), sh = (float)(r * s);
      wtf[t * B->denom + q] = make_float4(ch, (float)(r * c - (double)ch), sh, (float)(r * s - (double)sh));
    }
  // chi of the lower half's element: [half][512] (flip bit above the element number)
  std::vector<double> chi(2 * 1024, 0.0);
  for (int half = 0; half < 2; half++)
    for (size_t j = 0; j < nl; j++) {
      const int g = half ? listB[j] : listA[j];
      const uint32_t e = (half ? codeB[j] : codeA[j]) & (kElem | kFlip);
      ed_character(B->phase[g], B->denom, &chi[2 * (512 * half + e)], &chi[2 * (512 * half + e) + 1]);
    }
  // bonds as flipped bits of the two halves
  std::vector<uint2> bond(B->bond_pad.size() / 2, make_uint2(0, 0));
  for (size_t b = 0; b < bond.size(); b++) {
    const int pe[2] = {B->bond_pad[2 * b], B->bond_pad[2 * b + 1]};
    if (pe[0] == pe[1]) continue;
    for (int q = 0; q < 2; q++) {
      const int l = N - 1 - pe[q];
      (half[l] ? bond[b].y : bond[b].x) |= 1u << pos[l];
    }
  }
  // tables of the row order, staged in shared memory as one block of words: per bond the
  // flipped bits (of A across the halves and within A; of the upper representative's half
  // within that half) and the bit of B; antiparallel masks by nibbles (bit k is set for every
  // endpoint of bond k that is up) of A and of B or the upper representative; images of B's bits
  // under the elements of half B's list; the left multiplication table of H
  std::vector<uint32_t> rt;
  {
    std::vector<uint32_t> f;
    std::vector<uint8_t> bpos;
    std::vector<uint32_t> mA, mB;   // bits of the bond that count in A, and in B or R(c)
    for (int pass = 0; pass < 2; pass++) {   // bonds across and within A first
      for (int c = 0; c < B->n_classes; c++)
        for (int kind = pass ? 2 : 0; kind < (pass ? 3 : 2); kind++) {
          p->kw[c][pass ? 3 : kind] = (int)f.size() / 32;
          for (size_t b = (size_t)B->cls_word[c] * 32; b < (size_t)B->cls_word[c + 1] * 32; b++) {
            const uint32_t fa = bond[b].x, fb = bond[b].y;
            if (!fa && !fb) continue;   // padding
            const uint32_t fu = up_half ? fb : fa;
            const bool across = fa && fb;
            if (kind == 0 && across) {
              f.push_back(fa); bpos.push_back((uint8_t)__builtin_ctz(fb)); mA.push_back(fa); mB.push_back(fb);
            } else if (kind == 1 && !across && fa) {
              f.push_back(fa); bpos.push_back(0); mA.push_back(fa); mB.push_back(0);
            } else if (kind == 2 && !across && fu) {
              f.push_back(fu); bpos.push_back(0); mA.push_back(0); mB.push_back(fu);
            }
          }
          while (f.size() % 32) { f.push_back(0); bpos.push_back(0); mA.push_back(0); mB.push_back(0); }
          p->kw[c][pass ? 4 : kind + 1] = (int)f.size() / 32;
          if (kind == 0) p->rt_across = std::max(p->rt_across, (uint32_t)(p->kw[c][1] - p->kw[c][0]));
        }
      if (!pass) p->rt_wa = (uint32_t)f.size() / 32;
    }
    p->rt_w = (uint32_t)f.size() / 32;
    p->n_hnib = (uint32_t)(m + 3) / 4;
    auto words = [&](const void *v, size_t bytes) -> uint32_t {
      const uint32_t o = (uint32_t)rt.size();
      rt.resize(rt.size() + (bytes + 3) / 4, 0u);
      if (bytes) memcpy(rt.data() + o, v, bytes);
      return o;
    };
    auto nibbles = [&](const std::vector<uint32_t> &mk) {
      std::vector<uint32_t> t((size_t)p->rt_w * p->n_hnib * 16, 0u);
      for (size_t b = 0; b < mk.size(); b++)
        for (int q = 0; q < m; q++)
          if ((mk[b] >> q) & 1u)
            for (int v = 0; v < 16; v++)
              if ((v >> (q % 4)) & 1) t[((b / 32) * p->n_hnib + q / 4) * 16 + v] ^= 1u << (b % 32);
      return t;
    };
    const std::vector<uint32_t> tA = nibbles(mA), tB = nibbles(mB);
    std::vector<uint8_t> lm((size_t)h0 * h0);
    for (uint32_t x = 0; x < h0; x++)
      for (uint32_t y = 0; y < h0; y++) {
        const int e = mul(H0[x], H0[y]);
        if (e < 0 || num[e] < 0) { ed_free_pair(B); return ED_OK; }
        lm[(size_t)x * h0 + y] = (uint8_t)num[e];
      }
    p->rt_f = words(f.data(), f.size() * 4);
    p->rt_nibA = words(tA.data(), tA.size() * 4);
    p->rt_nibB = words(tB.data(), tB.size() * 4);
    p->rt_pos = words(bpos.data(), bpos.size());
    p->rt_img = words(imB.data(), (size_t)h0 * m);
    p->rt_left = words(lm.data(), lm.size());
    p->rt_words = (uint32_t)rt.size();
  }
  Blob blob;
  const size_t o_off = blob.add(off), o_low = blob.add(cls[0]), o_mult = blob.add(mult), o_bond = blob.add(bond),
               o_chi = blob.add(chi), o_w = blob.add(wt), o_rw = blob.add(rwt), o_wf = blob.add(wtf), o_rt = blob.add(rt), o_start = blob.add(start),
               o_fup = blob.add(first_up), o_up = blob.add(up), o_tc = blob.add(tcode);
  // halves that are no blocks: their bits by the state's nibbles, and back by their bytes
  std::vector<uint32_t> half_x;
  std::vector<uint64_t> spread;
  if (!blocks) {
    half_x.assign(2 * (size_t)B->n_nib * 16, 0u);
    spread.assign(2 * 768, 0);
    for (int l = 0; l < N; l++) {
      const int bit = N - 1 - l;
      for (int v = 0; v < 16; v++)
        if ((v >> (bit % 4)) & 1) half_x[((size_t)half[l] * B->n_nib + bit / 4) * 16 + v] |= 1u << pos[l];
      for (int v = 0; v < 256; v++)
        if ((v >> (pos[l] % 8)) & 1) spread[half[l] * 768 + pos[l] / 8 * 256 + v] |= 1ULL << bit;
    }
  }
  const size_t o_hx = blob.add(half_x), o_sp = blob.add(spread);
  const uint32_t zero = 0;
  const size_t o_any = blob.add(&zero, 1);
  p->d_small = keep(blob.bytes.size());
  p->d_slots = keep(6 * (size_t)acc);
  if (!p->d_small || !p->d_slots) { ed_free_pair(B); return ED_OK; }
  unsigned char *sb = (unsigned char *)p->d_small;
  ED_CK(cudaMemcpyAsync(sb, blob.bytes.data(), blob.bytes.size(), cudaMemcpyHostToDevice, st));
  p->off = (uint32_t *)(sb + o_off); p->low = (uint32_t *)(sb + o_low); p->mult = sb + o_mult;
  p->bond = (uint2 *)(sb + o_bond); p->chi = (double *)(sb + o_chi); p->w = (double *)(sb + o_w); p->rw = (double *)(sb + o_rw); p->wf = (float4 *)(sb + o_wf);
  p->rt = (uint32_t *)(sb + o_rt);
  p->half_x = (uint32_t *)(sb + o_hx);
  p->up = (uint32_t *)(sb + o_up);
  p->t_up = has_swap ? p->ta : p->tb;
  p->ubase = ubase;
  p->n_ucls = (uint32_t)up.size();
  p->no_swap = !has_swap;
  p->any_flip = any_flip;
  p->idx = (uint32_t *)p->d_slots;
  p->meta = (uint16_t *)(p->idx + acc);
  uint32_t *d_any = (uint32_t *)(sb + o_any);
  PairSlots Q{};
  Q.start = (uint32_t *)(sb + o_start); Q.first_up = (uint32_t *)(sb + o_fup); Q.low = p->low; Q.up = (uint32_t *)(sb + o_up);
  Q.n_low = nA; Q.n_slots = p->n_slots;
  Q.K = K; Q.kel = d_list; Q.tcode = sb + o_tc;
  for (int q = 0; q < 4; q++) Q.hb[q] = hb[q];
  Q.up_half = up_half;
  Q.idx = p->idx; Q.meta = p->meta; Q.any_weight = d_any;
  // the row order pays when xs outgrows the L2 and a class fills many warps
  const bool want_rows = room.rows && B->D >= kRowOrderMinDim && B->D / nA >= 256 && ubase + up.size() <= 1u << (kPosShift - kClassShift);
  if (want_rows) Q.pat = (uint32_t *)sc.get(4 * (size_t)acc);   // null without memory: no row order
  int rc = blocks ? ed_launch_pair_slots(B, Q, st) : ED_ERR_UNSUPPORTED;
  if (rc == ED_ERR_UNSUPPORTED) {
    if (blocks) { ed_free_pair(B); return ED_OK; }
    pair_slots_any<<<(int)std::min<uint32_t>((p->n_slots + 255) / 256, (uint32_t)B->sm_count * 8), 256, 0, st>>>(
        B->T, B->I, Q, B->n_up, d_img + 2 * 768 * nl, (const uint64_t *)(sb + o_sp));
    ED_CK(cudaGetLastError());
    rc = ED_OK;
  }
  if (rc) return rc;
  uint32_t any = 0;
  ED_CK(cudaMemcpyAsync(&any, d_any, 4, cudaMemcpyDeviceToHost, st));
  ED_CK(cudaStreamSynchronize(st));
  p->weights = any != 0;
  if (Q.pat)
    if ((rc = build_rows(B, p, start, Q.start, Q.pat, st))) return rc;
  // The memory of xs: large sectors keep a pool of their own, gone with the basis; small ones
  // take it from the device's shared one.
  const size_t first = 8 * ((size_t)p->n_slots + 1) + 256;
  p->own_pool = first > kSharedPoolMax;
  if (p->own_pool) p->pool = ed_make_pool(B->device, pair_rules::pool_keep(p->n_slots, B->is_real));
  else p->pool = ed_shared_pool(B->device);
  if (!p->pool) { ed_free_pair(B); return ED_OK; }
  // small sectors: the pool takes its first memory here rather than in the first product,
  // where mapping it would cost several times the product itself
  if (first <= ((size_t)64 << 20)) {
    void *q = nullptr;
    if (cudaMallocFromPoolAsync(&q, first, p->pool, st) == cudaSuccess) ED_CK(cudaFreeAsync(q, st));
    else cudaGetLastError();
  }
  B->table_bytes += p->bytes + (p->own_pool ? pair_rules::xs_most(p->n_slots, B->is_real) : 0);
  return ED_OK;
}

namespace {

size_t al16(size_t x) { return (x + 15) & ~(size_t)15; }

template <typename V>
int launch_expand(const ed_basis *B, const PairParams &P, cudaStream_t st) {
  const uint32_t blocks = pair_rules::expand_blocks(P.n_slots, (uint32_t)B->sm_count);
  expand_kernel<V><<<blocks, pair_rules::kExpandThreads, 0, st>>>(
      (const V *)P.x, P.slot_idx, P.slot_meta, P.w, P.wf, P.n_slots, (V *)const_cast<void *>(P.xs),
      const_cast<float *>(P.xslo), P.next);
  ED_CK(cudaGetLastError());
  return ED_OK;
}

template <typename V, bool kChi, bool kFlips, int kMode>
int launch_pair_t(const ed_basis *B, PairParams &P, bool rows, cudaStream_t st, int *n_blocks) {
  auto k = rows ? pair_rows_kernel<V, kChi, kFlips, kMode>
                : P.xs ? pair_kernel<V, kChi, kFlips, kMode, false> : pair_kernel<V, kChi, kFlips, kMode, true>;
  const int threads = rows ? kRowThreads : kThreads, per_sm = rows ? kRowBlocks : kMinBlocks;
  const int64_t blocks = rows ? (int64_t)P.n_chunks : (P.r1 - P.r0 + threads - 1) / threads;
  const int grid = (int)std::min<int64_t>(blocks, (int64_t)B->sm_count * per_sm);
  // small calls are held by the host: 48 KB need no permission, and a block per SM no split
  if (P.smem_bytes > 48 * 1024)
    if (const int rc = ed_allow_smem(k, rows ? kRowsMaxSmem : kPairMaxSmem)) return rc;
  if (grid > B->sm_count || rows) {
    const int need = per_sm * ((int)P.smem_bytes + 1536);
    const int pct = std::min(100, (need * 100 + 228 * 1024 - 1) / (228 * 1024));
    ED_CK(cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, pct));
  }
  if (n_blocks) *n_blocks = grid;
  k<<<grid, threads, P.smem_bytes, st>>>(P);
  ED_CK(cudaGetLastError());
  if (rows && P.partial) {
    chunk_sum_kernel<<<grid, 256, 0, st>>>(P, kMode == 1 ? P.n_classes : Pv<V>::cplx ? 2 : 1);
    ED_CK(cudaGetLastError());
  }
  return ED_OK;
}

template <typename V, int kMode>
int launch_pair_m(const ed_basis *B, PairParams &P, bool chi, bool flips, bool rows, cudaStream_t st, int *n_blocks) {
  if constexpr (Pv<V>::cplx) {
    if (chi)
      return flips ? launch_pair_t<V, true, true, kMode>(B, P, rows, st, n_blocks) : launch_pair_t<V, true, false, kMode>(B, P, rows, st, n_blocks);
  }
  return flips ? launch_pair_t<V, false, true, kMode>(B, P, rows, st, n_blocks) : launch_pair_t<V, false, false, kMode>(B, P, rows, st, n_blocks);
}

template <typename V>
int launch_pair_v(const ed_basis *B, PairParams &P, bool chi, bool flips, bool rows, int mode, cudaStream_t st,
                  int *n_blocks) {
  return mode == 1 ? launch_pair_m<V, 1>(B, P, chi, flips, rows, st, n_blocks) : launch_pair_m<V, 0>(B, P, chi, flips, rows, st, n_blocks);
}

// Shared memory of a block, as offsets in P and in bytes.
size_t pair_layout(const ed_basis *B, bool cplx, bool chi, bool rows, PairParams &P) {
  const PairPlan *p = B->pair;
  size_t off = 0;
  auto put = [&](uint32_t &o, size_t bytes) { o = (uint32_t)off; off += al16(bytes); };
  int words = 0;
  for (int c = 0; c < B->n_classes; c++) words = std::max(words, B->cls_word[c + 1] - B->cls_word[c]);
  put(P.off_off, 4 * (size_t)p->n_cls);
  put(P.off_mult, p->mult_bytes);
  put(P.off_bond, 8 * 32 * (size_t)B->cls_word[B->n_classes]);
  put(P.off_rs, 8 * ((size_t)B->nsym + 1));
  put(P.off_chi, chi ? 16 * 1024 : 0);
  if (rows) {
    put(P.off_rt, 4 * (size_t)p->rt_words);
    put(P.off_mask, 4 * std::max<size_t>(p->rt_across, cplx ? 4 : 2) * kRowThreads);   // or a row's <x, y>
    P.n_tab = p->K >= 32 ? 2 : 0;   // 32 rows span two classes at most (without stabilisers)
    P.et_words = (uint32_t)(65 * p->rt_wa + P.n_tab * (32 * (p->rt_w - p->rt_wa) + p->m) + 3) / 4 * 4;
    put(P.off_et, 4 * (size_t)P.et_words * (kRowThreads / 32));
  } else {
    put(P.off_nib, 4 * B->nib.size());
    put(P.off_hx, p->blocks ? 0 : 128 * (size_t)B->n_nib);
    put(P.off_mask, 4 * (size_t)words * kThreads);
  }
  P.smem_bytes = (uint32_t)off;
  return off;
}

size_t elem_bytes(int dtype) { return dtype == ED_F32 ? 4 : dtype == ED_C128 ? 16 : 8; }

}  // namespace

int ed_pair_route(const ed_basis *B, int dtype, int64_t r0, int64_t r1, int mode) {
  const PairPlan *p = B->pair;
  if (!p || r1 <= r0) return ED_ROUTE_SEARCH;
  const bool cplx = dtype == ED_C128 || dtype == ED_C64, chi = cplx && !B->is_real;
  const pair_rules::Route way = pair_rules::route(r1 - r0, B->D, B->terms_per_row, p->n_slots, dtype == ED_C128,
                                                  B->T.full && B->N <= 22 && mode == 0 && !B->is_real && dtype == ED_C64);
  PairParams P{};
  if (way == pair_rules::kSearch || pair_layout(B, cplx, chi, false, P) > kPairMaxSmem) return ED_ROUTE_SEARCH;
  if (way == pair_rules::kDirect) return ED_ROUTE_DIRECT;
  const size_t least = p->rt_w > p->rt_wa ? kRowOrderMinBytes : kRowOrderMinBytesAcross;
  if (p->n_slices && r0 == 0 && r1 == B->D && al16(elem_bytes(dtype) * ((size_t)p->n_slots + 1)) >= least &&
      pair_layout(B, cplx, chi, true, P) <= kRowsMaxSmem)
    return ED_ROUTE_SLOT_ORDER;
  return ED_ROUTE_EXPANDED;
}

int ed_launch_apply_pair(const ed_basis *B, const double *J, const double *Jz, const void *x, void *y,
                         int dtype, int64_t r0, int64_t r1, double *partial, cudaStream_t st, int mode,
                         void *ylo, bool *ylo_done, int *n_blocks) {
  const PairPlan *p = B->pair;
  int route = ed_pair_route(B, dtype, r0, r1, mode);
  if (route == ED_ROUTE_SEARCH) return ED_ERR_UNSUPPORTED;
  bool rows = route == ED_ROUTE_SLOT_ORDER;
  const size_t xs_bytes = al16(elem_bytes(dtype) * ((size_t)p->n_slots + 1));
  PairParams P{};
  P.n_classes = B->n_classes;
  for (int c = 0; c <= B->n_classes; c++) P.cls_word[c] = B->cls_word[c];
  for (int c = 0; c < B->n_classes; c++) {
    P.nb_cls[c] = B->cls_off[c + 1] - B->cls_off[c];
    P.jh[c] = 0.5 * J[c];
    P.jzq[c] = 0.25 * J[c] * Jz[c];
  }
  P.n = p->n;
  P.shA0 = p->shA0; P.shA1 = p->shA1; P.shB0 = p->shB0; P.shB1 = p->shB1;
  P.bmask_hi = p->bmask_hi; P.bmask = p->bmask;
  P.blocks = p->blocks; P.half_x = p->half_x;
  P.ta = p->ta; P.tb = p->tb; P.off = p->off;
  P.n_cls = p->n_cls; P.K = p->K; P.h0 = p->h0; P.sel_off = p->sel_off;
  P.mult = p->mult; P.mult_bytes = p->mult_bytes;
  P.bond = p->bond;
  P.nib = B->d_nib; P.n_nib = (uint32_t)B->n_nib;
  P.rsqrt_tab = B->d_rsqrt; P.n_sq = (uint32_t)B->nsym + 1;
  const bool cplx = dtype == ED_C128 || dtype == ED_C64;
  const bool chi = cplx && !B->is_real;
  P.chi = p->chi;
  P.basis = B->d_basis; P.stab = B->d_stab;
  P.up = p->up; P.t_up = p->t_up; P.ubase = p->ubase; P.n_ucls = p->n_ucls; P.rt = p->rt; P.rt_words = p->rt_words;
  memcpy(P.kw, p->kw, sizeof(P.kw));
  P.n_w = p->rt_w; P.n_wa = p->rt_wa; P.n_up = B->n_up; P.no_swap = p->no_swap; P.by_popcount = !p->any_flip;
  P.n_hnib = p->n_hnib; P.m = (uint32_t)p->m;
  P.rt_f = p->rt_f; P.rt_pos = p->rt_pos; P.rt_nibA = p->rt_nibA; P.rt_nibB = p->rt_nibB; P.rt_img = p->rt_img;
  P.rt_left = p->rt_left;
  P.low = p->low; P.row0 = p->row0; P.slice0 = p->slice0; P.chunk_cls = p->chunk_cls; P.n_slices = p->n_slices;
  P.row_b = p->row_b; P.row_i = p->row_i; P.row_m = p->row_m; P.rw = (const double2 *)p->rw;
  P.x = x; P.y = y; P.r0 = r0; P.r1 = r1; P.partial = partial;
  P.ylo = (dtype == ED_F32 || dtype == ED_C64) ? ylo : nullptr;
  pair_layout(B, cplx, chi, rows, P);
  const bool lo = dtype == ED_F32 && p->weights;
  P.lo_special = lo ? kSpecial : 0u;
  P.lo_same = lo ? 1u << kClassShift : 0u;
  P.n_slots = p->n_slots;
  P.slot_idx = p->idx; P.slot_meta = p->meta; P.w = (const double2 *)p->w; P.wf = p->wf;
  P.n_chunks = (p->n_slices + kRowThreads / 32 - 1) / (kRowThreads / 32);
  P.n_sums = P.n_chunks * (mode == 1 ? 1 : kSumWarps);
  // xs (and its remainders) for this call, from the basis's own pool in stream order, so
  // calls on several streams or threads never share it.  Without memory for it terms read x
  // through the slots; the largest sectors are searched sooner than that (pair_rules.h).
  char *ws = nullptr;
  if (route != ED_ROUTE_DIRECT) {
    const size_t lo_bytes = lo ? al16(4 * ((size_t)p->n_slots + 1)) : 0;
    const size_t n_sums = !rows || !partial ? 0 : (mode == 1 ? (size_t)B->n_classes : cplx ? 2 : 1) * P.n_sums;
    if (cudaMallocFromPoolAsync((void **)&ws, 16 + xs_bytes + lo_bytes + 8 * n_sums, p->pool, st) != cudaSuccess) {
      cudaGetLastError();
      ws = nullptr;
      if (B->D > pair_rules::kMaxDirectDim) return ED_ERR_UNSUPPORTED;
      rows = false;
      pair_layout(B, cplx, chi, false, P);
    } else {
      P.xs = ws;
      P.next = reinterpret_cast<uint32_t *>(ws + xs_bytes);
      if (lo) P.xslo = reinterpret_cast<float *>(ws + 16 + xs_bytes);
      P.chunk_part = reinterpret_cast<double *>(ws + 16 + xs_bytes + lo_bytes);
    }
  }
  int rc = ED_OK;
  switch (dtype) {
#define PCASE(D, V)                                                     \
  case D:                                                               \
    rc = ws ? launch_expand<V>(B, P, st) : ED_OK;                       \
    if (!rc) rc = launch_pair_v<V>(B, P, chi, p->flips, rows, mode, st, n_blocks); \
    break;
    PCASE(ED_F64, double)
    PCASE(ED_F32, float)
    PCASE(ED_C128, double2)
    PCASE(ED_C64, float2)
#undef PCASE
    default: rc = ed_fail(ED_ERR_INVALID, "unknown dtype");
  }
  if (ws) {
    const cudaError_t fe = cudaFreeAsync(ws, st);
    if (!rc && fe != cudaSuccess) rc = ed_cuda_fail(fe, "cudaFreeAsync");
  }
  if (!rc && ylo_done) *ylo_done = P.ylo != nullptr;
  return rc;
}
