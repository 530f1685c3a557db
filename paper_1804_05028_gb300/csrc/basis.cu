// basis.cu -- construction of the symmetry-adapted basis on one GPU (Alg. 3 of
// arXiv:1804.05028 without the process split) and of its prefix index (Basis and
// Limits, Sec. IV).
//
// Enumeration.  A representative's top block equals MinRep = min_X Rep_X, and MinRep
// is its own Rep_0; so only top blocks v with Rep_0(v) == v are enumerated (for a
// single sublattice: every top-P-bit prefix).  For each such v the remaining bits run
// over all patterns with the right number of up spins, in increasing order, split into
// work items of 1024 consecutive ranks.  One warp owns an item; lane l owns ranks
// [32 l, 32 l + 32) of it, so lanes are ordered like the states they produce.
//   pass 1 (count): every kept representative is counted per item;
//   scan: exclusive prefix sums of the item counts give each item's output offset;
//   pass 2 (fill): each lane records a 32-bit hit mask, the warp scans the popcounts,
//   and every lane writes its hits in order -- the output is sorted with no sort.
// Index.  top_rank compresses the occupied values of the top r bits to a dense rank;
// key = rank << q | next q bits; limits[key] = first position whose key is >= key
// (marked where keys begin, then filled from the end); the remaining low bits go to a narrow postfix
// array searched inside the bucket.  Where they fit (4x the basis's bytes, or 64 MB),
// ranked records replace the search: one record per prefix rank and value of every bit
// but the low 6, holding the first basis position and a 64-bit bitmap of the low-6-bit
// values present, so that the index is first + popcount(bitmap below the value) -- one
// 16-byte load.
#include "sced_internal.cuh"
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstring>
#include <vector>

namespace {

constexpr int kRun = 32;               // ranks per lane
constexpr int kItem = 32 * kRun;       // ranks per work item (one warp)

struct EnumParams {
  DevTables T;
  int S;                 // suffix bits (below the enumerated prefix)
  int n_tops;
  const uint32_t *top_v;       // prefix value
  const uint8_t *top_k;        // up spins in the suffix
  const uint64_t *top_total;   // C(S, k)
  const uint64_t *top_item0;   // first item of this prefix (exclusive scan of item counts)
  uint64_t n_items;
  const uint64_t *binom;       // [65][65]
};

__device__ __forceinline__ uint64_t unrank(const uint64_t *binom, int S, int k, uint64_t r) {
  // r-th S-bit pattern with k ones in increasing order: patterns whose bit pos is 0
  // come first and there are C(pos, k) of them.
  uint64_t x = 0;
  for (int pos = S - 1; pos >= 0 && k > 0; pos--) {
    const uint64_t c = __ldg(binom + pos * 65 + k);
    if (r >= c) { x |= 1ULL << pos; r -= c; k--; }
  }
  return x;
}

// next larger integer with the same number of ones: move the lowest run of ones up by
// one place, keeping all but one of its ones at the bottom
__device__ __forceinline__ uint64_t next_comb(uint64_t x) {
  if (x == 0) return 0;
  const int p = __ffsll((long long)x) - 1;
  const uint64_t y = x >> p;
  const int run = __ffsll((long long)~y) - 1;   // length of the run of ones
  const int q = p + run;                          // first zero above the run
  uint64_t hi = (q >= 64) ? 0 : (x & ~((q >= 63 ? ~0ULL : ((1ULL << (q + 1)) - 1ULL))));
  hi |= (q >= 64) ? 0 : (1ULL << q);
  return hi | ((run - 1) >= 64 ? ~0ULL : ((1ULL << (run - 1)) - 1ULL));
}

__device__ __forceinline__ int find_top(const EnumParams &E, uint64_t item) {
  int lo = 0, hi = E.n_tops - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (E.top_item0[mid] <= item) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// hit_s (may be null): the count pass leaves every lane's 32-bit hit mask there, so that the
// fill pass only has to look at the states it writes.
template <bool kFill>
__global__ void __launch_bounds__(256) enum_kernel(const EnumParams E, uint32_t *counts,
                                                   const uint64_t *offsets, uint64_t *basis,
                                                   uint16_t *stab, uint32_t *hit_s) {
  const DevTables &T = E.T;
  const int lane = threadIdx.x & 31;
  const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  for (uint64_t item = (((uint64_t)blockIdx.x * blockDim.x) >> 5) + (threadIdx.x >> 5);
       item < E.n_items; item += nwarps) {
    const int t = find_top(E, item);
    const uint64_t base = (item - E.top_item0[t]) * kItem;
    const uint64_t total = E.top_total[t];
    const int k = E.top_k[t];
    const uint64_t pre = (uint64_t)E.top_v[t] << E.S;
    const uint64_t r0 = base + (uint64_t)lane * kRun;
    int len = 0;
    if (r0 < total) len = (total - r0 < (uint64_t)kRun) ? (int)(total - r0) : kRun;
    uint32_t hits = 0;
    const bool known = kFill && hit_s;
    if (known) hits = hit_s[item * 32 + lane];
    uint64_t x = (known ? hits != 0 : len != 0) ? unrank(E.binom, E.S, k, r0) : 0;
    const uint64_t x0 = x;
    for (int u = 0; u < len && !known; u++) {
      int tt;
      if (is_kept_rep(T, T.rep, T.sym_off, T.sym_list, T.dest, T.phase, pre | x, &tt))
        hits |= 1u << u;
      x = next_comb(x);
    }
    if (!kFill && hit_s) hit_s[item * 32 + lane] = hits;
    const int c = __popc(hits);
    if (!kFill) {
      int tot = c;
      for (int o = 16; o > 0; o >>= 1) tot += __shfl_down_sync(0xFFFFFFFFu, tot, o);
      if (lane == 0) counts[item] = (uint32_t)tot;
    } else {
      int incl = c;
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += v;
      }
      uint64_t w = offsets[item] + (uint64_t)(incl - c);
      x = x0;
      for (int u = 0; u < len && (hits >> u); u++) {
        if (hits & (1u << u)) {
          int tt = 0;
          is_kept_rep(T, T.rep, T.sym_off, T.sym_list, T.dest, T.phase, pre | x, &tt);
          basis[w] = pre | x;
          stab[w] = (uint16_t)tt;
          w++;
        }
        x = next_comb(x);
      }
    }
  }
}

// ------------------------------ exclusive scan -------------------------------------
constexpr int kScanBlock = 1024;   // elements per CTA (256 threads x 4)

template <typename T>
__device__ T block_exclusive_scan(T v, T *total) {
  __shared__ T ws[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  T incl = v;
  for (int o = 1; o < 32; o <<= 1) {
    const T u = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= o) incl += u;
  }
  if (lane == 31) ws[wid] = incl;
  __syncthreads();
  if (wid == 0) {
    const int nw = blockDim.x >> 5;
    T a = lane < nw ? ws[lane] : 0;
    T ai = a;
    for (int o = 1; o < 32; o <<= 1) {
      const T u = __shfl_up_sync(0xFFFFFFFFu, ai, o);
      if (lane >= o) ai += u;
    }
    if (lane < nw) ws[lane] = ai - a;
    if (lane == nw - 1) ws[31] = ai;
  }
  __syncthreads();
  const T r = ws[wid] + incl - v;
  if (total) *total = ws[31];
  __syncthreads();
  return r;
}

template <typename TI>
__global__ void scan_block_sums(const TI *in, uint64_t n, uint64_t *sums) {
  const uint64_t b0 = (uint64_t)blockIdx.x * kScanBlock + threadIdx.x * 4;
  uint64_t s = 0;
  for (int u = 0; u < 4; u++) if (b0 + u < n) s += in[b0 + u];
  uint64_t tot;
  block_exclusive_scan<uint64_t>(s, &tot);
  if (threadIdx.x == 0) sums[blockIdx.x] = tot;
}

template <typename TI>
__global__ void scan_block_apply(const TI *in, uint64_t n, const uint64_t *block_off,
                                 uint64_t *out) {
  const uint64_t b0 = (uint64_t)blockIdx.x * kScanBlock + threadIdx.x * 4;
  uint64_t v[4], s = 0;
  for (int u = 0; u < 4; u++) { v[u] = (b0 + u < n) ? (uint64_t)in[b0 + u] : 0; s += v[u]; }
  uint64_t run = block_exclusive_scan<uint64_t>(s, nullptr) + (block_off ? block_off[blockIdx.x] : 0);
  for (int u = 0; u < 4; u++) {
    if (b0 + u < n) out[b0 + u] = run;
    run += v[u];
  }
}

// out[i] = sum_{j<i} in[j] (uint64), returns the total.  Scratch is allocated here.
template <typename TI>
int exclusive_scan(const TI *in, uint64_t n, uint64_t *out, uint64_t *total, cudaStream_t st) {
  if (n == 0) { *total = 0; return ED_OK; }
  const uint64_t nb = (n + kScanBlock - 1) / kScanBlock;
  if (nb == 1) {
    scan_block_apply<TI><<<1, 256, 0, st>>>(in, n, nullptr, out);
    ED_CK(cudaGetLastError());
  } else {
    Scratch sc(st);
    uint64_t *sums = (uint64_t *)sc.get(nb * 8), *offs = (uint64_t *)sc.get(nb * 8);
    if (!sums || !offs) return ed_fail(ED_ERR_OOM, "cannot allocate the scan's block sums");
    scan_block_sums<TI><<<(unsigned)nb, 256, 0, st>>>(in, n, sums);
    ED_CK(cudaGetLastError());
    uint64_t sub_total = 0;
    int rc = exclusive_scan<uint64_t>(sums, nb, offs, &sub_total, st);
    if (rc) return rc;
    scan_block_apply<TI><<<(unsigned)nb, 256, 0, st>>>(in, n, offs, out);
    ED_CK(cudaGetLastError());
  }
  // total = out[n-1] + in[n-1]
  uint64_t last_out = 0;
  TI last_in = 0;
  ED_CK(cudaMemcpyAsync(&last_out, out + n - 1, 8, cudaMemcpyDeviceToHost, st));
  ED_CK(cudaMemcpyAsync(&last_in, in + n - 1, sizeof(TI), cudaMemcpyDeviceToHost, st));
  ED_CK(cudaStreamSynchronize(st));
  *total = last_out + (uint64_t)last_in;
  return ED_OK;
}

// ------------------------------ index kernels --------------------------------------
__global__ void mark_tops(const uint64_t *basis, int64_t D, int shift, uint32_t *flags) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < D;
       i += (int64_t)gridDim.x * blockDim.x)
    flags[basis[i] >> shift] = 1u;   // every writer stores the same value
}

__global__ void make_rank(const uint32_t *flags, const uint64_t *scan, uint64_t n,
                          uint32_t *top_rank, uint32_t *rank_top) {
  for (uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (uint64_t)gridDim.x * blockDim.x) {
    if (flags[v]) { top_rank[v] = (uint32_t)scan[v]; rank_top[scan[v]] = (uint32_t)v; }
    else top_rank[v] = ED_NO_RANK;
  }
}

// limits[k] = first position whose key is >= k.  mark_limits notes the first position of every
// key that occurs; fill_limits gives the others that of the next key that does: a block owns
// 4096 keys, finds the first position beyond them by one search, and takes minima from the
// end.  (A search per key took 43 ms on the 8.6e8-state sector.)
__global__ void mark_limits(const uint64_t *basis, int64_t D, const uint32_t *top_rank, int r_shift,
                            int q_bits, int post_bits, uint32_t *limits) {
  const uint64_t qm = (1ULL << q_bits) - 1ULL;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < D;
       i += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t s = basis[i];
    const uint64_t k = ((uint64_t)top_rank[s >> r_shift] << q_bits) | ((s >> post_bits) & qm);
    if (i) {
      const uint64_t p = basis[i - 1];
      if ((((uint64_t)top_rank[p >> r_shift] << q_bits) | ((p >> post_bits) & qm)) == k) continue;
    }
    limits[k] = (uint32_t)i;
  }
}

constexpr int kLimitsTile = 4096;

__global__ void __launch_bounds__(256) fill_limits(const uint64_t *basis, int64_t D, const uint32_t *rank_top,
                                                   int r_shift, int q_bits, int post_bits, uint64_t n_keys,
                                                   uint32_t *limits) {
  constexpr int kPer = kLimitsTile / 256;
  __shared__ uint32_t next_s[256];
  __shared__ uint32_t beyond;
  const uint64_t n_tiles = (n_keys + kLimitsTile) / kLimitsTile;   // keys 0 .. n_keys
  for (uint64_t t = blockIdx.x; t < n_tiles; t += gridDim.x) {
    const uint64_t k0 = t * kLimitsTile, end = k0 + kLimitsTile;
    if (threadIdx.x == 0) {
      int64_t lo = D;
      if (end < n_keys) {   // first state whose key is >= end
        const uint64_t thr = ((uint64_t)rank_top[end >> q_bits] << r_shift) |
                             ((end & ((1ULL << q_bits) - 1ULL)) << post_bits);
        int64_t hi = D;
        lo = 0;
        while (lo < hi) {
          const int64_t m = (lo + hi) >> 1;
          if (basis[m] < thr) lo = m + 1; else hi = m;
        }
      }
      beyond = (uint32_t)lo;
    }
    // a thread owns kPer consecutive keys
    const uint64_t mine = k0 + (uint64_t)threadIdx.x * kPer;
    uint32_t v[kPer], first = 0xFFFFFFFFu;
#pragma unroll
    for (int q = kPer - 1; q >= 0; q--) {
      v[q] = mine + q < n_keys ? limits[mine + q] : 0xFFFFFFFFu;
      first = min(first, v[q]);
    }
    next_s[threadIdx.x] = first;
    __syncthreads();
    for (int o = 1; o < 256; o <<= 1) {   // suffix minima over the threads
      const uint32_t u = threadIdx.x + o < 256 ? next_s[threadIdx.x + o] : 0xFFFFFFFFu;
      __syncthreads();
      next_s[threadIdx.x] = min(next_s[threadIdx.x], u);
      __syncthreads();
    }
    uint32_t run = min(threadIdx.x < 255 ? next_s[threadIdx.x + 1] : 0xFFFFFFFFu, beyond);
#pragma unroll
    for (int q = kPer - 1; q >= 0; q--) {
      run = min(run, v[q]);
      if (mine + q <= n_keys) limits[mine + q] = run;
    }
    __syncthreads();
  }
}

// Ranked Limits (Sec. IV's Limits with the in-bucket search replaced by a rank): with at
// most 6 postfix bits a bucket is a subset of 64 values, kept as a 64-bit occupancy
// bitmap next to the bucket's first index; the index of a state is then
// start + popcount(bitmap below its postfix).  One 16-byte record per key:
// {start, 0, bitmap low word, bitmap high word}; a key that does not occur has an empty
// bitmap, which no lookup passes, and needs no start (the records are zeroed before).  The
// first state of a bucket writes its record.
__global__ void ranked_records(const uint64_t *basis, int64_t D, const uint32_t *top_rank,
                               int r_shift, int q_bits, int post_bits, uint4 *rec) {
  const uint64_t pm = (1ULL << post_bits) - 1ULL;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < D;
       i += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t s = basis[i];
    if (i && (basis[i - 1] >> post_bits) == (s >> post_bits)) continue;
    uint64_t bits = 0;
    for (int64_t j = i; j < D; j++) {
      const uint64_t u = basis[j];
      if ((u >> post_bits) != (s >> post_bits)) break;
      bits |= 1ULL << (u & pm);
    }
    const uint64_t k = ((uint64_t)top_rank[s >> r_shift] << q_bits) | ((s >> post_bits) & ((1ULL << q_bits) - 1ULL));
    rec[k] = make_uint4((uint32_t)i, 0u, (uint32_t)bits, (uint32_t)(bits >> 32));
  }
}

__global__ void max_bucket_kernel(const uint32_t *limits, uint64_t n_keys,
                                  unsigned long long *out) {
  unsigned long long m = 0;
  for (uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n_keys;
       k += (uint64_t)gridDim.x * blockDim.x)
    m = max(m, (unsigned long long)(limits[k + 1] - limits[k]));
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_down_sync(0xFFFFFFFFu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}

template <typename PT>
__global__ void make_postfix(const uint64_t *basis, int64_t D, uint64_t mask, PT *post) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < D;
       i += (int64_t)gridDim.x * blockDim.x)
    post[i] = (PT)(basis[i] & mask);
}

// The whole lookup table of a one-sublattice split: every configuration s < 2^N gets its
// representative (Eq. 4, every group element applied), the first minimising element and
// the number of minimisers.  pbit[g*N + b] is the bit that g carries bit b to.  A block takes
// kHigh x 256 configurations, a thread those with its low 8 bits: an image is the OR of the
// image of the high bits (one per element and high part, shared memory) and that of the low
// bits (a 256-entry table per element, read by neighbouring threads in one line), where
// moving the spins bit by bit took 26 ms for 50 elements on 25 sites.
__global__ void low_images(const uint8_t *pbit, int N, int nsym, uint32_t *low) {
  const int nl = min(N, 8);
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < nsym * 256; t += gridDim.x * blockDim.x) {
    const int g = t >> 8, v = t & 255;
    uint32_t m = 0;
    for (int b = 0; b < nl; b++)
      if ((v >> b) & 1) m |= 1u << pbit[g * N + b];
    low[t] = m;
  }
}

template <int kHigh>
__global__ void __launch_bounds__(256) full_table_kernel(const uint8_t *pbit, const uint8_t *flip, int N, int nsym,
                                                         const uint32_t *low, uint64_t *out) {
  extern __shared__ uint32_t hi_s[];   // [nsym][kHigh]
  const uint32_t total = 1u << N, all = total - 1u;   // N <= 26
  const uint32_t n_high = N > 8 ? 1u << (N - 8) : 1u;
  for (uint32_t h0 = blockIdx.x * kHigh; h0 < n_high; h0 += gridDim.x * kHigh) {
    for (int t = threadIdx.x; t < nsym * kHigh; t += 256) {
      const int g = t / kHigh;
      uint32_t v = flip && flip[g] ? all : 0u;   // the element also reverses every spin
      for (uint32_t m = h0 + t % kHigh; m; m &= m - 1) {
        const int b = 8 + __ffs(m) - 1;
        if (b < N) v ^= 1u << pbit[g * N + b];
      }
      hi_s[t] = v;
    }
    __syncthreads();
    uint32_t best[kHigh], gb[kHigh], cnt[kHigh];
#pragma unroll
    for (int q = 0; q < kHigh; q++) { best[q] = 0xFFFFFFFFu; gb[q] = cnt[q] = 0; }
    for (int g = 0; g < nsym; g++) {
      const uint32_t lo = __ldg(low + g * 256 + threadIdx.x);
#pragma unroll
      for (int q = 0; q < kHigh; q++) {
        const uint32_t v = hi_s[g * kHigh + q] ^ lo;
        if (v < best[q]) { best[q] = v; gb[q] = g; cnt[q] = 1; }
        else if (v == best[q]) cnt[q]++;
      }
    }
#pragma unroll
    for (int q = 0; q < kHigh; q++) {
      const uint64_t s = (uint64_t)(h0 + q) * 256 + threadIdx.x;
      if (h0 + q < n_high && s < total) out[s] = best[q] | ((uint64_t)gb[q] << 32) | ((uint64_t)cnt[q] << 48);
    }
    __syncthreads();
  }
}

uint64_t binom_host(int n, int k) {
  if (k < 0 || k > n) return 0;
  uint64_t r = 1;
  for (int i = 1; i <= k; i++) r = r * (uint64_t)(n - k + i) / (uint64_t)i;
  return r;
}

}  // namespace

int ed_exclusive_scan(const uint32_t *in, uint64_t n, uint64_t *out, uint64_t *total, cudaStream_t st) {
  return exclusive_scan<uint32_t>(in, n, out, total, st);
}

int ed_build_full_table(const uint8_t *d_pbit, const uint8_t *d_flip, int N, int nsym,
                        uint64_t *out, cudaStream_t st) {
  constexpr size_t kMaxImages = 200 * 1024;
  if ((size_t)nsym * N + nsym > kMaxImages) return ed_fail(ED_ERR_UNSUPPORTED, "group too large for the one-block table");
  // four high parts per block, one where the group's images would not fit in shared memory
  const bool four = sizeof(uint32_t) * 4 * (size_t)nsym <= 64 * 1024;
  const size_t sm = sizeof(uint32_t) * (size_t)nsym * (four ? 4 : 1);
  auto k = four ? full_table_kernel<4> : full_table_kernel<1>;
  if (sm > 48 * 1024)
    if (const int rc = ed_allow_smem(k, kMaxImages)) return rc;
  int dev = 0, nsm = 0;
  ED_CK(cudaGetDevice(&dev));
  ED_CK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  Scratch sc(st);
  uint32_t *low = (uint32_t *)sc.get(1024 * (size_t)nsym);
  if (!low) return ed_fail(ED_ERR_OOM, "cannot allocate the images of the one-block table");
  low_images<<<(nsym + 3) / 4, 256, 0, st>>>(d_pbit, N, nsym, low);
  k<<<nsm * 8, 256, sm, st>>>(d_pbit, d_flip, N, nsym, low, out);
  ED_CK(cudaGetLastError());
  return ED_OK;
}

// Build Basis, |Stab| and the index on the device.  Tables (B->T) must be in place.
int ed_build_device(ed_basis *B, cudaStream_t st, int bucket_target) {
  const int N = B->N;
  const int P = (B->nsub >= 2) ? B->n : std::min(N, 12);
  const int S = N - P;
  // prefixes to enumerate: Rep_0(v) == v when there are several sublattices
  std::vector<uint32_t> rep0;
  if (B->nsub >= 2) {
    rep0.resize((size_t)1 << B->n);
    ED_CK(cudaMemcpyAsync(rep0.data(), B->d_rep, rep0.size() * 4, cudaMemcpyDeviceToHost, st));
    ED_CK(cudaStreamSynchronize(st));
  }
  std::vector<uint32_t> tv;
  std::vector<uint8_t> tk;
  std::vector<uint64_t> ttot, titem;
  uint64_t n_items = 0;
  for (uint64_t v = 0; v < (1ULL << P); v++) {
    if (B->nsub >= 2 && rep0[v] != v) continue;
    const int k = B->n_up - __builtin_popcountll(v);
    if (k < 0 || k > S) continue;
    const uint64_t tot = binom_host(S, k);
    tv.push_back((uint32_t)v);
    tk.push_back((uint8_t)k);
    ttot.push_back(tot);
    titem.push_back(n_items);
    n_items += (tot + kItem - 1) / kItem;
  }
  B->D = 0;
  if (n_items == 0) return ED_OK;
  std::vector<uint64_t> binom(65 * 65);
  for (int a = 0; a <= 64; a++)
    for (int b = 0; b <= 64; b++) binom[a * 65 + b] = binom_host(a, b);

  // the small inputs in one upload, then the items' counts and offsets
  const size_t nt = tv.size();
  std::vector<unsigned char> blob;
  auto add = [&](const void *v, size_t bytes) {
    const size_t o = (blob.size() + 15) / 16 * 16;
    blob.resize(o + bytes);
    memcpy(blob.data() + o, v, bytes);
    return o;
  };
  const size_t o_tv = add(tv.data(), nt * 4), o_tk = add(tk.data(), nt), o_tt = add(ttot.data(), nt * 8),
               o_ti = add(titem.data(), nt * 8), o_bi = add(binom.data(), binom.size() * 8);
  const size_t o_off = (blob.size() + 15) / 16 * 16, o_cnt = o_off + n_items * 8;
  Scratch sc(st);
  unsigned char *d_in = (unsigned char *)sc.get(o_cnt + n_items * 4);
  if (!d_in) return ed_fail(ED_ERR_OOM, "cannot allocate the enumeration's scratch");
  ED_CK(cudaMemcpyAsync(d_in, blob.data(), blob.size(), cudaMemcpyHostToDevice, st));
  uint64_t *d_off = reinterpret_cast<uint64_t *>(d_in + o_off);
  uint32_t *d_counts = reinterpret_cast<uint32_t *>(d_in + o_cnt);

  EnumParams E{};
  E.T = B->T;
  E.S = S;
  E.n_tops = (int)nt;
  E.top_v = reinterpret_cast<const uint32_t *>(d_in + o_tv);
  E.top_k = d_in + o_tk;
  E.top_total = reinterpret_cast<const uint64_t *>(d_in + o_tt);
  E.top_item0 = reinterpret_cast<const uint64_t *>(d_in + o_ti);
  E.n_items = n_items;
  E.binom = reinterpret_cast<const uint64_t *>(d_in + o_bi);
  const uint64_t warps_needed = n_items;
  uint64_t grid64 = (warps_needed + 7) / 8;
  const uint64_t cap = (uint64_t)B->sm_count * 16;
  if (grid64 > cap) grid64 = cap;
  const unsigned grid = (unsigned)std::max<uint64_t>(grid64, 1);
  // 4 bytes per 32 candidates (3 bytes per state at most, less than the index takes later);
  // without memory for them the fill pass searches again
  uint32_t *d_hits = (uint32_t *)sc.get(n_items * 128);
  enum_kernel<false><<<grid, 256, 0, st>>>(E, d_counts, nullptr, nullptr, nullptr, d_hits);
  ED_CK(cudaGetLastError());
  uint64_t D = 0;
  int rc = exclusive_scan<uint32_t>(d_counts, n_items, d_off, &D, st);
  if (rc) return rc;
  if (D >= 0xFFFFFFFFull)
    return ed_fail(ED_ERR_UNSUPPORTED, "sector dimension must be below 2^32");
  B->D = (int64_t)D;
  if (D > 0) {
    if (ed_malloc(&B->d_basis, D * 8) != cudaSuccess || ed_malloc(&B->d_stab, D * 2) != cudaSuccess) {
      cudaGetLastError();
      return ed_fail(ED_ERR_OOM, "cannot allocate the basis on the device");
    }
    enum_kernel<true><<<grid, 256, 0, st>>>(E, nullptr, d_off, B->d_basis, B->d_stab, d_hits);
    ED_CK(cudaGetLastError());
  }
  sc.release(d_hits);
  sc.release(d_in);
  if (D == 0) return ED_OK;

  // ---- prefix index ----
  const int r_bits = std::min(N, 12);
  const uint64_t ntop = 1ULL << r_bits;
  const auto no_scratch = [] { return ed_fail(ED_ERR_OOM, "cannot allocate the index's scratch"); };
  uint32_t *d_flags = (uint32_t *)sc.get(ntop * 4);
  uint64_t *d_scan = (uint64_t *)sc.get(ntop * 8);
  if (!d_flags || !d_scan) return no_scratch();
  ED_CK(cudaMemsetAsync(d_flags, 0, ntop * 4, st));
  const int g1 = B->sm_count * 8;
  mark_tops<<<g1, 256, 0, st>>>(B->d_basis, B->D, N - r_bits, d_flags);
  ED_CK(cudaGetLastError());
  uint64_t R = 0;
  rc = exclusive_scan<uint32_t>(d_flags, ntop, d_scan, &R, st);
  if (rc) return rc;
  if (ed_malloc(&B->d_top_rank, ntop * 4) != cudaSuccess) {
    cudaGetLastError();
    return ed_fail(ED_ERR_OOM, "cannot allocate the prefix rank table");
  }
  uint32_t *d_rank_top = (uint32_t *)sc.get(R * 4);
  if (!d_rank_top) return no_scratch();
  make_rank<<<g1, 256, 0, st>>>(d_flags, d_scan, ntop, B->d_top_rank, d_rank_top);
  ED_CK(cudaGetLastError());
  // q: about bucket_target states per key, limited by the bits left
  int q = 0;
  const double want = (double)D / ((double)std::max(1, bucket_target) * (double)R);
  if (want > 1.0) q = (int)std::lround(std::log2(want));
  q = std::max(0, std::min(q, N - r_bits));
  while ((double)R * std::ldexp(1.0, q) > 4.0e9) q--;   // keys must fit in uint32
  const int post_bits = N - r_bits - q;
  const uint64_t n_keys = R << q;
  if (ed_malloc(&B->d_limits, (n_keys + 1) * 4) != cudaSuccess) {
    cudaGetLastError();
    return ed_fail(ED_ERR_OOM, "cannot allocate Limits");
  }
  ED_CK(cudaMemsetAsync(B->d_limits, 0xFF, (n_keys + 1) * 4, st));
  mark_limits<<<g1, 256, 0, st>>>(B->d_basis, B->D, B->d_top_rank, N - r_bits, q, post_bits, B->d_limits);
  ED_CK(cudaGetLastError());
  fill_limits<<<g1, 256, 0, st>>>(B->d_basis, B->D, d_rank_top, N - r_bits, q, post_bits, n_keys, B->d_limits);
  ED_CK(cudaGetLastError());
  unsigned long long *d_max = (unsigned long long *)sc.get(8);
  if (!d_max) return no_scratch();
  ED_CK(cudaMemsetAsync(d_max, 0, 8, st));
  max_bucket_kernel<<<g1, 256, 0, st>>>(B->d_limits, n_keys, d_max);
  ED_CK(cudaGetLastError());
  unsigned long long mb = 0;
  ED_CK(cudaMemcpyAsync(&mb, d_max, 8, cudaMemcpyDeviceToHost, st));
  const int post_bytes = post_bits <= 8 ? 1 : post_bits <= 16 ? 2 : post_bits <= 32 ? 4 : 8;
  const uint64_t pmask = post_bits >= 64 ? ~0ULL : ((1ULL << post_bits) - 1ULL);
  if (post_bytes == 8) {
    B->d_postfix = B->d_basis;   // full states are the postfixes
  } else {
    // 32 bytes of zero padding: the bucket reader loads whole 16-byte chunks
    if (ed_malloc(&B->d_postfix, (size_t)D * post_bytes + 32) != cudaSuccess) {
      cudaGetLastError();
      return ed_fail(ED_ERR_OOM, "cannot allocate postfixes");
    }
    ED_CK(cudaMemsetAsync((char *)B->d_postfix + (size_t)D * post_bytes, 0, 32, st));
    if (post_bytes == 1)
      make_postfix<uint8_t><<<g1, 256, 0, st>>>(B->d_basis, B->D, pmask, (uint8_t *)B->d_postfix);
    else if (post_bytes == 2)
      make_postfix<uint16_t><<<g1, 256, 0, st>>>(B->d_basis, B->D, pmask, (uint16_t *)B->d_postfix);
    else
      make_postfix<uint32_t><<<g1, 256, 0, st>>>(B->d_basis, B->D, pmask, (uint32_t *)B->d_postfix);
    ED_CK(cudaGetLastError());
  }
  // ranked Limits: 6 postfix bits (fewer when N - r_bits < 6), if the records fit (one
  // record per key; at most 2^32 keys and 16 bytes per key, no more than 4x the basis)
  {
    const int rq = std::max(0, N - r_bits - 6);
    const int rpost = N - r_bits - rq;
    const uint64_t rkeys = R << rq;
    if (rkeys < (1ULL << 32) && rkeys * 16 <= std::max<uint64_t>(4 * (uint64_t)D * 8, 1ULL << 26)) {
      if (ed_malloc(&B->d_rlim, rkeys * 16) == cudaSuccess) {
        ED_CK(cudaMemsetAsync(B->d_rlim, 0, rkeys * 16, st));
        ranked_records<<<g1, 256, 0, st>>>(B->d_basis, B->D, B->d_top_rank, N - r_bits, rq, rpost,
                                           reinterpret_cast<uint4 *>(B->d_rlim));
        ED_CK(cudaGetLastError());
        B->rq_bits = rq;
        B->rpost_bits = rpost;
        B->n_rkeys = (int64_t)rkeys;
      } else {
        cudaGetLastError();   // no ranked index: the kernels search the buckets instead
        B->d_rlim = nullptr;
      }
    }
  }
  for (void *q : {(void *)d_flags, (void *)d_scan, (void *)d_rank_top, (void *)d_max}) sc.release(q);
  ED_CK(cudaStreamSynchronize(st));
  B->n_keys = (int64_t)n_keys;
  B->max_bucket = (int64_t)mb;
  B->index_bytes = ntop * 4 + (n_keys + 1) * 4 + (post_bytes == 8 ? 0 : (size_t)D * post_bytes) +
                   (size_t)B->n_rkeys * 16;
  DevIndex &I = B->I;
  I.N = N;
  I.r_bits = r_bits;
  I.q_bits = q;
  I.post_bits = post_bits;
  I.post_bytes = post_bytes;
  I.D = B->D;
  I.basis = B->d_basis;
  I.stab = B->d_stab;
  I.top_rank = B->d_top_rank;
  I.limits = B->d_limits;
  I.postfix = B->d_postfix;
  I.rlim = reinterpret_cast<const uint4 *>(B->d_rlim);
  I.rq_bits = B->rq_bits;
  I.rpost_bits = B->rpost_bits;
  return ED_OK;
}
