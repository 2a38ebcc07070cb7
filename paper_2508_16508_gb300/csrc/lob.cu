// Limit order books (ABMax Section 5.3): many books matched in parallel, and
// traders' new orders placed into each book's vacant slots (the add primitive
// of Section 4 per book).
//
// Matching rule (the paper gives none; the oracle restates the same): bids in
// priority order (price descending, then time, then slot), asks likewise
// (price ascending). The traded volume V is the largest share count v such
// that the bid holding share v is priced at or above the ask holding share v;
// the first V shares of each side trade, so an order fills clamp(V - shares
// ahead of it, 0, qty) and filled orders leave the book. The price is that of
// the ask holding share V.
//
// The paper matches by sorting both sides by price and taking cumulative sums
// of shares. Here most books need no sort: with D(p) = bid shares priced >= p
// and S(p) = ask shares priced <= p,
//   V = max over p of min(D(p), S(p)),
// because the bid holding share min(D(p), S(p)) is priced >= p and the ask
// holding it <= p, while at p = the price of the ask holding share V both sums
// reach V. Only prices in [lowest ask, highest bid] matter.
//
// Level path (k_lob_match_levels): a CTA of G warps matches one book at a
// time. It stages the book's active, side, price and qty words into shared
// memory with cp.async, moves each thread's slots into registers (and starts
// staging its next book), builds per-price histograms of the range (shares |
// orders << 21, one shared atomic per order), scans them into D and S, and
// takes V, the bid level pb holding share V (largest p with D(p) >= V) and the
// ask level pa holding it (smallest p with S(p) >= V). Bids above pb and asks
// below pa fill whole, those beyond fill nothing, and only the orders on the
// two marginal levels are ranked by (time, slot), by counting.
//
// Sort path (lob_sort_book): a book whose range is wider than kWarpLevels
// prices, whose marginal level holds more than kWarpMarginal orders, or whose
// bid or ask shares reach 2^21 is left untouched by the level path and matched
// by a bitonic sort of the whole book in shared memory, cumulative sums and a
// binary search per bid: by the same CTA where every book has one, else (its
// volume set to -1) by a second kernel, k_lob_deferred.
#include <algorithm>
#include <atomic>
#include <type_traits>

#include "common.cuh"

namespace abm {

constexpr int kLobThreads = 256;        // sort path: threads per book
constexpr int kWarpLevels = 256;        // level path: prices in [lowest ask, highest bid], at most
constexpr int kWarpMarginal = 64;       // level path: orders on one marginal level, at most
constexpr u32 kShareBits = 21;          // level words: shares in the low 21 bits, orders above
constexpr u32 kShareMask = (1u << kShareBits) - 1u;
constexpr int32_t kNoPrice = 0;         // level path: a dead slot's price in registers (prices start at 1): as a bid, far
                                        // below every level


// order-preserving map of int32 onto u32
__device__ __forceinline__ u32 ord32(int32_t p) { return (u32)p ^ 0x80000000u; }

// Block-wide exclusive scan of a u64 (every thread gets its prefix and the
// total). T threads. Three barriers; the buffer is free again when it returns.
template <int T>
__device__ __forceinline__ u64 block_sum_scan_u64(u64 v, u64& total, u64* s_warp /* [T / 32 + 1] */) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  u64 incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const u64 t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    const u64 w = lane < (T / 32) ? s_warp[lane] : 0ull;
    u64 wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const u64 t = __shfl_up_sync(0xFFFFFFFFu, wi, o);
      if (lane >= o) wi += t;
    }
    if (lane < (T / 32)) s_warp[lane] = wi - w;
    if (lane == (T / 32) - 1) s_warp[(T / 32)] = wi;
  }
  __syncthreads();
  const u64 ex = s_warp[warp] + incl - v;
  total = s_warp[(T / 32)];
  __syncthreads();
  return ex;
}

// One book's words in shared memory (n entries each; slots >= cap hold
// active = 0).
struct LobBook {
  int32_t* act;
  int32_t* sid;
  int32_t* px;
  int32_t* qt;
};

// The sort path for one book (see the file comment) by T threads. n padded slots
// (a power of two, a multiple of T); key/cum share one u64 array and ord a u32 array, both [n], in
// the work area. nbid/nask: live orders per side.
template <int T>
__device__ void lob_match_sorted(const LobBook& d, int n, int b, int cap, int nbid, int nask, int32_t* active,
                                 int32_t* qty, const int32_t* __restrict__ time, long long* out_volume,
                                 int32_t* out_price, u64* key, u32* ord, u64* s_scan, unsigned long long* s_v) {
  const size_t o = (size_t)b * cap;
  __syncthreads();  // the work area may still be read as level tables
  if (threadIdx.x == 0) *s_v = 0ull;
  // key: side | price (bids descending; prices positive) | time (signed
  // order); ties by slot, empty slots (slot + n) last
#pragma unroll 4
  for (int i = threadIdx.x; i < n; i += T) {
    u64 k = kNoKey;
    u32 r = (u32)(i + n);
    if (d.act[i]) {
      const u32 s = d.sid[i] != 0;
      const u32 p = s ? (u32)d.px[i] : 0x7FFFFFFFu - (u32)d.px[i];
      k = ((u64)s << 63) | ((u64)(p & 0x7FFFFFFFu) << 32) | (u64)ord32(time[o + i]);
      r = (u32)i;
    }
    key[i] = k;
    ord[i] = r;
  }
  __syncthreads();
  // bitonic sort, a thread's pairs four at a time: all their loads before the first exchange
  for (int kk = 2; kk <= n; kk <<= 1) {
    for (int j = kk >> 1; j > 0; j >>= 1) {
      for (int p0 = threadIdx.x; p0 < n / 2; p0 += 4 * T) {
        u64 ka[4], kb[4];
        u32 oa[4], ob[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int p = p0 + u * T;
          if (p >= n / 2) continue;
          const int i = 2 * p - (p & (j - 1));  // the pair's lower entry: p with a zero bit put in at j
          ka[u] = key[i];
          kb[u] = key[i + j];
          oa[u] = ord[i];
          ob[u] = ord[i + j];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int p = p0 + u * T;
          if (p >= n / 2) continue;
          const int i = 2 * p - (p & (j - 1));
          const bool up = (i & kk) == 0;
          if ((ka[u] > kb[u] || (ka[u] == kb[u] && oa[u] > ob[u])) == up) {
            key[i] = kb[u];
            key[i + j] = ka[u];
            ord[i] = ob[u];
            ord[i + j] = oa[u];
          }
        }
      }
      __syncthreads();
    }
  }
  // sorted: bids [0, nbid), asks [nbid, nbid + nask), empty slots after. The
  // keys are dead now: cum[e] (same array) = shares of entries [0, e].
  u64* cum = key;
  const int nl = nbid + nask, per = n / T;
  u64 local = 0;
  for (int e = threadIdx.x * per; e < (threadIdx.x + 1) * per; ++e)
    local += e < nl ? (u64)(u32)d.qt[ord[e]] : 0ull;
  u64 tot;
  u64 run = block_sum_scan_u64<T>(local, tot, s_scan);
  for (int e = threadIdx.x * per; e < (threadIdx.x + 1) * per; ++e) {
    run += e < nl ? (u64)(u32)d.qt[ord[e]] : 0ull;
    cum[e] = run;
  }
  int32_t* const spx = d.sid;  // prices in sorted order (the sides are in the order now)
#pragma unroll 4
  for (int e = threadIdx.x; e < nl; e += T) spx[e] = d.px[ord[e]];
  __syncthreads();
  const u64 bid_total = nbid > 0 ? cum[nbid - 1] : 0ull;
  // V: bid i may trade the shares in (QB_{i-1}, min(QB_i, QA(J_i))], J_i = the
  // asks priced at or below it
  u64 vbest = 0;
  for (int i = threadIdx.x; i < nbid; i += T) {
    const int32_t p = spx[i];
    int lo = 0, hi = nask;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (spx[nbid + mid] <= p) lo = mid + 1;
      else hi = mid;
    }
    const u64 qa = lo > 0 ? cum[nbid + lo - 1] - bid_total : 0ull;
    const u64 qb = cum[i], before = i > 0 ? cum[i - 1] : 0ull;
    const u64 c = qa < qb ? qa : qb;
    if (c > before && c > vbest) vbest = c;
  }
  if (vbest) atomicMax(s_v, (unsigned long long)vbest);
  __syncthreads();
  const u64 V = *s_v;
  if (threadIdx.x == 0) {
    out_volume[b] = (long long)V;
    if (V == 0) out_price[b] = -1;
  }
  for (int e = threadIdx.x; e < nl; e += T) {
    const bool is_bid = e < nbid;
    const u64 start = is_bid ? (e > 0 ? cum[e - 1] : 0ull) : (e > nbid ? cum[e - 1] - bid_total : 0ull);
    const u64 end = is_bid ? cum[e] : cum[e] - bid_total;
    const u64 q = end - start;
    const u64 fill = V > start ? (V - start < q ? V - start : q) : 0ull;
    if (!is_bid && V > start && V <= end) out_price[b] = spx[e];
    if (fill || q == 0) {
      const u32 s = ord[e];
      const int32_t left = (int32_t)(q - fill);
      qty[o + s] = left;
      if (left == 0) active[o + s] = 0;
    }
  }
}

// Loads a book and matches it by the sort path; `work`: 28 bytes per padded slot.
// A CTA of the level path has 32 to 128 threads for it, so each of them keeps several
// accesses in flight: one pair after another, one wide book of 1000 slots took 73 us
// (500 books) and 137 (1000 books), of 60 slots 42; now 34, 60 and 13 (by 256 threads in a
// launch of their own before: 56, 58 and 17).
template <int T>
__device__ __noinline__ void lob_sort_book(int n, int b, int cap, int32_t* active, const int32_t* __restrict__ side,
                                           const int32_t* __restrict__ price, int32_t* qty,
                                           const int32_t* __restrict__ time, long long* out_volume, int32_t* out_price,
                                           unsigned char* work) {
  __shared__ u64 s_scan[T / 32 + 1];
  __shared__ unsigned long long s_v;
  int32_t* w = reinterpret_cast<int32_t*>(work);
  const LobBook d{w, w + n, w + 2 * n, w + 3 * n};
  u64* key = reinterpret_cast<u64*>(w + 4 * n);
  const size_t o = (size_t)b * cap;
  u64 cnt = 0;  // live bids | asks << 32
#pragma unroll 4
  for (int i = threadIdx.x; i < n; i += T) {
    const bool in = i < cap;
    const int32_t a = in ? active[o + i] : 0;
    const int32_t s = in ? side[o + i] : 0;
    d.act[i] = a;
    d.sid[i] = s;
    d.px[i] = in ? price[o + i] : 0;
    d.qt[i] = in ? qty[o + i] : 0;
    if (a != 0) cnt += s == 0 ? 1ull : 1ull << 32;
  }
  block_sum_scan_u64<T>(cnt, cnt, s_scan);
  const int nbid = (int)(u32)cnt, nask = (int)(cnt >> 32);
  lob_match_sorted<T>(d, n, b, cap, nbid, nask, active, qty, time, out_volume, out_price, key,
                      reinterpret_cast<u32*>(key + n), s_scan, &s_v);
  __syncthreads();  // the work area is used again
}

// Shared memory of one CTA of the level path (one book at a time): the staged
// book (4 arrays of n words; slots >= cap hold active = 0), the level words of
// both sides, and the marginal lists (qty, key = time | slot) of both sides.
__host__ __device__ constexpr size_t grp_smem_bytes(int n) {
  return 16 * (size_t)n + 2 * kWarpLevels * sizeof(u32) + 2 * kWarpMarginal * (sizeof(u32) + sizeof(u64));
}

// The sort path's work area for n padded slots
__host__ __device__ constexpr size_t sort_smem_bytes(int pad) {
  return (size_t)pad * (4 * sizeof(int32_t) + sizeof(u64) + sizeof(u32));
}

__device__ __forceinline__ int popc_mask(u32 m) { return __popc(m); }
__device__ __forceinline__ int popc_mask(u64 m) { return __popcll(m); }
__device__ __forceinline__ int ffs_mask(u32 m) { return __ffs(m); }
__device__ __forceinline__ int ffs_mask(u64 m) { return __ffsll((long long)m); }

// Inclusive warp scan of a u32.
__device__ __forceinline__ u32 warp_incl_scan(u32 v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const u32 t = __shfl_up_sync(0xFFFFFFFFu, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

// Barrier of the G warps matching one book.
template <int G>
__device__ __forceinline__ void grp_sync() {
  if (G == 1) __syncwarp();
  else __syncthreads();
}

// Signed min and max, or, and "any" over the G warps (every thread gets them).
// One barrier; the exchange buffer alternates between calls.
struct Agg {
  int32_t mn, mx;
  u32 orr;
  bool any;
};
template <int G>
__device__ __forceinline__ Agg grp_agg(Agg a, u32 (*x)[G][4], int& par) {
  a.mn = __reduce_min_sync(0xFFFFFFFFu, a.mn);
  a.mx = __reduce_max_sync(0xFFFFFFFFu, a.mx);
  a.orr = __reduce_or_sync(0xFFFFFFFFu, a.orr);
  a.any = __any_sync(0xFFFFFFFFu, a.any);
  if (G == 1) return a;
  if ((threadIdx.x & 31) == 0)
    *reinterpret_cast<uint4*>(x[par][threadIdx.x >> 5]) = make_uint4((u32)a.mn, (u32)a.mx, a.orr, a.any ? 1u : 0u);
  __syncthreads();
  Agg r{INT32_MAX, INT32_MIN, 0u, false};
#pragma unroll
  for (int w = 0; w < G; ++w) {
    const uint4 d = *reinterpret_cast<const uint4*>(x[par][w]);
    r.mn = min(r.mn, (int32_t)d.x);
    r.mx = max(r.mx, (int32_t)d.y);
    r.orr |= d.z;
    r.any = r.any || d.w != 0u;
  }
  par ^= 1;
  return r;
}

// Max of a u32 over the G warps (every thread gets it). One barrier.
template <int G>
__device__ __forceinline__ u32 grp_max(u32 v, u32 (*x)[G][4], int& par) {
  v = __reduce_max_sync(0xFFFFFFFFu, v);
  if (G == 1) return v;
  if ((threadIdx.x & 31) == 0) x[par][threadIdx.x >> 5][0] = v;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < G; ++w) v = max(v, x[par][w][0]);
  par ^= 1;
  return v;
}

// Exclusive scan of two u32 over the G warps' threads, with the totals.
template <int G>
__device__ __forceinline__ void grp_scan2(u32 a, u32 b, u32& ex_a, u32& ex_b, u32& tot_a, u32& tot_b,
                                          u32 (*x)[G][4], int& par) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const u32 ia = warp_incl_scan(a, lane), ib = warp_incl_scan(b, lane);
  if (G == 1) {
    ex_a = ia - a;
    ex_b = ib - b;
    tot_a = __shfl_sync(0xFFFFFFFFu, ia, 31);
    tot_b = __shfl_sync(0xFFFFFFFFu, ib, 31);
    return;
  }
  if (lane == 31) {
    x[par][warp][0] = ia;
    x[par][warp][1] = ib;
  }
  __syncthreads();
  u32 pa = 0, pb = 0, ta = 0, tb = 0;
#pragma unroll
  for (int w = 0; w < G; ++w) {
    const u32 wa = x[par][w][0], wb = x[par][w][1];
    pa += w < warp ? wa : 0u;
    pb += w < warp ? wb : 0u;
    ta += wa;
    tb += wb;
  }
  ex_a = pa + ia - a;
  ex_b = pb + ib - b;
  tot_a = ta;
  tot_b = tb;
  par ^= 1;
}

// Book b's words into the staging arrays (asynchronous; committed). T
// threads copy.
template <int T, bool kVec16>
__device__ __forceinline__ void grp_stage(int32_t* s_act, int n, int b, int cap, const int32_t* active,
                                          const int32_t* side, const int32_t* price, const int32_t* qty) {
  const size_t o = (size_t)b * cap;
  if (kVec16) {
    for (int c = threadIdx.x; c < (cap >> 2); c += T) {
      cp_async16(s_act + 4 * c, active + o + 4 * c);
      cp_async16(s_act + n + 4 * c, side + o + 4 * c);
      cp_async16(s_act + 2 * n + 4 * c, price + o + 4 * c);
      cp_async16(s_act + 3 * n + 4 * c, qty + o + 4 * c);
    }
  } else {
    for (int c = threadIdx.x; c < cap; c += T) {
      cp_async4(s_act + c, active + o + c);
      cp_async4(s_act + n + c, side + o + c);
      cp_async4(s_act + 2 * n + c, price + o + c);
      cp_async4(s_act + 3 * n + c, qty + o + c);
    }
  }
  cp_async_commit();
}

// Level path: a CTA of G warps (T = 32 G threads) matches one book at a time;
// SPL = slots per thread (cap <= T * SPL), thread t holding slots
// 4 * (g * T + t) + c. The book's words move from the staging arrays into
// registers, and the next book is staged at once. Books for the sort path are left
// untouched and get out_volume = -1, or with FOLD (every CTA has one book) are
// handed to it at the end.
//
// Bound by the chain of a book's dependent steps at the occupancy that the staged
// words allow (10 CTAs per SM): 65536 books of 1024 slots take 299 us with four
// warps per book and move 1.66 GB (249 us at the copy rate); issue slots are half
// full. Levels written back and counted, marginal orders listed and fetched one by
// one: 326 us with two warps, and 454 before the loops over the slots were cut to
// what each needs. Loads straight into registers with the next book prefetched
// into L2 are no faster (297 to 315 us).
template <int G, int SPL, bool kVec16, bool FOLD>
__global__ void __launch_bounds__(G * 32)
    k_lob_match_levels(int n_books, int cap, int32_t* active, const int32_t* __restrict__ side,
                       const int32_t* __restrict__ price, int32_t* qty, const int32_t* __restrict__ time,
                       long long* out_volume, int32_t* out_price) {
  constexpr int T = G * 32;
  constexpr int LPT = kWarpLevels / T;  // levels per thread in the scan
  constexpr int n = T * SPL;            // staged words per array
  extern __shared__ __align__(16) unsigned char lob_smem[];
  __shared__ __align__(16) u32 s_x[2][G][4];
  __shared__ u32 s_mar[2][3];  // per side: the marginal level, the shares of the better ones, its orders
  __shared__ u32 s_cnt;        // marginal orders listed: bids | asks << 16
  int32_t* s_act = reinterpret_cast<int32_t*>(lob_smem);  // then side, price, qty at +n, +2n, +3n
  u32* lv = reinterpret_cast<u32*>(s_act + 4 * n);        // level words: bids, then asks
  u32* m_qty = lv + 2 * kWarpLevels;                      // [2][kWarpMarginal]: slots, then quantities
  u64* m_key = reinterpret_cast<u64*>(m_qty + 2 * kWarpMarginal);  // [2][kWarpMarginal]
  const int t = threadIdx.x;
  int par = 0;
  int defer = -1;  // FOLD: this CTA's book, if the sort path has to take it
  for (int i = cap + t; i < n; i += T) s_act[i] = 0;  // padding slots: never copied, never live
  griddep_wait();
  // the sort path's few CTAs may start (and the next call's beside those: 100 steps
  // of 500 books in two launches a round 761 -> 748 us). Not from k_lob_add: its
  // successor's CTAs then crowd the SMs that are free at that moment (968 us).
  griddep_launch();
  if ((int)blockIdx.x < n_books) grp_stage<T, kVec16>(s_act, n, blockIdx.x, cap, active, side, price, qty);
  for (int b = blockIdx.x; b < n_books; b += gridDim.x) {
    const size_t o = (size_t)b * cap;
    cp_async_wait_0();
    grp_sync<G>();

    // the level words are free since that barrier; the next one comes before they are used
#pragma unroll
    for (int l = t; l < 2 * kWarpLevels / 4; l += T) reinterpret_cast<uint4*>(lv)[l] = make_uint4(0u, 0u, 0u, 0u);
    if (t == 0) s_cnt = 0u;

    // this thread's slots into registers: price (kNoPrice: dead) and qty | ask in
    // the sign bit, dead slots as bids of one share (far below every level). The
    // loops over the slots are most of a book's instructions, so each keeps to what
    // it needs.
    int32_t px[SPL];
    u32 w[SPL];
    int32_t mn = INT32_MAX, mx = INT32_MIN;  // lowest ask, highest bid
    u32 qor = 0, qmin = 1;
#pragma unroll
    for (int g = 0; g < SPL / 4; ++g) {
      const int v = g * T + t;
      const int4 a4 = reinterpret_cast<const int4*>(s_act)[v];
      const int4 s4 = reinterpret_cast<const int4*>(s_act + n)[v];
      const int4 p4 = reinterpret_cast<const int4*>(s_act + 2 * n)[v];
      const int4 q4 = reinterpret_cast<const int4*>(s_act + 3 * n)[v];
      const int av[4] = {a4.x, a4.y, a4.z, a4.w}, sv[4] = {s4.x, s4.y, s4.z, s4.w};
      const int pv[4] = {p4.x, p4.y, p4.z, p4.w}, qv[4] = {q4.x, q4.y, q4.z, q4.w};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int k = 4 * g + c;
        const bool live = av[c] != 0, ask = live && sv[c] != 0;
        const u32 q = live ? (u32)qv[c] : 1u;
        px[k] = live ? pv[c] : kNoPrice;
        qor |= q;
        qmin = min(qmin, q);
        if (ask) mn = min(mn, px[k]);
        else mx = max(mx, px[k]);
        w[k] = ask ? q | 0x80000000u : q;
      }
    }
    // for G > 1 the barrier inside also frees the staging arrays
    const Agg r1 = grp_agg<G>(Agg{mn, mx, qor, qmin == 0}, s_x, par);
    if (G == 1) __syncwarp();
    if (b + (int)gridDim.x < n_books)
      grp_stage<T, kVec16>(s_act, n, b + gridDim.x, cap, active, side, price, qty);
    const bool zq = r1.any;
    const int32_t pmin = r1.mn, pmax = r1.mx;
    // (without asks or without bids the test can hold for one extreme price: no volume comes of it)
    const bool cross = pmax >= pmin;
    const long long L = cross ? (long long)pmax - (long long)pmin + 1 : 0;
    if (cross) {
      // a level word holds share sums below 2^kShareBits: certainly if every qty could be the or of them all, else by
      // the sums themselves (saturating per thread, so that they cannot wrap)
      bool wide = L > kWarpLevels || r1.orr > kShareMask;
      if (!wide && (u64)r1.orr * (u32)cap > kShareMask) {
        u32 sb = 0, sa = 0;
#pragma unroll
        for (int k = 0; k < SPL; ++k) {
          const u32 q = w[k] & kShareMask;
          if ((int32_t)w[k] < 0) sa += q;
          else sb += px[k] != kNoPrice ? q : 0u;
        }
        u32 ex_b, ex_a, tb, ta;
        grp_scan2<G>(min(sb, 1u << kShareBits), min(sa, 1u << kShareBits), ex_b, ex_a, tb, ta, s_x, par);
        wide = tb > kShareMask || ta > kShareMask;
      }
      if (wide) {
        if (FOLD) defer = b;  // the sort path takes it
        else if (t == 0) out_volume[b] = -1;
        continue;
      }
    }
    u32 V = 0;
    int lb = 0, la = 0;  // the marginal levels
    u32 Dn = 0, Sp = 0;  // bid shares priced above pb, ask shares priced below pa
    if (cross) {
      // live asks lie at or above pmin and live bids at or below pmax, so one
      // unsigned comparison tells an order in the range from the others and the
      // dead. (Quantities below 2^kShareBits: w >> 23 is 256 for asks, 0 for bids.)
      static_assert(kWarpLevels == 256 && kShareBits <= 23, "level word of an order");
#pragma unroll
      for (int k = 0; k < SPL; ++k) {
        const u32 l = (u32)px[k] - (u32)pmin;
        if (l < (u32)L) atomicAdd(lv + (l + (w[k] >> 23)), (w[k] & kShareMask) | (1u << kShareBits));
      }
      grp_sync<G>();
      // D(l) = bid shares at levels >= l, S(l) = ask shares at levels <= l;
      // thread t owns levels [LPT * t, LPT * t + LPT). Levels from L on hold no
      // order: D = 0 there.
      u32 hb[LPT], ha[LPT];
      u32 tb = 0, ta = 0;
      const int l0 = t * LPT;
#pragma unroll
      for (int j = 0; j < LPT; j += 2) {
        const uint2 vb = *reinterpret_cast<const uint2*>(lv + l0 + j);
        const uint2 va = *reinterpret_cast<const uint2*>(lv + kWarpLevels + l0 + j);
        hb[j] = vb.x;
        hb[j + 1] = vb.y;
        ha[j] = va.x;
        ha[j + 1] = va.y;
      }
#pragma unroll
      for (int j = 0; j < LPT; ++j) {
        tb += hb[j] & kShareMask;
        ta += ha[j] & kShareMask;
      }
      u32 pre_b, pre_a, BT, AT;
      grp_scan2<G>(tb, ta, pre_b, pre_a, BT, AT, s_x, par);
      u32 best = 0, D = BT - pre_b, S = pre_a;
#pragma unroll
      for (int j = 0; j < LPT; ++j) {
        S += ha[j] & kShareMask;
        best = max(best, min(D, S));
        D -= hb[j] & kShareMask;
      }
      V = grp_max<G>(best, s_x, par);
      if (V > 0) {
        // D falls and S rises with the level: the one bid level with D >= V and less
        // above it, the one ask level with S >= V and less below it
        D = BT - pre_b;
        S = pre_a;
#pragma unroll
        for (int j = 0; j < LPT; ++j) {
          const u32 Dnext = D - (hb[j] & kShareMask), Snext = S + (ha[j] & kShareMask);
          if (D >= V && Dnext < V) {
            s_mar[0][0] = (u32)(l0 + j);
            s_mar[0][1] = Dnext;
            s_mar[0][2] = hb[j] >> kShareBits;
          }
          if (Snext >= V && S < V) {
            s_mar[1][0] = (u32)(l0 + j);
            s_mar[1][1] = S;
            s_mar[1][2] = ha[j] >> kShareBits;
          }
          D = Dnext;
          S = Snext;
        }
        grp_sync<G>();
        lb = (int)s_mar[0][0];
        la = (int)s_mar[1][0];
        Dn = s_mar[0][1];
        Sp = s_mar[1][1];
        if (max(s_mar[0][2], s_mar[1][2]) > kWarpMarginal) {
          if (FOLD) defer = b;  // a crowded marginal level: the sort path takes it
          else if (t == 0) out_volume[b] = -1;
          continue;
        }
      }
    }
    if (V == 0 && !zq) {
      if (t == 0) {
        out_volume[b] = 0;
        out_price[b] = -1;
      }
      continue;
    }
    // whole fills (and zero-qty orders) written here; marginal orders marked
    // in per-thread bit masks (bit k = this thread's slot k), listed below
    using Mask = typename std::conditional<(SPL > 32), u64, u32>::type;
    Mask mmb = 0, mma = 0;
    if (V > 0) {
      // d = levels past the marginal one minus 1. Whole fills have d in [0, L), the
      // marginal orders d = -1; the others and the dead (price 0) are far outside.
      const u32 cb = (u32)pmin + (u32)lb + 1u, ca = (u32)pmin + (u32)la - 1u;
#pragma unroll
      for (int k = 0; k < SPL; ++k) {
        const int i = 4 * ((k >> 2) * T + t) + (k & 3);
        const bool ask = (int32_t)w[k] < 0;
        const u32 d = ask ? ca - (u32)px[k] : (u32)px[k] - cb;
        if (d < (u32)L) {
          qty[o + i] = 0;
          active[o + i] = 0;
        }
        if (d == 0xFFFFFFFFu) {
          if (ask) mma |= (Mask)1 << k;
          else mmb |= (Mask)1 << k;
        }
      }
    }
    if (zq) {  // live orders without shares leave the book, whatever their price
#pragma unroll
      for (int k = 0; k < SPL; ++k) {
        const int i = 4 * ((k >> 2) * T + t) + (k & 3);
        if ((w[k] & 0x7FFFFFFFu) == 0) {
          active[o + i] = 0;
          mmb &= ~((Mask)1 << k);
          mma &= ~((Mask)1 << k);
        }
      }
    }
    if (V > 0) {
      // the marginal orders' slots listed in any order, then their qty and time from
      // global memory (neither written by this kernel) in one round trip
      if (mmb | mma) {
        const u32 at = atomicAdd(&s_cnt, (u32)popc_mask(mmb) | ((u32)popc_mask(mma) << 16));
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          Mask m = s ? mma : mmb;
          u32* list = m_qty + (s ? kWarpMarginal + (at >> 16) : (at & 0xFFFFu));
          while (m) {
            const int k = ffs_mask(m) - 1;
            m &= m - 1;
            *list++ = 4u * (u32)((k >> 2) * T + t) + (u32)(k & 3);
          }
        }
      }
      grp_sync<G>();
      const u32 nm0 = s_cnt & 0xFFFFu, nm1 = s_cnt >> 16;
      for (u32 e = t; e < nm0 + nm1; e += T) {
        const u32 f = e < nm0 ? e : e - nm0 + kWarpMarginal, i = m_qty[f];
        const u32 q = (u32)qty[o + i];
        m_key[f] = ((u64)ord32(time[o + i]) << 32) | i;
        m_qty[f] = q;
      }
      grp_sync<G>();
      for (u32 e = t; e < nm0 + nm1; e += T) {
        const int s = e >= nm0, f = (int)e - (s ? (int)nm0 : 0), m = s ? (int)nm1 : (int)nm0;
        const u32* mq = m_qty + s * kWarpMarginal;
        const u64* mk = m_key + s * kWarpMarginal;
        const u64 mine = mk[f];
        u32 before = s ? Sp : Dn;
        for (int h = 0; h < m; ++h) before += mk[h] < mine ? mq[h] : 0u;
        const u32 q = mq[f];
        const u32 fill = V > before ? min(V - before, q) : 0u;
        if (fill) {
          const u32 slot = (u32)mine;
          qty[o + slot] = (int32_t)(q - fill);
          if (fill == q) active[o + slot] = 0;
        }
      }
    }
    if (t == 0) {
      out_volume[b] = (long long)V;
      out_price[b] = V > 0 ? pmin + la : -1;
    }
  }
  cp_async_wait_0();
  if constexpr (FOLD) {
    if (defer >= 0) {
      grp_sync<G>();  // the level path's shared memory becomes the work area
      lob_sort_book<T>(n, defer, cap, active, side, price, qty, time, out_volume, out_price, lob_smem);
    }
  }
}

// Sort path for the books the level path deferred (out_volume < 0), one CTA
// per book; n = R * kLobThreads padded slots. Shared memory: the book's words
// (4 x n int32), then key u64[n] and ord u32[n].
template <int R>
__global__ void __launch_bounds__(kLobThreads)
    k_lob_deferred(int n_books, int cap, int32_t* active, const int32_t* __restrict__ side,
                   const int32_t* __restrict__ price, int32_t* qty, const int32_t* __restrict__ time,
                   long long* out_volume, int32_t* out_price) {
  extern __shared__ __align__(16) unsigned char lob_smem[];
  __shared__ int s_list[kLobThreads];
  __shared__ int s_cnt;
  griddep_wait();
  griddep_launch();
  for (int c0 = blockIdx.x * kLobThreads; c0 < n_books; c0 += gridDim.x * kLobThreads) {
    if (threadIdx.x == 0) s_cnt = 0;
    __syncthreads();
    const int bq = c0 + threadIdx.x;
    if (bq < n_books && out_volume[bq] < 0) s_list[atomicAdd(&s_cnt, 1)] = bq;
    __syncthreads();
    const int m = s_cnt;
    for (int j = 0; j < m; ++j)
      lob_sort_book<kLobThreads>(R * kLobThreads, s_list[j], cap, active, side, price, qty, time, out_volume, out_price,
                                 lob_smem);
    __syncthreads();
  }
}

// New orders into each book's lowest free slots: order j < k[b] -> j-th free
// slot. One warp per book takes 128 slots at a time (four per lane) and stops
// as soon as its orders are placed, so a book costs the first few slots of its
// live flags, not all of them. The warp lists a chunk's free slots in shared
// memory and lane j then places order j; a chunk's first 32 orders are fetched
// together with its flags. (A CTA per book that read every flag twice and
// ranked them by a block scan: 3.7 us for 500 books of 1000 slots and 10 orders
// each; now 2.5.)
constexpr int kAddWarps = 4;

template <bool kVec16>
__global__ void __launch_bounds__(kAddWarps * 32) k_lob_add(int n_books, int cap, int32_t* active, int32_t* side,
                                                            int32_t* price, int32_t* qty, int32_t* time,
                                                            const int32_t* __restrict__ orders,
                                                            const int32_t* __restrict__ k, int kmax,
                                                            int32_t* out_added) {
  __shared__ unsigned short s_free[kAddWarps][128];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned short* fl = s_free[warp];
  griddep_wait();
  for (int b = blockIdx.x * kAddWarps + warp; b < n_books; b += gridDim.x * kAddWarps) {
    const size_t o = (size_t)b * cap;
    const int32_t* act = active + o;
    const int32_t* ord = orders + (size_t)b * kmax * 4;
    const int kb = min(max(k[b], 0), kmax);
    int placed = 0;
    for (int c0 = 0; c0 < cap && placed < kb; c0 += 128) {
      const int i0 = c0 + 4 * lane;
      // the next orders in flight beside the flags
      int r[4] = {0, 0, 0, 0};
      if (placed + lane < kmax)
#pragma unroll
        for (int f = 0; f < 4; ++f) r[f] = ord[4 * (size_t)(placed + lane) + f];
      u32 fr = 0;
      if (kVec16 && i0 < cap) {  // cap is a multiple of 4
        const int4 a = *reinterpret_cast<const int4*>(act + i0);
        fr = (u32)(a.x == 0) | ((u32)(a.y == 0) << 1) | ((u32)(a.z == 0) << 2) | ((u32)(a.w == 0) << 3);
      } else if (!kVec16) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (i0 + j < cap) fr |= (u32)(act[i0 + j] == 0) << j;
      }
      const u32 n = (u32)__popc(fr);
      const u32 inc = warp_incl_scan(n, lane);
      const int found = (int)__shfl_sync(0xFFFFFFFFu, inc, 31);
      u32 pos = inc - n;
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if ((fr >> j) & 1u) fl[pos++] = (unsigned short)(i0 + j);
      __syncwarp();
      const int take = min(found, kb - placed);
      for (int e = lane; e < take; e += 32) {
        if (e >= 32) {
#pragma unroll
          for (int f = 0; f < 4; ++f) r[f] = ord[4 * (size_t)(placed + e) + f];
        }
        const size_t i = o + fl[e];
        side[i] = r[0];
        price[i] = r[1];
        qty[i] = r[2];
        time[i] = r[3];
        active[i] = 1;
      }
      placed += max(take, 0);
      __syncwarp();
    }
    if (lane == 0) out_added[b] = placed;
  }
}


static int lob_pad(int cap) {
  int n = kLobThreads;
  while (n < cap) n <<= 1;
  return n;
}

static std::atomic<int> g_lob_warps_per_book{0};  // level path: warps per book (1, 2 or 4; 0: by the capacity)

// FOLD: every book has a CTA of its own at once, which also takes it by the sort
// path where that is called for. grid = 0: as many CTAs as the device holds.
template <int G, int SPL, bool kVec16, bool FOLD>
static abm_status lob_levels(int& grid, int n_books, int cap, int32_t* active, const int32_t* side,
                             const int32_t* price, int32_t* qty, const int32_t* time, long long* vol, int32_t* px,
                             cudaStream_t st) {
  // the shared-memory limit and the occupancy are per device: looked up once for each
  static std::atomic<unsigned long long> attr{0};
  static std::atomic<int> occ_dev[64];
  constexpr int n = G * 32 * SPL;
  const size_t smem = std::max(grp_smem_bytes(n), FOLD ? sort_smem_bytes(n) : 0);
  const auto kernel = k_lob_match_levels<G, SPL, kVec16, FOLD>;
  ABM_CUDA_TRY(smem_attr_once(kernel, (int)smem, attr));
  int dev = 0;
  ABM_CUDA_TRY(cudaGetDevice(&dev));
  int blocks_per_sm = (dev >= 0 && dev < 64) ? occ_dev[dev].load(std::memory_order_relaxed) : 0;
  if (!blocks_per_sm) {
    int occ = 0;
    ABM_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, G * 32, smem));
    blocks_per_sm = std::max(occ, 1);
    if (dev >= 0 && dev < 64) occ_dev[dev].store(blocks_per_sm, std::memory_order_relaxed);
  }
  const long long held = (long long)num_sms() * blocks_per_sm;
  grid = (int)std::min<long long>(n_books, held);
  if (FOLD && n_books > held) return ABM_OK;
  ABM_CUDA_TRY(launch_pdl_smem(kernel, grid, G * 32, smem, st, n_books, cap, active, side, price, qty, time, vol, px));
  return ABM_OK;
}

// Books that all have a CTA at once are matched in one launch; with more of them the
// sort path is a launch of its own, whose work area does not cost the level path
// its occupancy. 100 steps of orders and matching: 500 books of 1000 slots 740 -> 692
// us, 1000 books 890 -> 808, 100 books of 300 slots 643 -> 540. A book for the sort path
// is also taken at once instead of one after another by the CTA of its 256 books.
template <int G, int SPL, bool kVec16>
static abm_status lob_launch_levels(bool& folded, int n_books, int cap, int32_t* active, const int32_t* side,
                                    const int32_t* price, int32_t* qty, const int32_t* time, long long* vol, int32_t* px,
                                    cudaStream_t st) {
  int grid = 0;
  abm_status e = lob_levels<G, SPL, kVec16, true>(grid, n_books, cap, active, side, price, qty, time, vol, px, st);
  folded = grid == n_books;
  if (e != ABM_OK || folded) return e;
  return lob_levels<G, SPL, kVec16, false>(grid, n_books, cap, active, side, price, qty, time, vol, px, st);
}

// the smallest slots-per-thread (a multiple of 4) that covers cap
template <int G, bool kVec16>
static abm_status lob_launch_g(bool& folded, int n_books, int cap, int32_t* active, const int32_t* side, const int32_t* price,
                               int32_t* qty, const int32_t* time, long long* vol, int32_t* px, cudaStream_t st) {
  constexpr int T = G * 32;
  if (cap <= 4 * T) return lob_launch_levels<G, 4, kVec16>(folded, n_books, cap, active, side, price, qty, time, vol, px, st);
  if (cap <= 8 * T) return lob_launch_levels<G, 8, kVec16>(folded, n_books, cap, active, side, price, qty, time, vol, px, st);
  if (cap <= 16 * T)
    return lob_launch_levels<G, 16, kVec16>(folded, n_books, cap, active, side, price, qty, time, vol, px, st);
  if (G <= 2 && cap <= 32 * T)
    return lob_launch_levels<G, (G <= 2 ? 32 : 16), kVec16>(folded, n_books, cap, active, side, price, qty, time, vol, px,
                                                             st);
  return lob_launch_levels<G, (G == 1 ? 64 : 16), kVec16>(folded, n_books, cap, active, side, price, qty, time, vol, px,
                                                           st);
}

template <int R>
static abm_status lob_launch_deferred(int n_books, int cap, int32_t* active, const int32_t* side,
                                      const int32_t* price, int32_t* qty, const int32_t* time, long long* vol,
                                      int32_t* px, cudaStream_t st) {
  constexpr size_t smem = sort_smem_bytes(R * kLobThreads);
  static std::atomic<unsigned long long> attr{0};
  ABM_CUDA_TRY(smem_attr_once(k_lob_deferred<R>, (int)smem, attr));
  const long long chunks = ((long long)n_books + kLobThreads - 1) / kLobThreads;
  const int grid = (int)std::min<long long>(chunks, (long long)num_sms() * 2);
  ABM_CUDA_TRY(launch_pdl_smem(k_lob_deferred<R>, grid, kLobThreads, smem, st, n_books, cap, active, side, price, qty,
                               time, vol, px));
  return ABM_OK;
}

static abm_status lob_launch(bool vec16, int n_books, int cap, int32_t* active, const int32_t* side,
                             const int32_t* price, int32_t* qty, const int32_t* time, long long* vol, int32_t* px,
                             cudaStream_t st) {
  abm_status e;
  bool folded = false;
  int g = g_lob_warps_per_book.load(std::memory_order_relaxed);
  // One warp matches a book of up to 256 slots (8 per lane) faster than two that
  // meet at a barrier after every step (20,000 books of 128 slots 22 us against 35,
  // 50,000 of 256 slots 73 against 89; 20,000 of 512 57 against 56, of 768 93 against
  // 82), and four share more than 768 slots better than two (65536 books of 1024
  // slots 299 against 313, 16384 of 2048 158 against 169; 768 slots the same).
  // With few books a book's own chain counts, which more warps shorten until the SMs
  // fill up; so the lines lie at books per SM. A placement and a matching round, us with
  // 1 / 2 / 4 warps: 300 books of 200 slots 5.7 / 5.3 / 5.5, of 400 6.6 / 5.7 / 5.6, of 1000
  // 8.2 / 6.3 / 6.0; 500 books of 400 6.7 / 5.8 / 5.9, of 1000 8.3 / 6.8 / 6.8; 1000 books of 200
  // 6.0 / 5.9 / 6.5, of 1000 9.5 / 8.2 / 8.8; 1700 books of 200 6.4 / 6.6 / 9.0, of 400 7.7 / 7.4 /
  // 9.1, of 768 14.7 / 11.9 / 11.3. Books of 513 to 1024 slots take two warps between the first
  // lines (four of them no longer find room on the SMs) and four again above seven books
  // per SM, where the books do not all have a CTA at once and a round is two launches.
  if (g == 0) {
    const int sms = num_sms();
    const int one = n_books <= 8 * sms ? 128 : 256;
    const int two = 2 * n_books <= 7 * sms ? 256 : n_books <= 7 * sms ? 1024 : 2 * n_books <= 27 * sms ? 512 : 768;
    g = cap <= one ? 1 : (cap <= two ? 2 : 4);
  }
  switch (g) {
    case 1:
      e = vec16 ? lob_launch_g<1, true>(folded, n_books, cap, active, side, price, qty, time, vol, px, st)
                : lob_launch_g<1, false>(folded, n_books, cap, active, side, price, qty, time, vol, px, st);
      break;
    case 4:
      e = vec16 ? lob_launch_g<4, true>(folded, n_books, cap, active, side, price, qty, time, vol, px, st)
                : lob_launch_g<4, false>(folded, n_books, cap, active, side, price, qty, time, vol, px, st);
      break;
    default:
      e = vec16 ? lob_launch_g<2, true>(folded, n_books, cap, active, side, price, qty, time, vol, px, st)
                : lob_launch_g<2, false>(folded, n_books, cap, active, side, price, qty, time, vol, px, st);
  }
  if (e != ABM_OK || folded) return e;
  switch (lob_pad(cap) / kLobThreads) {
    case 1: return lob_launch_deferred<1>(n_books, cap, active, side, price, qty, time, vol, px, st);
    case 2: return lob_launch_deferred<2>(n_books, cap, active, side, price, qty, time, vol, px, st);
    case 4: return lob_launch_deferred<4>(n_books, cap, active, side, price, qty, time, vol, px, st);
    default: return lob_launch_deferred<8>(n_books, cap, active, side, price, qty, time, vol, px, st);
  }
}

}  // namespace abm

using namespace abm;

extern "C" abm_status abm_lob_match(int32_t n_books, int32_t cap, int32_t* active, const int32_t* side,
                                    const int32_t* price, int32_t* qty, const int32_t* time, int64_t* out_volume,
                                    int32_t* out_price, void* stream) {
  if (n_books < 0 || cap < 1 || cap > ABM_LOB_MAX_CAP) return ABM_ERR_ARG;
  if (n_books == 0) return ABM_OK;
  if (!active || !side || !price || !qty || !time || !out_volume || !out_price) return ABM_ERR_ARG;
  // 16-byte copies need every book's rows 16-byte aligned
  const bool vec16 =
      cap % 4 == 0 && ((uintptr_t)active | (uintptr_t)side | (uintptr_t)price | (uintptr_t)qty) % 16 == 0;
  long long* vol = reinterpret_cast<long long*>(out_volume);
  const cudaStream_t st = (cudaStream_t)stream;
  return lob_launch(vec16, n_books, cap, active, side, price, qty, time, vol, out_price, st);
}

extern "C" abm_status abm_lob_tune(int32_t warps_per_book) {
  if (warps_per_book != 0 && warps_per_book != 1 && warps_per_book != 2 && warps_per_book != 4) return ABM_ERR_ARG;
  g_lob_warps_per_book.store(warps_per_book, std::memory_order_relaxed);
  return ABM_OK;
}

extern "C" abm_status abm_lob_add(int32_t n_books, int32_t cap, int32_t* active, int32_t* side, int32_t* price,
                                  int32_t* qty, int32_t* time, const int32_t* new_orders, const int32_t* k,
                                  int32_t kmax, int32_t* out_added, void* stream) {
  if (n_books < 0 || cap < 1 || cap > ABM_LOB_MAX_CAP || kmax < 0) return ABM_ERR_ARG;
  if (n_books == 0) return ABM_OK;
  if (!active || !side || !price || !qty || !time || !k || !out_added || (kmax > 0 && !new_orders))
    return ABM_ERR_ARG;
  const int grid = (int)std::min<long long>(((long long)n_books + kAddWarps - 1) / kAddWarps, (long long)num_sms() * 16);
  const bool vec16 = cap % 4 == 0 && (uintptr_t)active % 16 == 0;
  ABM_CUDA_TRY(launch_pdl(vec16 ? k_lob_add<true> : k_lob_add<false>, grid, kAddWarps * 32, (cudaStream_t)stream, n_books,
                          cap, active, side, price, qty, time, new_orders, k, kmax, out_added));
  return ABM_OK;
}
