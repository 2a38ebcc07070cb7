// sort_agents (ABMax Section 2 API list): reorder a slab so that its live
// agents come first, ascending by one int32 field with ties kept in slot
// order, and the placeholders after them in slot order.
//
// The live slots are first packed, in slot order, as (key, slot) pairs, key =
// the field with its sign bit flipped (so unsigned order is signed order);
// placeholders need no sorting, so they are only listed. The packing pass also
// collects the keys' set and cleared bits, which shows which bytes hold one value
// only (the high bytes of cells, ids and ages): their passes are left out. An LSD
// radix sort of the pairs then runs one pass per byte that is left: digit counts
// per chunk and in all, a scan over the chunks, and a stable scatter. Finally every agent's row (fields + live flag) is gathered
// into spare arrays, which then become the slab's arrays.
//
// Every pass splits the pairs over the same number of CTAs, a contiguous chunk
// each, so a position is a prefix over chunk counts: no CTA waits for another,
// and the passes are chained with programmatic dependent launch. The number of
// pairs is known on the device only; nothing is read back.
#include <algorithm>
#include <new>

#include "slab.cuh"

namespace abm {

constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSortItems = 16;
constexpr int kSortTile = kSortThreads * kSortItems;
constexpr int kWarpItems = 32 * kSortItems;
constexpr int kBins = 256;
constexpr int kPasses = 4;
constexpr int kSortCtasPerSm = 4;  // resident scatter CTAs (45 KB of shared memory, at most 64 registers a thread)

struct SortScratch {
  int cap, n_pad, Fp, G;  // G: CTAs (= chunks) of every pass
  u32* key[2];
  u32* val[2];
  u32* hist;        // [kBins][G]: a pass's digit counts per chunk, then its positions
  u32* counts;      // [G] live slots per chunk
  u32* info;        // [0] pairs, [1] or of the keys, [2] or of their complements, [3] set when a live flag is
                    // neither 0 nor 1 (the gather then copies the flags)
  u32* digits;      // = info + 4: [kPasses][kBins] digit counts over all pairs
  int32_t* fields;  // [n_pad * Fp]: the next fields array
  int32_t* active;  // [n_pad]: the next live-flag array
};

void sort_scratch_free(SortScratch* p) {
  if (!p) return;
  for (int b = 0; b < 2; ++b) {
    cudaFree(p->key[b]);
    cudaFree(p->val[b]);
  }
  cudaFree(p->hist);
  cudaFree(p->counts);
  cudaFree(p->info);
  cudaFree(p->fields);
  cudaFree(p->active);
  delete p;
}

// chunk length of n items over G CTAs: whole tiles
__device__ __forceinline__ int chunk_of(int n, int G) {
  return (int)(((long long)n + (long long)G * kSortTile - 1) / ((long long)G * kSortTile)) * kSortTile;
}

// sum over the block of one value per thread, in every thread (s: kSortWarps words)
__device__ __forceinline__ u32 block_total(u32 v, u32* s) {
  v = __reduce_add_sync(0xFFFFFFFFu, v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = v;
  __syncthreads();
  u32 t = 0;
#pragma unroll
  for (int w = 0; w < kSortWarps; ++w) t += s[w];
  return t;
}

// live slots per chunk; also notes flags other than 0 and 1
__global__ void __launch_bounds__(kSortThreads) k_sort_count(SlabDev s, SortScratch p) {
  __shared__ u32 s_red[kSortWarps];
  const int chunk = chunk_of(s.cap, gridDim.x);
  const long long lo = (long long)blockIdx.x * chunk;
  const int hi = (int)min((long long)s.cap, lo + chunk);
  u32 n = 0;
  bool other = false;
  // flags are padded to whole tiles, with zeros
  for (int i = (int)min(lo, (long long)s.cap) + 4 * (int)threadIdx.x; i < hi; i += 4 * kSortThreads) {
    const int4 f = *reinterpret_cast<const int4*>(s.active + i);
    n += (f.x != 0) + (f.y != 0) + (f.z != 0) + (f.w != 0);
    other |= ((f.x | f.y | f.z | f.w) & ~1) != 0;
  }
  const u32 t = block_total(n, s_red);
  if (threadIdx.x == 0) p.counts[blockIdx.x] = t;
  if (other) p.info[3] = 1u;  // (emptied by the memset before this launch)
}

// live slots before this chunk, and in all, in every thread
__device__ __forceinline__ void live_prefix(const SortScratch& p, u32& before, u32& total, u32* s_red) {
  u32 b = 0, t = 0;
  for (int j = threadIdx.x; j < (int)gridDim.x; j += kSortThreads) {
    const u32 c = p.counts[j];
    t += c;
    if (j < (int)blockIdx.x) b += c;
  }
  before = block_total(b, s_red);
  total = block_total(t, s_red);
}

// Pack the live slots' (key, slot) pairs in slot order; placeholder r goes to
// entry cap - 1 - r of the same list (the pairs never reach it). The keys of a
// tile are strided loads of one sector each, 16 in flight per thread.
__global__ void __launch_bounds__(kSortThreads, kSortCtasPerSm) k_sort_pack(SlabDev s, SortScratch p, int field) {
  __shared__ u32 s_red[kSortWarps];
  __shared__ u32 s_wcnt[kSortWarps];
  __shared__ u32 s_bits[2];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x < 2) s_bits[threadIdx.x] = 0u;
  griddep_wait();
  u32 before, total;
  live_prefix(p, before, total, s_red);
  if (blockIdx.x == 0 && threadIdx.x == 0) p.info[0] = total;
  const int chunk = chunk_of(s.cap, gridDim.x);
  const long long lo = (long long)blockIdx.x * chunk;
  const u32 lt = (1u << lane) - 1u;
  u32 ones = 0, zeros = 0;
  for (long long t0 = lo; t0 < lo + chunk && t0 < s.cap; t0 += kSortTile) {
    const int w0 = (int)t0 + warp * kWarpItems;
    u32 live[kSortItems], key[kSortItems];
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
      const int i = w0 + 32 * j + lane;
      live[j] = i < s.cap && s.active[i] != 0;
    }
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
      const int i = w0 + 32 * j + lane;
      key[j] = 0u;
      if (live[j]) {
        key[j] = (u32)s.fields[(size_t)i * s.Fp + field] ^ 0x80000000u;
        ones |= key[j];
        zeros |= ~key[j];
      }
    }
    u32 n = 0;
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
      live[j] = __ballot_sync(0xFFFFFFFFu, live[j]);
      n += __popc(live[j]);
    }
    __syncthreads();  // s_wcnt of the previous tile is read
    if (lane == 0) s_wcnt[warp] = n;
    __syncthreads();
    u32 rank = before;
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) {
      if (w < warp) rank += s_wcnt[w];
      before += s_wcnt[w];
    }
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
      const int i = w0 + 32 * j + lane;
      const u32 r = rank + __popc(live[j] & lt);
      if ((live[j] >> lane) & 1u) {
        p.key[0][r] = key[j];
        p.val[0][r] = (u32)i;
      } else if (i < s.cap) {
        p.val[0][s.cap - 1 - (i - (int)r)] = (u32)i;
      }
      rank += __popc(live[j]);
    }
  }
  ones = __reduce_or_sync(0xFFFFFFFFu, ones);
  zeros = __reduce_or_sync(0xFFFFFFFFu, zeros);
  if (lane == 0) {
    atomicOr(&s_bits[0], ones);
    atomicOr(&s_bits[1], zeros);
  }
  __syncthreads();
  if (threadIdx.x < 2) atomicOr(&p.info[1 + threadIdx.x], s_bits[threadIdx.x]);
}

// What a pass has to know: the number of pairs, whether the pass's byte varies,
// which of the two buffers holds the pairs before it, and whether a later byte
// varies.
struct PassInfo {
  int n;
  bool run, last;
  bool odd;  // the pairs lie in the second buffer
  __device__ __forceinline__ u32* in(u32* const (&b)[2]) const { return odd ? b[1] : b[0]; }
  __device__ __forceinline__ u32* out(u32* const (&b)[2]) const { return odd ? b[0] : b[1]; }
};

__device__ __forceinline__ PassInfo pass_info(const SortScratch& p, int pass) {
  const u32 diff = p.info[1] & p.info[2];
  u32 varies = 0;
#pragma unroll
  for (int b = 0; b < kPasses; ++b) varies |= ((diff >> (8 * b)) & 0xFFu) ? 1u << b : 0u;
  PassInfo f;
  f.n = (int)p.info[0];
  f.odd = __popc(varies & ((1u << pass) - 1u)) & 1;
  f.run = (varies >> pass) & 1u;
  f.last = (varies >> pass) == 1u;
  return f;
}

// lanes of the warp with the same digit d < 256 (ok lanes only): eight ballots, a
// third of what a warp match of the digits takes
__device__ __forceinline__ u32 digit_peers(u32 d, bool ok) {
  u32 peers = __ballot_sync(0xFFFFFFFFu, ok);
#pragma unroll
  for (int b = 0; b < 8; ++b) {
    const u32 set = __ballot_sync(0xFFFFFFFFu, (d >> b) & 1u);
    peers &= (d >> b) & 1u ? set : ~set;
  }
  return peers;
}

// a pass's digit counts per chunk
__global__ void __launch_bounds__(kSortThreads) k_sort_hist(SortScratch p, int pass) {
  __shared__ u32 s_cnt[kBins];
  s_cnt[threadIdx.x] = 0u;
  griddep_wait();
  const PassInfo f = pass_info(p, pass);
  if (!f.run) return;
  const int chunk = chunk_of(f.n, gridDim.x);
  const long long lo = (long long)blockIdx.x * chunk;
  const u32* key = f.in(p.key);
  __syncthreads();
  for (long long t0 = lo; t0 < lo + chunk && t0 < f.n; t0 += kSortTile) {
    u32 k[kSortItems];
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
      const long long i = t0 + j * kSortThreads + threadIdx.x;
      k[j] = i < f.n ? key[i] : 0u;
    }
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
      const long long i = t0 + j * kSortThreads + threadIdx.x;
      if (i < f.n) atomicAdd(&s_cnt[(k[j] >> (8 * pass)) & 0xFFu], 1u);
    }
  }
  __syncthreads();
  const u32 c = s_cnt[threadIdx.x];
  p.hist[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = c;
  if (c) atomicAdd(&p.digits[pass * kBins + threadIdx.x], c);
}

// digit counts per chunk -> positions: a digit's first position (a scan of the
// digit counts, in every CTA) plus the counts of the chunks before; one warp
// per digit
__global__ void __launch_bounds__(kSortThreads) k_sort_scan(SortScratch p, int pass, int G) {
  __shared__ u64 s_warp[kSortWarps + 1];
  __shared__ u32 s_first[kBins];
  griddep_wait();
  const PassInfo f = pass_info(p, pass);
  if (!f.run) return;
  u32 ex, ex2, tot, tot2;
  block_scan2<kSortThreads>(p.digits[pass * kBins + threadIdx.x], 0u, ex, ex2, tot, tot2, s_warp);
  s_first[threadIdx.x] = ex;
  __syncthreads();
  const int lane = threadIdx.x & 31, d = blockIdx.x * kSortWarps + (threadIdx.x >> 5);
  u32* row = p.hist + (size_t)d * G;
  u32 carry = s_first[d];
  for (int j0 = 0; j0 < G; j0 += 128) {  // four chunks per lane at a time
    u32 v[4], sum = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int j = j0 + 4 * lane + u;
      v[u] = j < G ? row[j] : 0u;
      sum += v[u];
    }
    u32 inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const u32 x = __shfl_up_sync(0xFFFFFFFFu, inc, o);
      if (lane >= o) inc += x;
    }
    u32 at = carry + inc - sum;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int j = j0 + 4 * lane + u;
      if (j < G) row[j] = at;
      at += v[u];
    }
    carry += __shfl_sync(0xFFFFFFFFu, inc, 31);
  }
}

// Stable scatter of one pass, tile by tile of the CTA's chunk. Each warp ranks
// its 512 consecutive pairs on its own (ballots of the digit's bits; its digit
// counts in shared memory), without block barriers; the warps' counts then give every pair its
// place in the tile's (digit, rank) order. The pairs are placed there in shared
// memory and written out in that order, so that consecutive threads write
// consecutive addresses of one digit's run.
__global__ void __launch_bounds__(kSortThreads, kSortCtasPerSm) k_sort_scatter(SortScratch p, int pass) {
  __shared__ u32 s_key[kSortTile], s_val[kSortTile];
  __shared__ u32 s_wc[kSortWarps][kBins];  // per warp: pairs of each digit, then its first place in the tile order
  __shared__ u32 s_off[kBins];             // global position of a digit's place 0 of the tile order
  __shared__ u64 s_warp[kSortWarps + 1];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  griddep_wait();
  const PassInfo f = pass_info(p, pass);
  if (!f.run) return;
  const u32 *key = f.in(p.key), *val = f.in(p.val);
  u32 *key_out = f.out(p.key), *val_out = f.out(p.val);
  const int chunk = chunk_of(f.n, gridDim.x);
  const long long lo = (long long)blockIdx.x * chunk;
  const u32 lt = (1u << lane) - 1u;
  u32 pos = p.hist[(size_t)threadIdx.x * gridDim.x + blockIdx.x];  // digit threadIdx.x's next position
  for (long long t0 = lo; t0 < lo + chunk && t0 < f.n; t0 += kSortTile) {
    const int n_tile = (int)min((long long)kSortTile, f.n - t0);
    u32 k[kSortItems], rank[kSortItems / 2];  // ranks below 512: two to a register
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
      const int i = warp * kWarpItems + 32 * j + lane;
      k[j] = i < n_tile ? key[t0 + i] : 0u;
    }
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) s_wc[w][threadIdx.x] = 0u;
    __syncthreads();
    u32* wc = s_wc[warp];
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
      const bool ok = warp * kWarpItems + 32 * j + lane < n_tile;
      const u32 d = (k[j] >> (8 * pass)) & 0xFFu;
      const u32 peers = digit_peers(d, ok);
      const u32 below = (u32)__popc(peers & lt);
      const u32 c = ok ? wc[d] : 0u;
      __syncwarp();
      if (ok && below == 0) wc[d] = c + (u32)__popc(peers);
      __syncwarp();
      if (j & 1) rank[j >> 1] |= (c + below) << 16;
      else rank[j >> 1] = c + below;
    }
    __syncthreads();
    u32 cnt = 0;
    {
      u32 c[kSortWarps];
#pragma unroll
      for (int w = 0; w < kSortWarps; ++w) {
        c[w] = s_wc[w][threadIdx.x];
        cnt += c[w];
      }
      u32 ex, ex2, tot, tot2;
      block_scan2<kSortThreads>(cnt, 0u, ex, ex2, tot, tot2, s_warp);
      s_off[threadIdx.x] = pos - ex;
      pos += cnt;
#pragma unroll
      for (int w = 0; w < kSortWarps; ++w) {
        s_wc[w][threadIdx.x] = ex;
        ex += c[w];
      }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
      const int i = warp * kWarpItems + 32 * j + lane;
      if (i < n_tile) {
        const u32 at = wc[(k[j] >> (8 * pass)) & 0xFFu] + ((rank[j >> 1] >> (16 * (j & 1))) & 0xFFFFu);
        s_key[at] = k[j];
        s_val[at] = val[t0 + i];
      }
    }
    __syncthreads();
#pragma unroll 4
    for (int i = threadIdx.x; i < n_tile; i += kSortThreads) {
      const u32 kk = s_key[i];
      const u32 at = s_off[(kk >> (8 * pass)) & 0xFFu] + (u32)i;
      if (!f.last) key_out[at] = kk;
      val_out[at] = s_val[i];
    }
    __syncthreads();
  }
}

// Small sets: pack and sort in one CTA, pairs in shared memory, every pass with
// the pairs in registers in between. Leaves the values in val[0] (as k_sort_pack
// does) with no pass left to run, for the gather. (With the
// memset and the fourteen launches that it takes the place of 78 us for 3000 slots, now 46.)
constexpr int kOneThreads = 1024;
constexpr int kOneWarps = kOneThreads / 32;
constexpr int kOneMax = kOneThreads * kSortItems;
constexpr size_t kOneSmem = (size_t)kOneMax * 8 + (size_t)kOneWarps * kBins * 4;

__global__ void __launch_bounds__(kOneThreads, 1) k_sort_one(SlabDev s, SortScratch p, int field) {
  extern __shared__ __align__(16) u32 s_one[];
  u32 *s_key = s_one, *s_val = s_one + kOneMax, *s_wc = s_one + 2 * kOneMax;
  __shared__ u64 s_warp[kOneWarps + 1];
  __shared__ u32 s_bits[3];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const u32 lt = (1u << lane) - 1u;
  const int w0 = warp * kWarpItems;
  u32 k[kSortItems], v[kSortItems], rank[kSortItems / 2];
  if (threadIdx.x < 3) s_bits[threadIdx.x] = 0u;
  griddep_wait();
  u32 ones = 0, zeros = 0, other = 0, mine = 0;
#pragma unroll
  for (int j = 0; j < kSortItems; ++j) {
    const int i = w0 + 32 * j + lane;
    v[j] = i < s.cap ? (u32)s.active[i] : 0u;
  }
#pragma unroll
  for (int j = 0; j < kSortItems; ++j) {
    const int i = w0 + 32 * j + lane;
    k[j] = 0u;
    if (v[j]) {
      k[j] = (u32)s.fields[(size_t)i * s.Fp + field] ^ 0x80000000u;
      ones |= k[j];
      zeros |= ~k[j];
    }
    other |= v[j] & ~1u;
    v[j] = __ballot_sync(0xFFFFFFFFu, v[j] != 0u);
    mine += __popc(v[j]);
  }
  u32 at, at2, total, total2;
  block_scan2<kOneThreads>(lane == 0 ? mine : 0u, 0u, at, at2, total, total2, s_warp);
  at = __shfl_sync(0xFFFFFFFFu, at, 0);
#pragma unroll
  for (int j = 0; j < kSortItems; ++j) {
    const int i = w0 + 32 * j + lane;
    const u32 r = at + __popc(v[j] & lt);
    if ((v[j] >> lane) & 1u) {
      s_key[r] = k[j];
      s_val[r] = (u32)i;
    } else if (i < s.cap) {
      p.val[0][s.cap - 1 - (i - (int)r)] = (u32)i;
    }
    at += __popc(v[j]);
  }
  ones = __reduce_or_sync(0xFFFFFFFFu, ones);
  zeros = __reduce_or_sync(0xFFFFFFFFu, zeros);
  other = __reduce_or_sync(0xFFFFFFFFu, other);
  if (lane == 0) {
    atomicOr(&s_bits[0], ones);
    atomicOr(&s_bits[1], zeros);
    atomicOr(&s_bits[2], other);
  }
  __syncthreads();
  const u32 diff = s_bits[0] & s_bits[1];
  const int n = (int)total;
  u32* wc = s_wc + warp * kBins;
  for (int sh = 0; sh < 32; sh += 8) {
    if (!((diff >> sh) & 0xFFu)) continue;
    for (int d = lane; d < kBins; d += 32) wc[d] = 0u;
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
      const int i = w0 + 32 * j + lane;
      k[j] = i < n ? s_key[i] : 0u;
      v[j] = i < n ? s_val[i] : 0u;
    }
    __syncwarp();
    if (w0 < n) {
#pragma unroll
      for (int j = 0; j < kSortItems; ++j) {
        const bool ok = w0 + 32 * j + lane < n;
        const u32 d = (k[j] >> sh) & 0xFFu;
        const u32 peers = digit_peers(d, ok);
        const u32 below = (u32)__popc(peers & lt);
        const u32 c = ok ? wc[d] : 0u;
        __syncwarp();
        if (ok && below == 0) wc[d] = c + (u32)__popc(peers);
        __syncwarp();
        if (j & 1) rank[j >> 1] |= (c + below) << 16;
        else rank[j >> 1] = c + below;
      }
    }
    __syncthreads();
    // a digit's counts over the warps (four threads each, eight warps of counts a thread) -> first places
    {
      const int d = threadIdx.x >> 2, g = threadIdx.x & 3;
      u32 c[kOneWarps / 4], sum = 0;
#pragma unroll
      for (int w = 0; w < kOneWarps / 4; ++w) {
        c[w] = s_wc[(g * (kOneWarps / 4) + w) * kBins + d];
        sum += c[w];
      }
      u32 ex, ex2, tot, tot2;
      block_scan2<kOneThreads>(sum, 0u, ex, ex2, tot, tot2, s_warp);  // digit-major, warps ascending
#pragma unroll
      for (int w = 0; w < kOneWarps / 4; ++w) {
        s_wc[(g * (kOneWarps / 4) + w) * kBins + d] = ex;
        ex += c[w];
      }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
      if (w0 + 32 * j + lane < n) {
        const u32 to = wc[(k[j] >> sh) & 0xFFu] + ((rank[j >> 1] >> (16 * (j & 1))) & 0xFFFFu);
        s_key[to] = k[j];
        s_val[to] = v[j];
      }
    }
    __syncthreads();
  }
  for (int i = threadIdx.x; i < n; i += kOneThreads) p.val[0][i] = s_val[i];
  if (threadIdx.x < 4) p.info[threadIdx.x] = threadIdx.x == 0 ? total : (threadIdx.x == 3 ? s_bits[2] : 0u);
}

// Row i of the sorted slab <- its old row. A thread moves 16-byte quads of
// rows, four in flight; the quads of one row go to neighbouring threads. Bound
// by the random rows' DRAM bursts.
__global__ void __launch_bounds__(kSortThreads) k_sort_gather(SlabDev s, SortScratch p, int32_t* perm_out) {
  griddep_wait();
  // after the last pass: the buffer that holds the pairs, and their number
  const PassInfo f = pass_info(p, kPasses);
  const u32* val = f.in(p.val);
  const bool exact = p.info[3] != 0u;
  constexpr int U = 4;
  const u32 q = (u32)s.Fp >> 2, sh = q == 4 ? 2 : q - 1;  // 1 to 4 quads a row
  const u32 n = (u32)s.cap * q, T = gridDim.x * kSortThreads;
  for (u32 e0 = blockIdx.x * kSortThreads + threadIdx.x; e0 < n; e0 += U * T) {
    int src[U];
    u32 row[U];
    int4 r[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const u32 e = e0 + u * T;
      src[u] = -1;
      row[u] = q == 3 ? e / 3u : e >> sh;
      if (e < n) {
        const int i = (int)row[u];
        src[u] = (int)(i < f.n ? val[i] : p.val[0][s.cap - 1 - (i - f.n)]);
        if (!in_range(src[u], s.cap, s.err)) src[u] = -1;
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (src[u] >= 0)
        r[u] = __ldcs(reinterpret_cast<const int4*>(s.fields) + (u32)src[u] * q + (e0 + u * T - row[u] * q));
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (src[u] < 0) continue;
      const u32 e = e0 + u * T;
      reinterpret_cast<int4*>(p.fields)[e] = r[u];
      if (e == row[u] * q) {
        p.active[row[u]] = exact ? s.active[src[u]] : ((int)row[u] < f.n ? 1 : 0);
        if (perm_out) perm_out[row[u]] = src[u];
      }
    }
  }
}

static abm_status sort_scratch(abm_slab* s, SortScratch** out) {
  if (s->sort) {
    *out = s->sort;
    return ABM_OK;
  }
  SortScratch* p = new (std::nothrow) SortScratch();
  if (!p) return ABM_ERR_OOM;
  p->cap = s->d.cap;
  p->n_pad = s->n_pad;
  p->Fp = s->d.Fp;
  p->G = std::min((s->d.cap + kSortTile - 1) / kSortTile, num_sms() * kSortCtasPerSm);
  bool ok = true;
  for (int b = 0; b < 2 && ok; ++b)
    ok = cudaMalloc(&p->key[b], sizeof(u32) * (size_t)p->cap) == cudaSuccess &&
         cudaMalloc(&p->val[b], sizeof(u32) * (size_t)p->cap) == cudaSuccess;
  ok = ok && cudaMalloc(&p->hist, sizeof(u32) * (size_t)kBins * p->G) == cudaSuccess;
  ok = ok && cudaMalloc(&p->counts, sizeof(u32) * (size_t)p->G) == cudaSuccess;
  ok = ok && cudaMalloc(&p->info, sizeof(u32) * (4 + kPasses * kBins)) == cudaSuccess;
  p->digits = p->info + 4;
  ok = ok && cudaMalloc(&p->fields, sizeof(int32_t) * (size_t)p->n_pad * p->Fp) == cudaSuccess;
  ok = ok && cudaMalloc(&p->active, sizeof(int32_t) * (size_t)p->n_pad) == cudaSuccess;
  // rows past the capacity are never gathered: keep them as the slab keeps its own
  ok = ok && cudaMemset(p->fields, 0, sizeof(int32_t) * (size_t)p->n_pad * p->Fp) == cudaSuccess;
  ok = ok && cudaMemset(p->active, 0, sizeof(int32_t) * (size_t)p->n_pad) == cudaSuccess;
  if (kCheck && ok)  // check builds: the spare arrays carry the canaries too (they become the slab's)
    ok = slab_canary_fill(p->fields, p->Fp, s->d.cap, p->n_pad, 0) == ABM_OK && cudaDeviceSynchronize() == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    sort_scratch_free(p);
    return ABM_ERR_OOM;
  }
  s->sort = p;
  *out = p;
  return ABM_OK;
}

}  // namespace abm

using namespace abm;

extern "C" abm_status abm_sort(abm_slab* s, int32_t field, int32_t* out_perm, void* stream) {
  if (!s || field < 0 || field >= s->d.F) return ABM_ERR_ARG;
  if (s->view) return ABM_ERR_STATE;  // the sort swaps the slab's arrays, which a world's view does not own
  SortScratch* p = nullptr;
  abm_status e = sort_scratch(s, &p);
  if (e != ABM_OK) return e;
  cudaStream_t st = (cudaStream_t)stream;
  const int G = p->G;
  if (s->d.cap <= kOneMax) {
    static std::atomic<unsigned long long> attr{0};
    ABM_CUDA_TRY(smem_attr_once(k_sort_one, (int)kOneSmem, attr));
    ABM_CUDA_TRY(launch_pdl_smem(k_sort_one, 1, kOneThreads, kOneSmem, st, s->d, *p, (int)field));
  } else {
    ABM_CUDA_TRY(cudaMemsetAsync(p->info, 0, sizeof(u32) * (4 + kPasses * kBins), st));
    k_sort_count<<<G, kSortThreads, 0, st>>>(s->d, *p);
    ABM_LAUNCH_CHECK();
    ABM_CUDA_TRY(launch_pdl(k_sort_pack, G, kSortThreads, st, s->d, *p, (int)field));
    for (int pass = 0; pass < kPasses; ++pass) {
      ABM_CUDA_TRY(launch_pdl(k_sort_hist, G, kSortThreads, st, *p, pass));
      ABM_CUDA_TRY(launch_pdl(k_sort_scan, kBins / kSortWarps, kSortThreads, st, *p, pass, G));
      ABM_CUDA_TRY(launch_pdl(k_sort_scatter, G, kSortThreads, st, *p, pass));
    }
  }
  const long long quads = (long long)s->d.cap * (s->d.Fp >> 2);
  const int grid = (int)std::min<long long>((quads + kSortThreads - 1) / kSortThreads, (long long)num_sms() * 8);
  ABM_CUDA_TRY(launch_pdl(k_sort_gather, grid, kSortThreads, st, s->d, *p, out_perm));
  // the gathered arrays become the slab's; the old ones are the next sort's targets
  std::swap(s->d.fields, p->fields);
  std::swap(s->d.active, p->active);
  return ABM_OK;
}
