// Generic fixed-capacity agent set ("Set", ABMax Section 2) and the selection /
// compaction / distinct-update primitives of Section 4 (Algorithms 1 and 2).
//
// Every rank-matched operation is count -> scatter -> apply over a static
// partition of the slab: pass 1 evaluates the per-slot flags (from 128-bit
// loads of live flags) into bit-planes and per-warp / per-CTA counts; pass 2
// turns a slot's position into its rank (prefix of the CTA counts + prefix of
// the warp counts + a warp scan) and writes rank-ordered slot lists; pass 3
// moves the records. The i-th selected slot receiving the i-th record is
// exactly Rank-Match's pairing (cumsum(mask) * mask on both sides, matched on
// equal nonzero ranks), computed in O(n + k) instead of O(n * k). The passes
// are chained with programmatic dependent launch; no pass spins on another CTA.
#include <algorithm>
#include <atomic>
#include <cstdlib>
#include <cstring>
#include <new>

#include "slab.cuh"

namespace abm {

// SM count per device, looked up once per device (a process may drive
// several GPUs from several host threads: relaxed atomics, idempotent writes)
constexpr int kSmCacheDevices = 64;
static std::atomic<int> g_num_sms[kSmCacheDevices];
int num_sms() {
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 1;
  if (dev >= 0 && dev < kSmCacheDevices) {
    n = g_num_sms[dev].load(std::memory_order_relaxed);
    if (n > 0) return n;
  }
  if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) return 1;
  if (dev >= 0 && dev < kSmCacheDevices) g_num_sms[dev].store(n, std::memory_order_relaxed);
  return n;
}

constexpr int kSlabThreads = 256;    // default CTA size of the slab passes
constexpr int kMaxFields = 16;



struct PredDev {
  int kind;
  u32 threshold, step, purpose, species;
  const int32_t* mask;
  int field, cmp, and_mask, value;
};

// The N slots from `base` on (those below n) that satisfy the predicate, as a
// bit mask. live: their live flags. The words of the live slots are all
// requested before the first is used: fetched slot by slot behind a test of the
// flag, sixteen fields a lane took 8 us of round trips.
template <int N>
__device__ __forceinline__ u32 pred_mask(const PredDev& p, const SlabDev& s, int base, int n, const int (&live)[N]) {
  u32 on = 0;
#pragma unroll
  for (int j = 0; j < N; ++j) on |= (u32)(live[j] != 0) << j;
  const u32 valid = n - base >= N ? (N == 32 ? 0xFFFFFFFFu : (1u << (N & 31)) - 1u) : (n > base ? (1u << (n - base)) - 1u : 0u);
  if (p.kind == ABM_PRED_FREE) return ~on & valid;
  on &= valid;
  if (p.kind == ABM_PRED_LIVE || on == 0u) return on;
  u32 m = 0;
  switch (p.kind) {
    case ABM_PRED_BERNOULLI:
#pragma unroll
      for (int j = 0; j < N; ++j)
        m |= (u32)(draw(s.seed, s.model, p.step, (u32)(base + j), p.purpose, p.species) < p.threshold) << j;
      return m & on;
    case ABM_PRED_MASK: {
      int v[N];
#pragma unroll
      for (int j = 0; j < N; ++j) v[j] = (on >> j) & 1u ? p.mask[base + j] : 0;
#pragma unroll
      for (int j = 0; j < N; ++j) m |= (u32)(v[j] != 0) << j;
      return m & on;
    }
    case ABM_PRED_FIELD: {
      int v[N];
#pragma unroll
      for (int j = 0; j < N; ++j) v[j] = (on >> j) & 1u ? s.fields[(size_t)(base + j) * s.Fp + p.field] : 0;
#pragma unroll
      for (int j = 0; j < N; ++j) {
        const int x = v[j] & p.and_mask;
        const bool f = p.cmp == ABM_CMP_EQ   ? x == p.value
                       : p.cmp == ABM_CMP_NE ? x != p.value
                       : p.cmp == ABM_CMP_LT ? x < p.value
                                             : x >= p.value;
        m |= (u32)f << j;
      }
      return m & on;
    }
  }
  return 0;
}

enum Op { OP_SELECT = 0, OP_REMOVE = 1, OP_ADD = 2, OP_UPDATE = 3, OP_FUSED = 4, OP_ARRAY = 5 };

struct ScanArgs {
  SlabDev s;
  PredDev pred;
  u32* ctrl;               // [1] CTAs finished, [2] epoch (last-CTA-out bookkeeping)
  u32* planeA;             // n/32 words each: selected / free
  u32* planeB;             // chosen (fused call)
  u32* planeL;             // the flags in memory after pass 1 that are 1 (fused call)
  u32* totals;             // [2 * G] per-CTA counts
  u32* wtotals;            // [2 * G * warps] per-warp counts
  int n;                   // slots (or array entries for OP_ARRAY)
  int chunk;               // slots per CTA (a multiple of the sub-tile)
  int G;                   // CTAs = number of chunks
  const int32_t* src;      // OP_ARRAY: mask array
  const int32_t* rec;      // records [k][F]
  const int32_t* rec2;     // OP_FUSED: deltas [k][F]
  int k;
  int op_kind;             // ABM_OP_ADD / ABM_OP_SET for OP_UPDATE
  int id_field;            // OP_ADD
  int use_rec_idx;         // OP_UPDATE with a record mask
  u32 step, threshold;     // OP_FUSED
  u32 rk[20];              // OP_FUSED: Philox round keys of the slab's key (seed, model), round r at 2r, 2r+1
  u32 mk[5];               // OP_FUSED: the call's mask draws' constant parts (mask_pair_consts)
  int32_t* list_a;         // slots by rank: selected / free (caller's out_idx or scratch)
  int32_t* list_b;         // slots by rank: chosen (fused call)
  int32_t* out_count;      // device outputs (nullable)
  int negate;              // OP_SELECT: select where the predicate is false
  const int32_t* list_base;  // OP_SELECT: device offset added to every rank (nullable)
  int* crowded;              // OP_FUSED: the slab's word (nullable)
  int crowded_known;         // its value at the launch
  int wave;                  // slots of the first wave of a ranking pass that moves records
  u32 div1, div4;            // one launch: 65536 / units of a row, rounded up, in words and in 16 bytes
};

template <int THREADS>
__device__ __forceinline__ void block_sum2(u32& a, u32& b, u64* s_red) {
  u64 v = ((u64)a << 32) | b;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) s_red[warp] = v;
  __syncthreads();
  u64 t = 0;
#pragma unroll
  for (int w = 0; w < THREADS / 32; ++w) t += s_red[w];
  a = (u32)(t >> 32);
  b = (u32)t;
}

// 32-byte (256-bit) global accesses: one instruction moves a whole 8-field
// row, so a row written to DRAM is one full sector (two 16-byte stores to a
// sector make L2 fetch it first when the first half arrives alone)
__device__ __forceinline__ void ld_v8_nc(const int32_t* p, int (&r)[8]) {
  asm volatile("ld.global.nc.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "l"(p));
}
__device__ __forceinline__ void ld_v8(const int32_t* p, int (&r)[8]) {
  asm volatile("ld.global.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "l"(p)
               : "memory");
}
__device__ __forceinline__ void st_v8(int32_t* p, const int (&r)[8]) {
  asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(r[0]), "r"(r[1]), "r"(r[2]),
               "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}

// Flags live in two bit-planes of one bit per slot: A = selected / free,
// B = chosen (fused call); word w of a plane covers slots [32w, 32w + 32).
//
// Both passes use the same static partition: CTA b owns the slots
// [b*chunk, (b+1)*chunk) and warp w of it the contiguous segment
// [b*chunk + w*seg, ... + seg), seg a multiple of 512 slots. In each 512-slot
// step, lane l handles the 16 consecutive slots [16l, 16l + 16).
constexpr int kLaneSlots = 16;
constexpr int kWarpStep = 32 * kLaneSlots;

// Pass 1: flags from four 128-bit loads of live flags per lane; the lane's
// 16-bit masks are paired with the neighbour lane's into plane words.
template <int OP, int THREADS>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS) k_count(ScanArgs a) {
  constexpr int WARPS = THREADS / 32;
  __shared__ u64 s_red[WARPS];
  const SlabDev& s = a.s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int seg = a.chunk / WARPS;
  const int wlo = blockIdx.x * a.chunk + warp * seg;
  const int whi = min(a.n, wlo + seg);
  const int32_t* flag_src = OP == OP_ARRAY ? a.src : s.active;
  const bool vec = (((uintptr_t)flag_src) & 15) == 0;  // a caller's mask array may start anywhere
  u32 ca = 0, cb = 0;
  for (int b0 = wlo; b0 < whi; b0 += kWarpStep) {
    const int base = b0 + lane * kLaneSlots;
    int live[kLaneSlots];
#pragma unroll
    for (int v = 0; v < kLaneSlots / 4; ++v) {
      const int b = base + 4 * v;
      int4 q = make_int4(0, 0, 0, 0);
      if (vec && b + 3 < a.n) {
        q = *reinterpret_cast<const int4*>(flag_src + b);
      } else {
        if (b + 0 < a.n) q.x = flag_src[b + 0];
        if (b + 1 < a.n) q.y = flag_src[b + 1];
        if (b + 2 < a.n) q.z = flag_src[b + 2];
        if (b + 3 < a.n) q.w = flag_src[b + 3];
      }
      live[4 * v + 0] = q.x; live[4 * v + 1] = q.y; live[4 * v + 2] = q.z; live[4 * v + 3] = q.w;
    }
    const u32 valid = a.n - base >= kLaneSlots ? 0xFFFFu : (a.n > base ? (1u << (a.n - base)) - 1u : 0u);
    u32 ma = 0, mr = 0;  // 16-bit masks over the lane's slots
    if (OP == OP_ARRAY || OP == OP_ADD) {
#pragma unroll
      for (int j = 0; j < kLaneSlots; ++j) ma |= (u32)((live[j] != 0) == (OP == OP_ARRAY)) << j;
      ma &= valid;
    } else {
      ma = pred_mask<kLaneSlots>(a.pred, s, base, a.n, live);
      if (a.negate) ma = ~ma & valid;
    }
    if (OP == OP_REMOVE) mr = ma;
    // removed slots become placeholders now: rewrite only the 4-slot groups
    // that changed (the other flags keep their values)
    if (OP == OP_REMOVE) {
#pragma unroll
      for (int v = 0; v < kLaneSlots / 4; ++v) {
        const u32 g = (mr >> (4 * v)) & 0xFu;
        if (!g) continue;
        const int b = base + 4 * v;
        const int4 q = make_int4((g & 1u) ? 0 : live[4 * v], (g & 2u) ? 0 : live[4 * v + 1],
                                 (g & 4u) ? 0 : live[4 * v + 2], (g & 8u) ? 0 : live[4 * v + 3]);
        if (b + 3 < a.n) {
          *reinterpret_cast<int4*>(s.active + b) = q;
        } else {
          if (b + 0 < a.n) s.active[b + 0] = q.x;
          if (b + 1 < a.n) s.active[b + 1] = q.y;
          if (b + 2 < a.n) s.active[b + 2] = q.z;
        }
      }
    }
    ca += __popc(ma);
    if (OP != OP_REMOVE) {
      const u32 na = __shfl_down_sync(0xFFFFFFFFu, ma, 1);
      if (!(lane & 1) && base < a.n) a.planeA[base >> 5] = ma | (na << 16);
    }
  }
  u64 v = ((u64)ca << 32) | cb;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  if (lane == 0) {
    a.wtotals[2 * (blockIdx.x * WARPS + warp)] = (u32)(v >> 32);
    a.wtotals[2 * (blockIdx.x * WARPS + warp) + 1] = (u32)v;
  }
  block_sum2<THREADS>(ca, cb, s_red);
  if (threadIdx.x == 0) {
    a.totals[2 * blockIdx.x] = ca;
    a.totals[2 * blockIdx.x + 1] = cb;
  }
  if (OP == OP_REMOVE) {
    __shared__ bool s_last;
    const bool last = last_cta_out(a.ctrl);
    if (threadIdx.x == 0) s_last = last;
    __syncthreads();
    if (!s_last) return;
    u32 A = 0, B = 0;
    for (int b = threadIdx.x; b < a.G; b += THREADS) A += ld_relaxed32(a.totals + 2 * b);
    block_sum2<THREADS>(A, B, s_red);
    if (threadIdx.x == 0) {
      s.counters[0] -= (int)A;
      if (a.out_count) *a.out_count = (int)A;
    }
  }
}

// The selective-update call's mask draws are Philox4x32-10 blocks on the
// counter (step, j, MASK, 0), j = slot >> 1: only the second word varies
// within a call, so the first round, one multiply of the second and one of
// the third depend on the call alone. mask_pair_consts works them out on the
// host (round r: (hi(M1 c2) ^ c1 ^ k0, lo(M1 c2), hi(M0 c0) ^ c3 ^ k1,
// lo(M0 c0)), M0 = 0xD2511F53, M1 = 0xCD9E8D57, round keys k = rk); the
// device finishes the block from them. Same outputs as philox.
static void mask_pair_consts(u32 step, const u32 (&rk)[20], u32 (&mk)[5]) {
  const auto wide = [](u32 m, u32 x, u32& hi, u32& lo) {
    const uint64_t p = (uint64_t)m * (uint64_t)x;
    hi = (u32)(p >> 32);
    lo = (u32)p;
  };
  u32 h0, l0, h1, l1;
  // round 0 on (step, j, MASK, 0) -> (A ^ j, B, C, D)
  wide(0xD2511F53u, step, h0, l0);
  wide(0xCD9E8D57u, (u32)ABM_P_MASK, h1, l1);
  const u32 A = h1 ^ rk[0], B = l1, C = h0 ^ 0u ^ rk[1], D = l0;
  // round 1: the third word C is constant -> (E, F, hi(M0 (A ^ j)) ^ G, lo(M0 (A ^ j)))
  wide(0xCD9E8D57u, C, h1, l1);
  const u32 E = h1 ^ B ^ rk[2], F = l1, G = D ^ rk[3];
  // round 2: the first word E is constant -> (hi(M1 z) ^ H, lo(M1 z), I ^ w, J)
  wide(0xD2511F53u, E, h0, l0);
  mk[0] = A;
  mk[1] = G;
  mk[2] = F ^ rk[4];  // H
  mk[3] = h0 ^ rk[5];  // I
  mk[4] = l0;          // J
}

__device__ __forceinline__ uint4 mask_pair_draw(u32 j, const u32 (&mk)[5], const u32 (&rk)[20]) {
  const u32 x = mk[0] ^ j;                                         // round 0
  const u32 a_lo = 0xD2511F53u * x, a_hi = __umulhi(0xD2511F53u, x);  // round 1
  const u32 z = a_hi ^ mk[1];
  const u32 b_lo = 0xCD9E8D57u * z, b_hi = __umulhi(0xCD9E8D57u, z);  // round 2
  uint4 c = make_uint4(b_hi ^ mk[2], b_lo, mk[3] ^ a_lo, mk[4]);
#pragma unroll
  for (int r = 3; r < 10; ++r) {
    const u32 p0_lo = 0xD2511F53u * c.x, p0_hi = __umulhi(0xD2511F53u, c.x);
    const u32 p1_lo = 0xCD9E8D57u * c.z, p1_hi = __umulhi(0xCD9E8D57u, c.z);
    c = make_uint4(p1_hi ^ c.y ^ rk[2 * r], p1_lo, p0_hi ^ c.w ^ rk[2 * r + 1], p0_lo);
  }
  return c;
}

// Pass 1 of the selective-update call: as k_count, with the live flags as a
// 16-bit mask per lane (any nonzero flag is live) read by two 32-byte loads;
// the lane's eight draws are independent and all in flight together. The pass
// is bound by the Philox draws (one per pair of slots): fewer draws in flight
// at a higher occupancy measured slower.
// Flags of removed slots (whole 8-slot groups, as 0/1): with few records they are
// written here. LATE (see kLateShare): most removed slots are refilled by the same
// call, so the ranking pass, which knows every final flag, writes the groups
// that end up different. It compares with plane L; flags other than 0 and 1
// are put right here.
template <int THREADS, bool LATE>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS) k_count_fused(ScanArgs a) {
  constexpr int WARPS = THREADS / 32;
  __shared__ u64 s_red[WARPS];
  const SlabDev& s = a.s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int seg = a.chunk / WARPS;
  const int wlo = blockIdx.x * a.chunk + warp * seg;
  const int whi = min(a.n, wlo + seg);
  u32 ca = 0, cb = 0;
  for (int b0 = wlo; b0 < whi; b0 += kWarpStep) {
    const int base = b0 + lane * kLaneSlots;
    u32 ml = 0;
    int odd = 0;
    if (base + kLaneSlots <= a.n) {
      int f[8];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        ld_v8(s.active + base + 8 * h, f);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          ml |= (u32)(f[j] != 0) << (8 * h + j);
          odd |= f[j];
        }
      }
    } else {
      for (int j = 0; j < kLaneSlots; ++j)
        if (base + j < a.n) {
          ml |= (u32)(s.active[base + j] != 0) << j;
          odd |= s.active[base + j];
        }
    }
    // the draws' outcomes as 16-bit masks (bit j: slot base + j), combined
    // with the live mask once per 16 slots
    u32 dr = 0, dc = 0;
#pragma unroll
    for (int m = 0; m < kLaneSlots / 2; ++m) {
      const int slot = base + 2 * m;
      // slots 2j and 2j+1 share draw j: words (x, y) and (z, w) = (remove, choose)
      const uint4 u = mask_pair_draw((u32)slot >> 1, a.mk, a.rk);
      dr |= (u.x < a.threshold ? 1u << (2 * m) : 0u) | (u.z < a.threshold ? 2u << (2 * m) : 0u);
      dc |= (u.y < a.threshold ? 1u << (2 * m) : 0u) | (u.w < a.threshold ? 2u << (2 * m) : 0u);
    }
    const u32 valid = base + kLaneSlots <= a.n ? 0xFFFFu : (base < a.n ? (1u << (a.n - base)) - 1u : 0u);
    const u32 mr = ml & dr;         // removed: live and drawn
    const u32 al = ml & ~dr;        // still live
    const u32 ma = valid & ~al;     // free after the removals
    const u32 mb = al & dc;         // chosen among the live
    const u32 nl = ml & ~mr;
    u32 fl = ml;  // LATE: flags that are 1 in memory
    if (LATE && (odd & ~1)) {
      fl = 0;
      for (int j = 0; j < kLaneSlots; ++j) {
        if (base + j >= a.n) break;
        if ((mr >> (j & 8)) & 0xFFu) {
          s.active[base + j] = (int)((nl >> j) & 1u);
          fl |= nl & (1u << j);
        } else if (s.active[base + j] == 1) {
          fl |= 1u << j;
        }
      }
    }
    if (!LATE) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (!((mr >> (8 * h)) & 0xFFu)) continue;
        const int b = base + 8 * h;
        if (b + 8 <= a.n) {
          int f[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) f[j] = (int)((nl >> (8 * h + j)) & 1u);
          st_v8(s.active + b, f);
        } else {
          for (int j = 0; j < 8; ++j)
            if (b + j < a.n) s.active[b + j] = (int)((nl >> (8 * h + j)) & 1u);
        }
      }
    }
    ca += __popc(ma);
    cb += __popc(mb);
    const u32 na = __shfl_down_sync(0xFFFFFFFFu, ma, 1);
    const u32 nb = __shfl_down_sync(0xFFFFFFFFu, mb, 1);
    const u32 nf = LATE ? __shfl_down_sync(0xFFFFFFFFu, fl, 1) : 0u;
    if (!(lane & 1) && base < a.n) {
      a.planeA[base >> 5] = ma | (na << 16);
      a.planeB[base >> 5] = mb | (nb << 16);
      if (LATE) a.planeL[base >> 5] = fl | (nf << 16);
    }
  }
  u64 v = ((u64)ca << 32) | cb;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  if (lane == 0) {
    a.wtotals[2 * (blockIdx.x * WARPS + warp)] = (u32)(v >> 32);
    a.wtotals[2 * (blockIdx.x * WARPS + warp) + 1] = (u32)v;
  }
  block_sum2<THREADS>(ca, cb, s_red);
  if (threadIdx.x == 0) {
    a.totals[2 * blockIdx.x] = ca;
    a.totals[2 * blockIdx.x + 1] = cb;
  }
}

// The selective-update call's records moved by the pass that ranks them: the
// staged slots (offsets from slot0) take records r0 + i, i < n (ADDROW: added to
// the row, wrapping), U 32-byte rows per lane in flight. Ranks are consecutive
// over a warp's steps, so a warp stages slots over several steps until it has
// kMoveBatch of them: four rows per lane, also where few slots are touched (see
// kMoveShare for what that is worth).
constexpr int kMoveBatch = 128;
constexpr int kMoveStage = kMoveBatch + kWarpStep;
// CTAs of such a pass resident on an SM (126 registers a thread).
template <int THREADS>
constexpr int move_resident() {
  return 512 / THREADS;
}

template <bool ADDROW>
__device__ __forceinline__ void move_staged(const ScanArgs& a, const unsigned short* stage, int slot0, u32 n, u32 r0,
                                            const int32_t* rec, int lane) {
  constexpr int U = ADDROW ? 2 : 4;
  for (u32 i0 = lane; i0 < n; i0 += 32 * U) {
    int slot[U];
    int r[U][8];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const u32 i = i0 + 32 * u;
      slot[u] = -1;
      if (i < n) {
        slot[u] = slot0 + stage[i];
        if (!in_range(slot[u], a.s.cap, a.s.err)) slot[u] = -1;
        ld_v8_nc(rec + (size_t)(r0 + i) * 8, r[u]);
      }
    }
    if (ADDROW) {
      int o[U][8];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (slot[u] >= 0) ld_v8(a.s.fields + (size_t)slot[u] * 8, o[u]);
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int f = 0; f < 8; ++f) r[u][f] = (int)((u32)o[u][f] + (u32)r[u][f]);
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (slot[u] >= 0) st_v8(a.s.fields + (size_t)slot[u] * 8, r[u]);
  }
}

// a lane's flagged slots (bits of m, offsets from off0) to stage[pos ...), those below place `end`. Dense steps go
// through all 16 places, sparse ones through the set bits only.
template <typename S>
__device__ __forceinline__ void stage_bits(S* stage, u32 m, u32 pos, u32 end, int off0, bool dense) {
  if (dense) {
#pragma unroll
    for (int j = 0; j < kLaneSlots; ++j) {
      const u32 at = pos + (u32)__popc(m & ((1u << j) - 1u));
      if (((m >> j) & 1u) && at < end) stage[at] = (S)(off0 + j);
    }
  } else {
    while (m && pos < end) {
      stage[pos++] = (S)(off0 + __ffs(m) - 1);
      m &= m - 1;
    }
  }
}

// Pass 2: ranks from the CTA prefix + warp prefix + a warp scan per step.
// Each 512-slot step of a warp stages its flagged slots in shared memory in
// rank order (each lane writes its own, 16 slots at most) and the warp copies
// them out coalesced; steps with no rank below the limit are skipped. The add
// passes also write the final live flags of every 16-slot group that receives
// a new agent, whole (0/1), so no flag sector is written in part.
// MOVE (selective-update call, 8 fields, 32-byte aligned records): the pass
// moves the records itself instead of writing the rank-ordered slot lists, and
// no apply pass follows. LATE (selective-update call): see k_count_fused.
template <int OP, int THREADS, bool MOVE = false, bool LATE = false>
__global__ void __launch_bounds__(THREADS, MOVE ? move_resident<THREADS>() : 1) k_scatter(ScanArgs a) {
  constexpr int WARPS = THREADS / 32;
  __shared__ u64 s_red[WARPS];
  __shared__ int s_stage[MOVE ? 1 : WARPS * kWarpStep];
  __shared__ unsigned short s_move[MOVE ? WARPS * 2 * kMoveStage : 1];
  griddep_wait();
  const SlabDev& s = a.s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int seg = a.chunk / WARPS;
  const int wlo = blockIdx.x * a.chunk + warp * seg;
  const int whi = min(a.n, wlo + seg);
  // the plane words of the warp's first step, requested ahead of the prefix
  // sums; each step then requests the next step's words before its own work,
  // so a warp waits for one round trip in all, not one per step
  u32 wa_next = 0, wb_next = 0, wl_next = 0;
  {
    const int base = wlo + lane * kLaneSlots;
    if (wlo < whi && base < a.n) {
      wa_next = a.planeA[base >> 5];
      if (OP == OP_FUSED) wb_next = a.planeB[base >> 5];
      if (LATE) wl_next = a.planeL[base >> 5];
    }
  }
  u32 pa = 0, pb = 0, ta = 0, tb = 0;
  for (int j = threadIdx.x; j < a.G; j += THREADS) {
    const u32 x = a.totals[2 * j], y = a.totals[2 * j + 1];
    if (j < (int)blockIdx.x) {
      pa += x;
      pb += y;
    }
    ta += x;
    tb += y;
  }
  block_sum2<THREADS>(pa, pb, s_red);
  block_sum2<THREADS>(ta, tb, s_red);
  {
    u32 x = 0, y = 0;
    if (lane < warp) {
      x = a.wtotals[2 * (blockIdx.x * WARPS + lane)];
      y = a.wtotals[2 * (blockIdx.x * WARPS + lane) + 1];
    }
    u64 v = ((u64)x << 32) | y;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    pa += (u32)(v >> 32);
    pb += (u32)v;
  }
  const int nrec = (OP == OP_UPDATE && a.use_rec_idx) ? s.counters[3] : a.k;
  const u32 limit = (u32)(OP == OP_UPDATE ? nrec : (OP == OP_SELECT || OP == OP_ARRAY ? 0x7FFFFFFF : a.k));
  const u32 limit_b = (u32)a.k;
  if (OP == OP_FUSED && a.crowded && blockIdx.x == (unsigned)(a.wave / a.chunk) && threadIdx.x == 0) {
    // (pa: the free slots in front of this CTA) adds reach the slots of a second wave and leave much free
    const u32 added = min(limit, ta);
    const int crowded = pa < added && 2 * (u64)ta > 5 * (u64)added;
    if (crowded != a.crowded_known) *reinterpret_cast<volatile int*>(a.crowded) = crowded;
  }
  // ranks land at list_a + *list_base (the permutation's second half)
  int32_t* const list_a = a.list_a + (OP == OP_SELECT && a.list_base ? *a.list_base : 0);
  int* const stage = s_stage + (MOVE ? 0 : warp * kWarpStep);
  // MOVE: the slots staged for adds (0) and updates (1): how many, the first one's step and rank
  unsigned short* const mst[2] = {s_move + (MOVE ? warp * 2 * kMoveStage : 0),
                                  s_move + (MOVE ? (warp * 2 + 1) * kMoveStage : 0)};
  u32 mcnt[2] = {0, 0}, mrank[2] = {0, 0};
  int mbase[2] = {0, 0};
  for (int b0 = wlo; b0 < whi; b0 += kWarpStep) {
    const int base = b0 + lane * kLaneSlots;
    const u32 wa = wa_next, wb = wb_next, wl = wl_next;
    {
      const int nbase = base + kWarpStep;
      wa_next = wb_next = wl_next = 0;
      if (b0 + kWarpStep < whi && nbase < a.n) {
        wa_next = a.planeA[nbase >> 5];
        if (OP == OP_FUSED) wb_next = a.planeB[nbase >> 5];
        if (LATE) wl_next = a.planeL[nbase >> 5];
      }
    }
    u32 ma = 0, mb = 0;
    if (base < a.n) {
      ma = (wa >> (16 * (lane & 1))) & 0xFFFFu;
      if (OP == OP_FUSED) mb = (wb >> (16 * (lane & 1))) & 0xFFFFu;
    }
    const u32 c = (u32)__popc(ma) | ((u32)__popc(mb) << 16);
    u32 inc = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const u32 t = __shfl_up_sync(0xFFFFFFFFu, inc, o);
      if (lane >= o) inc += t;
    }
    const u32 tot = __shfl_sync(0xFFFFFFFFu, inc, 31);
    const u32 ex = inc - c;
    const u32 sa = pa, sb = pb;  // ranks of the step's first flagged slots
    pa += tot & 0xFFFFu;
    pb += tot >> 16;
    // plane A: the step's ranks [sa, sa + na) are below the limit
    const u32 na = sa < limit ? min(tot & 0xFFFFu, limit - sa) : 0u;
    const u32 nb = OP == OP_FUSED && sb < limit_b ? min(tot >> 16, limit_b - sb) : 0u;
    if constexpr (MOVE) {
      const u32 n2[2] = {na, nb}, r2[2] = {sa, sb}, m2[2] = {ma, mb}, o2[2] = {ex & 0xFFFFu, ex >> 16};
      // staged offsets are 16 bits; the next step's must still fit
      const bool last = b0 + kWarpStep >= whi;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        if (n2[k]) {
          if (mcnt[k] == 0) {
            mbase[k] = b0;
            mrank[k] = r2[k];
          }
          stage_bits(mst[k], m2[k], mcnt[k] + o2[k], mcnt[k] + n2[k], base - mbase[k], n2[k] > kWarpStep / 4);
          mcnt[k] += n2[k];
        }
        if (mcnt[k] && (mcnt[k] >= kMoveBatch || last || b0 - mbase[k] + 2 * kWarpStep > 65536)) {
          __syncwarp();
          if (k == 0) move_staged<false>(a, mst[0], mbase[0], mcnt[0], mrank[0], a.rec, lane);
          else move_staged<true>(a, mst[1], mbase[1], mcnt[1], mrank[1], a.rec2, lane);
          mcnt[k] = 0;
          __syncwarp();  // the stage is rewritten next
        }
      }
    } else if (na) {
      stage_bits(stage, ma, ex & 0xFFFFu, na, base, na > kWarpStep / 4);
      __syncwarp();
      for (u32 i = lane; i < na; i += 32) list_a[sa + i] = stage[i];
    }
    if (OP == OP_ADD || OP == OP_FUSED) {
      // flags of the lane's 16 slots after the adds: live 1, free 0, and the
      // free slots with a rank below the limit 1. Written are the groups that
      // receive an agent, or LATE the 8-slot halves that an add or a removal left
      // different from memory: a removed slot that is refilled costs no write
      // (2^24 slots, half of them touched: two passes over 64 MB of flags less).
      const u32 off = ex & 0xFFFFu;
      const u32 mine = off < na ? min((u32)__popc(ma), na - off) : 0u;
      if (LATE || mine) {
        const u32 added = mine == (u32)__popc(ma) ? ma : (mine ? ma & ((1u << __fns(ma, 0, (int)mine + 1)) - 1u) : 0u);
        const u32 valid = base + kLaneSlots <= a.n ? 0xFFFFu : (base < a.n ? (1u << (a.n - base)) - 1u : 0u);
        const u32 nl = ((~ma & valid) | added) & valid;
        u32 halves = 3u;
        if (LATE) {
          const u32 ml = (wl >> (16 * (lane & 1))) & valid;
          const u32 touched = mine ? 0xFFFFu : ma & ml, diff = nl ^ ml;
          halves = ((touched & 0xFFu) && (diff & 0xFFu) ? 1u : 0u) | ((touched >> 8) && (diff >> 8) ? 2u : 0u);
        }
        if (halves && valid == 0xFFFFu) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (!((halves >> h) & 1u)) continue;
            int f[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) f[j] = (int)((nl >> (8 * h + j)) & 1u);
            st_v8(s.active + base + 8 * h, f);
          }
        } else if (halves) {
          for (int j = 0; j < kLaneSlots; ++j)
            if (((valid >> j) & 1u) && ((halves >> (j >> 3)) & 1u)) s.active[base + j] = (int)((nl >> j) & 1u);
        }
      }
    }
    // plane B (the fused call's chosen survivors), the same way
    if (!MOVE && nb) {
      __syncwarp();
      stage_bits(stage, mb, ex >> 16, nb, base, nb > kWarpStep / 4);
      __syncwarp();
      for (u32 i = lane; i < nb; i += 32) a.list_b[sb + i] = stage[i];
    }
    if (!MOVE) __syncwarp();  // the stage is rewritten next
  }
  if (last_cta_out(a.ctrl)) {
    const int A = (int)ta, B = (int)tb;
    if (OP == OP_SELECT || OP == OP_ARRAY) {
      if (a.out_count) *a.out_count = A;
      if (OP == OP_ARRAY) s.counters[3] = A;
    } else if (OP == OP_ADD) {
      const int r = min(a.k, A);
      s.meta[0] = r;
      s.meta[1] = 0;
      s.meta[2] = s.counters[1];  // first id of this batch
      s.counters[0] += r;
      if (a.id_field >= 0) s.counters[1] += r;
      if (a.k > A) s.counters[2] = 1;
      if (a.out_count) *a.out_count = r;
    } else if (OP == OP_UPDATE) {
      const int r = min(A, nrec);
      s.meta[0] = r;
      s.meta[1] = 0;
      if (a.out_count) *a.out_count = r;
    } else if (OP == OP_FUSED) {  // A = free after removal, B = chosen survivors
      const int n_before = s.counters[0];
      const int added = min(a.k, A);
      s.meta[0] = added;
      s.meta[1] = min(a.k, B);
      s.counters[0] = s.cap - A + added;
      if (a.k > A) s.counters[2] = 1;
      if (a.out_count) {
        a.out_count[0] = A - (s.cap - n_before);
        a.out_count[1] = added;
        a.out_count[2] = min(a.k, B);
      }
    }
    __threadfence();
  }
}

// Whole 8-field rows, 32-byte aligned: records [j0, j1) of `rec` (or their
// rec_idx entries) go to the slots list[j], U rows in flight per thread, all
// loads issued before the stores. ADDROW: the slot's row is read and the
// record added to it field-wise (wrapping).
template <int U, bool ADDROW, bool STAMP, bool IDX>
__device__ __forceinline__ void move_rows_v8(const ScanArgs& a, const int32_t* rec, const int32_t* list, int j1,
                                             int id_field, int id0) {
  const SlabDev& s = a.s;
  const int stride = gridDim.x * blockDim.x;
  for (int j0 = blockIdx.x * blockDim.x + threadIdx.x; j0 < j1; j0 += U * stride) {
    int slot[U];
    int r[U][8];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int j = j0 + u * stride;
      slot[u] = -1;
      if (j < j1) {
        slot[u] = list[j];
        if (!in_range(slot[u], s.cap, s.err)) slot[u] = -1;
        ld_v8_nc(rec + (size_t)(IDX ? s.rec_idx[j] : j) * 8, r[u]);
      }
    }
    if (ADDROW) {
      int o[U][8];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (slot[u] >= 0) ld_v8(s.fields + (size_t)slot[u] * 8, o[u]);
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int f = 0; f < 8; ++f) r[u][f] = (int)((u32)o[u][f] + (u32)r[u][f]);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (slot[u] < 0) continue;
      if (STAMP) {  // the id of an added agent: next id + its rank
        const int id = (int)((u32)id0 + (u32)(j0 + u * stride));
#pragma unroll
        for (int f = 0; f < 8; ++f)
          if (f == id_field) r[u][f] = id;
      }
      st_v8(s.fields + (size_t)slot[u] * 8, r[u]);
    }
  }
}

__device__ __forceinline__ int wrap_add(int a, int b) { return (int)((u32)a + (u32)b); }
__device__ __forceinline__ int4 wrap_add(int4 a, int4 b) {
  return make_int4(wrap_add(a.x, b.x), wrap_add(a.y, b.y), wrap_add(a.z, b.z), wrap_add(a.w, b.w));
}
__device__ __forceinline__ void set_word(int& v, int, int x) { v = x; }
__device__ __forceinline__ void set_word(int4& v, int c, int x) {
  if (c == 0) v.x = x;
  else if (c == 1) v.y = x;
  else if (c == 2) v.z = x;
  else v.w = x;
}

// Rows of any other shape: records [0, n) of `rec` (or their rec_idx entries) in
// units V (int4 where the fields are a multiple of four and the records 16-byte
// aligned, else words), a warp taking 32 records and neighbouring lanes
// neighbouring units: a record's words are read and written together, U of a
// lane's in flight. (A record per thread, field by field: the loads of one warp 32
// records apart, each waited for before its store. 199,000 records of 11 fields
// added to a set of 931,561 slots 89 -> 9 us;
// the fused call's 1.4 M moves of 12 fields on 4 M slots 76 -> 64.)
template <typename V, bool ADDROW, bool STAMP, bool IDX>
__device__ __forceinline__ void move_rows(const ScanArgs& a, const int32_t* rec, const int32_t* list, int n, int id_field,
                                          int id0) {
  constexpr int W = sizeof(V) / 4, U = 16 / (2 * W) > 4 ? 8 : 4;
  const SlabDev& s = a.s;
  const V* const src = reinterpret_cast<const V*>(rec);
  V* const dst = reinterpret_cast<V*>(s.fields);
  const int F = s.F / W, Fp = s.Fp / W, lane = threadIdx.x & 31;
  if (F == 1) {  // a unit a row: U records per thread in flight
    const int stride = gridDim.x * blockDim.x;
    for (int j0 = blockIdx.x * blockDim.x + threadIdx.x; j0 < n; j0 += U * stride) {
      V v[U], o[U];
      int slot[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int j = j0 + u * stride;
        slot[u] = j < n ? list[j] : -1;
        if (j < n && !in_range(slot[u], s.cap, s.err)) slot[u] = -1;
        if (slot[u] >= 0) v[u] = __ldg(src + (IDX ? s.rec_idx[j] : j));
        if (STAMP && slot[u] >= 0) set_word(v[u], id_field, (int)((u32)id0 + (u32)j));
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (ADDROW && slot[u] >= 0) o[u] = dst[(size_t)slot[u] * Fp];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (slot[u] >= 0) dst[(size_t)slot[u] * Fp] = ADDROW ? wrap_add(o[u], v[u]) : v[u];
    }
    return;
  }
  const int rq = 32 / F, rm = 32 % F, r0 = lane / F, f0 = lane % F;
  const int warps = gridDim.x * (blockDim.x >> 5);
  for (int j0 = 32 * (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)); j0 < n; j0 += 32 * warps) {
    const int m = min(32, n - j0);
    int slot = -1, from = j0 + lane;
    if (lane < m) {
      slot = list[j0 + lane];
      if (!in_range(slot, s.cap, s.err)) slot = -1;
      if (IDX) from = s.rec_idx[j0 + lane];
    }
    int r = r0, f = f0;
    for (int e0 = 0; e0 < m * F; e0 += 32 * U) {
      V v[U], o[U];
      size_t at[U];
      bool ok[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int sl = __shfl_sync(0xFFFFFFFFu, slot, r & 31), sr = __shfl_sync(0xFFFFFFFFu, from, r & 31);
        ok[u] = e0 + 32 * u + lane < m * F && sl >= 0;
        at[u] = (size_t)(ok[u] ? sl : 0) * Fp + f;
        if (ok[u]) v[u] = __ldg(src + (size_t)sr * F + f);
        if (ADDROW && ok[u]) o[u] = dst[at[u]];
        if (STAMP && ok[u] && f == id_field / W) set_word(v[u], id_field % W, (int)((u32)id0 + (u32)(j0 + r)));
        r += rq;
        f += rm;
        if (f >= F) {
          f -= F;
          ++r;
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (ok[u]) dst[at[u]] = ADDROW ? wrap_add(o[u], v[u]) : v[u];
    }
  }
}

template <int OP, typename V>
__device__ __forceinline__ void apply_rows(const ScanArgs& a, int ra, int rb, int id0) {
  if (OP == OP_UPDATE) {
    const bool idx = a.use_rec_idx != 0;
    if (a.op_kind == ABM_OP_ADD) {
      if (idx) move_rows<V, true, false, true>(a, a.rec, a.list_a, ra, -1, 0);
      else move_rows<V, true, false, false>(a, a.rec, a.list_a, ra, -1, 0);
    } else {
      if (idx) move_rows<V, false, false, true>(a, a.rec, a.list_a, ra, -1, 0);
      else move_rows<V, false, false, false>(a, a.rec, a.list_a, ra, -1, 0);
    }
  } else if (OP == OP_ADD && a.id_field >= 0) {
    move_rows<V, false, true, false>(a, a.rec, a.list_a, ra, a.id_field, id0);
  } else {
    move_rows<V, false, false, false>(a, a.rec, a.list_a, ra, -1, 0);
  }
  if (OP == OP_FUSED) move_rows<V, true, false, false>(a, a.rec2, a.list_b, rb, -1, 0);
}

// Pass 3: record j goes to (or is added to) the slot at rank j, several in flight
// per thread, all loads issued before the stores; coalesced record reads, one
// field run written per slot (one 32-byte store for 8 fields). Two CTAs of 256
// threads per SM (96 registers) measured faster than three with two rows in flight
// where rows are read.
template <int OP>
__global__ void __launch_bounds__(256, 2) k_apply(ScanArgs a) {
  griddep_wait();
  const SlabDev& s = a.s;
  const int ra = s.meta[0], rb = s.meta[1];
  const int id0 = s.meta[2];
  const uintptr_t al = (uintptr_t)a.rec | (uintptr_t)a.rec2;
  // 8 fields, records 32-byte aligned (the rows always are): whole rows per instruction
  if (s.F == 8 && s.Fp == 8 && ((al | (uintptr_t)s.fields) & 31) == 0) {
    if (OP == OP_UPDATE) {
      const bool idx = a.use_rec_idx != 0;
      if (a.op_kind == ABM_OP_ADD) {
        if (idx) move_rows_v8<4, true, false, true>(a, a.rec, a.list_a, ra, -1, 0);
        else move_rows_v8<4, true, false, false>(a, a.rec, a.list_a, ra, -1, 0);
      } else {
        if (idx) move_rows_v8<4, false, false, true>(a, a.rec, a.list_a, ra, -1, 0);
        else move_rows_v8<4, false, false, false>(a, a.rec, a.list_a, ra, -1, 0);
      }
    } else if (OP == OP_ADD && a.id_field >= 0) {
      move_rows_v8<4, false, true, false>(a, a.rec, a.list_a, ra, a.id_field, id0);
    } else {
      move_rows_v8<4, false, false, false>(a, a.rec, a.list_a, ra, -1, 0);
    }
    if (OP == OP_FUSED) move_rows_v8<4, true, false, false>(a, a.rec2, a.list_b, rb, -1, 0);
  } else if ((s.F & 3) == 0 && (al & 15) == 0) {
    apply_rows<OP, int4>(a, ra, rb, id0);
  } else {
    apply_rows<OP, int>(a, ra, rb, id0);
  }
}

// ---------------------------------------------------------------------------
// Small sets: one launch per operation. Up to kSmallMax slots are held by one
// thread-block cluster, LS consecutive slots per lane, so that flags, ranks and
// record moves happen in one kernel: the CTAs' counts are exchanged through
// distributed shared memory between two cluster barriers. Three launches that
// each touch 0.4 MB cost their launches and round trips, not their bytes. GPU
// time of a select / update / remove / add back to back, three launches against
// one, few records: 1000 slots 9.2 / 11.0 / 9.2 / 8.2 -> 2.2 / 2.8 / 2.1 / 1.8 us; 100,003
// slots 10.2 / 14.3 / 10.3 / 8.2 -> 5.5 / 7.0 / 5.0 / 3.2; at 262,144 slots,
// where 16 SMs do what 64 CTAs do above it, 8.4 / 11.0 / 7.7 / 4.2 (three
// launches at 300,000: 8.2 / 12.3 / 8.2 / 8.2). For many records see small_moves.
constexpr int kSmallThreads = 1024;
constexpr int kSmallWarps = kSmallThreads / 32;
constexpr int kSmallCtas = 16;  // cluster size, at most (above 8: opt-in)
constexpr int kSmallMax = kSmallCtas * kSmallThreads * 16;

// word c of v, if it has one
__device__ __forceinline__ void stamp_word(int& v, int c, int x) { v = c == 0 ? x : v; }
__device__ __forceinline__ void stamp_word(int4& v, int c, int x) {
  v = make_int4(c == 0 ? x : v.x, c == 1 ? x : v.y, c == 2 ? x : v.z, c == 3 ? x : v.w);
}

// Records r0 .. r0 + n - 1, their slots staged by the warp (offsets from slot0) or, with
// LIST, in a list that the cluster wrote (list[r0] on), in units V (int4 where the fields are a multiple of four and the records 16-byte aligned, else
// words), neighbouring lanes on neighbouring units of a record, U of a lane's in flight.
// ADD: added to the row (wrapping); id_field >= 0: that field is id0 + r instead.
template <typename V, int U, bool ADD, bool LIST>
__device__ __forceinline__ void move_small_units(const SlabDev& s, const unsigned short* stage, const int32_t* list,
                                                 int slot0, u32 n, u32 r0, const int32_t* rec, const int32_t* rec_idx,
                                                 int id_field, int id0, int lane, u32 div1, u32 div4) {
  constexpr int W = sizeof(V) / 4;
  const V* const src = reinterpret_cast<const V*>(rec);
  V* const dst = reinterpret_cast<V*>(s.fields);
  const u32 F = (u32)s.F / W, Fp = (u32)s.Fp / W;
  const u32 inv = W == 4 ? div4 : div1;  // x / F = x * inv >> 16 for x <= 32
  const u32 rq = (32u * inv) >> 16, rm = 32u - rq * F;
  u32 i = ((u32)lane * inv) >> 16, f = (u32)lane - i * F;
  for (u32 e0 = lane; e0 < n * F; e0 += 32 * U) {
    V v[U], o[U];
    u32 at[U];
    bool ok[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      ok[u] = e0 + 32 * u < n * F;
      if (ok[u]) {
        const int slot = LIST ? __ldcg(list + r0 + i) : slot0 + stage[i];
        ok[u] = in_range(slot, s.cap, s.err);
        at[u] = (u32)slot * Fp + f;
        const u32 j = rec_idx ? (u32)rec_idx[r0 + i] : r0 + i;
        v[u] = __ldg(src + (size_t)j * F + f);
        if (ADD && ok[u]) o[u] = dst[at[u]];
        if (!ADD) stamp_word(v[u], id_field - W * (int)f, (int)((u32)id0 + r0 + i));
      }
      i += rq;
      f += rm;
      if (f >= F) {
        f -= F;
        ++i;
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (ok[u]) dst[at[u]] = ADD ? wrap_add(o[u], v[u]) : v[u];
  }
}

// U: four words, or two int4 where rows are read; one int4 where they are only written (the next store does not wait for
// the one before, and a CTA that runs once pays for every instruction it fetches).
template <bool ADD, bool LIST>
__device__ __forceinline__ void move_small(const SlabDev& s, const unsigned short* stage, const int32_t* list, int slot0,
                                           u32 n, u32 r0, const int32_t* rec, const int32_t* rec_idx, int id_field, int id0,
                                           int lane, u32 div1, u32 div4) {
  if ((s.F & 3) == 0 && ((uintptr_t)rec & 15) == 0)
    move_small_units<int4, ADD ? 2 : 1, ADD, LIST>(s, stage, list, slot0, n, r0, rec, rec_idx, id_field, id0, lane, div1,
                                                   div4);
  else
    move_small_units<int, 4, ADD, LIST>(s, stage, list, slot0, n, r0, rec, rec_idx, id_field, id0, lane, div1, div4);
}

// Adds fall to the lowest free slots, updates to the first that satisfy a predicate, so
// on a set that is not in its steady state one CTA can own most of a call's records. The
// cluster then lists the slots and splits the records evenly, at a cluster barrier and a
// round trip more (3.5 us), where the CTA with most records has this much more to do than
// the average: in ns, a record costs a CTA 0.72 + 0.04 F, and a warp, which may own half its
// slots, 2 to 4 a unit. Without and with: adds of 7864 records to 262,144 half-live slots
// 11.9 and 10.0 us (4 fields), 13.6 and 10.0 (8), 23.1 and 11.0 (11); of 3932 records to
// 131,072 slots 7.3 and 7.6 (4), 8.3 and 7.6 (8); updates of 262 of those 10.0 and 6.3 (11).
__device__ __forceinline__ bool small_crowded(u32 most, u32 all, int F, u32 units, u32 half_warp) {
  const u32 more = most - all / gridDim.x;
  return more * (18u + (u32)F) / 25u > 3500u || min(more, half_warp) * units > 1000u;
}

// This warp's run of the na records of the first list and the nb of the second. (Out of
// line: the kernel's usual way is as short as without it.)
template <int OP>
__device__ __noinline__ void move_even(const ScanArgs& a, u32 na, u32 nb, int id0) {
  const int lane = threadIdx.x & 31;
  const u32 warps = gridDim.x * kSmallWarps, w = blockIdx.x * kSmallWarps + (threadIdx.x >> 5);
  u32 per = (na + warps - 1) / warps, r0 = min(na, per * w);
  u32 n = min(per, na - r0);
  if (OP == OP_UPDATE && a.op_kind == ABM_OP_ADD)
    move_small<true, true>(a.s, nullptr, a.list_a, 0, n, r0, a.rec, a.use_rec_idx ? a.s.rec_idx : nullptr, -1, 0, lane, a.div1, a.div4);
  else
    move_small<false, true>(a.s, nullptr, a.list_a, 0, n, r0, a.rec, OP == OP_UPDATE && a.use_rec_idx ? a.s.rec_idx : nullptr,
                            OP == OP_ADD ? a.id_field : -1, id0, lane, a.div1, a.div4);
  if (OP == OP_FUSED) {
    per = (nb + warps - 1) / warps;
    r0 = min(nb, per * w);
    n = min(per, nb - r0);
    move_small<true, true>(a.s, nullptr, a.list_b, 0, n, r0, a.rec2, nullptr, -1, 0, lane, a.div1, a.div4);
  }
}

template <int OP, int LS>
__global__ void __launch_bounds__(kSmallThreads, 1) k_small(const __grid_constant__ ScanArgs a) {
  constexpr int STEP = 32 * LS;  // slots of a warp
  constexpr bool MOVES = OP == OP_ADD || OP == OP_UPDATE || OP == OP_FUSED;
  __shared__ u64 s_w[kSmallWarps];
  __shared__ u64 s_tot;     // this CTA's counts: A << 32 | B
  __shared__ u64 s_pre[2];  // the CTAs before, all
  __shared__ int s_even;    // the cluster splits the records evenly
  __shared__ unsigned short s_stage[kSmallWarps * STEP];
  const SlabDev& s = a.s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int slot0 = ((int)blockIdx.x * kSmallWarps + warp) * STEP;
  const int base = slot0 + LS * lane;
  griddep_wait();
  const int32_t* flag_src = OP == OP_ARRAY ? a.src : s.active;
  int live[LS];
  if (base + LS <= a.n && (((uintptr_t)flag_src) & 15) == 0) {
#pragma unroll
    for (int v = 0; v < LS / 4; ++v) {
      const int4 q = *reinterpret_cast<const int4*>(flag_src + base + 4 * v);
      live[4 * v] = q.x; live[4 * v + 1] = q.y; live[4 * v + 2] = q.z; live[4 * v + 3] = q.w;
    }
  } else {
#pragma unroll
    for (int j = 0; j < LS; ++j) live[j] = base + j < a.n ? flag_src[base + j] : 0;
  }
  // read before the barrier after which CTA 0 changes them
  const int id0 = s.counters[1];
  const int nrec = (OP == OP_UPDATE && a.use_rec_idx) ? s.counters[3] : a.k;
  const u32 valid = a.n - base >= LS ? (1u << LS) - 1u : (a.n > base ? (1u << (a.n - base)) - 1u : 0u);
  u32 on = 0, ma = 0, mb = 0, mr = 0;  // live; selected / free; chosen; removed
#pragma unroll
  for (int j = 0; j < LS; ++j) on |= (u32)(live[j] != 0) << j;
  on &= valid;
  if (OP == OP_ARRAY) {
    ma = on;
  } else if (OP == OP_ADD) {
    ma = ~on & valid;
  } else if (OP == OP_FUSED) {
    u32 dr = 0, dc = 0;
#pragma unroll
    for (int m = 0; m < LS / 2; ++m) {
      const uint4 u = mask_pair_draw((u32)(base >> 1) + m, a.mk, a.rk);
      dr |= (u.x < a.threshold ? 1u << (2 * m) : 0u) | (u.z < a.threshold ? 2u << (2 * m) : 0u);
      dc |= (u.y < a.threshold ? 1u << (2 * m) : 0u) | (u.w < a.threshold ? 2u << (2 * m) : 0u);
    }
    mr = on & dr;
    on &= ~dr;
    ma = ~on & valid;
    mb = on & dc;
  } else {
    ma = pred_mask<LS>(a.pred, s, base, a.n, live);
    if (a.negate) ma = ~ma & valid;
    if (OP == OP_REMOVE) mr = ma;
  }
  // ranks: lanes, warps, CTAs
  const u32 c = (u32)__popc(ma) | ((u32)__popc(mb) << 16);
  u32 inc = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const u32 t = __shfl_up_sync(0xFFFFFFFFu, inc, o);
    if (lane >= o) inc += t;
  }
  const u32 ex = inc - c, tot = __shfl_sync(0xFFFFFFFFu, inc, 31);
  if (lane == 0) s_w[warp] = ((u64)(tot & 0xFFFFu) << 32) | (tot >> 16);
  __syncthreads();
  u64 wv = s_w[lane], wpre = lane < warp ? wv : 0ull;  // kSmallWarps == 32
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    wv += __shfl_xor_sync(0xFFFFFFFFu, wv, o);
    wpre += __shfl_xor_sync(0xFFFFFFFFu, wpre, o);
  }
  const u32 limit = (u32)(OP == OP_UPDATE ? nrec : (OP == OP_SELECT || OP == OP_ARRAY ? 0x7FFFFFFF : a.k));
  u64 pre = 0, all = wv;
  bool even = false;
  if (gridDim.x > 1) {
    if (threadIdx.x == 0) s_tot = wv;
    cluster_arrive();
    cluster_wait();
    if (warp == 0) {
      const u64 t = lane < (int)gridDim.x ? ld_cluster(&s_tot, (u32)lane) : 0ull;
      u64 p = t;
#pragma unroll
      for (int o = 1; o < kSmallCtas; o <<= 1) {
        const u64 x = __shfl_up_sync(0xFFFFFFFFu, p, o);
        if (lane >= o) p += x;
      }
      if (lane == (int)gridDim.x - 1) s_pre[1] = p;
      p -= t;
      if (lane == (int)blockIdx.x) s_pre[0] = p;
      if (MOVES) {  // the records of each list that a CTA has to move, by its slots' ranks
        const u32 before = (u32)(p >> 32), mine = before < limit ? min((u32)(t >> 32), limit - before) : 0u;
        const u32 before2 = (u32)p, mine2 = before2 < (u32)a.k ? min((u32)t, (u32)a.k - before2) : 0u;
        const u32 most = __reduce_max_sync(0xFFFFFFFFu, mine), sum = __reduce_add_sync(0xFFFFFFFFu, mine);
        const u32 most2 = __reduce_max_sync(0xFFFFFFFFu, mine2), sum2 = __reduce_add_sync(0xFFFFFFFFu, mine2);
        const u32 units = (s.F & 3) == 0 && (((uintptr_t)a.rec | (uintptr_t)a.rec2) & 15) == 0 ? s.F >> 2 : s.F;
        const bool crowded = small_crowded(most, sum, s.F, units, STEP / 2);
        const bool crowded2 = OP == OP_FUSED && small_crowded(most2, sum2, s.F, units, STEP / 2);
        if (lane == 0) s_even = crowded || crowded2;
      }
    }
    __syncthreads();
    cluster_arrive();  // the others' counts are read; waited for before leaving
    pre = s_pre[0];
    all = s_pre[1];
    if (MOVES) even = s_even != 0;
  } else {
    __syncthreads();  // every thread has read the counters that are changed below
  }
  pre += wpre;
  const u32 sa = (u32)(pre >> 32), sb = (u32)pre;
  const int A = (int)(all >> 32), B = (int)all;
  // removed slots become placeholders: k_count's (4-slot groups, other flags kept) and k_count_fused's (8-slot groups
  // as 0/1) writes
  if (OP == OP_REMOVE) {
#pragma unroll
    for (int v = 0; v < LS / 4; ++v) {
      const u32 g = (mr >> (4 * v)) & 0xFu;
      if (!g) continue;
      const int b = base + 4 * v;
      const int4 q = make_int4((g & 1u) ? 0 : live[4 * v], (g & 2u) ? 0 : live[4 * v + 1],
                               (g & 4u) ? 0 : live[4 * v + 2], (g & 8u) ? 0 : live[4 * v + 3]);
      if (b + 3 < a.n) {
        *reinterpret_cast<int4*>(s.active + b) = q;
      } else {
        if (b + 0 < a.n) s.active[b + 0] = q.x;
        if (b + 1 < a.n) s.active[b + 1] = q.y;
        if (b + 2 < a.n) s.active[b + 2] = q.z;
      }
    }
  }
  u32 na = 0;
  if (OP != OP_REMOVE && sa < limit) na = min(tot & 0xFFFFu, limit - sa);
  if (OP == OP_ADD || OP == OP_FUSED) {
    // final flags: live, or free with a rank below the limit. Written as 0/1 in whole groups: the 16 slots around an
    // added agent, the 8 around a removed one
    const u32 e0 = ex & 0xFFFFu;
    const u32 mine = e0 < na ? min((u32)__popc(ma), na - e0) : 0u;
    const u32 added = mine == (u32)__popc(ma) ? ma : (mine ? ma & ((1u << __fns(ma, 0, (int)mine + 1)) - 1u) : 0u);
    const u32 nl = on | added;
    const u32 ab = __ballot_sync(0xFFFFFFFFu, added != 0u);
    u32 wr = LS == 16 ? (added ? valid : 0u)
                      : (((ab >> (lane & ~(16 / LS - 1))) & ((1u << (16 / LS)) - 1u)) ? valid : 0u);
    if (OP == OP_FUSED) {
      if (LS >= 8) {
#pragma unroll
        for (int h = 0; h < LS / 8; ++h)
          if ((mr >> (8 * h)) & 0xFFu) wr |= valid & (0xFFu << (8 * h));
      } else {
        const u32 rb = __ballot_sync(0xFFFFFFFFu, mr != 0u);
        if ((rb >> (lane & ~1)) & 3u) wr = valid;
      }
    }
#pragma unroll
    for (int v = 0; v < LS / 4; ++v) {
      if (!((wr >> (4 * v)) & 0xFu)) continue;
      const u32 g = nl >> (4 * v);
      const int b = base + 4 * v;
      if (b + 3 < a.n) {
        *reinterpret_cast<int4*>(s.active + b) =
            make_int4((int)(g & 1u), (int)((g >> 1) & 1u), (int)((g >> 2) & 1u), (int)((g >> 3) & 1u));
      } else {
#pragma unroll
        for (int j = 0; j < 3; ++j)
          if (b + j < a.n) s.active[b + j] = (int)((g >> j) & 1u);
      }
    }
  }
  // the selected slots in rank order, then lists and records
  unsigned short* stage = s_stage + warp * STEP;
  const int32_t* const idx = OP == OP_UPDATE && a.use_rec_idx ? s.rec_idx : nullptr;
  const bool add = OP == OP_UPDATE && a.op_kind == ABM_OP_ADD;
  const int idf = OP == OP_ADD ? a.id_field : -1;
  if (OP != OP_REMOVE && na) {
    u32 pos = ex & 0xFFFFu;
#pragma unroll
    for (int j = 0; j < LS; ++j)
      if ((ma >> j) & 1u) stage[pos++] = (unsigned short)(LS * lane + j);
    __syncwarp();
    int32_t* const list = a.list_a + (OP == OP_SELECT && a.list_base ? *a.list_base : 0);
    if (OP != OP_FUSED || even)  // (the selective-update call hands no list out)
      for (u32 i = lane; i < na; i += 32) list[sa + i] = slot0 + stage[i];
    if (MOVES && !even) {
      if (add) move_small<true, false>(s, stage, nullptr, slot0, na, sa, a.rec, idx, -1, 0, lane, a.div1, a.div4);
      else move_small<false, false>(s, stage, nullptr, slot0, na, sa, a.rec, idx, idf, id0, lane, a.div1, a.div4);
    }
    __syncwarp();
  }
  if (OP == OP_FUSED && sb < (u32)a.k && (tot >> 16)) {
    const u32 nb = min(tot >> 16, (u32)a.k - sb);
    u32 pos = ex >> 16;
#pragma unroll
    for (int j = 0; j < LS; ++j)
      if ((mb >> j) & 1u) stage[pos++] = (unsigned short)(LS * lane + j);
    __syncwarp();
    if (even)
      for (u32 i = lane; i < nb; i += 32) a.list_b[sb + i] = slot0 + stage[i];
    else
      move_small<true, false>(s, stage, nullptr, slot0, nb, sb, a.rec2, nullptr, -1, 0, lane, a.div1, a.div4);
  }
  if (MOVES && even) {
    __syncwarp();
    cluster_wait();
    cluster_arrive();  // the lists are complete
    cluster_wait();
    move_even<OP>(a, min((u32)A, limit), OP == OP_FUSED ? min((u32)B, (u32)a.k) : 0u, id0);
    cluster_arrive();  // (the wait at the end)
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    if (OP == OP_SELECT || OP == OP_ARRAY) {
      if (a.out_count) *a.out_count = A;
      if (OP == OP_ARRAY) s.counters[3] = A;
    } else if (OP == OP_REMOVE) {
      s.counters[0] -= A;
      if (a.out_count) *a.out_count = A;
    } else if (OP == OP_ADD) {
      const int r = min(a.k, A);
      s.counters[0] += r;
      if (a.id_field >= 0) s.counters[1] = (int)((u32)id0 + (u32)r);
      if (a.k > A) s.counters[2] = 1;
      if (a.out_count) *a.out_count = r;
    } else if (OP == OP_UPDATE) {
      if (a.out_count) *a.out_count = min(A, nrec);
    } else {  // A = free after removal, B = chosen survivors
      const int n_before = s.counters[0];
      const int added = min(a.k, A);
      s.counters[0] = s.cap - A + added;
      if (a.k > A) s.counters[2] = 1;
      if (a.out_count) {
        a.out_count[0] = A - (s.cap - n_before);
        a.out_count[1] = added;
        a.out_count[2] = min(a.k, B);
      }
    }
  }
  if (gridDim.x > 1) cluster_wait();
}

// --------------------------------------------------------------------------
// check builds: the fields past the capacity hold the canary, the live flags
// there stay 0; k_canary_check records kErrCheck if either changed
__global__ void k_canary_fill(int32_t* fields, int Fp, int cap, int n_pad) {
  const long long n = (long long)(n_pad - cap) * Fp;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    fields[(long long)cap * Fp + i] = kCanary;
}

__global__ void k_canary_check(const int32_t* active, const int32_t* fields, int Fp, int cap, int n_pad, int* err) {
  const long long n = (long long)(n_pad - cap) * Fp;
  bool bad = false;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    bad |= fields[(long long)cap * Fp + i] != kCanary;
  for (int i = cap + blockIdx.x * blockDim.x + threadIdx.x; i < n_pad; i += gridDim.x * blockDim.x)
    bad |= active[i] != 0;
  if (bad) atomicCAS(err, 0, kErrCheck);
}

__global__ void k_check_index(long long i, long long n, int* err) { in_range(i, n, err); }

__global__ void k_slab_init(SlabDev s, int init, int n_pad) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_pad; i += gridDim.x * blockDim.x) {
    const bool inside = i < s.cap;
    int live = 0;
    if (inside && init == ABM_INIT_HALF_LIVE)
      live = draw(s.seed, s.model, ABM_INIT_STEP, (u32)i, ABM_P_INIT_ACTIVE, 0u) < 0x80000000u;
    s.active[i] = live;
    int32_t* dst = s.fields + (size_t)i * s.Fp;
    uint4 w0 = make_uint4(0, 0, 0, 0), w1 = w0, w2 = w0, w3 = w0;
    if (inside && init == ABM_INIT_HALF_LIVE) {
      w0 = draw4(s.seed, s.model, ABM_INIT_STEP, (u32)i, ABM_P_NEWREC0, 0u);
      if (s.F > 4) w1 = draw4(s.seed, s.model, ABM_INIT_STEP, (u32)i, ABM_P_NEWREC1, 0u);
      if (s.F > 8) w2 = draw4(s.seed, s.model, ABM_INIT_STEP, (u32)i, ABM_P_NEWREC1 + 1, 0u);
      if (s.F > 12) w3 = draw4(s.seed, s.model, ABM_INIT_STEP, (u32)i, ABM_P_NEWREC1 + 2, 0u);
    }
    const uint4 w[4] = {w0, w1, w2, w3};
    for (int f = 0; f < s.Fp; f += 4) {
      const uint4 q = f < s.F ? w[f >> 2] : make_uint4(0, 0, 0, 0);
      int4 o = make_int4((int)q.x, (int)q.y, (int)q.z, (int)q.w);
      if (f + 1 >= s.F) o.y = 0;
      if (f + 2 >= s.F) o.z = 0;
      if (f + 3 >= s.F) o.w = 0;
      if (f >= s.F) o.x = 0;
      *reinterpret_cast<int4*>(dst + f) = o;
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    s.counters[1] = 0;
    s.counters[2] = 0;
    s.counters[3] = 0;
  }
}

// One field of agent-major records to or from a contiguous array, four
// elements per thread in flight. Bound by the sectors of the records: every
// element moves the 32-byte sector it lies in. (A 2D copy with rows of one
// int32 moves them one by one: 415 us for 4 M rows of 32 bytes; this kernel 38.)
constexpr int kStridedU = 4;
__global__ void __launch_bounds__(256) k_strided_copy(int32_t* dst, int dst_stride, const int32_t* src, int src_stride,
                                                      size_t n) {
  const size_t T = (size_t)gridDim.x * blockDim.x;
  for (size_t i0 = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i0 < n; i0 += kStridedU * T) {
    int32_t v[kStridedU];
#pragma unroll
    for (int u = 0; u < kStridedU; ++u)
      if (i0 + u * T < n) v[u] = src[(i0 + u * T) * src_stride];
#pragma unroll
    for (int u = 0; u < kStridedU; ++u)
      if (i0 + u * T < n) dst[(i0 + u * T) * dst_stride] = v[u];
  }
}

// n_active after init (a plain count)
__global__ void k_count_live(SlabDev s) {
  int c = 0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < s.cap; i += gridDim.x * blockDim.x)
    c += s.active[i] != 0;
  warp_add(&s.counters[0], c);
}

// live flags from src (the first n slots), counted on the way; the flags past
// n are only counted
__global__ void __launch_bounds__(256) k_write_flags(SlabDev s, const int32_t* src, int n) {
  int c = 0;
  const int T = gridDim.x * blockDim.x;
  for (int i0 = blockIdx.x * blockDim.x + threadIdx.x; i0 < s.cap; i0 += 4 * T) {
    int v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = i0 + u * T;
      v[u] = i < n ? src[i] : (i < s.cap ? s.active[i] : 0);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = i0 + u * T;
      if (i < n) s.active[i] = v[u];
      c += v[u] != 0;
    }
  }
  warp_add(&s.counters[0], c);
}

__global__ void k_philox_records(SlabDev s, u32 step, u32 p0, u32 p1, int k, int32_t* out) {
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < k; j += gridDim.x * blockDim.x) {
    int32_t* dst = out + (size_t)j * s.F;
    const uint4 a = draw4(s.seed, s.model, step, (u32)j, p0, 0u);
    const u32 wa[4] = {a.x, a.y, a.z, a.w};
    uint4 b = make_uint4(0, 0, 0, 0);
    if (s.F > 4) b = draw4(s.seed, s.model, step, (u32)j, p1, 0u);
    const u32 wb[4] = {b.x, b.y, b.z, b.w};
    for (int f = 0; f < s.F && f < 8; ++f) dst[f] = (int)(f < 4 ? wa[f] : wb[f - 4]);
  }
}

}  // namespace abm

// ============================================================================
// host side
using namespace abm;



extern "C" const char* abm_strerror(abm_status st) {
  switch (st) {
    case ABM_OK: return "ok";
    case ABM_ERR_ARG: return "invalid argument";
    case ABM_ERR_OOM: return "device allocation failed";
    case ABM_ERR_CUDA: return "CUDA runtime error";
    case ABM_ERR_DEVICE_TIMEOUT: return "device-side wait timed out";
    case ABM_ERR_OVERFLOW: return "more agents asked for a slot than were free";
    case ABM_ERR_STATE: return "operation not valid for this handle";
    case ABM_ERR_TOO_LARGE: return "size beyond the fixed maximum of this entry point";
    case ABM_ERR_CHECK: return "check build: an index out of range or a damaged canary was recorded";
  }
  return "unknown status";
}

extern "C" int32_t abm_version(void) { return kCheck ? -101 : 101; }

static void slab_free(abm_slab* s) {
  if (!s->view) {
    cudaFree(s->d.active);
    cudaFree(s->d.fields);
  }
  cudaFree(s->d.counters);
  cudaFree(s->d.rec_idx);
  cudaFree(s->d.err);
  cudaFree(s->planes);
  cudaFree(s->planes2);
  cudaFree(s->totals);
  cudaFree(s->totals2);
  cudaFree(s->wtotals);
  cudaFree(s->wtotals2);
  cudaFree(s->lista);
  cudaFree(s->listb);
  cudaFree(s->d.meta);
  cudaFree(s->ctrl);
  if (s->crowded) cudaFreeHost(s->crowded);  // (the frees above waited for every launch)
  sort_scratch_free(s->sort);
  delete s;
}

extern "C" abm_status abm_slab_destroy(abm_slab* s) {
  if (!s) return ABM_ERR_ARG;
  if (s->view) return ABM_ERR_STATE;  // a world's view lives as long as the world
  slab_free(s);
  return ABM_OK;
}

void abm::slab_free_view(abm_slab* s) {
  if (s) slab_free(s);
}

// host part of slab creation: the struct, its scratch and counters, and the
// live flags and fields unless they are borrowed (active != nullptr)
static abm_status slab_alloc(int capacity, int n_fields, u32 seed, u32 model, int32_t* active, int32_t* fields,
                             abm_slab** out) {
  abm_slab* s = new (std::nothrow) abm_slab();
  if (!s) return ABM_ERR_OOM;
  std::memset(s, 0, sizeof(*s));
  s->d.cap = capacity;
  s->d.F = n_fields;
  s->d.Fp = (n_fields + 3) & ~3;
  s->d.seed = seed;
  s->d.model = model;
  s->n_pad = ((capacity + kSlabTileMax - 1) / kSlabTileMax) * kSlabTileMax;
  s->max_ctas = num_sms() * 16;
  s->fused_threads = 256;
  s->fused_ctas_per_sm = 0;  // by the path taken
  s->view = active != nullptr;
  bool ok = true;
  if (s->view) {
    s->d.active = active;
    s->d.fields = fields;
  } else {
    ok = cudaMalloc(&s->d.active, sizeof(int32_t) * (size_t)s->n_pad) == cudaSuccess &&
         cudaMalloc(&s->d.fields, sizeof(int32_t) * (size_t)s->n_pad * s->d.Fp) == cudaSuccess;
  }
  ok = ok && cudaMalloc(&s->d.counters, sizeof(int32_t) * 4) == cudaSuccess &&
            cudaMalloc(&s->d.rec_idx, sizeof(int32_t) * (size_t)capacity) == cudaSuccess &&
            cudaMalloc(&s->d.err, sizeof(int)) == cudaSuccess &&
            cudaMalloc(&s->planes, sizeof(u32) * 2 * (size_t)(s->n_pad / 32)) == cudaSuccess &&
            cudaMalloc(&s->planes2, sizeof(u32) * (size_t)(s->n_pad / 32)) == cudaSuccess &&
            cudaMalloc(&s->totals, sizeof(u32) * 2 * (size_t)s->max_ctas) == cudaSuccess &&
            cudaMalloc(&s->totals2, sizeof(u32) * 2 * (size_t)s->max_ctas) == cudaSuccess &&
            cudaMalloc(&s->wtotals, sizeof(u32) * 32 * (size_t)s->max_ctas) == cudaSuccess &&
            cudaMalloc(&s->wtotals2, sizeof(u32) * 32 * (size_t)s->max_ctas) == cudaSuccess &&
            cudaMalloc(&s->lista, sizeof(int32_t) * (size_t)capacity) == cudaSuccess &&
            cudaMalloc(&s->listb, sizeof(int32_t) * (size_t)capacity) == cudaSuccess &&
            cudaMalloc(&s->d.meta, sizeof(int32_t) * 4) == cudaSuccess &&
            cudaMalloc(&s->ctrl, sizeof(u32) * 8) == cudaSuccess;
  if (ok && n_fields == 8 && capacity > kSmallMax) {
    ok = cudaHostAlloc(&s->crowded, sizeof(int), cudaHostAllocPortable | cudaHostAllocMapped) == cudaSuccess;
    if (ok) *s->crowded = 0;
  }
  if (!ok) {
    cudaGetLastError();
    slab_free(s);
    return ABM_ERR_OOM;
  }
  *out = s;
  return ABM_OK;
}

abm_status abm::slab_create_view(int cap, u32 seed, u32 model, int32_t* active, int32_t* fields, abm_slab** out) {
  if (!active || !fields || !out || cap < 1 || cap > (1 << 28) - 1) return ABM_ERR_ARG;
  abm_slab* s = nullptr;
  const abm_status e = slab_alloc(cap, 4, seed, model, active, fields, &s);
  if (e != ABM_OK) return e;
  // zeroed synchronously: a view is made once, outside any stream order
  if (cudaMemset(s->d.counters, 0, sizeof(int32_t) * 4) != cudaSuccess ||
      cudaMemset(s->d.err, 0, sizeof(int)) != cudaSuccess || cudaMemset(s->ctrl, 0, sizeof(u32) * 8) != cudaSuccess) {
    slab_free(s);
    return ABM_ERR_CUDA;
  }
  *out = s;
  return ABM_OK;
}

extern "C" abm_status abm_slab_create(int32_t capacity, int32_t n_fields, uint32_t seed,
                                      uint32_t model, int32_t init, void* stream, abm_slab** out) {
  if (!out || capacity < 1 || capacity > (1 << 28) - 1 || n_fields < 1 || n_fields > kMaxFields ||
      (init != ABM_INIT_EMPTY && init != ABM_INIT_HALF_LIVE))
    return ABM_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  abm_slab* s = nullptr;
  const abm_status e = slab_alloc(capacity, n_fields, seed, model, nullptr, nullptr, &s);
  if (e != ABM_OK) return e;
  if (cudaMemsetAsync(s->d.counters, 0, sizeof(int32_t) * 4, st) != cudaSuccess ||
      cudaMemsetAsync(s->d.err, 0, sizeof(int), st) != cudaSuccess ||
      cudaMemsetAsync(s->ctrl, 0, sizeof(u32) * 8, st) != cudaSuccess) {
    slab_free(s);
    return ABM_ERR_CUDA;
  }
  k_slab_init<<<num_sms() * 4, 256, 0, st>>>(s->d, init, s->n_pad);
  k_count_live<<<num_sms() * 4, 256, 0, st>>>(s->d);
  if (kCheck) k_canary_fill<<<num_sms() * 4, 256, 0, st>>>(s->d.fields, s->d.Fp, s->d.cap, s->n_pad);
  if (cudaGetLastError() != cudaSuccess) {
    slab_free(s);
    return ABM_ERR_CUDA;
  }
  *out = s;
  return ABM_OK;
}

extern "C" abm_status abm_slab_check(abm_slab* s, void* stream) {
  if (!s) return ABM_ERR_ARG;
  // check builds: the padding of a slab's own arrays (a world's view has none of its own)
  if (kCheck && !s->view && s->n_pad > s->d.cap) {
    k_canary_check<<<num_sms() * 4, 256, 0, (cudaStream_t)stream>>>(s->d.active, s->d.fields, s->d.Fp, s->d.cap,
                                                                    s->n_pad, s->d.err);
    ABM_LAUNCH_CHECK();
  }
  ABM_CUDA_TRY(cudaStreamSynchronize((cudaStream_t)stream));
  int err = 0;
  ABM_CUDA_TRY(cudaMemcpy(&err, s->d.err, sizeof(int), cudaMemcpyDeviceToHost));
  return ABM_ERR_OF(err);
}

abm_status abm::slab_canary_fill(int32_t* fields, int Fp, int cap, int n_pad, cudaStream_t st) {
  if (!kCheck || n_pad <= cap) return ABM_OK;
  k_canary_fill<<<num_sms() * 4, 256, 0, st>>>(fields, Fp, cap, n_pad);
  ABM_LAUNCH_CHECK();
  return ABM_OK;
}

abm_status abm::canary_check(const int32_t* active, const int32_t* fields, int Fp, int cap, int n_pad, int* err,
                             cudaStream_t st) {
  if (!kCheck || n_pad <= cap) return ABM_OK;
  k_canary_check<<<num_sms() * 4, 256, 0, st>>>(active, fields, Fp, cap, n_pad, err);
  ABM_LAUNCH_CHECK();
  return ABM_OK;
}

abm_status abm::strided_copy(int32_t* dst, int dst_stride, const int32_t* src, int src_stride, size_t n,
                             cudaStream_t st) {
  if (n == 0) return ABM_OK;
  const size_t per = 256 * kStridedU;
  const int grid = (int)std::min<size_t>((n + per - 1) / per, (size_t)num_sms() * 8);
  k_strided_copy<<<grid, 256, 0, st>>>(dst, dst_stride, src, src_stride, n);
  ABM_LAUNCH_CHECK();
  return ABM_OK;
}

extern "C" abm_status abm_diag_check_index(int64_t i, int64_t n, void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  int* err = nullptr;
  ABM_CUDA_TRY(cudaMalloc(&err, sizeof(int)));
  abm_status rc = ABM_OK;
  int h = 0;
  if (cudaMemsetAsync(err, 0, sizeof(int), st) != cudaSuccess) rc = ABM_ERR_CUDA;
  if (rc == ABM_OK) {
    k_check_index<<<1, 1, 0, st>>>((long long)i, (long long)n, err);
    if (cudaGetLastError() != cudaSuccess ||
        cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
      rc = ABM_ERR_CUDA;
  }
  cudaFree(err);
  return rc != ABM_OK ? rc : ABM_ERR_OF(h);
}

extern "C" abm_status abm_slab_arrays(abm_slab* s, int32_t** active, int32_t** fields, int32_t* stride) {
  if (!s) return ABM_ERR_ARG;
  if (active) *active = s->d.active;
  if (fields) *fields = s->d.fields;
  if (stride) *stride = s->d.Fp;
  return ABM_OK;
}

extern "C" abm_status abm_slab_read(abm_slab* s, int32_t field, int32_t* dst, int32_t n, void* stream) {
  if (!s || !dst || n < 0 || n > s->d.cap || field < -1 || field >= s->d.F) return ABM_ERR_ARG;
  if (n == 0) return ABM_OK;
  cudaStream_t st = (cudaStream_t)stream;
  if (field < 0) {
    ABM_CUDA_TRY(cudaMemcpyAsync(dst, s->d.active, sizeof(int32_t) * (size_t)n, cudaMemcpyDeviceToDevice, st));
  } else {
    return strided_copy(dst, 1, s->d.fields + field, s->d.Fp, (size_t)n, st);
  }
  return ABM_OK;
}

extern "C" abm_status abm_slab_write(abm_slab* s, int32_t field, const int32_t* src, int32_t n, void* stream) {
  if (!s || !src || n < 0 || n > s->d.cap || field < -1 || field >= s->d.F) return ABM_ERR_ARG;
  if (n == 0) return ABM_OK;
  cudaStream_t st = (cudaStream_t)stream;
  if (field < 0) {
    ABM_CUDA_TRY(cudaMemsetAsync(s->d.counters, 0, sizeof(int32_t), st));
    k_write_flags<<<std::max(1, std::min((s->d.cap + 1023) / 1024, num_sms() * 8)), 256, 0, st>>>(s->d, src, n);
    ABM_LAUNCH_CHECK();
  } else {
    return strided_copy(s->d.fields + field, s->d.Fp, src, 1, (size_t)n, st);
  }
  return ABM_OK;
}

static bool pred_ok(const abm_slab* s, const abm_pred* p) {
  if (!p) return false;
  switch (p->kind) {
    case ABM_PRED_LIVE:
    case ABM_PRED_FREE:
    case ABM_PRED_BERNOULLI: return true;
    case ABM_PRED_MASK: return p->mask != nullptr;
    case ABM_PRED_FIELD: return p->field >= 0 && p->field < s->d.F && p->cmp >= 0 && p->cmp <= 3;
  }
  return false;
}

static PredDev to_dev(const abm_pred* p) {
  PredDev d;
  std::memset(&d, 0, sizeof(d));
  if (!p) return d;
  d.kind = p->kind;
  d.threshold = p->threshold;
  d.step = p->step;
  d.purpose = p->purpose;
  d.species = p->species;
  d.mask = p->mask;
  d.field = p->field;
  d.cmp = p->cmp;
  d.and_mask = p->and_mask;
  d.value = p->value;
  return d;
}

// The apply pass runs one wave: as many CTAs as fit on the device at once
// (looked up once per device), each striding over the records.
template <int OP>
static int apply_grid() {
  static std::atomic<int> per_sm[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) dev = -1;
  int b = (dev >= 0 && dev < 64) ? per_sm[dev].load(std::memory_order_relaxed) : 0;
  if (!b) {
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_apply<OP>, 256, 0) != cudaSuccess || b < 1) b = 1;
    if (dev >= 0 && dev < 64) per_sm[dev].store(b, std::memory_order_relaxed);
  }
  return num_sms() * b;
}

// The selective-update call with at least capacity / kLateShare records writes the flags
// of removed slots late. A call pays 1 to 2 us for plane L and saves the writes of the removed
// slots that it refills, all of them once the set is full (after some 3 / p calls). 2^24
// slots, early and late, first calls and full set: p = 0.001 45.5 and 47.5 us, 47.5 and 47.5;
// 0.003 47.5 and 49.1, 52.1 and 50.6; 0.005 49.1 and 50.1, 55.2 and 52.6; 0.01 52.7 and 53.7,
// 61.3 and 57.8.
// The selective-update call with many records, 8 fields and 32-byte aligned records and
// deltas: the ranking pass moves them (four CTAs per SM: two leave the count pass short of
// warps, eight cost a second wave). Lists and an apply pass against moving at once on full
// sets of 2^24 slots: p = 0.01 57.8 us against 67, 0.0157 62 and 62, 0.02 68 and 66, 0.03 79 and
// 76, 0.05 101 and 93, 0.1 145 and 126, 0.3 246 and 192. What is left at p = 0.05 is the draws
// (30 us) and random 32-byte rows, of which DRAM moves 64 bytes each way. While a set fills
// up, the adds that refill no removed slot go to the lowest free ones, to a few CTAs with much
// to do, where an apply pass spreads them. That costs little while these are in the first
// wave of CTAs, and much once they are in the second and run on alone: 2^24 slots at p = 0.03
// after 12, 20 and 60 calls 69, 84 and 90 us moved and 70, 71 and 77 with lists, 0.05 after 3,
// 9 and 20 calls 75, 94 and 102 against 81, 85 and 94 (1.4 times the adds left free from call
// 40 on: 104 and 100), 0.1 after 4, 20 and 60 calls 123, 132 and 126 against 121, 141 and
// 145. Sets of one wave (2^20 slots: 13 to 15 us) never lose. So from kMoveShare on records
// are moved at once unless the last call filled slots of a second wave and left more than 1.5
// times its adds free, from kMoveAlways on always.
constexpr int kMoveShare = 64;
constexpr int kMoveAlways = 12;
constexpr int kLateShare = 256;
constexpr int kMoveCtasPerSm = 4;
static bool fused_moves(const abm_slab* s, const ScanArgs& a) {
  if (s->d.F != 8 || s->d.Fp != 8 || ((((uintptr_t)a.rec) | ((uintptr_t)a.rec2)) & 31) != 0) return false;
  if ((long long)a.k * kMoveAlways >= (long long)s->d.cap) return true;
  return (long long)a.k * kMoveShare >= (long long)s->d.cap && !a.crowded_known;
}

// Where one cluster is faster than the passes, for a call on n slots that moves up to k
// records of F fields (16-byte units where `quads`): its SMs are at most sixteen, and the
// more slots a lane has, the less time is left for records. What a CTA moves at most, in ns,
// against lines drawn from 1 to 16 fields and k from 0.002 to 0.5 n (adds to half-live and
// nearly full sets, updates of the first slots and of slots spread over the set). 131,072 slots, us of the passes and of the cluster: adds of 0.1 n to a
// half-live set, 5 fields 10.5 and 8.3, 11 fields 11.9 and 9.3, of 0.5 n 8 fields 10.9 and
// 9.0, 16 fields 12.4 and 11.4 (its updates 10.7 and 13.1), 11 fields 12.9 and 14.1; 262,144
// slots: adds of 0.03 n 10.7 and 10.3 (1 field), 10.0 and 10.3 (8), 12.2 and 11.0 (11), of
// 0.1 n 10.7 and 12.1 (8; to a nearly full set 10.7 and 8.3), 11.9 and 13.2 (11); the
// selective-update call at p = 0.01 12.4 and 11.7 (8), at 0.03 11.6 and 13.8. Up to 65,536 slots
// the cluster is always faster (11 fields, 0.5 n: 12.6 and 9.0).
// The slots of a lane (4, 8 or 16) of one cluster of at most `most` CTAs, or 0: the passes.
static int small_lanes(int n, long long k, int F, bool quads, bool fused, int most) {
  int lanes = 4;
  while (lanes <= 16 && (long long)n > (long long)most * kSmallThreads * lanes) lanes *= 2;
  if (lanes > 16) return 0;
  if (lanes == 4) return lanes;
  const long long ctas = (n + kSmallThreads * lanes - 1) / (kSmallThreads * lanes);
  const long long ns = std::min<long long>(k, n / 2) / ctas * (18 + (quads ? F : 2 * F)) / 25;
  return ns <= (lanes == 8 ? (fused ? 3700 : 4700) : (fused ? 300 : 1750)) ? lanes : 0;
}

// One cluster of as few CTAs as hold the slots, LS slots per lane.
template <int OP, int LS>
static abm_status launch_small(const ScanArgs& a, cudaStream_t st) {
  static std::atomic<unsigned long long> wide{0};  // devices on which the kernel may use clusters above 8
  const int ctas = (a.n + kSmallThreads * LS - 1) / (kSmallThreads * LS);
  if (ctas > 8) {
    int dev = 0;
    ABM_CUDA_TRY(cudaGetDevice(&dev));
    const unsigned long long bit = (dev >= 0 && dev < 64) ? 1ull << dev : 0ull;
    if (!bit || !(wide.load(std::memory_order_acquire) & bit)) {
      ABM_CUDA_TRY(cudaFuncSetAttribute(k_small<OP, LS>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
      wide.fetch_or(bit, std::memory_order_release);
    }
  }
  ScanArgs b = a;
  b.div1 = (65536u + (u32)a.s.F - 1u) / (u32)a.s.F;
  b.div4 = a.s.F >= 4 ? (65536u + (u32)(a.s.F / 4) - 1u) / (u32)(a.s.F / 4) : 0u;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)ctas);
  cfg.blockDim = dim3(kSmallThreads);
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = (unsigned)ctas;
  at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  ABM_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_small<OP, LS>, b));
  return ABM_OK;
}

// Up to three launches per operation: flags + per-warp / per-CTA counts, then
// ranks + slot lists, then the record moves. Each warp owns one static
// segment of slots in the first two passes; no CTA waits for another.
template <int OP, int THREADS = kSlabThreads>
static abm_status launch_scan(abm_slab* s, const ScanArgs& a, bool aux, cudaStream_t st,
                              int ctas_per_sm = 8) {
  ScanArgs b = a;
  const size_t words = (size_t)(s->n_pad / 32);
  b.planeA = aux ? s->planes2 : s->planes;
  b.planeB = s->planes + words;
  b.planeL = s->planes2;  // (free: only record masks use it, in other calls)
  b.totals = aux ? s->totals2 : s->totals;
  b.wtotals = aux ? s->wtotals2 : s->wtotals;
  b.ctrl = aux ? s->ctrl + 4 : s->ctrl;
  constexpr int SUB = (THREADS / 32) * kWarpStep;  // chunks are whole warp steps
  if (b.n <= 0) {
    if (b.out_count) ABM_CUDA_TRY(cudaMemsetAsync(b.out_count, 0, sizeof(int32_t), st));
    if (OP == OP_ARRAY) ABM_CUDA_TRY(cudaMemsetAsync(s->d.counters + 3, 0, sizeof(int32_t), st));
    return ABM_OK;
  }
  // small sets: one launch (see k_small); few slots per lane while one cluster has the lanes
  constexpr bool MOVES = OP == OP_ADD || OP == OP_UPDATE || OP == OP_FUSED;
  const bool quads = (s->d.F & 3) == 0 && (((uintptr_t)b.rec | (uintptr_t)b.rec2) & 15) == 0;
  if (b.n <= kSmallMax) {
    static std::atomic<int> most[64];
    switch (small_lanes(b.n, MOVES ? b.k : 0, s->d.F, quads, OP == OP_FUSED,
                        std::min(kSmallCtas, cluster_limit(k_small<OP, 16>, kSmallThreads, most)))) {
      case 4: return launch_small<OP, 4>(b, st);
      case 8: return launch_small<OP, 8>(b, st);
      case 16: return launch_small<OP, 16>(b, st);
    }
  }
  const auto chunk_at = [&](int ctas) {
    const int target = std::max(1, std::min(num_sms() * ctas, s->max_ctas));
    const long per = ((long)b.n + target - 1) / target;
    return (int)(((per + SUB - 1) / SUB) * SUB);
  };
  if (OP == OP_FUSED && s->crowded) {
    const long wave = (long)chunk_at(ctas_per_sm ? ctas_per_sm : kMoveCtasPerSm) * num_sms() * move_resident<THREADS>();
    if (wave < b.n) {
      b.wave = (int)wave;
      b.crowded = s->crowded;
      b.crowded_known = *reinterpret_cast<volatile int*>(s->crowded);
    }
  }
  const bool move = OP == OP_FUSED && fused_moves(s, b);
  if (ctas_per_sm == 0) ctas_per_sm = move ? kMoveCtasPerSm : 8;
  b.chunk = chunk_at(ctas_per_sm);
  b.G = (int)(((long)b.n + b.chunk - 1) / b.chunk);
  // the next passes may launch while the previous one drains; they wait on
  // it (griddepcontrol) before reading its results
  if constexpr (OP == OP_FUSED) {
    const bool late = move || (long long)b.k * kLateShare >= (long long)s->d.cap;
    if (late) k_count_fused<THREADS, true><<<b.G, THREADS, 0, st>>>(b);
    else k_count_fused<THREADS, false><<<b.G, THREADS, 0, st>>>(b);
    ABM_LAUNCH_CHECK();
    if (move) {
      ABM_CUDA_TRY(launch_pdl(k_scatter<OP, THREADS, true, true>, b.G, THREADS, st, b));
      return ABM_OK;
    }
    if (late) ABM_CUDA_TRY(launch_pdl(k_scatter<OP, THREADS, false, true>, b.G, THREADS, st, b));
    else ABM_CUDA_TRY(launch_pdl(k_scatter<OP, THREADS>, b.G, THREADS, st, b));
    ABM_CUDA_TRY(launch_pdl(k_apply<OP>, apply_grid<OP>(), 256, st, b));
    return ABM_OK;
  }
  k_count<OP, THREADS><<<b.G, THREADS, 0, st>>>(b);
  ABM_LAUNCH_CHECK();
  if (OP != OP_REMOVE) ABM_CUDA_TRY(launch_pdl(k_scatter<OP, THREADS>, b.G, THREADS, st, b));
  if constexpr (OP == OP_ADD || OP == OP_UPDATE)
    ABM_CUDA_TRY(launch_pdl(k_apply<OP>, apply_grid<OP>(), 256, st, b));
  return ABM_OK;
}

static abm_status launch_fused(abm_slab* s, const ScanArgs& a, cudaStream_t st) {
  const int c = s->fused_ctas_per_sm;
  switch (s->fused_threads) {
    case 128: return launch_scan<OP_FUSED, 128>(s, a, false, st, c);
    case 256: return launch_scan<OP_FUSED, 256>(s, a, false, st, c);
    case 512: return launch_scan<OP_FUSED, 512>(s, a, false, st, c);
  }
  return ABM_ERR_ARG;
}

static ScanArgs base_args(abm_slab* s) {
  ScanArgs a;
  std::memset(&a, 0, sizeof(a));
  a.s = s->d;
  a.n = s->d.cap;
  a.id_field = -1;
  return a;
}

extern "C" abm_status abm_select(abm_slab* s, const abm_pred* pred, int32_t* out_idx, int32_t* out_count,
                                 void* stream) {
  if (!s || !pred_ok(s, pred) || !out_idx || !out_count) return ABM_ERR_ARG;
  ScanArgs a = base_args(s);
  a.pred = to_dev(pred);
  a.list_a = out_idx;
  a.out_count = out_count;
  return launch_scan<OP_SELECT>(s, a, false, (cudaStream_t)stream);
}

extern "C" abm_status abm_select_permutation(abm_slab* s, const abm_pred* pred, int32_t* out_perm,
                                             int32_t* out_count, void* stream) {
  if (!s || !pred_ok(s, pred) || !out_perm || !out_count) return ABM_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  ScanArgs a = base_args(s);
  a.pred = to_dev(pred);
  a.list_a = out_perm;
  a.out_count = out_count;
  abm_status e = launch_scan<OP_SELECT>(s, a, false, st);
  if (e != ABM_OK) return e;
  // the complement, ranked from *out_count on (read on the device by the
  // second compaction, after the first one has finished in stream order)
  ScanArgs b = base_args(s);
  b.pred = to_dev(pred);
  b.negate = 1;
  b.list_a = out_perm;
  b.list_base = out_count;
  b.out_count = s->d.meta + 3;
  return launch_scan<OP_SELECT>(s, b, false, st);
}

extern "C" abm_status abm_remove(abm_slab* s, const abm_pred* pred, int32_t* out_removed, void* stream) {
  if (!s || !pred_ok(s, pred) || pred->kind == ABM_PRED_FREE) return ABM_ERR_ARG;
  ScanArgs a = base_args(s);
  a.pred = to_dev(pred);
  a.out_count = out_removed;
  return launch_scan<OP_REMOVE>(s, a, false, (cudaStream_t)stream);
}

extern "C" abm_status abm_add(abm_slab* s, const int32_t* records, int32_t k, int32_t id_field,
                              int32_t* out_slots, int32_t* out_added, void* stream) {
  if (!s || k < 0 || (k > 0 && !records) || id_field < -1 || id_field >= s->d.F) return ABM_ERR_ARG;
  ScanArgs a = base_args(s);
  a.rec = records;
  a.k = k;
  a.id_field = id_field;
  a.list_a = out_slots ? out_slots : s->lista;
  a.out_count = out_added;
  return launch_scan<OP_ADD>(s, a, false, (cudaStream_t)stream);
}

extern "C" abm_status abm_update_distinct(abm_slab* s, const abm_pred* pred, const int32_t* records,
                                          const int32_t* record_mask, int32_t k, int32_t op,
                                          int32_t* out_slots, int32_t* out_applied, void* stream) {
  if (!s || !pred_ok(s, pred) || k < 0 || (k > 0 && !records) || (op != ABM_OP_ADD && op != ABM_OP_SET))
    return ABM_ERR_ARG;
  if (record_mask && k > s->d.cap) return ABM_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  if (record_mask) {
    ScanArgs r = base_args(s);
    r.n = k;
    r.src = record_mask;
    r.list_a = s->d.rec_idx;
    abm_status e = launch_scan<OP_ARRAY>(s, r, true, st);
    if (e != ABM_OK) return e;
  }
  ScanArgs a = base_args(s);
  a.pred = to_dev(pred);
  a.rec = records;
  a.k = k;
  a.op_kind = op;
  a.use_rec_idx = record_mask != nullptr;
  a.list_a = out_slots ? out_slots : s->lista;
  a.out_count = out_applied;
  return launch_scan<OP_UPDATE>(s, a, false, st);
}

extern "C" abm_status abm_selective_update(abm_slab* s, uint32_t step, uint32_t threshold,
                                           const int32_t* records, const int32_t* deltas, int32_t k,
                                           int32_t* out_counts, void* stream) {
  if (!s || k < 0 || (k > 0 && (!records || !deltas))) return ABM_ERR_ARG;
  ScanArgs a = base_args(s);
  philox_round_keys(s->d.seed, s->d.model, a.rk);
  mask_pair_consts(step, a.rk, a.mk);
  a.rec = records;
  a.rec2 = deltas;
  a.k = k;
  a.step = step;
  a.threshold = threshold;
  a.out_count = out_counts;
  a.list_a = s->lista;
  a.list_b = s->listb;
  return launch_fused(s, a, (cudaStream_t)stream);
}

extern "C" int32_t abm_diag_small_lanes(int32_t n, int32_t k, int32_t n_fields, int32_t quads, int32_t fused,
                                        int32_t most_ctas) {
  return small_lanes(n, k, n_fields, quads != 0, fused != 0, std::min(kSmallCtas, most_ctas));
}

extern "C" abm_status abm_slab_tune(abm_slab* s, int32_t threads, int32_t ctas_per_sm, void* stream) {
  (void)stream;
  if (!s || (threads != 128 && threads != 256 && threads != 512) || ctas_per_sm < 1 || ctas_per_sm > 16 ||
      threads * ctas_per_sm > 2048)
    return ABM_ERR_ARG;
  s->fused_threads = threads;
  s->fused_ctas_per_sm = ctas_per_sm;
  return ABM_OK;
}

extern "C" abm_status abm_philox_records(abm_slab* s, uint32_t step, uint32_t purpose0, uint32_t purpose1,
                                         int32_t k, int32_t* out, void* stream) {
  if (!s || k < 0 || (k > 0 && !out) || s->d.F > 8) return ABM_ERR_ARG;
  if (k == 0) return ABM_OK;
  const int grid = std::min((k + 255) / 256, num_sms() * 8);
  k_philox_records<<<grid, 256, 0, (cudaStream_t)stream>>>(s->d, step, purpose0, purpose1, k, out);
  ABM_LAUNCH_CHECK();
  return ABM_OK;
}

extern "C" abm_status abm_slab_counters_get(abm_slab* s, abm_slab_counters* out, void* stream) {
  if (!s || !out) return ABM_ERR_ARG;
  int32_t c[4];
  ABM_CUDA_TRY(cudaMemcpyAsync(c, s->d.counters, sizeof(c), cudaMemcpyDeviceToHost, (cudaStream_t)stream));
  ABM_CUDA_TRY(cudaStreamSynchronize((cudaStream_t)stream));
  out->n_active = c[0];
  out->next_id = c[1];
  out->overflow = c[2];
  out->reserved = 0;
  return ABM_OK;
}
