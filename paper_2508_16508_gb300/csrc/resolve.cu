// Conflict resolution: several agents claim one resource (ABMax Section 1;
// the per-cell priority of Section 5.2). Winner per resource = the claim with
// the smallest packed key (priority << 32 | claim index), i.e. the
// lexicographic minimum of (priority, index). atomicMin on a unique 64-bit
// key is order-independent, so the result is deterministic.
//
// Skewed (Zipf) claim distributions put a large share of the claims on a few
// resources, whose table entries would then serialise the atomics. Each CTA
// therefore keeps the best claim of up to kHash resources in shared memory and
// issues one global atomicMin for each of them at its end; claims on resources
// that found their place taken go to the global table at once.
#include <algorithm>
#include <mutex>

#include "common.cuh"

namespace abm {

constexpr int kResThreads = 1024;
constexpr int kResPerThread = 4;
constexpr int kResChunk = kResThreads * kResPerThread;
constexpr int kHashBits = 13;
constexpr int kHash = 1 << kHashBits;  // 8192 entries x 12 B = 96 KiB of shared memory

__global__ void k_table_fill(u64* table, int R) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < R; i += gridDim.x * blockDim.x) table[i] = kNoKey;
}

// A place of the shared table belongs to the first resource that takes it. A
// chunk of claims goes through two rounds with a barrier after each: take
// places and lower the priorities (32-bit shared atomics, only by claims below the
// priority of the chunks before: an equal one loses to the earlier index); then
// lower the index among the claims that hold a new priority. 4 M Zipf(1.1) claims
// on 262144 resources: 33 us, bound by the scattered global atomics that are
// left (about two million; reading an entry first to spare its atomic costs as
// much as the atomic: 43 us; one CTA per SM with twice the places: 38 us). (Open
// addressing with contended 64-bit shared atomics on packed keys: 39 us, and 147
// instead of 62 us for the whole call where all resources are equally popular. A
// shared filter of seen priorities with every unbeaten claim going to global memory:
// 70 us, the hot entries' first claims serialise in L2.)
//
// A resource that finds its place taken has a second one: with one place, two hot
// resources that share it cost one global atomic per claim on the loser, all on one
// address (4 M claims on two such resources 713 us, now 18). Only a chunk's first
// kResThreads claims take second places, which is enough for a resource that is
// hot: cold ones cost more in the table than as an atomic (all claims taking them:
// 4 M claims on resources of equal popularity 42.9 us against 41.8; one place 41.1).
// A resource's two places; the complement moves resource 0, which every multiplier leaves at 0.
__device__ __forceinline__ int first_place(int r) { return (int)(((u32)r * 2654435761u) >> (32 - kHashBits)); }
__device__ __forceinline__ int second_place(int r) {
  const int h = (int)((~(u32)r * 2246822519u) >> (32 - kHashBits));
  return h == first_place(r) ? h ^ (kHash / 2) : h;
}
// place h, if it is resource r's (it was, or it was free and now is), else -1
__device__ __forceinline__ int take_place(volatile int* s_res, int r, int h) {
  int v = s_res[h];
  if (v == -1) v = atomicCAS(const_cast<int*>(s_res) + h, -1, r);
  return v == r || v == -1 ? h : -1;
}

__global__ void __launch_bounds__(kResThreads, 2) k_claims(const int32_t* __restrict__ res,
                                                           const u32* __restrict__ prio, int M, int R, u64* table) {
  extern __shared__ __align__(16) unsigned char smem[];
  volatile int* s_res = reinterpret_cast<int*>(smem);       // the resource of a place, -1: free
  u32* s_prio = reinterpret_cast<u32*>(smem) + kHash;       // its smallest priority
  u32* s_idx = reinterpret_cast<u32*>(smem) + 2 * kHash;    // and the smallest claim index with it
  for (int h = threadIdx.x; h < kHash; h += kResThreads) {
    s_res[h] = -1;
    s_prio[h] = 0xFFFFFFFFu;
    s_idx[h] = 0xFFFFFFFFu;
  }
  // a contiguous run of claims per CTA, in chunks of kResChunk (the last one ragged)
  const long long run = ((long long)M + gridDim.x - 1) / gridDim.x;
  const int lo = (int)min((long long)M, run * blockIdx.x), hi = (int)min((long long)M, run * (blockIdx.x + 1));
  __syncthreads();
  for (long long m0 = lo; m0 < hi; m0 += kResChunk) {
    int r[kResPerThread];
    u32 p[kResPerThread];
#pragma unroll
    for (int j = 0; j < kResPerThread; ++j) {
      const long long m = m0 + j * kResThreads + threadIdx.x;  // coalesced, all in flight
      r[j] = m < hi ? res[m] : -1;
      p[j] = m < hi ? prio[m] : 0u;
      if (r[j] >= R) r[j] = -1;
    }
    int h[kResPerThread];  // the place of the claim's resource, -1: no claim, none, or already beaten
#pragma unroll
    for (int j = 0; j < kResPerThread; ++j) {
      h[j] = -1;
      if (r[j] < 0) continue;
      int at = take_place(s_res, r[j], first_place(r[j]));
      if (at < 0) {
        const int h2 = second_place(r[j]);
        at = j == 0 ? take_place(s_res, r[j], h2) : (s_res[h2] == r[j] ? h2 : -1);
      }
      if (at < 0) {
        atomicMin(&table[r[j]], ((u64)p[j] << 32) | ((u32)m0 + j * kResThreads + threadIdx.x));
      } else if (p[j] < *(volatile u32*)&s_prio[at] || *(volatile u32*)&s_idx[at] == 0xFFFFFFFFu) {
        // below every earlier chunk's claim (or none came before, or this chunk is lowering the entry already). The
        // index of the priority that no longer counts goes first, so that whoever sees a priority of this chunk sees
        // that too and stays in
        *(volatile u32*)&s_idx[at] = 0xFFFFFFFFu;
        __threadfence_block();
        atomicMin(&s_prio[at], p[j]);
        h[j] = at;
      }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kResPerThread; ++j) {
      if (h[j] < 0) continue;
      if (p[j] == *(volatile u32*)&s_prio[h[j]]) atomicMin(&s_idx[h[j]], (u32)m0 + j * kResThreads + threadIdx.x);
    }
    __syncthreads();
  }
#pragma unroll 4
  for (int h = threadIdx.x; h < kHash; h += kResThreads) {
    const int r = s_res[h];
    if (r >= 0) atomicMin(&table[r], ((u64)s_prio[h] << 32) | s_idx[h]);
  }
}

// winner per resource, then restore the table to "no claim"
__global__ void k_winners(u64* table, int R, int32_t* winner) {
  griddep_wait();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < R; i += gridDim.x * blockDim.x) {
    const u64 v = table[i];
    winner[i] = v == kNoKey ? -1 : (int32_t)(u32)v;
    if (v != kNoKey) table[i] = kNoKey;
  }
}

__global__ void k_is_winner(const int32_t* __restrict__ res, int M, int R, const int32_t* __restrict__ winner,
                            uint8_t* is_winner) {
  griddep_wait();
  // 4 claims per thread: one 128-bit load of resource ids, one 32-bit store of flags
  const int n4 = M >> 2;
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < n4; q += gridDim.x * blockDim.x) {
    const int4 r = reinterpret_cast<const int4*>(res)[q];
    const int m = q << 2;
    u32 f = 0;
    f |= (u32)(r.x >= 0 && r.x < R && winner[r.x] == m + 0) << 0;
    f |= (u32)(r.y >= 0 && r.y < R && winner[r.y] == m + 1) << 8;
    f |= (u32)(r.z >= 0 && r.z < R && winner[r.z] == m + 2) << 16;
    f |= (u32)(r.w >= 0 && r.w < R && winner[r.w] == m + 3) << 24;
    reinterpret_cast<u32*>(is_winner)[q] = f;
  }
  if (blockIdx.x == 0 && threadIdx.x < (M & 3)) {
    const int m = (n4 << 2) + threadIdx.x;
    const int r = res[m];
    is_winner[m] = (r >= 0 && r < R && winner[r] == m) ? 1 : 0;
  }
}

__global__ void k_is_winner_scalar(const int32_t* __restrict__ res, int M, int R,
                                   const int32_t* __restrict__ winner, uint8_t* is_winner) {
  griddep_wait();
  for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < M; m += gridDim.x * blockDim.x) {
    const int r = res[m];
    is_winner[m] = (r >= 0 && r < R && winner[r] == m) ? 1 : 0;
  }
}

static std::atomic<unsigned long long> g_res_attr{0};  // devices whose k_claims has its smem limit

abm_status resolve_launch(const int32_t* claim_res, const uint32_t* claim_prio, int32_t M, int32_t R,
                          uint64_t* table, int32_t* out_winner, uint8_t* out_is_winner, cudaStream_t st) {
  const size_t smem = (size_t)kHash * 3 * sizeof(u32);
  ABM_CUDA_TRY(smem_attr_once(k_claims, (int)smem, g_res_attr));
  const int sms = num_sms();
  if (M > 0) {
    const int nchunks = (M + kResChunk - 1) / kResChunk;
    const int grid = std::max(1, std::min(nchunks, sms * 2));
    k_claims<<<grid, kResThreads, smem, st>>>(claim_res, claim_prio, M, R, (u64*)table);
    ABM_LAUNCH_CHECK();
  }
  ABM_CUDA_TRY(launch_pdl(k_winners, std::max(1, std::min((R + 255) / 256, sms * 8)), 256, st, (u64*)table, (int)R,
                          out_winner));
  if (out_is_winner && M > 0) {
    if ((((uintptr_t)claim_res) & 15) == 0 && (((uintptr_t)out_is_winner) & 3) == 0) {
      ABM_CUDA_TRY(launch_pdl(k_is_winner, std::max(1, std::min((M / 4 + 255) / 256, sms * 8)), 256, st, claim_res,
                              (int)M, (int)R, (const int32_t*)out_winner, out_is_winner));
    } else {
      ABM_CUDA_TRY(launch_pdl(k_is_winner_scalar, std::max(1, std::min((M + 255) / 256, sms * 8)), 256, st, claim_res,
                              (int)M, (int)R, (const int32_t*)out_winner, out_is_winner));
    }
  }
  return ABM_OK;
}

}  // namespace abm

using namespace abm;

extern "C" abm_status abm_resolve_table_init(uint64_t* table, int32_t R, void* stream) {
  if (!table || R < 1) return ABM_ERR_ARG;
  k_table_fill<<<std::max(1, std::min((R + 255) / 256, num_sms() * 8)), 256, 0, (cudaStream_t)stream>>>(
      (u64*)table, R);
  ABM_LAUNCH_CHECK();
  return ABM_OK;
}

extern "C" abm_status abm_resolve(const int32_t* claim_res, const uint32_t* claim_prio, int32_t M, int32_t R,
                                  uint64_t* table, int32_t* out_winner, uint8_t* out_is_winner, void* stream) {
  if (M < 0 || R < 1 || !table || !out_winner || (M > 0 && (!claim_res || !claim_prio))) return ABM_ERR_ARG;
  return resolve_launch(claim_res, claim_prio, M, R, table, out_winner, out_is_winner, (cudaStream_t)stream);
}

// ----------------------------------------------------------------------------
// Resolve without allocation: the scratch table lives in a fixed-size
// file-scope device array instead of caller- or library-allocated memory.
namespace abm {

static __device__ __align__(256) unsigned long long g_resolve_scratch[ABM_RESOLVE_STATIC_MAX_R];

constexpr int kMaxDevices = 64;
static std::mutex g_scratch_mu;
static u64* g_scratch_ptr[kMaxDevices] = {};

// Device address of this device's copy of the array, looked up once per
// device (the array's name is only a host-side handle in host code).
static abm_status static_scratch(u64** out) {
  int dev = 0;
  ABM_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return ABM_ERR_ARG;
  std::lock_guard<std::mutex> lock(g_scratch_mu);
  if (!g_scratch_ptr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_resolve_scratch) != cudaSuccess || !p) return ABM_ERR_CUDA;
    g_scratch_ptr[dev] = (u64*)p;
  }
  *out = g_scratch_ptr[dev];
  return ABM_OK;
}

}  // namespace abm

extern "C" abm_status abm_resolve_static(const int32_t* claim_res, const uint32_t* claim_prio, int32_t M, int32_t R,
                                         int32_t* out_winner, uint8_t* out_is_winner, void* stream) {
  if (M < 0 || R < 1 || !out_winner || (M > 0 && (!claim_res || !claim_prio))) return ABM_ERR_ARG;
  if (R > ABM_RESOLVE_STATIC_MAX_R) return ABM_ERR_TOO_LARGE;
  u64* table = nullptr;
  abm_status e = static_scratch(&table);
  if (e != ABM_OK) return e;
  cudaStream_t st = (cudaStream_t)stream;
  // the array keeps whatever the previous call left: empty the R entries used here
  k_table_fill<<<std::max(1, std::min((R + 255) / 256, num_sms() * 8)), 256, 0, st>>>(table, R);
  ABM_LAUNCH_CHECK();
  return resolve_launch(claim_res, claim_prio, M, R, (uint64_t*)table, out_winner, out_is_winner, st);
}
