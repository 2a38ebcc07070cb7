// Device state of one predation world, shared by the per-phase kernels
// (predation.cu) and the persistent step kernel (pred_persistent.cu).
#pragma once

#include "pred_rules.cuh"

namespace abm {

constexpr int kPredThreads = 256;
constexpr int kPredItems = 4;  // one 128-bit load of live flags per thread
constexpr int kPredTile = kPredThreads * kPredItems;

struct SpeciesDev {
  int32_t* active;   // [cap_pad]
  int4* agent;       // [cap_pad]: cell, energy, id, age
  int32_t* parents;  // [cap] compacted parent slots
  int32_t* freel;    // [cap] compacted free slots (only the first n_active are written)
  u64* tiles;        // decoupled look-back states
  u32* ctrl;         // [0..4) scan control, [4..8) births exit counter
  int cap;
};

struct WorldCtr {
  int n_active[2], next_id[2], hw[2], overflow[2], extent[2], step;
  int parents[2], free_in[2];
  int starved[2], eaten, grass_eaten;
  int n_start[2];
  u32 energy_exit[4];
  long long energy[2];
};

// scratch of the persistent step kernel
struct PersistDev {
  u32* plane[2][2];   // per species: [0] free, [1] parent bit-planes (cap/32 words)
  u64* blk[2];        // per species: (free << 32 | parents) of each 128-slot unit (cap/128)
  u64* seg[2];        // per species: the same summed over each CTA's run of units (max CTAs)
  u32* bar;           // [0] grid-barrier arrivals (monotonic, wraps)
  int* acc;           // [2][4] per-step accumulators by step parity: starved0, starved1, eaten, grass
};

struct WorldDev {
  SpeciesDev sp[2];
  PersistDev ps;
  int32_t* regrow;  // first step at which the cell's grass is edible
  u64* gclaim;      // per-cell grass claims (sheep)
  u64* victim;      // per-cell victim keys (sheep)
  u64* wclaim;      // per-cell wolf claims
  WorldCtr* ctr;
  // size class of the extents, which chooses the launch of the next steps (never the results): pinned host word, set by
  // a launch that ends in another class than the one it was given (class_known), so that other launches write nothing
  int* class_host;
  int class_known, class_small, class_cluster, class_round;
  int* err;
  int side, ncells;
  u32 seed, model;
  u32 bar_base;     // barrier arrivals before this launch (persistent kernel)
  int params[8];
  // ABM_VARIANT_MANY_WOLVES: per-cell lists of this step's live sheep and
  // wolves. Heads reuse `victim` (sheep) and `wclaim` (wolves); a head or link
  // is (step << 32 | slot), so entries of earlier steps end a list and no list
  // is ever cleared. key = the agent's (draw, slot) key.
  int variant;
  u64* skey;        // [cap sheep]
  u64* snext;       // [cap sheep]
  u64* wkey;        // [cap wolves]
  u64* wnext;       // [cap wolves]
  // a call of two launches: the first stops once the extents exceed stop_at slots and leaves the rest of its steps in
  // *left (device), which the second one (follow) runs
  int* left;
  int stop_at, follow;
};

// 0: few enough slots for one CTA's shared memory to be faster; 1: for one cluster to be; 2: the sheep units fit one round
// of one CTA per SM; 3: more
__host__ __device__ inline int extent_class(const WorldDev& w, int ext0, int ext1) {
  if (ext0 + ext1 <= w.class_small) return 0;
  if (ext0 + ext1 <= w.class_cluster) return 1;
  return ext0 <= w.class_round ? 2 : 3;
}
constexpr int kNoStop = 0x7FFFFFFF;
__device__ __forceinline__ void note_class(const WorldDev& w, int ext0, int ext1) {
  const int k = extent_class(w, ext0, ext1);
  if (k != w.class_known) *reinterpret_cast<volatile int*>(w.class_host) = k;
}

// persistent step kernel (pred_persistent.cu)
int persistent_max_ctas();
int persistent_warps();
// whether the one-cluster launch can be placed on the current device
bool persistent_cluster_fits();
// units (128 slots) of a species that one CTA takes in one round of the persistent kernel's sheep phases
int persistent_round_units();
abm_status launch_persistent(const WorldDev& d, u32* bar_next, int grid, bool cluster, int nsteps, abm_step_stats* stats,
                             cudaStream_t st,
                             unsigned long long* phase_ns = nullptr);

// steps of a world whose state fits one CTA's shared memory (pred_resident.cu)
bool resident_fits(const WorldDev& d);
abm_status launch_resident(const WorldDev& d, int nsteps, abm_step_stats* stats, cudaStream_t st);

}  // namespace abm
