// Predation steps of a small world (ABMax Section 5.1) with its whole state in
// one CTA's shared memory: all phases of all requested steps in one launch.
//
// A step is a chain of dependent accesses -- flags, agents, cells, claims,
// ranks -- with a barrier between the phases. For a few hundred agents the
// persistent kernel spends its time in that chain's round trips to L2 and in
// its grid barriers, whatever the number of CTAs (40 x 40 cells: 14.5 us a step
// with 1 to 152 CTAs). Here the chain runs in shared memory and the barrier is
// the CTA's: the same world takes 3.2 us a step. The state is read once
// and written back once per launch.
//
// The phases, their hazards and the results are those of k_persistent
// (pred_persistent.cu): wolf ranks and births run one step late beside the
// sheep phases, on the last warp.
#include <algorithm>

#include "pred_world.cuh"

namespace abm {

constexpr int kRT = 512;              // threads
constexpr int kRWarps = kRT / 32;
constexpr int kRTeam = kRWarps - 1;   // warps of the sheep phases; the last one serves the wolves' ranks and births

// shared-memory layout, in bytes
struct ResidentLayout {
  int regrow, gclaim, victim, wclaim;          // per cell
  int agent[2];                                // int4 per slot
  int live[2], par[2], fre[2], born[2], pre[2]; // one word per 32 slots
  int bytes;
};

static ResidentLayout resident_layout(int ncells, const int (&cap)[2]) {
  ResidentLayout l;
  long long at = 0;
  const auto take = [&](long long n, int align) {
    at = (at + align - 1) / align * align;
    const long long o = at;
    at += n;
    return (int)std::min<long long>(o, 1 << 30);
  };
  for (int s = 0; s < 2; ++s) l.agent[s] = take(16ll * cap[s], 16);
  l.gclaim = take(8ll * ncells, 8);
  l.victim = take(8ll * ncells, 8);
  l.wclaim = take(8ll * ncells, 8);
  l.regrow = take(4ll * ncells, 4);
  for (int s = 0; s < 2; ++s) {
    const long long words = 4ll * ((cap[s] + 31) / 32);
    l.live[s] = take(words, 4);
    l.par[s] = take(words, 4);
    l.fre[s] = take(words, 4);
    l.born[s] = take(words, 4);
    l.pre[s] = take(words, 4);
  }
  l.bytes = (int)std::min<long long>(at, 1 << 30);
  return l;
}

// bookkeeping that no phase reads (kept by thread 0)
struct ResidentBook {
  int nact[2], hw[2], ovf[2];
  int nstart0, r0p, P0p, starved0p, grassp;  // of the previous step's sheep
};

// TWO: the first of a call's two launches (WorldDev::stop_at).
template <bool TWO>
__global__ void __launch_bounds__(kRT, 1) k_resident(WorldDev w, ResidentLayout lay, int nsteps,
                                                     abm_step_stats* stats) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ int s_acc[4];    // starved sheep, starved wolves, eaten, grass eaten
  __shared__ int s_tot[2][2]; // per species: free slots, parents
  int4* const ag[2] = {reinterpret_cast<int4*>(sm + lay.agent[0]), reinterpret_cast<int4*>(sm + lay.agent[1])};
  u64* const gclaim = reinterpret_cast<u64*>(sm + lay.gclaim);
  u64* const victim = reinterpret_cast<u64*>(sm + lay.victim);
  u64* const wclaim = reinterpret_cast<u64*>(sm + lay.wclaim);
  int* const regrow = reinterpret_cast<int*>(sm + lay.regrow);
  const auto words = [&](const int (&off)[2], int s) { return reinterpret_cast<u32*>(sm + off[s]); };
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool last_warp = warp == kRTeam;
  const u32 lt = (1u << lane) - 1u;
  const int L = w.side;
  const bool grass_on = !(w.variant & ABM_VARIANT_GRASS_OFF);
  WorldCtr* const c = w.ctr;
  int t = c->step;
  int ext[2] = {c->extent[0], c->extent[1]};
  int nid[2] = {c->next_id[0], c->next_id[1]};
  ResidentBook bk;
  for (int s = 0; s < 2; ++s) {
    bk.nact[s] = c->n_active[s];
    bk.hw[s] = c->hw[s];
    bk.ovf[s] = c->overflow[s];
  }
  bk.nstart0 = bk.r0p = bk.P0p = bk.starved0p = bk.grassp = 0;
  // ---- the state into shared memory (between launches no cell holds a claim)
  for (int i = tid; i < w.ncells; i += kRT) {
    regrow[i] = w.regrow[i];
    victim[i] = w.victim[i];
    gclaim[i] = kNoKey;
    wclaim[i] = kNoKey;
  }
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const int nw = (w.sp[s].cap + 31) >> 5;
    for (int wd = warp; wd < nw; wd += kRWarps) {
      const int i = 32 * wd + lane;
      const int f = i < ext[s] ? w.sp[s].active[i] : 0;
      if (i < ext[s]) ag[s][i] = w.sp[s].agent[i];
      const u32 m = __ballot_sync(0xFFFFFFFFu, f != 0);
      if (lane == 0) {
        words(lay.live, s)[wd] = m;
        words(lay.born, s)[wd] = 0u;
      }
    }
  }
  if (tid < 4) s_acc[tid] = 0;
  __syncthreads();

  // ranks of species s on one warp: the free and parent counts before each word (16 bits each), and the totals
  auto ranks = [&](int s) {
    const u32 *fre = words(lay.fre, s), *par = words(lay.par, s);
    u32* pre = words(lay.pre, s);
    const int nw = (ext[s] + 31) >> 5;
    u32 carry = 0;
    for (int b = 0; b < nw; b += 32) {
      const int wd = b + lane;
      const u32 v = wd < nw ? ((u32)__popc(fre[wd]) << 16) | (u32)__popc(par[wd]) : 0u;
      u32 inc = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const u32 x = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= o) inc += x;
      }
      if (wd < nw) pre[wd] = carry + inc - v;
      carry += __shfl_sync(0xFFFFFFFFu, inc, 31);
    }
    if (lane == 0) {
      s_tot[s][0] = (int)(carry >> 16);
      s_tot[s][1] = (int)(carry & 0xFFFFu);
    }
  };
  // births of species s by warps w0, w0 + nwarps, ...: the parent of rank i < r fills the free slot of rank i, or the
  // slots past the extent once those are used up
  auto births = [&](int s, int tb, int r, int F, int ext_s, int id0, int w0, int nwarps) {
    const u32 *fre = words(lay.fre, s), *par = words(lay.par, s), *pre = words(lay.pre, s);
    u32 *live = words(lay.live, s), *born = words(lay.born, s);
    const int nw = (ext_s + 31) >> 5;
    for (int wd = w0; wd < nw; wd += nwarps) {
      const u32 pw = par[wd];
      if (!((pw >> lane) & 1u)) continue;
      const int i = (int)(pre[wd] & 0xFFFFu) + __popc(pw & lt);
      if (i >= r) continue;
      int slot;
      if (i < F) {
        int lo = 0, hi = nw - 1;  // the last word with at most i free slots before it
        while (lo < hi) {
          const int mid = (lo + hi + 1) >> 1;
          if ((int)(pre[mid] >> 16) <= i) lo = mid;
          else hi = mid - 1;
        }
        u32 m = fre[lo];
        for (int k = i - (int)(pre[lo] >> 16); k > 0; --k) m &= m - 1;
        slot = 32 * lo + __ffs(m) - 1;
      } else {
        slot = ext_s + (i - F);
      }
      int4 pa = ag[s][32 * wd + lane];
      const int half = pa.y >> 1;
      ag[s][32 * wd + lane].y = pa.y - half;
      ag[s][slot] = make_int4(pa.x, half, (int)((u32)id0 + (u32)i), 0);
      atomicOr(&live[slot >> 5], 1u << (slot & 31));
      atomicOr(&born[slot >> 5], 1u << (slot & 31));
      if (s == 0 && in_range(pa.x, w.ncells, w.err))
        atomicMin(&victim[pa.x], claim_key(draw(w.seed, w.model, (u32)tb, (u32)slot, ABM_P_VICTIM, 0u), slot));
    }
  };
  // move the live agents of species s; claims for the cell's grass (sheep) or the cell's victim (wolves)
  auto move = [&](int s, int w0, int nwarps) {
    const u32* live = words(lay.live, s);
    const int metab = (s == 0 && !grass_on) ? 0 : w.params[PRM_SHEEP_METAB + s];
    const int nw = (ext[s] + 31) >> 5;
    for (int wd = w0; wd < nw; wd += nwarps) {
      if (!((live[wd] >> lane) & 1u)) continue;
      const int slot = 32 * wd + lane;
      int4 a = ag[s][slot];
      if (!in_range(a.x, w.ncells, w.err)) continue;  // check builds: a cell outside the lattice
      // both draws at once: with a few warps per SM, their serial chains are what a phase takes
      const u32 dir = draw(w.seed, w.model, (u32)t, (u32)slot, ABM_P_MOVE, (u32)s) >> 29;
      u32 prio = draw(w.seed, w.model, (u32)t, (u32)slot, ABM_P_PRIO, (u32)s);
      asm volatile("" : "+r"(prio));
      if (s == 0) victim[a.x] = kNoKey;  // last step's victim entry here
      const int cell = step_cell(a.x, L, dir);
      a.x = cell;
      a.y -= metab;
      a.w += 1;
      ag[s][slot] = a;
      if (s == 0 ? (grass_on && regrow[cell] <= t) : victim[cell] != kNoKey)
        atomicMin(&(s == 0 ? gclaim : wclaim)[cell], claim_key(prio, slot));
    }
  };
  // eat if the claim was won, then die or be drawn as a parent; the words of free slots (before the deaths) and parents
  auto count = [&](int s, int w0, int nwarps) {
    u32 *live = words(lay.live, s), *par = words(lay.par, s), *fre = words(lay.fre, s);
    u64* const claim = s == 0 ? gclaim : wclaim;
    const int gain = w.params[s];
    const u32 Tr = (u32)w.params[PRM_SHEEP_T + s];
    const int nw = (ext[s] + 31) >> 5;
    int starved = 0, won = 0;
    for (int wd = w0; wd < nw; wd += nwarps) {
      const u32 lw = live[wd];
      const int slot = 32 * wd + lane;
      bool dead = false, parent = false, ate = false;
      if ((lw >> lane) & 1u) {
        u32 rep = draw(w.seed, w.model, (u32)t, (u32)slot, ABM_P_REPRO, (u32)s);
        u32 vic = s == 0 ? draw(w.seed, w.model, (u32)t, (u32)slot, ABM_P_VICTIM, 0u) : 0u;
        asm volatile("" : "+r"(rep), "+r"(vic));  // both draws at once, as in the move
        const int4 a = ag[s][slot];
        int e = a.y;
        const int cell = a.x;
        if (in_range(cell, w.ncells, w.err)) {
          const u64 cl = claim[cell];
          ate = cl != kNoKey && (u32)cl == (u32)slot;
          if (ate) {
            e += gain;
            ag[s][slot].y = e;
            claim[cell] = kNoKey;
            if (s == 0) {
              regrow[cell] = t + w.params[PRM_REGROWTH];
            } else {
              const u32 v = (u32)victim[cell];
              if (in_range(v, w.sp[0].cap, w.err)) atomicAnd(&words(lay.live, 0)[v >> 5], ~(1u << (v & 31)));
              victim[cell] = kNoKey;
            }
          }
          dead = e < 0;
          if (!dead) {
            parent = rep < Tr;
            if (s == 0) atomicMin(&victim[cell], claim_key(vic, slot));
          }
        }
      }
      const u32 dw = __ballot_sync(0xFFFFFFFFu, dead), pw = __ballot_sync(0xFFFFFFFFu, parent);
      won += __popc(__ballot_sync(0xFFFFFFFFu, ate));
      starved += __popc(dw);
      if (lane == 0) {
        live[wd] = lw & ~dw;
        par[wd] = pw;
        fre[wd] = ~lw & (ext[s] - 32 * wd >= 32 ? 0xFFFFFFFFu : (1u << (ext[s] - 32 * wd)) - 1u);
      }
    }
    if (lane == 0) {
      if (starved) atomicAdd(&s_acc[s], starved);
      if (won) atomicAdd(&s_acc[s == 0 ? 3 : 2], won);
    }
  };
  // the counters after step tw's wolf births (every thread), bookkeeping and that step's statistics (thread 0)
  auto wolf_counters = [&](int tw, abm_step_stats* st, int& r1, int& F1, int& ext1, int& id1) {
    F1 = s_tot[1][0];
    const int P1 = s_tot[1][1];
    const int avail = F1 + (w.sp[1].cap - ext[1]);
    r1 = min(P1, avail);
    ext1 = ext[1];
    id1 = nid[1];
    nid[1] += r1;
    if (r1 > F1) ext[1] += r1 - F1;
    if (tid == 0) {
      const int starved = s_acc[1], eaten = s_acc[2];
      s_acc[1] = s_acc[2] = 0;  // next added to in the wolves' meal phase
      const int n_after = bk.nact[1] + r1;
      if (n_after > bk.hw[1]) bk.hw[1] = n_after;
      bk.nact[1] = n_after - starved;
      if (P1 > avail) bk.ovf[1] = 1;
      bk.nact[0] -= eaten;
      if (st) {
        st->parents[0] = bk.P0p;
        st->parents[1] = P1;
        st->births[0] = bk.r0p;
        st->births[1] = r1;
        st->starved[0] = bk.starved0p;
        st->starved[1] = starved;
        st->eaten = eaten;
        st->grass_eaten = bk.grassp;
        for (int s = 0; s < 2; ++s) {
          st->n_end[s] = bk.nact[s];
          st->hw[s] = bk.hw[s];
          st->overflow[s] = bk.ovf[s];
        }
        st->step = tw;
      }
    }
  };

  int done = TWO ? 0 : nsteps;
  for (int it = 0; it < nsteps; ++it, ++t) {
    if (TWO) {
      if (ext[0] + ext[1] > w.stop_at) break;
      done = it + 1;
    }
    // P1: sheep move | wolf ranks of the previous step
    if (!last_warp) move(0, warp, kRTeam);
    else if (it > 0) ranks(1);
    __syncthreads();
    // P2: sheep eat / select / die | wolf births of the previous step
    int r1 = 0, F1 = 0, ext1 = 0, id1 = 0;
    if (it > 0) wolf_counters(t - 1, stats ? stats + it - 1 : nullptr, r1, F1, ext1, id1);
    if (tid == 0) {
      bk.nstart0 = bk.nact[0];
      if (stats) {
        abm_step_stats* st = stats + it;
        for (int s = 0; s < 2; ++s) {
          st->n_start[s] = bk.nact[s];
          st->extent[s] = ext[s];
        }
      }
    }
    if (!last_warp) count(0, warp, kRTeam);
    else births(1, t - 1, r1, F1, ext1, id1, 0, 1);
    __syncthreads();
    // P3: wolves move + victim claims | sheep ranks
    if (!last_warp) move(1, warp, kRTeam);
    else ranks(0);
    __syncthreads();
    // P4: sheep births
    const int F0 = s_tot[0][0], P0 = s_tot[0][1];
    const int avail0 = F0 + (w.sp[0].cap - ext[0]);
    const int r0 = min(P0, avail0);
    births(0, t, r0, F0, ext[0], nid[0], warp, kRWarps);
    if (tid == 0) {
      const int n_after = bk.nstart0 + r0;
      if (n_after > bk.hw[0]) bk.hw[0] = n_after;
      bk.starved0p = s_acc[0];
      bk.grassp = s_acc[3];
      s_acc[0] = s_acc[3] = 0;  // next added to in the sheep's meal phase
      bk.nact[0] = n_after - bk.starved0p;
      if (P0 > avail0) bk.ovf[0] = 1;
      bk.r0p = r0;
      bk.P0p = P0;
    }
    nid[0] += r0;
    if (r0 > F0) ext[0] += r0 - F0;
    __syncthreads();
    // P5: wolves eat / kill / select / die
    count(1, warp, kRWarps);
    __syncthreads();
  }
  if (done > 0) {  // the last step's wolf ranks and births
    if (warp == 0) ranks(1);
    __syncthreads();
    int r1, F1, ext1, id1;
    wolf_counters(t - 1, stats ? stats + done - 1 : nullptr, r1, F1, ext1, id1);
    births(1, t - 1, r1, F1, ext1, id1, warp, kRWarps);
    __syncthreads();
  }
  // ---- the state back
  for (int i = tid; i < w.ncells; i += kRT) {
    w.regrow[i] = regrow[i];
    w.victim[i] = victim[i];
  }
#pragma unroll
  for (int s = 0; s < 2; ++s)
    for (int i = tid; i < ext[s]; i += kRT) {
      w.sp[s].agent[i] = ag[s][i];
      const u32 bit = 1u << (i & 31);
      // a live flag that was there keeps its value (any nonzero flag is live)
      if (!(words(lay.live, s)[i >> 5] & bit)) w.sp[s].active[i] = 0;
      else if (words(lay.born, s)[i >> 5] & bit) w.sp[s].active[i] = 1;
    }
  if (tid == 0) {
    if (TWO) *w.left = nsteps - done;
    c->step = t;
    for (int s = 0; s < 2; ++s) {
      c->extent[s] = ext[s];
      c->n_active[s] = bk.nact[s];
      c->next_id[s] = nid[s];
      c->hw[s] = bk.hw[s];
      c->overflow[s] = bk.ovf[s];
    }
    note_class(w, ext[0], ext[1]);
  }
}

constexpr int kResidentMaxSmem = 226 * 1024;  // dynamic shared memory (the kernel's static arrays are a few words)

bool resident_fits(const WorldDev& d) {
  if (d.variant & ABM_VARIANT_MANY_WOLVES) return false;  // per-cell lists
  if (d.sp[0].cap > 32767 || d.sp[1].cap > 32767) return false;  // 16-bit ranks
  const int cap[2] = {d.sp[0].cap, d.sp[1].cap};
  return resident_layout(d.ncells, cap).bytes <= kResidentMaxSmem;
}

abm_status launch_resident(const WorldDev& d, int nsteps, abm_step_stats* stats, cudaStream_t st) {
  static std::atomic<unsigned long long> attr[2];
  const int cap[2] = {d.sp[0].cap, d.sp[1].cap};
  const ResidentLayout lay = resident_layout(d.ncells, cap);
  const bool two = d.stop_at != kNoStop;
  const auto kernel = two ? k_resident<true> : k_resident<false>;
  ABM_CUDA_TRY(smem_attr_once(kernel, kResidentMaxSmem, attr[two]));
  kernel<<<1, kRT, (size_t)lay.bytes, st>>>(d, lay, nsteps, stats);
  ABM_LAUNCH_CHECK();
  return ABM_OK;
}

}  // namespace abm
