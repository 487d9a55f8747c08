// k_commit.cu — ro_gather_commit kernels (Section 4.4, Eq. 3; Section 4.2, Reduce).
//
// commit_scatter  one thread per report.  The fence of Eq. (3) is a single
//                 compare-and-swap of the child's slot from IN-FLIGHT(gen) to
//                 SEALED(gen) that publishes the outcome with it (one sector;
//                 with several Calls, of its phase word, the outcome after
//                 it); the winner counts the member down at its parent with
//                 one 64-bit atomic add on (remaining | bad << 32).  Lanes of a
//                 warp that hit
//                 the same parent are merged first (__match_any_sync), so a
//                 hot parent sees one atomic per warp.  Members of heavy
//                 parents (>= HEAVY_CHILDREN children, whose reports seldom
//                 share a warp) are first summed per CTA in a shared-memory
//                 table and added to the parent once per CTA.  The add that
//                 takes `remaining` to zero completes the parent and sets its
//                 bit in a completion bitmap (the counter's high half then
//                 tells whether a member Failed or was Suppressed).
// commit_fix      after the scatter, on the same stream: when the call
//                 carried two reports for one Grain or a GroupFailure (rare)
//                 the grid orders the repeats and applies the barriers, so the
//                 result equals applying the reports one by one in array
//                 order; otherwise it returns at once.
// The completed list and its copy plan come next, from commit_list
// (k_complete.cu) and asm_members, which may run on another stream while later commits'
// scatters run (commits take completion bitmaps in turn).
#include <algorithm>

#include "ro_internal.h"

namespace ro {

// commit_fix's marks on the reports of a repeated Grain
constexpr uint8_t V_WIN_SEALER = 7, V_WIN_CAND = 8, V_LOSE_SEALER = 9, V_LOSE_CAND = 10, V_SEALER = 11;
// and on an accepted GroupFailure whose barrier is still to seal its siblings
constexpr uint8_t V_SEALS = 12;
// The GroupFailure barrier table: per parent (seq << 32) | ~r, r the lowest
// accepted GroupFailure report of commit seq (atomicMax keeps the lowest r of
// the newest commit); an entry of an older commit means no barrier, so no
// commit clears the table.  (The expansion's scan does, for replays of captured
// commits; a call that orders repeats clears its own GroupFailures' entries.)
__device__ __forceinline__ unsigned long long gb_tag(uint32_t seq, uint32_t r) {
  return ((unsigned long long)seq << 32) | (unsigned long long)(uint32_t)~r;
}
__device__ __forceinline__ bool gb_get(const CommitArgs& a, uint32_t p, uint32_t* r) {
  const unsigned long long v = __ldcg(a.gb + p);
  if ((uint32_t)(v >> 32) != a.seq) return false;
  *r = ~(uint32_t)v;
  return true;
}
__device__ __forceinline__ uint32_t fix_slot(const CommitArgs& a) { return a.seq & 1u; }
__device__ __forceinline__ void stat_add(unsigned long long* s, unsigned long long d) {
  if (d) atomicAdd(s, d);   // d may be a negative delta in two's complement
}


// record word read past L1 (other threads update it with atomics at L2)
__device__ __forceinline__ uint64_t ld_w(const Slot* rc) {
  return __ldcg((const unsigned long long*)&rc->w);
}

__device__ __forceinline__ uint64_t commit_count(const CommitArgs& a) {
  if (!a.d_n) return a.n_host;
  const uint64_t n = *a.d_n;
  return n < a.n_host ? n : a.n_host;
}

__device__ void seal_parents(const CommitArgs& a, bool mine, uint32_t p, int lane, unsigned long long* n_wait,
                             unsigned long long* n_fly);

#ifndef RO_CM_GROUPS
#define RO_CM_GROUPS 1
#endif
constexpr int CM_GROUPS = RO_CM_GROUPS;   // groups of 32 reports a warp has in flight per step (2 and 4 measured slower)

// Warm L2 with the lines of this warp's first CM_GROUPS groups of 32 reports while the previous
// kernel drains (addresses inside the report arrays' host-given length; L2 is
// coherent, so nothing read later can be stale).
__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}
__device__ __forceinline__ void prefetch_reports(const CommitArgs& a) {
  const int lane = threadIdx.x & 31;
  if (lane >= 6 * CM_GROUPS) return;
  const uint64_t n_warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  const uint64_t w = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint64_t r0 = (w + (uint64_t)(lane / 6) * n_warps) * 32;   // this lane's group
  if (r0 >= a.n_host) return;
  switch (lane % 6) {
    case 0: prefetch_l2(a.child + r0); break;
    case 1: prefetch_l2(a.len + r0); break;
    case 2: prefetch_l2(a.off + r0); break;
    case 3: if (r0 + 16 < a.n_host) prefetch_l2(a.off + r0 + 16); break;
    case 4: prefetch_l2(a.state + r0); break;
    default: if (a.gen) prefetch_l2(a.gen + r0); break;
  }
}

// 16-byte compare-and-swap of a slot (phase word, length and w at once).
__device__ __forceinline__ ulonglong2 cas_slot(Slot* p, ulonglong2 want, ulonglong2 put) {
  ulonglong2 old;
  asm volatile(
      "{\n .reg .b128 w, q, o;\n mov.b128 w, {%2, %3};\n mov.b128 q, {%4, %5};\n"
      " atom.relaxed.gpu.global.cas.b128 o, [%6], w, q;\n mov.b128 {%0, %1}, o;\n}"
      : "=l"(old.x), "=l"(old.y)
      : "l"(want.x), "l"(want.y), "l"(put.x), "l"(put.y), "l"(p)
      : "memory");
  return old;
}

// Per-CTA table of heavy parents' member counts (open addressing on the
// parent id): value = bad members << 32 | members, added to the parent's
// counter (as bad << 32 - members) when the CTA is done.
constexpr int HT_SIZE = 2048;
constexpr int HT_PROBES = 32;
constexpr uint32_t HT_EMPTY = 0xFFFFFFFFu;   // no parent has this id (P < 2^32)
struct HeavyTable {
  uint32_t key[HT_SIZE];
  unsigned long long val[HT_SIZE];
};
size_t commit_scatter_smem(int heavy) { return heavy ? sizeof(HeavyTable) : 0; }

// Count n_tot members (n_bad of them Failed or Suppressed) down at parent p;
// the add that takes `remaining` to zero completes the parent.
__device__ __forceinline__ void count_down(const CommitArgs& a, uint32_t p, uint32_t n_tot, uint32_t n_bad) {
  const unsigned long long delta = ((unsigned long long)n_bad << 32) - (unsigned long long)n_tot;
  const unsigned long long old = atomicAdd(a.pw + p, delta);
  if ((uint32_t)old == n_tot)   // the last members: the parent is complete
    atomicOr(a.bitmap + (p >> 5), 1u << (p & 31));
}

// Add to heavy parent p's entry of the CTA's table; false when no entry was
// found within HT_PROBES slots (the caller counts down directly).
__device__ __forceinline__ bool table_add(HeavyTable* t, uint32_t p, unsigned long long v) {
  uint32_t h = (p * 2654435761u) >> (32 - 11);   // HT_SIZE = 2^11
  for (int i = 0; i < HT_PROBES; ++i) {
    const uint32_t k = atomicCAS(&t->key[h], HT_EMPTY, p);
    if (k == HT_EMPTY || k == p) {
      atomicAdd(&t->val[h], v);
      return true;
    }
    h = (h + 1) & (HT_SIZE - 1);
  }
  return false;
}

// Bound by random accesses to the slots (one per report, a DRAM line each once
// they outgrow L2) and, for small commits, by the chain report -> slot and
// parent -> parent counter.  ONE: in a context with one Call an in-flight
// slot's 16 bytes are known, so the fence and the publish are one 16-byte
// compare-and-swap: 110M reports 8.4 -> 5.3 ms against the CAS of the phase
// word with a store of the length and an OR of w after it, a pass of 256
// commits of 64,000 reports 7.87 -> 7.63 ms.  With several Calls the slot's
// Call is not known, a second transaction would wait for the first, and the
// three separate ones stay (50,000 reports of 4 Calls per commit: a pass of 200
// takes 5.28 ms so, 5.37 with the Call guessed, 5.40 with it loaded first).
// At most 56 registers: a CTA (256 threads) fits beside two copy CTAs.
template <bool ONE>
__global__ void __maxnreg__(56) commit_scatter_kernel(CommitArgs a) {
  prefetch_reports(a);
  wait_predecessor();
  allow_successor();
  extern __shared__ __align__(16) unsigned char cm_smem[];
  HeavyTable* ht = reinterpret_cast<HeavyTable*>(cm_smem);
  if (a.heavy)
    for (int i = threadIdx.x; i < HT_SIZE; i += blockDim.x) {
      ht->key[i] = HT_EMPTY;
      ht->val[i] = 0ull;
    }
  // verdict counts: accept, invalid, not in flight, stale, -, barrier,
  // duplicate candidates, accepted GroupFailures
  __shared__ unsigned long long s_cnt[8];
  DevScalars* ds = a.ds;
  if (threadIdx.x < 8) s_cnt[threadIdx.x] = 0;
  __syncthreads();
  const uint64_t n = commit_count(a);
  if (a.d_n && *a.d_n > a.n_host && blockIdx.x == 0 && threadIdx.x == 0)
    atomicOr(&ds->err, ERR_INVAL);
  if (blockIdx.x == 0 && threadIdx.x == 0) {   // the next commit's slot (its last reader is done)
    ds->cm_conflicts[fix_slot(a) ^ 1u] = 0ull;
    ds->cm_gf[fix_slot(a) ^ 1u] = 0ull;
  }
  const int lane = threadIdx.x & 31;
  const uint64_t warp_global = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint64_t n_warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  uint32_t cnt[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  // Each warp takes CM_GROUPS groups of 32 reports per step (group q at
  // base + q * stride): their loads, parents and fence CASes are all in flight
  // before the first verdict is used.
  const uint64_t stride = n_warps * 32;
  for (uint64_t base = warp_global * 32; base < n; base += CM_GROUPS * stride) {
    uint64_t c[CM_GROUPS], o[CM_GROUPS];
    uint64_t curw[CM_GROUPS], putp[CM_GROUPS];
    uint32_t lenp[CM_GROUPS];
    uint32_t l[CM_GROUPS], g[CM_GROUPS], par[CM_GROUPS], cur[CM_GROUPS];
    uint8_t st[CM_GROUPS], v[CM_GROUPS];
    bool heavy[CM_GROUPS], won[CM_GROUPS];
#pragma unroll
    for (int q = 0; q < CM_GROUPS; ++q) {
      const uint64_t r = base + q * stride + lane;
      v[q] = 255;   // inactive lane
      if (r < n) {
        c[q] = a.child[r];
        st[q] = a.state[r];
        l[q] = a.len[r];
        o[q] = a.off[r];
        g[q] = a.gen ? a.gen[r] : 0u;
      }
    }
#pragma unroll
    for (int q = 0; q < CM_GROUPS; ++q) {
      const uint64_t r = base + q * stride + lane;
      heavy[q] = won[q] = false;
      par[q] = cur[q] = 0u;
      curw[q] = 0ull;
      if (r >= n) continue;
      const uint8_t s = st[q];
      const bool valid_state = s >= ST_PRESENT && s <= ST_GROUP_FAILURE;
      const bool in_bounds =
          s != ST_PRESENT || (o[q] <= a.arena_bytes && (uint64_t)l[q] <= a.arena_bytes - o[q]);
      if (c[q] >= a.N || !valid_state || !in_bounds) {
        v[q] = V_INVALID;
        continue;
      }
      v[q] = 254;   // decided below
      // the parent, immutable.  A fill tile of FILL_TILE children that
      // starts with the same parent as the next one is one heavy parent's
      // (it has more than HEAVY_CHILDREN children): the small fill-tile
      // table, resident in L2, names it, and the report touches no sector
      // but its slot's.  Otherwise it is read alongside the fence.
      const uint64_t t = c[q] / FILL_TILE;
      if (a.heavy && t + 1 < a.n_fill_tiles) {
        const uint32_t f0 = __ldg(a.tfp + t), f1 = __ldg(a.tfp + t + 1);
        heavy[q] = f0 == f1;
        par[q] = heavy[q] ? f0 : a.par[c[q]];
      } else {
        par[q] = a.par[c[q]];
      }
      // Eq. (3): accept iff IN-FLIGHT at the report's generation
      const uint32_t want = ph_make(PH_INFLIGHT, g[q]);
      Slot* rc = a.slot + c[q];
      if (g[q] >> 30) {   // no Grain ever reaches such a generation
        const ulonglong2 v = __ldcg(reinterpret_cast<const ulonglong2*>(rc));
        cur[q] = (uint32_t)v.x;
        curw[q] = v.y;
      } else {
        const bool present = s == ST_PRESENT;
        const uint8_t outcome = (s == ST_GROUP_FAILURE) ? ST_FAILED : s;   // its own Grain failed
        const uint32_t len = present ? l[q] : 0u, sealed = ph_make(PH_SEALED, g[q]);
        const uint64_t put = (present ? (o[q] & W_OFF_MASK) : 0ull) | ((uint64_t)outcome << W_STATE_SHIFT);
        if (ONE) {
          ulonglong2 exp = make_ulonglong2(want, 0ull), old;
          for (;;) {
            old = cas_slot(rc, exp, make_ulonglong2(((uint64_t)len << 32) | sealed, put | (exp.y & W_CALL_MASK)));
            won[q] = old.x == exp.x && old.y == exp.y;
            if (won[q] || (uint32_t)old.x != want) break;   // done, or not in flight at this generation
            exp = old;   // (a Call other than 0)
          }
          cur[q] = (uint32_t)old.x;
          curw[q] = old.y;
        } else {
          cur[q] = atomicCAS(&rc->phase, want, sealed);
          won[q] = cur[q] == want;
          lenp[q] = len;
          putp[q] = put;
        }
      }
    }
#pragma unroll
    for (int q = 0; q < CM_GROUPS; ++q) {
      const uint64_t r = base + q * stride + lane;
      uint32_t p = 0;
      bool bad = false;
      if (v[q] == 254) {
        const uint8_t s = st[q];
        if (won[q]) {
          v[q] = V_ACCEPT;
          if (!ONE) {
            Slot* rc = a.slot + c[q];
            rc->len = lenp[q];
            atomicOr((unsigned long long*)&rc->w, (unsigned long long)putp[q]);
          }
          p = par[q];
          bad = (s == ST_FAILED || s == ST_SUPPRESSED || s == ST_GROUP_FAILURE);
          if (s == ST_GROUP_FAILURE) atomicMax(a.gb + p, gb_tag(a.seq, (uint32_t)r));   // barrier
        } else if ((cur[q] & 3u) == PH_WAITING || (cur[q] & 3u) == PH_READY) {
          v[q] = V_NOT_INFLIGHT;
        } else if ((cur[q] >> 2) != g[q]) {
          v[q] = V_STALE;
        } else if ((ONE ? curw[q] : ld_w(a.slot + c[q])) & W_BARRIER_BIT) {
          v[q] = V_BARRIER;   // suppressed by a sibling's GroupFailure in an earlier call
        } else {
          // SEALED at this generation: a duplicate, possibly of a report of
          // this same call with a higher index (ordered by commit_fix)
          v[q] = V_DUP_CANDIDATE;
          atomicOr((unsigned long long*)&a.slot[c[q]].w, (unsigned long long)W_CONFLICT_BIT);
        }
      }
      if (r < n) a.code[r] = v[q];
      // merge the accepted lanes of this warp by parent, one atomic per parent
      const unsigned acc = __ballot_sync(0xffffffffu, v[q] == V_ACCEPT);
      const unsigned badm = __ballot_sync(0xffffffffu, v[q] == V_ACCEPT && bad);
      if (v[q] == V_ACCEPT) {
        const unsigned grp = __match_any_sync(acc, p);
        if (lane == __ffs(grp) - 1) {
          const unsigned n_tot = __popc(grp), n_bad = __popc(grp & badm);
          if (!(heavy[q] && table_add(ht, p, ((unsigned long long)n_bad << 32) | n_tot)))
            count_down(a, p, n_tot, n_bad);
        }
      }
      if (v[q] <= V_DUP_CANDIDATE) cnt[v[q]] += 1;
      // any GroupFailure report (it may still win an ordering of duplicates)
      if (r < n && v[q] != V_INVALID && st[q] == ST_GROUP_FAILURE) cnt[7] += 1;
    }
  }
  // statistics: accepted, invalid, not in flight, stale, barrier (duplicates
  // are counted by the finish pass), candidates for ordering, GroupFailures
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    uint32_t x = cnt[k];
    for (int d = 16; d > 0; d >>= 1) x += __shfl_down_sync(0xffffffffu, x, d);
    if (lane == 0 && x) atomicAdd(&s_cnt[k], (unsigned long long)x);
  }
  __syncthreads();
  if (a.heavy)   // the CTA's heavy-parent counts, one add per parent
    for (int i = threadIdx.x; i < HT_SIZE; i += blockDim.x) {
      const uint32_t p = ht->key[i];
      if (p == HT_EMPTY) continue;
      const unsigned long long v = ht->val[i];
      count_down(a, p, (uint32_t)v, (uint32_t)(v >> 32));
    }
  if (threadIdx.x == 0) {
    for (int k = 0; k < 4; ++k)
      if (s_cnt[k]) atomicAdd(&ds->stats[k], s_cnt[k]);
    if (s_cnt[5]) atomicAdd(&ds->stats[7], s_cnt[5]);
    if (s_cnt[6]) atomicAdd(&ds->cm_conflicts[fix_slot(a)], s_cnt[6]);
    if (s_cnt[7]) atomicAdd(&ds->cm_gf[fix_slot(a)], s_cnt[7]);
  }
}

// A call's barriers, spread over the grid: each CTA takes tiles of FX_TILE
// reports.  A report after its parent's barrier report (table gb) is rejected:
// an accepted one's Grain becomes Suppressed by the barrier, one that met a
// WAITING or READY Grain meets a sealed one (the fence compares generations);
// and the warp holding a barrier's own GroupFailure report seals that parent's
// open siblings (SEAL: here; else the report is marked for a later pass).  The
// two touch disjoint Grains (sealed by this call vs still open), and the
// parent's counters are only added to, so no order between them is needed:
// the result is that of the reports taken in array order.
constexpr uint32_t FX_TILE = 2048;
constexpr int FX_U = 2;   // reports a thread has in flight
template <bool SEAL>
__device__ void apply_barriers_grid(const CommitArgs& a, uint64_t n) {
  DevScalars* ds = a.ds;
  // counter deltas: accepted, not in flight, stale, -, barrier, suppressed while
  // waiting or ready, suppressed while in flight
  __shared__ unsigned long long s_d[7];   // two's complement
  if (threadIdx.x < 7) s_d[threadIdx.x] = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const uint64_t tiles = ceil_div(n, (uint64_t)FX_TILE);
  for (uint64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    for (uint64_t base0 = t * FX_TILE; base0 < (t + 1) * FX_TILE; base0 += (uint64_t)FX_U * blockDim.x) {
      uint8_t vv[FX_U];
      uint32_t cv[FX_U], pv[FX_U];
      unsigned long long gv[FX_U];
#pragma unroll
      for (int u = 0; u < FX_U; ++u) {
        const uint64_t r = base0 + (uint64_t)u * blockDim.x + threadIdx.x;
        vv[u] = r < n ? a.code[r] : V_INVALID;
        cv[u] = r < n ? a.child[r] : 0u;
      }
#pragma unroll
      for (int u = 0; u < FX_U; ++u) pv[u] = vv[u] == V_ACCEPT || vv[u] == V_NOT_INFLIGHT ? a.par[cv[u]] : 0u;
#pragma unroll
      for (int u = 0; u < FX_U; ++u) gv[u] = vv[u] == V_ACCEPT || vv[u] == V_NOT_INFLIGHT ? __ldcg(a.gb + pv[u]) : 0ull;
#pragma unroll
      for (int u = 0; u < FX_U; ++u) {
        const uint64_t r = base0 + (uint64_t)u * blockDim.x + threadIdx.x;
        const uint8_t v = vv[u];
        const uint32_t p = pv[u], b = ~(uint32_t)gv[u];
        const uint64_t c = cv[u];
        const bool barrier = (uint32_t)(gv[u] >> 32) == a.seq;   // (gb_get's test; seq is never 0)
        const bool under = barrier && r > b;
        const bool trig = barrier && r == b;   // the barrier's own (accepted) GroupFailure report
        if (under) {
          if (v == V_ACCEPT) {
            Slot* rc = a.slot + c;
            const uint64_t keep = ld_w(rc) & ~(W_OFF_MASK | W_STATE_MASK);
            rc->len = 0u;
            rc->w = keep | ((uint64_t)ST_SUPPRESSED << W_STATE_SHIFT) | W_BARRIER_BIT;
            const uint8_t st = a.state[r];
            if (!(st == ST_FAILED || st == ST_SUPPRESSED || st == ST_GROUP_FAILURE))
              atomicAdd(a.pw + p, 1ull << 32);   // its outcome class is now bad
            a.code[r] = V_BARRIER;
            atomicAdd(&s_d[0], ~0ull);
            atomicAdd(&s_d[4], 1ull);
            atomicAdd(&s_d[6], 1ull);
          } else {
            const uint32_t ph = __ldcg(&a.slot[c].phase);
            const uint32_t gen_c = ((ph & 3u) == PH_WAITING) ? 0u : (ph >> 2);
            const uint32_t g = a.gen ? a.gen[r] : 0u;
            const bool same = g == gen_c;
            a.code[r] = same ? V_BARRIER : V_STALE;
            atomicAdd(&s_d[1], ~0ull);
            atomicAdd(&s_d[same ? 4 : 2], 1ull);
          }
        }
        if (SEAL)
          seal_parents(a, trig, p, lane, &s_d[5], &s_d[6]);
        else if (trig)
          a.code[r] = V_SEALS;
      }
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    stat_add(&ds->stats[0], s_d[0]);
    stat_add(&ds->stats[2], s_d[1]);
    stat_add(&ds->stats[3], s_d[2]);
    stat_add(&ds->stats[7], s_d[4]);
    stat_add(&ds->stats[8], s_d[5]);
    stat_add(&ds->stats[9], s_d[6]);
  }
}

// A barrier seals every sibling of parent pp that is still open (a whole
// warp, lane = its lane): Suppressed, barrier bit set, counted down at the
// parent; the parent then completes (with a failed member it gathers
// nothing).  Siblings sealed while WAITING or READY and while IN-FLIGHT are
// added to *n_wait and *n_fly (shared counters of the CTA).
__device__ void seal_open(const CommitArgs& a, uint32_t pp, int lane, unsigned long long* n_wait,
                          unsigned long long* n_fly) {
  const uint64_t c0 = a.offsets[pp], c1 = a.offsets[pp + 1];
  uint32_t k_wait = 0, k_fly = 0;
  for (uint64_t d = c0 + lane; d < c1; d += 32) {
    Slot* rc = a.slot + d;
    const uint32_t ph = __ldcg(&rc->phase);
    const uint32_t f = ph & 3u;
    if (f == PH_SEALED) continue;
    const uint32_t gen_d = (f == PH_WAITING) ? 0u : (ph >> 2);
    Slot sl;   // the whole slot in one store
    sl.phase = ph_make(PH_SEALED, gen_d);
    sl.len = 0u;
    sl.w = (ld_w(rc) & ~(W_OFF_MASK | W_STATE_MASK)) | ((uint64_t)ST_SUPPRESSED << W_STATE_SHIFT) |
           W_BARRIER_BIT;
    *rc = sl;
    if (f == PH_INFLIGHT) ++k_fly; else ++k_wait;
  }
  for (int sh = 16; sh > 0; sh >>= 1) {
    k_wait += __shfl_down_sync(0xffffffffu, k_wait, sh);
    k_fly += __shfl_down_sync(0xffffffffu, k_fly, sh);
  }
  if (lane == 0) {
    const unsigned long long k = (unsigned long long)k_wait + k_fly;
    if (k) {
      const unsigned long long old = atomicAdd(a.pw + pp, (k << 32) - k);
      if ((uint32_t)old == k)   // the barrier completes the parent
        atomicOr(a.bitmap + (pp >> 5), 1u << (pp & 31));
    }
    atomicAdd(n_wait, (unsigned long long)k_wait);
    atomicAdd(n_fly, (unsigned long long)k_fly);
  }
  __syncwarp();
}

// The same for the parents p of those lanes of a warp that have one (mine).
__device__ void seal_parents(const CommitArgs& a, bool mine, uint32_t p, int lane, unsigned long long* n_wait,
                             unsigned long long* n_fly) {
  unsigned m = __ballot_sync(0xffffffffu, mine);
  while (m) {
    const int src = __ffs(m) - 1;
    m &= m - 1;
    seal_open(a, __shfl_sync(0xffffffffu, p, src), lane, n_wait, n_fly);
  }
}

// f(r, verdict) for each of the call's reports, over the whole grid (each report
// always by the same thread), FX_U verdicts loaded at a time.
template <class F>
__device__ __forceinline__ void each_report(const CommitArgs& a, uint64_t n, const F& f) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t r0 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; r0 < n; r0 += FX_U * stride) {
    uint8_t v[FX_U];
#pragma unroll
    for (int u = 0; u < FX_U; ++u) v[u] = r0 + u * stride < n ? a.code[r0 + u * stride] : V_INVALID;
#pragma unroll
    for (int u = 0; u < FX_U; ++u)
      if (v[u] != V_INVALID) f(r0 + u * stride, v[u]);
  }
}

// Make the lowest-index report of each Grain that was reported more than once
// in this call the accepted one (the whole grid; sync() is its barrier).  With
// GroupFailures in the call (gfs) the barrier table is rebuilt on the way, from
// the verdicts as they become final (a GroupFailure may lose to an earlier
// report of its Grain): cleared in A, raised in D.
template <class Sync>
__device__ void order_repeats(const CommitArgs& a, uint64_t n, bool gfs, const Sync& sync) {
  DevScalars* ds = a.ds;
  __shared__ unsigned long long s_dups;
  if (threadIdx.x == 0) s_dups = 0;
  __syncthreads();
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  const uint64_t r_first = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  // A: this call's sealer of a conflicted Grain marks itself and opens the
  //    minimum-index election in the record's len field with its own index
  for (uint64_t r0 = r_first; r0 < n; r0 += FX_U * stride) {
    uint8_t v[FX_U], s[FX_U];
    uint32_t c[FX_U];
    uint64_t w[FX_U];
#pragma unroll
    for (int u = 0; u < FX_U; ++u) {
      const uint64_t r = r0 + u * stride;
      v[u] = r < n ? a.code[r] : V_INVALID;
      s[u] = gfs && r < n ? a.state[r] : 0;
      c[u] = r < n ? a.child[r] : 0u;
    }
#pragma unroll
    for (int u = 0; u < FX_U; ++u) w[u] = v[u] == V_ACCEPT ? ld_w(a.slot + c[u]) : 0ull;
#pragma unroll
    for (int u = 0; u < FX_U; ++u) {
      if (s[u] == ST_GROUP_FAILURE && c[u] < a.N) a.gb[a.par[c[u]]] = 0ull;
      if (!(w[u] & W_CONFLICT_BIT)) continue;
      const uint64_t r = r0 + u * stride;
      Slot* rc = a.slot + c[u];
      __stcg(&rc->len, (uint32_t)r);
      atomicOr((unsigned long long*)&rc->w, (unsigned long long)W_SEALER_BIT);
      a.code[r] = V_SEALER;
    }
  }
  sync();
  // B: candidates of Grains sealed in this call vote; the others are plain
  //    duplicates of an earlier call's publication
  each_report(a, n, [&](uint64_t r, uint8_t v) {
    if (v != V_DUP_CANDIDATE) return;
    Slot* rc = a.slot + a.child[r];
    if (ld_w(rc) & W_SEALER_BIT) {
      atomicMin(&rc->len, (uint32_t)r);
    } else {
      a.code[r] = V_DUPLICATE;
      atomicAnd((unsigned long long*)&rc->w, ~(unsigned long long)W_CONFLICT_BIT);
      atomicAdd(&s_dups, 1ull);
    }
  });
  sync();
  // C: every contender learns whether it won
  each_report(a, n, [&](uint64_t r, uint8_t v) {
    if (v != V_SEALER && v != V_DUP_CANDIDATE) return;
    const bool win = __ldcg(&a.slot[a.child[r]].len) == (uint32_t)r;
    a.code[r] = (v == V_SEALER) ? (win ? V_WIN_SEALER : V_LOSE_SEALER) : (win ? V_WIN_CAND : V_LOSE_CAND);
  });
  sync();
  // D: the winner writes the record; outcome classes move with it (a parent's
  //    moves with its counter, where the completion list reads it)
  each_report(a, n, [&](uint64_t r, uint8_t v) {
    const bool win = v == V_WIN_SEALER || v == V_WIN_CAND;
    if (gfs && (v == V_ACCEPT || win) && a.state[r] == ST_GROUP_FAILURE)
      atomicMax(a.gb + a.par[a.child[r]], gb_tag(a.seq, (uint32_t)r));
    if (v < V_WIN_SEALER || v > V_LOSE_CAND) return;
    const uint8_t s = a.state[r];
    const bool bad = (s == ST_FAILED || s == ST_SUPPRESSED || s == ST_GROUP_FAILURE);
    const uint64_t c = a.child[r];
    Slot* rc = a.slot + c;
    const uint32_t p = a.par[c];
    if (win) {
      const bool present = s == ST_PRESENT;
      const uint8_t outcome = (s == ST_GROUP_FAILURE) ? ST_FAILED : s;
      const uint64_t keep = ld_w(rc) & ~(W_OFF_MASK | W_STATE_MASK | W_SEALER_BIT | W_CONFLICT_BIT);
      __stcg(&rc->len, present ? a.len[r] : 0u);
      __stcg((unsigned long long*)&rc->w, (unsigned long long)(keep | (present ? (a.off[r] & W_OFF_MASK) : 0ull) |
                                                               ((uint64_t)outcome << W_STATE_SHIFT)));
      if (v == V_WIN_CAND && bad) atomicAdd(a.pw + p, 1ull << 32);
    } else {
      if (v == V_LOSE_SEALER && bad) atomicAdd(a.pw + p, ~((1ull << 32) - 1));   // -(1 << 32)
      atomicAdd(&s_dups, 1ull);
    }
    a.code[r] = win ? V_ACCEPT : V_DUPLICATE;
  });
  __syncthreads();
  if (threadIdx.x == 0 && s_dups) atomicAdd(&ds->stats[4], s_dups);
}

// The barriers of a call with repeated reports, once these are ordered: first
// the reports that they reject, then the duplicates after a barrier of a Grain
// whose accepted report the barrier rejected, and the siblings still open.  A
// duplicate's Grain was sealed before the barriers, so the last two need no
// order between them, and no grid barrier comes after the sealing: one warp
// seals a parent, and with 10^8 children that takes longer than the grid's
// waits last.
template <class Sync>
__device__ void barriers_after_repeats(const CommitArgs& a, uint64_t n, const Sync& sync) {
  DevScalars* ds = a.ds;
  sync();   // every verdict and barrier is final
  apply_barriers_grid<false>(a, n);
  sync();
  __shared__ unsigned long long s_sealed[2];   // while waiting or ready, while in flight
  if (threadIdx.x < 2) s_sealed[threadIdx.x] = 0;
  __syncthreads();
  uint32_t moved = 0;
  const int lane = threadIdx.x & 31;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t w0 = (uint64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); w0 < n; w0 += FX_U * stride) {   // by warp
    uint8_t v[FX_U];
#pragma unroll
    for (int u = 0; u < FX_U; ++u) v[u] = w0 + u * stride + lane < n ? a.code[w0 + u * stride + lane] : V_INVALID;
#pragma unroll
    for (int u = 0; u < FX_U; ++u) {
      const uint64_t r = w0 + u * stride + lane;
      uint32_t p = 0;
      if (v[u] == V_SEALS) {
        p = a.par[a.child[r]];
        a.code[r] = V_ACCEPT;
      } else if (v[u] == V_DUPLICATE) {
        const uint64_t c = a.child[r];
        uint32_t b;
        // (a Grain without the bit was sealed before the barrier)
        if (gb_get(a, a.par[c], &b) && r > b && (ld_w(a.slot + c) & W_BARRIER_BIT)) {
          a.code[r] = V_BARRIER;
          ++moved;
        }
      }
      seal_parents(a, v[u] == V_SEALS, p, lane, &s_sealed[0], &s_sealed[1]);
    }
  }
  if (moved) {
    atomicAdd(&ds->stats[4], ~(unsigned long long)moved + 1ull);
    atomicAdd(&ds->stats[7], (unsigned long long)moved);
  }
  __syncthreads();
  if (threadIdx.x < 2) stat_add(&ds->stats[8 + threadIdx.x], s_sealed[threadIdx.x]);
}

// After the scatter, on the same stream: reports of one Grain that met in
// this call are ordered and GroupFailure barriers applied, so the next commit
// and the completion list (which may run on another stream) see final
// outcomes.  Returns at once when the scatter saw neither.  Kept out of the
// scatter so that the scatter's registers and shared memory stay small.  The
// launch is cooperative, a CTA per FX_TILE reports, because the ordering's
// steps meet at grid barriers: one CTA took 1.2 ms for 105,000 reports with 2 %
// repeats, bound by one SM's loads in flight; the grid takes 50 us.  Nearly
// every launch returns at once, so its CTAs are few and small: twice the CTAs,
// or 512 threads each, took 10 % off a pass with repeats in every commit but
// added 0.5 to 1 % to passes without, as did 48 registers for four reports a
// thread in flight.
__global__ void __maxnreg__(32) commit_fix_kernel(CommitArgs a) {
  wait_predecessor();
  allow_successor();
  DevScalars* ds = a.ds;
  const unsigned long long dups = ds->cm_conflicts[fix_slot(a)], gfs = ds->cm_gf[fix_slot(a)];
  if (dups == 0ull && gfs == 0ull) return;
  const uint64_t n = commit_count(a);
  if (!dups) {
    apply_barriers_grid<true>(a, n);
    return;
  }
  // the barrier's generation, read before any barrier of this launch can complete
  uint32_t gen = __ldcg(&ds->cm_bar_gen);
  const auto sync = [&]() {
    gen = (gen + 1u) & ~BAR_FLAG;
    grid_barrier(&ds->cm_bar_count, &ds->cm_bar_gen, gen, &ds->err);
  };
  order_repeats(a, n, gfs != 0ull, sync);
  if (gfs) barriers_after_repeats(a, n, sync);
}

void launch_commit_scatter(const LaunchCfg& L, const CommitArgs& a) {
  const uint64_t warps = ceil_div(a.n_host, 32);
  const int grid =
      (int)std::max<uint64_t>(1, std::min<uint64_t>(ceil_div(warps, CM_THREADS / 32),
                                                    (uint64_t)L.grid_commit));
  launch_k(L, K_COMMIT, a.multi_call ? commit_scatter_kernel<false> : commit_scatter_kernel<true>, grid, CM_THREADS,
           commit_scatter_smem(a.heavy), a);
  // the fix returns at once unless the scatter flagged the call
  const int grid_fix = (int)std::max<uint64_t>(
      1, std::min<uint64_t>(ceil_div(a.n_host, (uint64_t)FX_TILE), (uint64_t)L.grid_cfix_coop));
  if (grid_fix == 1)   // (nothing to meet)
    launch_k(L, K_CFIX, commit_fix_kernel, 1, CM_THREADS, 0, a);
  else
    launch_coop(L, K_CFIX, commit_fix_kernel, grid_fix, CM_THREADS, a);
}

const void* kernel_ptr_commit(int which) {
  return which == K_CFIX ? (const void*)commit_fix_kernel : (const void*)commit_scatter_kernel<true>;
}

}  // namespace ro
