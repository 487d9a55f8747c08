// k_complete.cu — the completion list of a commit (Section 4.2: a parent's
// Reduce fires once every member outcome is resolved).
//
// commit_list  runs after a commit's scatter (and its fix-up), one pass over
//              the commit's completion bitmap in tiles of up to CL_WORDS
//              words (32 parents per word).  Per tile it lists the parents this
//              commit completed, takes each one's members to gather (the
//              parent's size from the offsets, or 0 when its counter records
//              a Failed or Suppressed member: it is then Suppressed), scans
//              them with one decoupled look-back over (parents | members <<
//              32) and writes the list in ascending parent order: parent,
//              outcome, member base, first child and the member-tile table.
// The list's copy plan follows on the same stream, from asm_members
// (k_assemble.cu), spread over tiles of AM_TILE members whatever parents they
// belong to.  One kernel for both, a tile's members walked by the CTA that
// held its parents, left the chip idle wherever few tiles held the members:
// 65 us for 11,781 members of 1,000 parents (one CTA), 106 us per wave of
// 50,000 parents (7 CTAs), 4.9 ms for parents of 100,000 members each.
#include <algorithm>

#include "ro_internal.h"

namespace ro {

namespace {

struct ClShared {
  uint32_t scan[33];
  uint16_t par[CL_PARENTS];   // the tile's completed parents, relative to its first
  uint32_t mb[CL_CAP + 1];    // a group's members, then their group-local bases (+ the total)
  unsigned long long prefix;
  uint32_t tile;
};

// Members to gather (0 for a parent with a Failed or Suppressed member) of the
// completed parents at local list positions [g0, g1), into sh.mb as bases
// within the group.  Returns their sum.
__device__ __forceinline__ uint32_t stage_members(const CommitArgs& a, ClShared& sh, uint64_t p0, uint32_t g0,
                                                  uint32_t g1) {
  for (uint32_t k0 = g0 + threadIdx.x; k0 < g1; k0 += CL_GROUP * CL_THREADS) {
    unsigned long long v[CL_GROUP];
    uint64_t o0[CL_GROUP], o1[CL_GROUP];
#pragma unroll
    for (int u = 0; u < CL_GROUP; ++u) {
      const uint32_t q = k0 + u * CL_THREADS;
      if (q >= g1) continue;
      const uint64_t p = p0 + sh.par[q];
      v[u] = __ldcg(a.pw + p);
      o0[u] = __ldg(a.offsets + p);
      o1[u] = __ldg(a.offsets + p + 1);
    }
#pragma unroll
    for (int u = 0; u < CL_GROUP; ++u) {
      const uint32_t q = k0 + u * CL_THREADS;
      if (q < g1) sh.mb[q - g0] = pw_bad(v[u]) ? 0u : (uint32_t)(o1[u] - o0[u]);
    }
  }
  __syncthreads();
  const uint32_t cnt = g1 - g0, per = (cnt + CL_THREADS - 1) / CL_THREADS;
  const uint32_t ka = min(threadIdx.x * per, cnt), kb = min(ka + per, cnt);
  uint32_t mine = 0;
  for (uint32_t q = ka; q < kb; ++q) mine += sh.mb[q];
  uint32_t total;
  uint32_t run = block_excl_scan(mine, sh.scan, &total);
  for (uint32_t q = ka; q < kb; ++q) {
    const uint32_t m = sh.mb[q];
    sh.mb[q] = run;
    run += m;
  }
  if (threadIdx.x == 0) sh.mb[cnt] = total;
  __syncthreads();
  return total;
}

}  // namespace

// Bound by its chain of dependent loads (bitmap word, counter and offsets,
// look-back); each step is spread over the CTA, its loads CL_GROUP at a time.
// 33 KB of shared memory and 56 registers, so that a CTA fits beside two
// asm_copy CTAs on one SM.  A tile with more than CL_CAP completed parents
// takes them in groups, reading their counters again (from L2) to place them.
__global__ void __maxnreg__(CL_MAXREG) commit_list_kernel(CommitArgs a) {
  wait_predecessor();   // (asm_members, its successor, launches after it: early, its CTAs would hold the scatters' room)
  __shared__ ClShared sh;
  DevScalars* ds = a.ds;
  const ListBufs& L = a.list;
  const uint64_t n_words = ceil_div(a.P, 32);
  const uint64_t n_tiles = ceil_div(n_words, (uint64_t)a.list_words);
  if (n_tiles == 0) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      ds->cm_n_done[a.pslot] = 0;
      L.hdr->n = 0;
      L.hdr->M = 0;
      L.hdr->err = 0u;
      L.hdr->incomplete = 0;
      L.mb[0] = 0;
      a.plan.hdr->err = 0u;
      a.plan.hdr->max_end = 0;
      if (a.n_done_out) *a.n_done_out = 0;
    }
    return;
  }
  const uint32_t n_part = participants(n_tiles);
  if (blockIdx.x >= n_part) return;
  const int slot = commit_slot(a.pslot);
  const unsigned long long epoch = ds->epoch[slot];

  for (;;) {
    if (threadIdx.x == 0) sh.tile = claim_tile(&ds->tile_ctr[slot]);
    __syncthreads();
    const uint32_t tile = sh.tile;
    if (tile >= n_tiles) break;
    const uint64_t w = (uint64_t)tile * a.list_words + threadIdx.x;
    const uint64_t p0 = (uint64_t)tile * a.list_words * 32;
    uint32_t bits = 0;
    if (threadIdx.x < a.list_words && w < n_words) {
      bits = __ldcg(a.bitmap + w);
      if (bits) a.bitmap[w] = 0u;   // the bitmap slot is clean for its next commit
    }
    uint32_t Pt;
    uint32_t k = block_excl_scan((uint32_t)__popc(bits), sh.scan, &Pt);
    for (; bits; bits &= bits - 1) sh.par[k++] = (uint16_t)(threadIdx.x * 32 + (__ffs(bits) - 1));
    __syncthreads();
    uint64_t Mt = 0;
    for (uint32_t g0 = 0; g0 < Pt; g0 += CL_CAP) Mt += stage_members(a, sh, p0, g0, min(Pt, g0 + CL_CAP));
    if (threadIdx.x < 32) {   // one warp looks back
      const unsigned long long local = (unsigned long long)Pt | (Mt << 32);
      const unsigned long long pfx = lookback_exclusive(a.ts_list, tile, local, epoch, &ds->err);
      if (threadIdx.x == 0) {
        sh.prefix = pfx;
        if (tile == n_tiles - 1) {   // the whole commit's totals
          const unsigned long long all = pfx + local;
          const uint64_t n = all & 0xFFFFFFFFull, M = all >> 32;
          ds->cm_n_done[a.pslot] = n;
          L.hdr->n = n;
          L.hdr->M = M;
          L.hdr->err = 0u;
          L.hdr->incomplete = 0;
          L.mb[n] = (uint32_t)M;
          a.plan.hdr->err = 0u;
          a.plan.hdr->max_end = 0;   // asm_members raises it
          if (a.n_done_out) *a.n_done_out = n;
        }
      }
    }
    __syncthreads();
    uint64_t gp = sh.prefix & 0xFFFFFFFFull, gm = sh.prefix >> 32;
    for (uint32_t g0 = 0; g0 < Pt; g0 += CL_CAP) {
      const uint32_t g1 = min(Pt, g0 + CL_CAP), cnt = g1 - g0;
      if (Pt > CL_CAP) stage_members(a, sh, p0, g0, g1);
      for (uint32_t q = threadIdx.x; q < cnt; q += CL_THREADS) {
        const uint64_t i = gp + q;
        const uint32_t p = (uint32_t)p0 + sh.par[g0 + q], m = sh.mb[q + 1] - sh.mb[q];
        const uint64_t mbg = gm + sh.mb[q];
        a.done_int[i] = p;
        if (a.done_user) a.done_user[i] = p;
        L.status[i] = m ? ST_PRESENT : ST_SUPPRESSED;
        L.mb[i] = (uint32_t)mbg;
        L.coff[i] = (uint32_t)__ldg(a.offsets + p);
        for (uint64_t t = ceil_div(mbg, AM_TILE); t * AM_TILE < mbg + m && t < L.mtfp_cap; ++t)
          L.mtfp[t] = (uint32_t)i;
      }
      gp += cnt;
      gm += sh.mb[cnt];
      __syncthreads();   // the next group restages
    }
  }
  if (threadIdx.x == 0) retire_cta(ds, slot, n_part);
}

// Words per tile: as few as give up to CL_TILES tiles (one look-back step), so
// that a small expansion's parents spread over the SMs and a large one's
// look-back and launches stay short (1M parents, 256 waves: 7.83 ms per pass
// with 122 tiles of 256 words, 8.17 with 245, 8.84 with 489; 400,000 parents,
// 200 waves: 5.43 ms with 98 tiles, 5.37 with 66, 5.30 with 49).
uint32_t commit_list_words(uint64_t P) {
  const uint64_t want = ceil_div(ceil_div(P, 32), CL_TILES);
  return (uint32_t)std::min<uint64_t>(CL_WORDS, std::max<uint64_t>(32, ceil_div(want, 32) * 32));
}

void launch_commit_list(const LaunchCfg& L, const CommitArgs& a) {
  const uint64_t n_tiles = ceil_div(ceil_div(a.P, 32), (uint64_t)a.list_words);
  const int grid = (int)std::max<uint64_t>(1, std::min<uint64_t>(n_tiles, (uint64_t)L.grid_cplan));
  launch_k(L, K_CPLAN, commit_list_kernel, grid, CL_THREADS, 0, a);
}

const void* kernel_ptr_complete() { return (const void*)commit_list_kernel; }

}  // namespace ro
