// k_assemble.cu — ro_assemble kernels (Section 4.2, Reduce).
//
// A completed parent is Suppressed if a member Failed or was Suppressed,
// otherwise Present with the Present members' payloads concatenated by
// ordinal (Dropped members add nothing).  The work is a segmented byte gather
// from the result arena in three steps:
//   asm_parents  (caller's lists only; commit_list does this for the
//                parents a commit completed) per listed parent: outcome,
//                members to gather (0 unless Present), their exclusive scan
//                (member bases), and for every AM_TILE-member tile the parent
//                holding its first member;
//   asm_members  per member, load-balanced over AM_TILE-member tiles so a
//                100k-member parent spreads over many CTAs: read the record,
//                scan the Present bytes (single-pass look-back) and write the
//                plan — each parent's relative output offset, each
//                contributing member's relative position and arena offset, and
//                for every 16 KB chunk of the output the member holding its
//                first byte;
//   asm_copy     per chunk: two producer warps stage chunks' member pieces
//                in shared memory with cp.async.bulk (a ring of AC_STAGES
//                stages, mbarrier completion, bounded waits) while eight
//                consumer warps turn staged chunks into aligned 16-byte
//                stores; source and destination alignments may differ
//                arbitrarily.
// The plan is independent of where the output starts, so planning (on the
// context's plan stream) can run ahead of the copies (copy stream).
#include <algorithm>

#include "copy_rounds.h"
#include "ro_internal.h"

namespace ro {

constexpr int TS_ASM_COPY = 5;

template <class V>
__device__ __forceinline__ uint32_t last_le_u(const V* v, uint32_t lo, uint32_t hi, uint64_t x) {
  while (hi - lo > 1) {
    const uint32_t mid = lo + ((hi - lo) >> 1);
    if ((uint64_t)v[mid] <= x)
      lo = mid;
    else
      hi = mid;
  }
  return lo;
}

// ---------------------------------------------------------------------------
// asm_parents: a caller's list -> outcomes, member bases, member-tile table.
__global__ void __launch_bounds__(AP_THREADS) asm_parents_kernel(AssembleArgs a) {
  wait_predecessor();
  __shared__ unsigned long long s_scan[33];
  __shared__ uint32_t s_tile;
  __shared__ unsigned long long s_prefix;
  __shared__ unsigned long long s_incomplete;
  DevScalars* ds = a.ds;
  const ListBufs& L = a.list;
  const uint64_t n_req = a.d_n ? *a.d_n : a.n_host;
  if (n_req > a.n_host) {   // a device count beyond the arrays' length
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      L.hdr->err = 1u;
      L.hdr->n = 0;
      atomicOr(&ds->err, ERR_INVAL);
    }
    return;
  }
  const uint64_t n = n_req;
  const uint64_t TILE = (uint64_t)AP_THREADS * AP_ITEMS;
  const uint64_t n_tiles = ceil_div(n, TILE);
  if (n_tiles == 0) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      L.mb[0] = 0;
      L.hdr->n = 0;
      L.hdr->M = 0;
      L.hdr->err = 0u;
    }
    return;
  }
  const uint32_t n_part = participants(n_tiles);
  if (blockIdx.x >= n_part) return;
  if (threadIdx.x == 0) s_incomplete = 0;
  for (;;) {
    if (threadIdx.x == 0) s_tile = claim_tile(&ds->tile_ctr[TS_ASM_PARENTS]);
    __syncthreads();
    const uint32_t tile = s_tile;
    __syncthreads();
    if (tile >= n_tiles) break;
    const uint64_t i0 = tile * TILE + (uint64_t)threadIdx.x * AP_ITEMS;
    uint32_t m[AP_ITEMS], cf[AP_ITEMS];
    unsigned long long mine = 0;
    uint32_t incomplete = 0;
#pragma unroll
    for (int k = 0; k < AP_ITEMS; ++k) {
      const uint64_t i = i0 + k;
      m[k] = 0;
      cf[k] = 0;
      if (i >= n) continue;
      const uint64_t p = L.parents[i];
      uint8_t st = ST_PENDING;
      if (p < a.P) {
        const unsigned long long v = a.pw[p];
        cf[k] = (uint32_t)a.offsets[p];
        if (pw_remaining(v) == 0u) {
          if (pw_bad(v) != 0u) {
            st = ST_SUPPRESSED;
          } else {
            st = ST_PRESENT;
            m[k] = (uint32_t)(a.offsets[p + 1] - a.offsets[p]);
          }
        }
      }
      if (st == ST_PENDING) ++incomplete;
      L.status[i] = st;
      mine += m[k];
    }
    if (incomplete) atomicAdd(&s_incomplete, (unsigned long long)incomplete);
    unsigned long long total;
    unsigned long long excl = block_excl_scan(mine, s_scan, &total);
    if (threadIdx.x < 32) {  // one warp looks back
      const auto pfx = lookback_exclusive(a.ts_parents, tile, total, ds->epoch[TS_ASM_PARENTS], &ds->err);
      if (threadIdx.x == 0) s_prefix = pfx;
    }
    __syncthreads();
    unsigned long long run = s_prefix + excl;
#pragma unroll
    for (int k = 0; k < AP_ITEMS; ++k) {
      const uint64_t i = i0 + k;
      if (i >= n) break;
      L.mb[i] = (uint32_t)run;
      L.coff[i] = cf[k];
      if (m[k]) {
        for (uint64_t b = ceil_div(run, AM_TILE); b * AM_TILE < run + m[k] && b < L.mtfp_cap; ++b)
          L.mtfp[b] = (uint32_t)i;
      }
      run += m[k];
    }
    if (tile == n_tiles - 1 && threadIdx.x == AP_THREADS - 1) {
      L.mb[n] = (uint32_t)run;
      L.hdr->n = n;
      L.hdr->M = run;
      // more members than the plan holds (a parent listed many times)
      L.hdr->err = run > a.plan.member_cap ? 1u : 0u;
      if (run > a.plan.member_cap) atomicOr(&ds->err, ERR_CAPACITY);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    // counted once the assembly succeeds (asm_copy)
    if (s_incomplete) atomicAdd(&L.hdr->incomplete, s_incomplete);
    retire_cta(ds, TS_ASM_PARENTS, n_part);
  }
}

// ---------------------------------------------------------------------------
// asm_members: list -> plan (relative offsets and member positions).  Tiles
// of AM_TILE members, whatever parents they belong to, so its time follows
// the members and not how they fall to parents.  Bound by the latency of a
// tile's steps (claim, list, records, look-back; about 14 us), so by the
// tiles in flight: 48 registers and 25 KB of shared memory let 5 CTAs share
// an SM (a pass of 110M members 12.85 ms; with 56 registers and 4 CTAs 13.1,
// with 40 and 6 12.8, but lists of 60,000 parents 1 % slower alone).
__global__ void __maxnreg__(48) asm_members_kernel(AssembleArgs a) {
  wait_predecessor();
  __shared__ uint32_t s_mb[AM_SMEM_CAP];
  __shared__ uint32_t s_coff[AM_SMEM_CAP];
  __shared__ Pair64 s_scan[33];
  __shared__ uint32_t s_tile;
  __shared__ Pair64 s_prefix;
  __shared__ unsigned long long s_pos[AM_TILE + 1];   // tile-relative position of each member (+ the end)
  __shared__ unsigned long long s_end;
  DevScalars* ds = a.ds;
  const ListBufs& L = a.list;
  const PlanBufs& pl = a.plan;
  const int slot = a.members_slot;
  const ListHdr lh = *L.hdr;
  const uint64_t n = lh.n, M = lh.M;
  // the list's entries must fit the caller's list-structure outputs
  const bool elems_too_many = a.elem_base && M > a.elem_cap;
  if (lh.err || elems_too_many) {   // nothing to plan
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      pl.hdr->n = n;
      pl.hdr->bytes = 0;
      pl.hdr->nnz = 0;
      pl.hdr->M = M;
      pl.hdr->incomplete = 0;
      pl.hdr->max_end = 0;
      pl.hdr->err = 1u;
      L.hdr->incomplete = 0;   // spent (asm_parents adds to it)
      if (elems_too_many) atomicOr(&ds->err, ERR_CAPACITY);
    }
    return;
  }
  const uint64_t n_tiles = ceil_div(M, AM_TILE);
  const uint64_t par_units = ceil_div(n, (uint64_t)AM_TILE);
  const uint32_t n_part = participants((n_tiles > par_units ? n_tiles : par_units) + 1);
  if (blockIdx.x >= n_part) return;
  if (a.elem_base) {   // each listed parent's first list entry (its member base)
    const uint64_t stride = (uint64_t)n_part * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i <= n; i += stride)
      a.elem_base[i] = L.mb[i];
  }

  if (M == 0) {   // nothing to gather: every listed parent starts at 0
    const uint64_t stride = (uint64_t)n_part * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i <= n; i += stride)
      pl.off[i] = 0;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      pl.hdr->n = n;
      pl.hdr->bytes = 0;
      pl.hdr->nnz = 0;
      pl.hdr->M = 0;
      pl.hdr->incomplete = lh.incomplete;
      pl.hdr->max_end = 0;
      pl.hdr->err = 0u;
      pl.hdr->chunks_ok = 1u;
      L.hdr->incomplete = 0;   // spent (asm_parents adds to it)
    }
    return;
  }

  unsigned long long end = 0;   // largest arena end of this thread's members
  if (threadIdx.x == 0) s_end = 0;
  for (;;) {
    if (threadIdx.x == 0) s_tile = claim_tile(&ds->tile_ctr[slot]);
    __syncthreads();
    const uint32_t tile = s_tile;
    __syncthreads();
    if (tile >= n_tiles) break;
    const uint64_t g0 = (uint64_t)tile * AM_TILE;
    const uint64_t i_lo = L.mtfp[tile];
    const uint64_t i_hi = (tile + 1 < n_tiles) ? L.mtfp[tile + 1] : n - 1;
    const uint64_t R = i_hi - i_lo + 1;
    const bool staged = R <= AM_SMEM_CAP;
    if (staged) {
#pragma unroll 4
      for (uint32_t k = threadIdx.x; k < (uint32_t)R; k += AM_THREADS) {
        s_mb[k] = __ldcg(L.mb + i_lo + k);
        s_coff[k] = __ldcg(L.coff + i_lo + k);
      }
    }
    __syncthreads();

    // my members gt .. gt+AM_ITEMS-1 are consecutive: one search finds the
    // list entry holding the first, a walk over the member bases the rest
    const uint64_t gt = g0 + (uint64_t)threadIdx.x * AM_ITEMS;
    constexpr uint64_t NONE = ~0ull;
    uint32_t ridx[AM_ITEMS];   // the member's child number (below 2^32 - 1), or ~0
    {
      uint64_t i = i_lo;
      if (gt < M) {
        if (staged) {
          i = i_lo + last_le_u(s_mb, 0u, (uint32_t)R, gt);
        } else {
          uint64_t lo = i_lo, hi = i_hi + 1;
          while (hi - lo > 1) {
            const uint64_t mid = lo + ((hi - lo) >> 1);
            if (L.mb[mid] <= gt) lo = mid; else hi = mid;
          }
          i = lo;
        }
      }
      // no member of this tile lies past entry i_hi
      auto mb_at = [&](uint64_t x) -> uint64_t { return staged ? s_mb[x - i_lo] : L.mb[x]; };
      uint64_t mbi = gt < M ? mb_at(i) : 0;
      uint64_t mbn = (gt < M && i < i_hi) ? mb_at(i + 1) : NONE;
      uint64_t cof = gt < M ? (staged ? s_coff[i - i_lo] : L.coff[i]) : 0;
#pragma unroll
      for (int k = 0; k < AM_ITEMS; ++k) {
        const uint64_t g = gt + k;
        ridx[k] = ~0u;
        if (g < M) {
          while (g >= mbn) {   // member-less entries have equal bases and are passed over
            ++i;
            mbi = mbn;
            mbn = (i < i_hi) ? mb_at(i + 1) : NONE;
            cof = staged ? s_coff[i - i_lo] : L.coff[i];
          }
          ridx[k] = (uint32_t)(cof + (g - mbi));
        }
      }
    }
    // all record loads first (no store in between), so they overlap
    Slot rr[AM_ITEMS];
#pragma unroll
    for (int k = 0; k < AM_ITEMS; ++k) {
      if (ridx[k] != ~0u) {
        rr[k] = a.slot[ridx[k]];
      } else {
        rr[k].len = 0;
        rr[k].w = 0;
      }
    }
    // len becomes the bytes the member contributes (0 unless Present)
    Pair64 mine{0, 0};
#pragma unroll
    for (int k = 0; k < AM_ITEMS; ++k) {
      if (w_state(rr[k].w) != ST_PRESENT) rr[k].len = 0;
      if (rr[k].len) {
        const uint64_t src = w_off(rr[k].w);
        // the arena of the assembly must hold what the commit accepted: for a
        // commit's own plan the copy checks the largest end
        if (a.for_commit) {
          const unsigned long long e = src + rr[k].len;
          end = e > end ? e : end;
        } else if (src > a.arena_bytes || (uint64_t)rr[k].len > a.arena_bytes - src) {
          atomicOr(&ds->err, ERR_INVAL);
          L.hdr->bad = 1u;
        }
      }
      mine.a += rr[k].len;
      mine.b += rr[k].len ? 1ull : 0ull;
    }
    Pair64 total;
    Pair64 excl = block_excl_scan_pair(mine, s_scan, &total);
    if (threadIdx.x < 32) {  // one warp looks back
      const auto pfx = lookback_exclusive(a.ts_members, tile, total, ds->epoch[slot], &ds->err);
      if (threadIdx.x == 0) s_prefix = pfx;
    }
    {
      unsigned long long at = excl.a;
#pragma unroll
      for (int k = 0; k < AM_ITEMS; ++k) {
        s_pos[threadIdx.x * AM_ITEMS + k] = at;
        at += rr[k].len;
      }
      if (threadIdx.x == AM_THREADS - 1) s_pos[AM_TILE] = at;
    }
    __syncthreads();
    // Output offsets of the listed parents that start in this tile (a parent
    // without members starts where its successor does): all of i_lo .. i_hi
    // but a parent that started in an earlier tile or starts the next one.
    for (uint64_t i = i_lo + threadIdx.x; i <= i_hi; i += AM_THREADS) {
      const uint64_t mb = staged ? s_mb[i - i_lo] : L.mb[i];
      if (i == i_lo && mb != g0) continue;
      if (i == i_hi && tile + 1 < n_tiles && mb == g0 + AM_TILE) continue;
      pl.off[i] = s_prefix.a + s_pos[mb - g0];
    }
    if (tile == 0)   // parents without members before the first that has some
      for (uint64_t i = threadIdx.x; i < i_lo; i += AM_THREADS) pl.off[i] = 0;
    Pair64 run = s_prefix + excl;   // (bytes, contributing members) before my first item
#pragma unroll
    for (int k = 0; k < AM_ITEMS; ++k) {
      const uint64_t g = gt + k;
      if (g >= M) break;
      const uint64_t pos = run.a;
      if (a.elem_base) {   // the member's list entry (offset relative until the copy)
        a.elem_state[g] = w_state(rr[k].w) == ST_PRESENT ? ST_PRESENT : ST_DROPPED;
        a.elem_len[g] = rr[k].len;
        a.elem_off[g] = pos;
      }
      if (rr[k].len) {
        const uint64_t j = run.b;
        if (j < pl.member_cap) {
          pl.cpos[j] = pos;
          pl.csrc[j] = w_off(rr[k].w);
        }
        const uint64_t e = pos + rr[k].len;
        for (uint64_t t = ceil_div(pos, AC_CHUNK); t * AC_CHUNK < e && t < pl.ctfp_cap; ++t)
          pl.ctfp[t] = (uint32_t)j;
        run.b += 1;
        run.a += rr[k].len;
      }
    }
    if (tile == n_tiles - 1 && threadIdx.x == AM_THREADS - 1) {
      pl.off[n] = run.a;
      pl.hdr->n = n;
      pl.hdr->bytes = run.a;
      pl.hdr->nnz = run.b;
      pl.hdr->M = M;
      pl.hdr->incomplete = lh.incomplete;
      if (!a.for_commit) pl.hdr->max_end = 0;   // checked here, member by member
      pl.hdr->chunks_ok = ceil_div(run.a, AC_CHUNK) <= pl.ctfp_cap ? 1u : 0u;
    }
    __syncthreads();
  }
  if (a.for_commit) {
    for (int d = 16; d > 0; d >>= 1) {
      const unsigned long long o = __shfl_xor_sync(0xffffffffu, end, d);
      end = o > end ? o : end;
    }
    if ((threadIdx.x & 31) == 0 && end) atomicMax(&s_end, end);
    __syncthreads();
    if (threadIdx.x == 0 && s_end) atomicMax(&pl.hdr->max_end, s_end);
  }
  if (threadIdx.x == 0 && ticket(&ds->exit_ctr[slot]) == n_part - 1) {
    ds->tile_ctr[slot] = 0u;
    ds->exit_ctr[slot] = 0u;
    ds->epoch[slot] += 1ull;
    L.hdr->incomplete = 0;   // spent (asm_parents adds to it)
    pl.hdr->err = __ldcg(&L.hdr->bad);
    L.hdr->bad = 0u;
  }
}

// ---------------------------------------------------------------------------
// Bytes sh .. sh+15 of the 32-byte window (x, y), sh in [0, 15].
__device__ __forceinline__ uint4 window16(const uint4 x, const uint4 y, uint32_t sh) {
  // branch-free: move the window by 8 bytes, then by 4, then funnel-shift
  // the remaining 0..3 bytes (lanes with different shifts do not diverge)
  const bool h8 = (sh & 8u) != 0u, h4 = (sh & 4u) != 0u;
  const uint32_t b0 = h8 ? x.z : x.x, b1 = h8 ? x.w : x.y, b2 = h8 ? y.x : x.z;
  const uint32_t b3 = h8 ? y.y : x.w, b4 = h8 ? y.z : y.x, b5 = h8 ? y.w : y.y;
  const uint32_t a0 = h4 ? b1 : b0, a1 = h4 ? b2 : b1, a2 = h4 ? b3 : b2;
  const uint32_t a3 = h4 ? b4 : b3, a4 = h4 ? b5 : b4;
  const uint32_t b = (sh & 3u) * 8u;
  uint4 r;
  r.x = __funnelshift_r(a0, a1, b);
  r.y = __funnelshift_r(a1, a2, b);
  r.z = __funnelshift_r(a2, a3, b);
  r.w = __funnelshift_r(a3, a4, b);
  return r;
}

// v with its bytes from position b (0..16) on replaced by those of u
__device__ __forceinline__ uint32_t keep_low(uint32_t v, uint32_t u, int b) {
  const int c = b < 0 ? 0 : (b > 4 ? 4 : b);
  const uint32_t m = (uint32_t)((1ull << (8 * c)) - 1ull);
  return (v & m) | (u & ~m);
}
__device__ __forceinline__ uint4 take_from(const uint4 v, const uint4 u, uint32_t b) {
  const int bi = (int)b;
  return make_uint4(keep_low(v.x, u.x, bi), keep_low(v.y, u.y, bi - 4), keep_low(v.z, u.z, bi - 8),
                    keep_low(v.w, u.w, bi - 12));
}

__device__ __forceinline__ uint4 shfl_down4(const uint4 v, int d) {
  return make_uint4(__shfl_down_sync(0xffffffffu, v.x, d), __shfl_down_sync(0xffffffffu, v.y, d),
                    __shfl_down_sync(0xffffffffu, v.z, d), __shfl_down_sync(0xffffffffu, v.w, d));
}
__device__ __forceinline__ uint4 shfl_idx4(const uint4 v, int l) {
  return make_uint4(__shfl_sync(0xffffffffu, v.x, l), __shfl_sync(0xffffffffu, v.y, l),
                    __shfl_sync(0xffffffffu, v.z, l), __shfl_sync(0xffffffffu, v.w, l));
}

constexpr int CP_UNROLL = 4;   // groups of 32 words in flight per warp

// One warp copies `len` bytes from src to dst (both any alignment).  Whole
// destination words are written with 16-byte stores, each lane's word built
// from its own aligned source block and its right neighbour's (shuffled in,
// or loaded by the lane at a group's edge); the partial first and last words
// are written byte by byte, so the bytes of neighbouring pieces are never
// touched.  Every block read holds at least one byte of the source range.
// (Used for chunks whose pieces do not fit the shared-memory stage.)
__device__ __forceinline__ void warp_copy(uint8_t* dst, const uint8_t* src, uint64_t len, int lane) {
  const uint64_t d = (uint64_t)(uintptr_t)dst, d_end = d + len;
  const uint64_t head_end = ((d + 15) & ~15ull) < d_end ? ((d + 15) & ~15ull) : d_end;
  if ((uint64_t)lane < head_end - d) dst[lane] = __ldg(src + lane);
  if (head_end == d_end) return;
  const uint64_t full_lo = head_end, full_hi = d_end & ~15ull;
  if (full_hi > full_lo) {
    const uint64_t nw = (full_hi - full_lo) >> 4;
    const uint8_t* s_full = src + (full_lo - d);
    const uint32_t sig = (uint32_t)((uintptr_t)s_full & 15u);
    const uint4* A0 = reinterpret_cast<const uint4*>((uintptr_t)s_full & ~(uintptr_t)15);
    uint4* D0 = reinterpret_cast<uint4*>((uintptr_t)full_lo);
    for (uint64_t g0 = 0; g0 < nw; g0 += 32 * CP_UNROLL) {
      uint4 x[CP_UNROLL], y[CP_UNROLL];
#pragma unroll
      for (int u = 0; u < CP_UNROLL; ++u) {
        const uint64_t k = g0 + (uint64_t)u * 32 + lane;
        x[u] = make_uint4(0u, 0u, 0u, 0u);
        y[u] = x[u];
        if (k < nw) {
          x[u] = __ldg(A0 + k);
          const bool edge = (lane == 31 && (u == CP_UNROLL - 1 || k + 1 >= nw)) || k + 1 >= nw;
          if (sig && edge) y[u] = __ldg(A0 + k + 1);
        }
      }
      if (sig) {
#pragma unroll
        for (int u = 0; u < CP_UNROLL; ++u) {
          const uint64_t k = g0 + (uint64_t)u * 32 + lane;
          const uint4 nb = shfl_down4(x[u], 1);
          const uint4 nx = (u + 1 < CP_UNROLL) ? shfl_idx4(x[(u + 1) % CP_UNROLL], 0) : nb;
          const bool edge = (lane == 31 && (u == CP_UNROLL - 1 || k + 1 >= nw)) || k + 1 >= nw;
          if (!edge) y[u] = (lane == 31) ? nx : nb;
        }
      }
#pragma unroll
      for (int u = 0; u < CP_UNROLL; ++u) {
        const uint64_t k = g0 + (uint64_t)u * 32 + lane;
        if (k < nw) D0[k] = sig ? window16(x[u], y[u], sig) : x[u];
      }
    }
  }
  const uint64_t tail_lo = full_hi > head_end ? full_hi : head_end;
  if ((uint64_t)lane < d_end - tail_lo) dst[(tail_lo - d) + lane] = __ldg(src + (tail_lo - d) + lane);
}

// ---- TMA staging --------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0u;
}
// The same wait, but the thread may sleep until the phase completes (or
// about `ns` nanoseconds pass) instead of returning at once.
__device__ __forceinline__ bool mbar_try_wait_sleep(uint64_t* bar, uint32_t parity, uint32_t ns) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity), "r"(ns)
      : "memory");
  return ok != 0u;
}
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
// bulk copy of `bytes` (multiple of 16) from 16-byte aligned global memory
// into 16-byte aligned shared memory, completing on `bar`
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}

// tx bytes the current phase of `bar` waits for, without arriving
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.expect_tx.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
// 16 bytes from 16-byte aligned global to 16-byte aligned shared memory,
// asynchronously (no register staging)
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
// the current phase of `bar` also waits for this thread's cp.async copies
// issued so far (the pending count goes up now and down when they land)
__device__ __forceinline__ void cp_async_track(uint64_t* bar) {
  asm volatile("cp.async.mbarrier.arrive.shared::cta.b64 [%0];" ::"r"(smem_addr(bar)) : "memory");
}

// Bounded wait on a stage barrier for the phase of parity `parity`; false
// (recording ERR_TIMEOUT and raising the CTA's abort flag) if it gave up or
// another warp of the CTA already did.  Called by every lane of a warp; the
// answer is the same for the whole warp (false if any lane gave up), so the
// warp's collective operations after it never see a split warp.
__device__ __forceinline__ bool stage_wait_lane(uint64_t* bar, uint32_t parity, uint32_t* err,
                                                volatile uint32_t* abort);
__device__ __forceinline__ bool stage_wait2(uint64_t* bar, uint32_t parity, uint32_t* err,
                                            volatile uint32_t* abort) {
  return __all_sync(0xffffffffu, stage_wait_lane(bar, parity, err, abort));
}
__device__ __forceinline__ bool stage_wait_lane(uint64_t* bar, uint32_t parity, uint32_t* err,
                                                volatile uint32_t* abort) {
  // at most 2^20 polls of up to ~1 us each
  for (uint32_t i = 0; i < (1u << 20); ++i) {
    if (mbar_try_wait_sleep(bar, parity, 1000u)) return true;
    if ((i & 255u) == 255u && (*abort || (ld_acquire(err) & ERR_TIMEOUT))) {
      *abort = 1u;
      return false;
    }
  }
  atomicOr(err, ERR_TIMEOUT);
  *abort = 1u;
  return false;
}

// One pipeline stage: the source bytes of one 16 KB output chunk, laid out
// piece by piece (each piece = the part of one member inside the chunk, read
// as the aligned 16-byte blocks that hold it).  Offsets inside the chunk are
// taken from wbase, the aligned word at or before the chunk's first byte.
struct CopyStage {
  uint32_t np;                    // pieces staged, or AC_FALLBACK
  uint32_t vbeg, vend;            // the chunk's bytes, relative to wbase
  uint32_t pad;
  unsigned long long wbase;       // absolute address of the chunk's first word
  unsigned long long rel_s, rel_e;   // the chunk's bytes, relative to the call's output
  unsigned long long j_lo;        // first member of the chunk
  // output start of each piece (+ end), relative to wbase (< 16400), and the
  // buffer offset of output byte wbase per piece (-16400 .. 24592)
  uint16_t pstart[AC_PIECES + 1];
  int16_t qbase[AC_PIECES];
  uint32_t pad2[3];
  // the 16 bytes before buf (the end of qbase) may be read and ignored: a
  // piece's first word can start before the piece's first staged block
  __align__(16) unsigned char buf[AC_BUF + 32];
};
constexpr uint32_t AC_FALLBACK = 0xFFFFFFFFu;
constexpr uint32_t AC_DONE = 0xFFFFFFFEu;      // no chunk: the consumers stop at this stage



struct CopyCtx {
  const AssembleArgs* a;
  const uint64_t* cpos;
  const uint64_t* csrc;
  const uint32_t* ctfp;   // chunk table, or NULL (search instead)
  uint64_t out_base;      // absolute address of the call's first output byte
  uint64_t S, Mnz, n_chunks;
};

__device__ __forceinline__ uint64_t cpos_at(const CopyCtx& c, uint64_t j) {
  return j < c.Mnz ? c.cpos[j] : c.S;
}

// Largest j in [0, n) with pos[j] <= x (pos[0] = 0 <= x): 32 probes a round.
__device__ __forceinline__ uint64_t warp_search(const uint64_t* pos, uint64_t n, uint64_t x, int lane) {
  uint64_t lo = 0, hi = n;
  while (hi - lo > 1) {
    const uint64_t step = (hi - lo + 31) / 32;
    const uint64_t probe = lo + step * (uint64_t)lane;
    const bool le = probe < hi && pos[probe] <= x;
    const unsigned m = __ballot_sync(0xffffffffu, le);
    const uint64_t last = (uint64_t)(31 - __clz((int)m));
    lo = lo + step * last;
    hi = (lo + step < hi) ? lo + step : hi;
  }
  return lo;
}

// A producer warp stages chunk k: finds its members, builds the piece table
// and issues one bulk copy per piece, completing on `bar`.
__device__ void stage_chunk(const CopyCtx& c, uint64_t k, CopyStage* st, uint64_t* bar, int lane) {
  const uint64_t rs = k * AC_CHUNK;
  const uint64_t re = (rs + AC_CHUNK < c.S) ? rs + AC_CHUNK : c.S;
  uint64_t j_lo, j_hi;
  if (c.ctfp) {
    j_lo = c.ctfp[k];
    j_hi = (k + 1 < c.n_chunks) ? c.ctfp[k + 1] : c.Mnz - 1;
  } else {
    j_lo = warp_search(c.cpos, c.Mnz, rs, lane);
    j_hi = warp_search(c.cpos, c.Mnz, re - 1, lane);
  }
  const uint64_t np = j_hi - j_lo + 1;
  const uint64_t wbase = (c.out_base + rs) & ~15ull;
  if (lane == 0) {
    st->wbase = wbase;
    st->rel_s = rs;
    st->rel_e = re;
    st->j_lo = j_lo;
    st->vbeg = (uint32_t)(c.out_base + rs - wbase);
    st->vend = (uint32_t)(c.out_base + re - wbase);
  }
  const uint64_t arena = (uint64_t)(uintptr_t)c.a->arena;
  // a chunk whose aligned blocks do not fit AC_BUF is read by the consumers
  // with plain loads
  // (a pinned host arena is staged like any other: 117 MB read and 117 MB
  // written back over the link per pass took 1.04 ms among other passes with
  // plain loads, 0.93 staged; the link copies both ways at 167 GB/s)
  const bool tabled = np <= AC_PIECES;
  uint32_t roff = 0;   // running buffer offset (warp-uniform)
  uint32_t tx = 0;     // bytes of the pieces staged by bulk copies (per lane)
  if (tabled) {
    constexpr int R = 4;   // rounds of 32 pieces whose loads go out together
    for (uint64_t g0 = 0; g0 < np; g0 += 32 * R) {
      uint64_t p0[R], p1[R], cs[R];
#pragma unroll
      for (int u = 0; u < R; ++u) {
        const uint64_t i = g0 + (uint64_t)u * 32 + lane;
        p0[u] = p1[u] = cs[u] = 0;
        if (i < np) {
          const uint64_t j = j_lo + i;
          p0[u] = c.cpos[j];
          p1[u] = cpos_at(c, j + 1);
          cs[u] = c.csrc[j];
        }
      }
#pragma unroll
      for (int u = 0; u < R; ++u) {
        const uint64_t i = g0 + (uint64_t)u * 32 + lane;
        uint32_t size = 0, sh = 0, ps = 0;
        if (i < np) {
          const uint64_t ob = p0[u] > rs ? p0[u] : rs, oe = p1[u] < re ? p1[u] : re;
          const uint64_t src = arena + cs[u] + (ob - p0[u]);
          const uint64_t a0 = src & ~15ull, a1 = (src + (oe - ob) + 15) & ~15ull;
          size = (uint32_t)(a1 - a0);
          sh = (uint32_t)(src & 15u);
          ps = (uint32_t)(c.out_base + ob - wbase);
          if (size > AC_SMALL) tx += size;
        }
        uint32_t inc = size;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const uint32_t t = __shfl_up_sync(0xffffffffu, inc, d);
          if (lane >= d) inc += t;
        }
        const uint32_t my_off = roff + inc - size;
        if (i < np) {
          st->pstart[i] = (uint16_t)ps;
          st->qbase[i] = (int16_t)((int32_t)(my_off + sh) - (int32_t)ps);
        }
        roff += __shfl_sync(0xffffffffu, inc, 31);
      }
    }
  }
  const bool fits = tabled && roff <= AC_BUF;
  if (!fits) {
    if (lane == 0) {
      st->np = AC_FALLBACK;
      mbar_arrive(bar);   // completes the phase; consumers copy from global
    }
    __syncwarp();
    return;
  }
  // the stage completes when the bulk copies' bytes have landed, every
  // lane's cp.async copies of small pieces too, and lane 0 has arrived
  for (int d = 16; d > 0; d >>= 1) tx += __shfl_xor_sync(0xffffffffu, tx, d);
  if (lane == 0) {
    st->np = (uint32_t)np;
    st->pstart[np] = (uint16_t)(c.out_base + re - wbase);
    mbar_expect_tx(bar, tx);
  }
  __syncwarp();
  fence_proxy_async_smem();   // earlier generic accesses of this stage before async writes
  bool small = false;
  constexpr int R = 4;
  for (uint64_t i0 = lane; i0 < np; i0 += 32 * R) {
    uint64_t p0[R], cs[R];
#pragma unroll
    for (int u = 0; u < R; ++u) {
      const uint64_t i = i0 + (uint64_t)u * 32;
      p0[u] = cs[u] = 0;
      if (i < np) {
        p0[u] = c.cpos[j_lo + i];
        cs[u] = c.csrc[j_lo + i];
      }
    }
#pragma unroll
    for (int u = 0; u < R; ++u) {
      const uint64_t i = i0 + (uint64_t)u * 32;
      if (i >= np) break;
      const uint64_t ob = wbase + st->pstart[i] - c.out_base;      // relative
      const uint64_t oe = wbase + st->pstart[i + 1] - c.out_base;
      const uint64_t src = arena + cs[u] + (ob - p0[u]);
      const uint64_t a0 = src & ~15ull, a1 = (src + (oe - ob) + 15) & ~15ull;
      const uint32_t off = (uint32_t)(st->qbase[i] + (int32_t)st->pstart[i]) - (uint32_t)(src & 15u);
      const uint32_t size = (uint32_t)(a1 - a0);   // 0: a member that starts at the chunk's end
      if (size > AC_SMALL) {
        bulk_g2s(st->buf + off, reinterpret_cast<const void*>((uintptr_t)a0), size, bar);
      } else {
        // small pieces: one 16-byte asynchronous copy per block, no bulk copy
        for (uint32_t b = 0; b < size; b += 16)
          cp_async16(st->buf + off + b, reinterpret_cast<const void*>((uintptr_t)(a0 + b)));
        small = small || size != 0;
      }
    }
  }
  if (small) cp_async_track(bar);
  __syncwarp();
  if (lane == 0) mbar_arrive(bar);
}

// A producer's plan entries of a chunk, fetched a round ahead with cp.async,
// so that the chunk can be staged without touching global memory: members j_lo
// .. j_lo + np - 1 and the position after them.
constexpr uint32_t AC_AHEAD = 64;
struct ChunkEntries {
  unsigned long long pos[AC_AHEAD + 2], src[AC_AHEAD + 2];
};
// the stages, then two rounds of entries per producer
constexpr size_t AC_SMEM = AC_STAGES * sizeof(CopyStage) + 2 * AC_PRODUCERS * sizeof(ChunkEntries);
size_t asm_copy_smem() { return AC_SMEM; }
struct ChunkRef {
  uint32_t k, j_lo, j_hi;   // chunk, its first member, the member holding the next chunk's first byte
  __device__ __forceinline__ bool ahead() const { return j_hi - j_lo <= AC_AHEAD; }
};
__device__ __forceinline__ void cp_async8(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}

__device__ __forceinline__ ChunkRef chunk_ref(const CopyCtx& c, uint32_t k, int lane) {
  ChunkRef r;
  r.k = k;
  const uint64_t rs = (uint64_t)k * AC_CHUNK, re = (rs + AC_CHUNK < c.S) ? rs + AC_CHUNK : c.S;
  if (c.ctfp) {
    r.j_lo = c.ctfp[k];
    r.j_hi = (k + 1 < c.n_chunks) ? c.ctfp[k + 1] : (uint32_t)c.Mnz - 1;
  } else {
    r.j_lo = (uint32_t)warp_search(c.cpos, c.Mnz, rs, lane);
    r.j_hi = (uint32_t)warp_search(c.cpos, c.Mnz, re - 1, lane);
  }
  return r;
}

// Fetch a chunk's entries (nothing for chunks of too many members).
__device__ __forceinline__ void fetch_entries(const CopyCtx& c, const ChunkRef& r, ChunkEntries* en, int lane) {
  if (!r.ahead()) return;
  const uint32_t n = r.j_hi - r.j_lo + 2;   // and the entry after the last
  for (uint32_t i = lane; i < n; i += 32) {
    const uint32_t j = r.j_lo + i;
    if (j < c.Mnz) {
      cp_async8(&en->pos[i], c.cpos + j);
      cp_async8(&en->src[i], c.csrc + j);
    } else {
      en->pos[i] = c.S;
    }
  }
}

// Stage a chunk whose entries are in shared memory: piece table, expected
// bytes and copies, 32 pieces at a time.  (At most AC_AHEAD + 1 pieces, each
// less than 32 bytes longer in the stage than in the output, always fit it.)
// Other chunks take stage_chunk's general path.
__device__ __forceinline__ void issue_chunk(const CopyCtx& c, const ChunkRef& r, const ChunkEntries* en, CopyStage* st, uint64_t* bar,
                            int lane) {
  if (!r.ahead()) {
    stage_chunk(c, r.k, st, bar, lane);
    return;
  }
  const uint64_t rs = (uint64_t)r.k * AC_CHUNK, re = (rs + AC_CHUNK < c.S) ? rs + AC_CHUNK : c.S;
  const uint64_t wbase = (c.out_base + rs) & ~15ull, arena = (uint64_t)(uintptr_t)c.a->arena;
  const uint32_t n = r.j_hi - r.j_lo + 1;
  // the last member may start at the chunk's end
  const uint32_t np = (n > 1 && en->pos[n - 1] >= re) ? n - 1 : n;
  if (lane == 0) {
    st->wbase = wbase;
    st->rel_s = rs;
    st->rel_e = re;
    st->j_lo = r.j_lo;
    st->vbeg = (uint32_t)(c.out_base + rs - wbase);
    st->vend = (uint32_t)(c.out_base + re - wbase);
    st->np = np;
    st->pstart[np] = (uint16_t)(c.out_base + re - wbase);
  }
  __syncwarp();
  fence_proxy_async_smem();   // earlier generic accesses of this stage before async writes
  uint32_t roff = 0;          // running buffer offset (warp-uniform)
  bool small = false;
  for (uint32_t i0 = 0; i0 < np; i0 += 32) {
    const uint32_t i = i0 + (uint32_t)lane;
    uint64_t a0 = 0;
    uint32_t size = 0, sh = 0, ps = 0;
    if (i < np) {
      const uint64_t p0 = en->pos[i], p1 = en->pos[i + 1];
      const uint64_t ob = p0 > rs ? p0 : rs, oe = p1 < re ? p1 : re;
      const uint64_t src = arena + en->src[i] + (ob - p0);
      a0 = src & ~15ull;
      size = (uint32_t)(((src + (oe - ob) + 15) & ~15ull) - a0);
      sh = (uint32_t)(src & 15u);
      ps = (uint32_t)(c.out_base + ob - wbase);
    }
    uint32_t inc = size, tx = size > AC_SMALL ? size : 0;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t t = __shfl_up_sync(0xffffffffu, inc, d);
      if (lane >= d) inc += t;
    }
    tx = __reduce_add_sync(0xffffffffu, tx);
    const uint32_t off = roff + inc - size;
    roff += __shfl_sync(0xffffffffu, inc, 31);
    if (i < np) {
      st->pstart[i] = (uint16_t)ps;
      st->qbase[i] = (int16_t)((int32_t)(off + sh) - (int32_t)ps);
    }
    if (lane == 0) mbar_expect_tx(bar, tx);
    __syncwarp();
    if (size > AC_SMALL) {
      bulk_g2s(st->buf + off, reinterpret_cast<const void*>((uintptr_t)a0), size, bar);
    } else if (size) {   // small pieces: one 16-byte asynchronous copy per block, no bulk copy
      for (uint32_t b = 0; b < size; b += 16)
        cp_async16(st->buf + off + b, reinterpret_cast<const void*>((uintptr_t)(a0 + b)));
      small = true;
    }
  }
  if (small) cp_async_track(bar);
  __syncwarp();
  if (lane == 0) mbar_arrive(bar);
}

__device__ __forceinline__ uint4 lds128(const unsigned char* p) {
  return *reinterpret_cast<const uint4*>(p);
}
// bytes A .. A+15 of the stage buffer (A may be down to -15)
__device__ __forceinline__ uint4 stage_word(const CopyStage* st, int32_t A) {
  const int32_t Aa = A & ~15;
  return window16(lds128(st->buf + Aa), lds128(st->buf + Aa + 16), (uint32_t)(A & 15));
}

// Consumer warp cw writes words [w0, w1) of a staged chunk, a lane per
// 16-byte word.  A word inside one piece is one shifted 16-byte read of the
// stage; a word that meets a piece boundary merges its pieces' bytes.  The
// chunk's first and last words may hold bytes of neighbouring chunks: only
// the chunk's own bytes of them are written, byte by byte.
__device__ void emit_range(const CopyStage* st, uint32_t cw, int lane) {
  const uint32_t np = st->np, vbeg = st->vbeg, vend = st->vend;
  const uint64_t wbase = st->wbase;
  const uint32_t nW = (vend + 15u) >> 4;
  const uint32_t w0 = (nW * cw) / AC_CONSUMERS, w1 = (nW * (cw + 1)) / AC_CONSUMERS;
  if (w0 >= w1) return;
  const uint32_t first = (w0 * 16u > vbeg) ? w0 * 16u : vbeg;
  uint32_t a = 0, b = np;   // the piece holding byte `first` (pstart[0] = vbeg)
  while (b - a > 1) {
    const uint32_t m = (a + b) >> 1;
    if (st->pstart[m] <= first) a = m; else b = m;
  }
  uint32_t icur = a;
#pragma unroll 1
  for (uint32_t g = w0; g < w1; g += 32) {
    const uint32_t w = g + (uint32_t)lane;
    uint32_t i = icur;
    if (w < w1) {
      const uint32_t wr = w * 16u;
      const uint32_t lo = wr > vbeg ? wr : vbeg;
      const uint32_t hi = (wr + 16u < vend) ? wr + 16u : vend;
      // the piece holding byte lo: the warp's last piece or the next (large
      // pieces), else a search of the rest (many small pieces per chunk)
      uint32_t pe = st->pstart[i + 1];
      if (pe <= lo) {
        ++i;
        pe = st->pstart[i + 1];
        if (pe <= lo) {
          uint32_t ia = i + 1, ib = np;   // pstart[ia] <= lo < pstart[np]
          while (ib - ia > 1) {
            const uint32_t m = (ia + ib) >> 1;
            if (st->pstart[m] <= lo) ia = m; else ib = m;
          }
          i = ia;
          pe = st->pstart[i + 1];
        }
      }
      // bytes [lo, pe) come from piece i; a word that reaches further takes
      // the rest from the following pieces, one boundary at a time
      uint4 v = stage_word(st, st->qbase[i] + (int32_t)wr);
      while (pe < hi) {
        ++i;
        v = take_from(v, stage_word(st, st->qbase[i] + (int32_t)wr), pe - wr);
        pe = st->pstart[i + 1];
      }
      uint4* dst = reinterpret_cast<uint4*>((uintptr_t)(wbase + wr));
      if (lo == wr && hi == wr + 16u) {
        *dst = v;
      } else {
        // the chunk's first or last word: only the chunk's own bytes
        const uint32_t vv[4] = {v.x, v.y, v.z, v.w};
        uint8_t* d8 = reinterpret_cast<uint8_t*>(dst);
#pragma unroll
        for (int t = 0; t < 16; ++t)
          if ((uint32_t)t >= lo - wr && (uint32_t)t < hi - wr) d8[t] = (uint8_t)(vv[t >> 2] >> (8 * (t & 3)));
      }
    }
    icur = __shfl_sync(0xffffffffu, i, 31);
  }
}

// ---- gather: copies of small records --------------------------------------------------
// Pieces of a few dozen bytes are not worth staging: their piece tables cost
// the two producer warps more than the copies.  When a call's members average
// at most AC_GATHER bytes (AC_GATHER_SMALL in a copy of few chunks, which
// otherwise takes a member at a time) every warp of the CTA copies on its own:
// a ring of the plan's entries in shared memory is kept ahead with cp.async,
// and each lane builds whole 16-byte output words from the members they fall
// into, loading the aligned blocks that hold them straight from the arena, two
// words in flight (in registers; four did not fit and took 1.7 times as long).
// Bound by the random reads: each fetches a 128-byte line from DRAM, 15 GB for
// 110M members of 32 bytes, 3.4 ms against 5.5 staged.  The lines, staged and
// gathered: 4.7M members of 48 bytes 278 and 233 us, of 128 592 and 521, of 160
// 617 and 650; few chunks, 11,781 members of 64 bytes 27 and 12 us, of 333 18.7
// and 15.8, 7,120 of 512 12.3 and 14.6.
constexpr uint64_t AC_GATHER = 140, AC_GATHER_SMALL = 384;
constexpr int GA_WORDS = 2;
constexpr uint32_t GA_RING = 512, GA_WINDOW = GA_RING / 2;   // plan entries of a warp's ring
struct GatherRing {
  unsigned long long p[GA_RING], s[GA_RING];
  __device__ __forceinline__ unsigned long long& pos(uint64_t j) { return p[(uint32_t)j & (GA_RING - 1)]; }
  __device__ __forceinline__ unsigned long long& src(uint64_t j) { return s[(uint32_t)j & (GA_RING - 1)]; }
};
static_assert((AC_THREADS / 32) * sizeof(GatherRing) <= AC_SMEM, "a ring per warp");

// The 16 bytes at a global address, or zero.
__device__ __forceinline__ uint4 ldg_if(uint64_t addr, bool on) {
  uint4 v = make_uint4(0u, 0u, 0u, 0u);
  if (on) v = __ldg(reinterpret_cast<const uint4*>((uintptr_t)addr));
  return v;
}

// An output word being built: its offset in the unit, the offsets of its first
// byte not copied yet and of its end, the member that byte is in, its bytes so
// far and the blocks loaded for them.
struct GatherWord {
  uint32_t wr, at, hi, it, end, sh;
  uint4 v, x, y;
};
__device__ __forceinline__ void gather_load(GatherRing& r, GatherWord& w, uint64_t arena, uint64_t ub,
                                            uint64_t j) {
  const bool on = w.at < w.hi;
  const uint64_t q = j + (on ? w.it : 0);
  const uint64_t p0 = r.pos(q), nx = r.pos(q + 1) - ub;
  w.end = on ? (nx < w.hi ? (uint32_t)nx : w.hi) : w.at;
  // the arena address of the word's byte 0, were it this member's, and its 16-byte block
  const uint64_t sw = arena + r.src(q) + (ub + w.wr - p0), blk = sw & ~15ull;
  w.sh = (uint32_t)sw & 15u;
  // only blocks that hold a byte of the member
  w.x = ldg_if(blk, on && blk + 16 > sw + (w.at - w.wr));
  w.y = ldg_if(blk + 16, on && blk + 16 < sw + (w.end - w.wr));
}
__device__ __forceinline__ bool gather_merge(GatherWord& w) {
  const bool on = w.at < w.hi;
  w.v = take_from(w.v, window16(w.x, w.y, w.sh), on ? w.at - w.wr : 16u);
  w.at = w.end;
  w.it += on ? 1u : 0u;
  return w.at < w.hi;
}

// One warp copies output bytes [p, e0) of the call; member j holds byte p.
// The ring holds entries [.., jl) of the plan, never more than half its size
// past the current unit's first member, so that entries written ahead replace
// none the unit still reads.
__device__ __forceinline__ void gather_range(const CopyCtx& c, GatherRing& r, uint64_t p, uint64_t e0, uint64_t j,
                                             int lane) {
  const uint64_t arena = (uint64_t)(uintptr_t)c.a->arena, out_base = c.out_base, Mnz = c.Mnz;
  const uint64_t n_ent = Mnz + 1;   // entry Mnz: the end, S
  uint64_t jl = j;
  const auto fill = [&](uint64_t upto) {
    upto = upto < n_ent ? upto : n_ent;
    for (uint64_t q = jl + lane; q < upto; q += 32) {
      if (q < Mnz) {
        cp_async8(&r.pos(q), c.cpos + q);
        cp_async8(&r.src(q), c.csrc + q);
      } else {
        r.pos(q) = c.S;
      }
    }
    jl = upto > jl ? upto : jl;
  };
  fill(j + GA_WINDOW);
  while (p < e0) {
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
    // the unit: up to 32 * GA_WORDS words from the aligned one holding byte p,
    // as far as the ring's entries reach.  Positions inside it are 32-bit
    // offsets from that word, relative to the call's output at ub.
    const uint64_t w0 = (out_base + p) & ~15ull, ub = w0 - out_base;   // (ub may be just below 0)
    uint64_t e = ub + 16ull * 32 * GA_WORDS;
    e = e < e0 ? e : e0;
    if (jl < n_ent) {
      const uint64_t known = r.pos(jl - 1);
      e = known < e ? known : e;   // (past p: the ring starts at the member holding p)
    }
    const uint32_t p_off = (uint32_t)(p - ub), e_off = (uint32_t)(e - ub), n_words = (e_off + 15) >> 4;
    const uint32_t nr = (uint32_t)(jl - j);
    const auto init = [&](GatherWord& w, uint32_t wi) {
      w.wr = 16 * wi;
      w.at = wi == 0 ? p_off : w.wr;
      w.hi = w.wr + 16 < e_off ? w.wr + 16 : e_off;
      w.v = make_uint4(0u, 0u, 0u, 0u);
      uint32_t a = 0, b = w.at < w.hi ? nr : 1;
      while (b - a > 1) {
        const uint32_t m = (a + b) >> 1;
        if (r.pos(j + m) <= ub + w.at) a = m; else b = m;
      }
      w.it = a;
    };
    const auto store = [&](const GatherWord& w) {
      const uint32_t lo = w.wr == 0 ? p_off : w.wr;
      if (lo >= e_off) return;
      uint8_t* d8 = reinterpret_cast<uint8_t*>((uintptr_t)(w0 + w.wr));
      if (lo == w.wr && w.wr + 16 <= e_off) {
        *reinterpret_cast<uint4*>(d8) = w.v;
      } else {   // an edge of the range: only its own bytes
#pragma unroll
        for (int q = 0; q < 16; ++q) {
          const uint32_t x = (q >> 2) == 0 ? w.v.x : (q >> 2) == 1 ? w.v.y : (q >> 2) == 2 ? w.v.z : w.v.w;
          if (w.wr + q >= lo && w.wr + q < e_off) d8[q] = (uint8_t)(x >> (8 * (q & 3)));
        }
      }
    };
    GatherWord wa, wb;   // (named: an array of them would not stay in registers)
    init(wa, lane);
    init(wb, 32 + lane);
    // the next unit starts in the last word's member or after it; its entries load meanwhile
    const uint32_t ja = __shfl_sync(0xffffffffu, wa.it, (n_words - 1) & 31u);
    const uint32_t jb = __shfl_sync(0xffffffffu, wb.it, (n_words - 1) & 31u);
    const uint32_t jn = n_words > 32 ? jb : ja;
    fill(j + jn + GA_WINDOW);
    bool more = true;
    while (more) {   // one member of each unfinished word per step (one step when words lie inside members)
      gather_load(r, wa, arena, ub, j);
      gather_load(r, wb, arena, ub, j);
      more = gather_merge(wa);
      more = gather_merge(wb) || more;
      more = __any_sync(0xffffffffu, more);
    }
    store(wa);
    store(wb);
    p = e;
    j += jn;
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncwarp();   // the ring is reused
}

// A chunk whose pieces do not fit a stage: consumer warps copy slices of it
// straight from global memory.
__device__ void emit_direct(const CopyCtx& c, const CopyStage* st, uint32_t cw, int lane) {
  constexpr uint64_t SLICE = (AC_CHUNK + AC_CONSUMERS - 1) / AC_CONSUMERS;
  const uint64_t rs = st->rel_s, re = st->rel_e;
  uint64_t ra = rs + (uint64_t)cw * SLICE;
  const uint64_t rb = (ra + SLICE < re) ? ra + SLICE : re;
  if (ra >= rb) return;
  uint64_t k = warp_search(c.cpos, c.Mnz, ra, lane);
  for (; ra < rb; ++k) {
    const uint64_t pk = c.cpos[k], pn = cpos_at(c, k + 1);
    const uint64_t e = pn < rb ? pn : rb;
    warp_copy(c.a->out + (c.out_base - (uint64_t)(uintptr_t)c.a->out) + ra,
              c.a->arena + c.csrc[k] + (ra - pk), e - ra, lane);
    ra = e;
  }
}

// A copy of at most AC_SMALL_CHUNKS chunks is latency-bound: every warp of
// the participating CTAs takes 2 KB slices of the output in turn and copies
// the member pieces inside each straight from the arena (no claims, staging
// or barriers), the slice's first member found from the chunk table and one
// warp-wide probe of the next 32 members.
constexpr uint64_t AC_SLICE = 2048;
__device__ void copy_small(const CopyCtx& c, uint64_t gw, uint64_t n_w, int lane) {
  const uint64_t n_sl = ceil_div(c.S, AC_SLICE);
  for (uint64_t sl = gw; sl < n_sl; sl += n_w) {
    uint64_t ra = sl * AC_SLICE;
    const uint64_t rb = (ra + AC_SLICE < c.S) ? ra + AC_SLICE : c.S;
    uint64_t k;
    if (c.ctfp) {   // the member holding the chunk's first byte holds or precedes ra
      const uint64_t k0 = c.ctfp[ra / AC_CHUNK], probe = k0 + (uint64_t)lane;
      const unsigned m = __ballot_sync(0xffffffffu, probe < c.Mnz && c.cpos[probe] <= ra);
      k = (m == 0xffffffffu) ? warp_search(c.cpos, c.Mnz, ra, lane) : k0 + (uint64_t)(__popc(m) - 1);
    } else {
      k = warp_search(c.cpos, c.Mnz, ra, lane);
    }
    for (; ra < rb; ++k) {
      const uint64_t pk = c.cpos[k], pn = cpos_at(c, k + 1);
      const uint64_t e = pn < rb ? pn : rb;
      warp_copy(c.a->out + (c.out_base - (uint64_t)(uintptr_t)c.a->out) + ra,
                c.a->arena + c.csrc[k] + (ra - pk), e - ra, lane);
      ra = e;
    }
  }
}

// The copy: the chunks of the call's output, claimed in rounds from a counter
// the grid shares, and the per-parent outputs beside them.  Warps
// 0..AC_PRODUCERS-1 stage chunks into a ring of AC_STAGES stages (producer p
// takes chunk p of each of the CTA's rounds), the other warps write them out in
// order; full and empty mbarriers per stage hand the stages back and forth.
// (Calls of small records: gather_range; few chunks: copy_small.)
// Sized to leave room beside it: two CTAs per SM take 2 x 320 threads x 80
// registers and 2 x 85 KB of shared memory (three stages and the producers'
// plan entries), so a CTA of a later wave's commit_list (56 registers, 33 KB)
// or asm_members (48, 25 KB) on another stream can be resident on the same SM
// while a copy runs.
__global__ void __maxnreg__(80) asm_copy_kernel(const __grid_constant__ AssembleArgs a) {
  wait_predecessor();
  extern __shared__ __align__(128) unsigned char ac_smem[];
  __shared__ __align__(8) uint64_t full_bar[AC_STAGES];
  __shared__ __align__(8) uint64_t empty_bar[AC_STAGES];
  __shared__ uint32_t s_issued[AC_STAGES];
  __shared__ uint32_t s_abort;
  __shared__ CopyRounds rounds;
  CopyStage* stages = reinterpret_cast<CopyStage*>(ac_smem);
  DevScalars* ds = a.ds;
  const PlanHdr hdr = *a.plan.hdr;
  const uint64_t n = hdr.n, S = hdr.bytes;
  const uint64_t base = a.cursor ? *a.cursor : 0ull;
  // Conditions every participating CTA sees the same way.  A CTA that starts
  // after the last of them is out may find the cursor advanced, and so conclude
  // anything but that it takes part: CTA 0, always a participant, reports.
  bool failed = hdr.err != 0u;
  if (!failed && hdr.max_end > a.arena_bytes) {   // the arena passed here must hold what was accepted
    failed = true;
    if (blockIdx.x + threadIdx.x == 0) atomicOr(&ds->err, ERR_INVAL);
  }
  const bool too_many = !a.user_list && n > a.n_host;   // outputs hold fewer parents
  const bool too_big = base + S > a.out_cap;
  if (!failed && (too_many || too_big)) {
    failed = true;
    if (blockIdx.x + threadIdx.x == 0) atomicOr(&ds->err, ERR_CAPACITY);
  }
  CopyCtx c;
  c.a = &a;
  c.cpos = a.plan.cpos;
  c.csrc = a.plan.csrc;
  c.ctfp = hdr.chunks_ok ? a.plan.ctfp : nullptr;
  c.out_base = (uint64_t)(uintptr_t)a.out + base;
  c.S = S;
  c.Mnz = hdr.nnz;
  const uint64_t n_chunks = (!failed && S) ? ceil_div(S, AC_CHUNK) : 0;
  c.n_chunks = n_chunks;
  const uint64_t par_units = failed ? 0 : ceil_div(n + 1, (uint64_t)AC_THREADS * 8);
  uint64_t units = n_chunks > par_units ? n_chunks : par_units;
  if (units == 0) units = 1;   // one CTA still finishes the call
  const uint32_t n_part = participants(units);
  if (blockIdx.x >= n_part) return;
  // Every warp of the CTA has read the cursor before its ticket is drawn: the
  // last CTA out rewrites it.
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

  if (!failed) {
    // per-parent outputs: status (commit plans), offsets, lengths, and the
    // list structure's entry offsets made absolute; by nt threads of each CTA.
    // Off the copy's way: the consumers write them while the first chunks
    // load, the warps of an unstaged copy after their bytes.
    const auto outputs = [&](uint32_t tid, uint32_t nt) {
      const uint64_t stride = (uint64_t)n_part * nt;
      const uint64_t gt0 = (uint64_t)blockIdx.x * nt + tid;
      if (a.elem_base)
        for (uint64_t g = gt0; g < hdr.M; g += stride) a.elem_off[g] += base;
      for (uint64_t i = gt0; i <= n; i += stride) {
        const uint64_t o = a.plan.off[i];
        a.out_off[i] = base + o;
        if (i == n) break;
        if (!a.user_list) a.status[i] = a.list.status[i];   // a caller's list has them already
        if (a.out_len) {
          const uint64_t len = a.plan.off[i + 1] - o;
          if (len > 0xFFFFFFFFull) atomicOr(&ds->err, ERR_OVERFLOW);
          a.out_len[i] = (uint32_t)len;
        }
      }
    };
    const bool gather = S <= (n_chunks <= a.small_chunks ? AC_GATHER_SMALL : AC_GATHER) * hdr.nnz;
    if (gather) {
      // Small copies: 2 KB slices in turn, as in copy_small; others: chunks
      // claimed by warp, the next claim and its first member ahead of the copy.
      GatherRing& ring = reinterpret_cast<GatherRing*>(ac_smem)[warp];
      const bool slices = n_chunks <= a.small_chunks;
      const uint64_t unit = slices ? AC_SLICE : AC_CHUNK, n_units = ceil_div(S, unit);
      const uint64_t n_w = (uint64_t)n_part * (AC_THREADS / 32);
      uint64_t k = slices ? (uint64_t)blockIdx.x * (AC_THREADS / 32) + warp : 0, j0 = 0;
      const auto advance = [&]() {
        if (slices) {
          k += n_w;
        } else {
          uint32_t q = 0;
          if (lane == 0) q = atomicAdd(&ds->tile_ctr[TS_ASM_COPY], 1u);
          k = __shfl_sync(0xffffffffu, q, 0);
          if (k < n_units && c.ctfp) j0 = c.ctfp[k];
        }
      };
      if (!slices) advance();
      while (k < n_units) {
        const uint64_t ra = k * unit, rb = (ra + unit < S) ? ra + unit : S;
        uint64_t j = j0;
        if (slices || !c.ctfp) {
          uint64_t lo = 0, hi = hdr.nnz;
          if (c.ctfp) {   // the members of the slice's chunk
            const uint64_t q = ra / AC_CHUNK;
            lo = c.ctfp[q];
            if (q + 1 < n_chunks) hi = (uint64_t)c.ctfp[q + 1] + 1;
          }
          j = lo + warp_search(c.cpos + lo, hi - lo, ra, lane);
        }
        advance();
        gather_range(c, ring, ra, rb, j, lane);
      }
      outputs(threadIdx.x, AC_THREADS);
      __syncthreads();   // every warp's claims are done before the counter is reset
    } else if (n_chunks <= a.small_chunks) {
      copy_small(c, (uint64_t)blockIdx.x * (AC_THREADS / 32) + warp, (uint64_t)n_part * (AC_THREADS / 32),
                 lane);
      outputs(threadIdx.x, AC_THREADS);
    } else {
    if (threadIdx.x == 0) {
      for (int s = 0; s < AC_STAGES; ++s) {
        mbar_init(&full_bar[s], 1);
        mbar_init(&empty_bar[s], AC_CONSUMERS);
        s_issued[s] = 0u;
      }
      s_abort = 0u;
      rounds.start(blockIdx.x * AC_PRODUCERS);
      mbar_fence_init();
    }
    volatile uint32_t* abort = &s_abort;
    ChunkEntries* en = reinterpret_cast<ChunkEntries*>(ac_smem + AC_STAGES * sizeof(CopyStage)) + 2 * warp;
    const uint32_t nc = (uint32_t)n_chunks, dyn = n_part * AC_PRODUCERS;   // (dyn: the counter's first chunk)
    uint32_t next = dyn;
    ChunkRef cur{};
    if (warp < AC_PRODUCERS) {   // the first round, before anything is waited for
      if (warp == 0 && lane == 0 && nc > dyn)
        next = dyn + atomicAdd(&ds->tile_ctr[TS_ASM_COPY], (uint32_t)AC_PRODUCERS);
      const uint32_t k0 = blockIdx.x * AC_PRODUCERS + warp;
      if (k0 < nc) {
        cur = chunk_ref(c, k0, lane);
        fetch_entries(c, cur, en, lane);
      }
    }
    __syncthreads();
    if (warp < AC_PRODUCERS) {
      // Chunks are claimed in rounds of AC_PRODUCERS, the first by CTA index
      // and the rest from a counter the grid shares, so a CTA that starts late
      // (its SM busy with another stream's work) takes fewer: producer 0
      // claims a round ahead and hands it to the other producer at a named
      // barrier; stage index AC_PRODUCERS * r + warp holds the round's chunk
      // warp.  While a round is staged the next one's place in the chunk table
      // is read, and its plan entries are fetched behind it, so a producer
      // seldom waits for more than a free stage.  (Reading table and entries
      // at the round's start made the producers pace the copy of 512-byte
      // records: 1.71 ms for 4.7 GB, 1.43 so.  Two rounds ahead instead of one
      // left late CTAs more to finish alone, 7.75 ms per pass of 256 waves
      // against 7.64.)  Both producers leave at the same round (the barrier
      // needs both), and the first stage index left unfilled is marked done
      // for the consumers.
      uint32_t r = 0;
      bool lost = false;   // a wait for a stage gave up: nothing more is staged, the rounds go on until both leave
      for (;; ++r) {
        if (warp == 0 && lane == 0) {
          rounds.publish(r, next, *abort);
          if (next < nc)   // the claim of the following round, ahead
            next = dyn + atomicAdd(&ds->tile_ctr[TS_ASM_COPY], (uint32_t)AC_PRODUCERS);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        asm volatile("bar.sync 1, %0;" ::"r"(AC_PRODUCERS * 32) : "memory");
        if (rounds.leave(r, nc)) break;
        const uint32_t k = rounds.chunk(r) + warp, k1 = rounds.chunk(r + 1) + warp;
        const uint32_t i = AC_PRODUCERS * r + (uint32_t)warp;
        const uint32_t s = i % AC_STAGES, u = i / AC_STAGES;
        ChunkRef nxt{};
        if (k1 < nc) nxt = chunk_ref(c, k1, lane);
        asm volatile("cp.async.wait_group 0;" ::: "memory");   // this round's entries
        __syncwarp();
        if (!lost && u > 0) lost = !stage_wait2(&empty_bar[s], (u - 1u) & 1u, &ds->err, abort);
        if (!lost) {
          if (k < nc) {
            issue_chunk(c, cur, en + (r & 1u), &stages[s], &full_bar[s], lane);
          } else if (lane == 0) {   // the last round is short: the consumers stop here
            stages[s].np = AC_DONE;
            mbar_arrive(&full_bar[s]);
          }
          if (lane == 0) s_issued[s] = u + 1u;
          __syncwarp();
        }
        if (k1 < nc) fetch_entries(c, nxt, en + ((r + 1) & 1u), lane);
        cur = nxt;
      }
      const bool aborted = __any_sync(0xffffffffu, *abort != 0u);
      if (warp == 0 && !aborted) {   // the first stage index left unfilled
        const uint32_t i = AC_PRODUCERS * r;
        const uint32_t s = i % AC_STAGES, u = i / AC_STAGES;
        if (u == 0 || stage_wait2(&empty_bar[s], (u - 1u) & 1u, &ds->err, abort)) {
          if (lane == 0) {
            stages[s].np = AC_DONE;
            mbar_arrive(&full_bar[s]);
            s_issued[s] = u + 1u;
          }
        }
        __syncwarp();
      }
      // this lane's cp.async copies of small pieces land before the CTA can
      // exit (on an abort nobody else waits for them)
      asm volatile("cp.async.wait_all;" ::: "memory");
    } else {
      const uint32_t cw = (uint32_t)(warp - AC_PRODUCERS);
      outputs(threadIdx.x - AC_PRODUCERS * 32, AC_CONSUMERS * 32);
      for (uint32_t i = 0;; ++i) {
        const uint32_t s = i % AC_STAGES, u = i / AC_STAGES;
        if (!stage_wait2(&full_bar[s], u & 1u, &ds->err, abort)) break;
        const uint32_t np = stages[s].np;
        if (np == AC_DONE) break;
        if (np == AC_FALLBACK)
          emit_direct(c, &stages[s], cw, lane);
        else
          emit_range(&stages[s], cw, lane);
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty_bar[s]);
      }
    }
    __syncthreads();
    // a wait that gave up: give the copies still in flight a bounded chance
    // to land before the CTA's shared memory is released
    if (s_abort && threadIdx.x == 0) {
      for (int s = 0; s < AC_STAGES; ++s) {
        if (!s_issued[s]) continue;
        bool landed = false;
        for (uint32_t t = 0; t < (1u << 20) && !landed; ++t)
          landed = mbar_try_wait(&full_bar[s], (s_issued[s] - 1u) & 1u);
        // bulk copies still in flight as the CTA exits: recorded apart
        if (!landed) atomicOr(&ds->err, ERR_DRAIN);
      }
    }
    }
  }
  // this CTA's bytes are done: the next copy on the stream may be scheduled
  // into the space it leaves (it waits for this grid before it reads anything)
  allow_successor();
  if (threadIdx.x == 0) {
    if (ticket(&ds->exit_ctr[TS_ASM_COPY]) == n_part - 1) {
      if (!failed && a.cursor) *a.cursor = base + S;
      if (!failed && hdr.incomplete) ds->stats[6] += hdr.incomplete;
      if (a.out_bytes) *a.out_bytes = S;
      if (a.n_elems_out) *a.n_elems_out = hdr.M;
      ds->as_bytes = S;
      ds->as_elems = hdr.M;
      ds->tile_ctr[TS_ASM_COPY] = 0u;   // the chunk counter, for the next copy
      ds->exit_ctr[TS_ASM_COPY] = 0u;
    }
  }
}

void launch_assemble_plan(const LaunchCfg& L, const AssembleArgs& a) {
  if (a.user_list) {
    const uint64_t tiles = ceil_div(a.n_host, (uint64_t)AP_THREADS * AP_ITEMS);
    const int grid = (int)std::max<uint64_t>(1, std::min<uint64_t>(tiles, (uint64_t)L.grid_aparents));
    launch_k(L, K_APARENTS, asm_parents_kernel, grid, AP_THREADS, 0, a);
  }
  launch_assemble_members(L, a);
}

void launch_assemble_members(const LaunchCfg& L, const AssembleArgs& a) {
  // No more CTAs than the tiles of all members, or of the list's offsets.  A
  // commit completes, on average over an expansion, as many members as it
  // reports: twice those tiles, so that small commits' plans leave the SMs to
  // the scatters and copies beside them.
  uint64_t units = ceil_div(std::max<uint64_t>(a.plan.member_cap, a.n_host), (uint64_t)AM_TILE) + 1;
  if (a.for_commit) units = std::min<uint64_t>(units, 2 * ceil_div(a.n_reports, (uint64_t)AM_TILE) + 8);
  launch_k(L, K_AMEMBERS, asm_members_kernel, (int)std::min<uint64_t>(units, (uint64_t)L.grid_amembers), AM_THREADS,
           0, a);
}

void launch_assemble_copy(const LaunchCfg& L, const AssembleArgs& a) {
  launch_k(L, K_ACOPY, asm_copy_kernel, L.grid_acopy, AC_THREADS, asm_copy_smem(), a);
}

// opt in to the copy kernel's dynamic shared memory (AC_STAGES pipeline stages)
cudaError_t prepare_assemble_kernels() {
  return cudaFuncSetAttribute(asm_copy_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)asm_copy_smem());
}

// F.filter (Table 3) on a report batch: Present with a false mask -> Dropped
__global__ void filter_kernel(uint8_t* state, const uint8_t* keep, uint64_t n) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t r = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += stride)
    if (state[r] == ST_PRESENT && !keep[r]) state[r] = ST_DROPPED;
}

void launch_filter(cudaStream_t s, uint8_t* state, const uint8_t* keep, uint64_t n, int grid) {
  const uint64_t need = ceil_div(n, 256);
  const int g = (int)(need < (uint64_t)grid ? (need ? need : 1) : grid);
  filter_kernel<<<g, 256, 0, s>>>(state, keep, n);
}

const void* kernel_ptr_assemble(int which) {
  if (which == K_APARENTS) return (const void*)asm_parents_kernel;
  if (which == K_AMEMBERS) return (const void*)asm_members_kernel;
  return (const void*)asm_copy_kernel;
}

}  // namespace ro
