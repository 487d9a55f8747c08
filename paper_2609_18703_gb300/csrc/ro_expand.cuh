// ro_expand.cuh — the expansion's scan and fill, shared by expand_scan and
// expand_fill (k_expand.cu) and their allocation-free variants
// (ro_expand_noalloc.cu).
#pragma once

#include "ro_internal.h"

namespace ro {

// What a scan reads and writes.  Lineage outputs (offsets2, pw, gb, bitmap, n_heavy) are
// NULL where no lineage state is kept.
struct ScanIo {
  const uint32_t* counts;
  uint64_t P;
  uint64_t* offsets;              // the caller's
  uint64_t* offsets2;             // the context's copy
  unsigned long long* pw;         // per parent: remaining = count, bad = 0
  unsigned long long* gb;         // per parent: no GroupFailure barrier (0)
  uint32_t* bitmap;               // the completion bitmaps, 32 slots of a bit per parent: cleared
  uint32_t* empty_out;            // optional: ascending empty parents
  uint32_t* tfp;                  // fill tile -> parent of its first child
  uint64_t tfp_cap;
  TileStatus<Pair64> ts;
  unsigned long long epoch;
  uint32_t* tile_ctr;
  uint32_t* err;
  unsigned long long* n_children;
  unsigned long long* n_empty;
  unsigned long long* n_heavy;    // children of parents with at least HEAVY_CHILDREN children
};

// Element i of a tile in shared memory, padded by one per 16 so that threads
// reading 16 (or 4) consecutive elements each meet different banks.
__device__ __forceinline__ uint32_t scan_at(uint32_t i) { return i + (i >> 4); }
template <int ITEMS>
struct ScanShared {
  static constexpr uint32_t TILE = EXP_THREADS * ITEMS;
  unsigned long long off[TILE + TILE / 16];   // counts (as 32-bit words) first, then tile-relative offsets
  Pair64 scan[33];
  Pair64 prefix;
  uint32_t tile;
};

// Exclusive scan of the child counts, TILE = EXP_THREADS * ITEMS parents a
// tile, claimed in order; single pass with decoupled look-back.  Bound by
// memory for millions of parents (28 bytes each), by its chain (counts, block
// scan, look-back, writes) below.  Global accesses are striped over the
// threads, one element each, so they coalesce at any alignment of the
// caller's arrays; each thread scans ITEMS consecutive parents, handed over in
// shared memory.  (Loading and storing those consecutive parents directly
// took 256 us for 10M parents and 20 us for 50,000 in 13 tiles of 4,096; this
// takes 117 and 13.)
template <int ITEMS>
__device__ void scan_tiles(const ScanIo& a, ScanShared<ITEMS>& sh) {
  constexpr uint32_t TILE = ScanShared<ITEMS>::TILE;
  const uint64_t n_tiles = ceil_div(a.P, (uint64_t)TILE);
  uint32_t* s_cnt = reinterpret_cast<uint32_t*>(sh.off);
  for (;;) {
    if (threadIdx.x == 0) sh.tile = claim_tile(a.tile_ctr);
    __syncthreads();
    const uint32_t tile = sh.tile;
    if (tile >= n_tiles) break;
    const uint64_t p0 = (uint64_t)tile * TILE;
    uint32_t c[ITEMS];
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
      const uint64_t p = p0 + (uint32_t)k * EXP_THREADS + threadIdx.x;
      c[k] = p < a.P ? __ldg(a.counts + p) : 0u;
    }
    unsigned long long heavy = 0;
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
      const uint32_t i = (uint32_t)k * EXP_THREADS + threadIdx.x;
      s_cnt[scan_at(i)] = c[k];
      if (a.pw && p0 + i < a.P) {
        a.pw[p0 + i] = c[k];
        a.gb[p0 + i] = 0ull;
      }
      // (32 slots of P / 32 words, rounded up: a word per parent)
      if (a.bitmap && p0 + i < ((a.P + 31) & ~31ull)) a.bitmap[p0 + i] = 0u;
      heavy += c[k] >= HEAVY_CHILDREN ? c[k] : 0u;
    }
    if (a.n_heavy) {
      heavy = warp_sum(heavy);
      if ((threadIdx.x & 31) == 0 && heavy) atomicAdd(a.n_heavy, heavy);
    }
    __syncthreads();
    // this thread's consecutive parents
    const uint32_t i0 = threadIdx.x * ITEMS;
    Pair64 mine{0, 0};
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
      c[k] = s_cnt[scan_at(i0 + k)];
      mine.a += c[k];
      mine.b += (p0 + i0 + k < a.P && c[k] == 0u) ? 1ull : 0ull;
    }
    Pair64 total;
    const Pair64 excl = block_excl_scan_pair(mine, sh.scan, &total);   // (its barriers: every count was read)
    {
      unsigned long long run = excl.a;
#pragma unroll
      for (int k = 0; k < ITEMS; ++k) {
        sh.off[scan_at(i0 + k)] = run;
        run += c[k];
      }
    }
    if (threadIdx.x < 32) {   // one warp looks back
      const Pair64 pfx = lookback_exclusive(a.ts, tile, total, a.epoch, a.err);
      if (threadIdx.x == 0) sh.prefix = pfx;
    }
    __syncthreads();
    const Pair64 pre = sh.prefix;
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
      const uint32_t i = (uint32_t)k * EXP_THREADS + threadIdx.x;
      if (p0 + i >= a.P) break;
      const uint64_t o = pre.a + sh.off[scan_at(i)];
      a.offsets[p0 + i] = o;
      if (a.offsets2) a.offsets2[p0 + i] = o;
    }
    Pair64 run = pre + excl;
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
      const uint64_t p = p0 + i0 + k, o = run.a, m = c[k];
      if (p >= a.P) break;
      if (m == 0) {
        if (a.empty_out) a.empty_out[run.b] = (uint32_t)p;
        run.b += 1;
      } else {
        // fill tiles whose first child is a child of p
        for (uint64_t b = ceil_div(o, FILL_TILE); b * FILL_TILE < o + m && b < a.tfp_cap; ++b)
          a.tfp[b] = (uint32_t)p;
      }
      run.a += m;
    }
    if (tile == n_tiles - 1 && threadIdx.x == 0) {
      const Pair64 all = pre + total;
      a.offsets[a.P] = all.a;
      if (a.offsets2) a.offsets2[a.P] = all.a;
      *a.n_children = all.a;
      *a.n_empty = all.b;
    }
    __syncthreads();   // the next tile reuses the shared memory
  }
}

// Up to this many parents a tile has 4 per thread, so that a small expansion
// spreads over the SMs; more have 16, which keeps the look-back short (128
// tiles of 1,024 at the line).
constexpr uint64_t SCAN_SMALL = 128ull * EXP_THREADS * 4;
__host__ __device__ __forceinline__ uint64_t scan_tile(uint64_t P) {
  return (uint64_t)EXP_THREADS * (P <= SCAN_SMALL ? 4 : EXP_ITEMS);
}

// What a fill reads and writes.  Lineage outputs (slot, par) are NULL where no
// lineage state is kept.
struct FillIo {
  const uint64_t* offsets;
  uint64_t P, N;
  const uint32_t* tfp;
  const uint8_t* parent_call;   // optional
  uint32_t* child_parent;
  uint32_t* child_ordinal;
  Slot* slot;
  uint32_t* par;
};
struct FillShared {
  uint32_t off[FILL_SMEM_CAP];   // offsets of the parents the tile touches (children number below 2^32)
};

// Largest index k in [lo, hi) with v[k] <= x (v non-decreasing, v[lo] <= x).
template <class V, class I>
__device__ __forceinline__ I last_le(const V* v, I lo, I hi, V x) {
  while (hi - lo > 1) {
    const I mid = lo + ((hi - lo) >> 1);
    if (v[mid] <= x)
      lo = mid;
    else
      hi = mid;
  }
  return lo;
}

// Every child of a FILL_TILE-child tile gets its parent and ordinal, and with
// lineage state its parent and its slot (WAITING, unclaimed).  Bound by memory
// once the search is cheap: a thread takes 4 consecutive children, finds the
// first one's parent by binary search among the tile's staged offsets and the
// others' from it (the same parent, the next, or a search past runs of empty
// ones), and stores 16 bytes per array where the caller's arrays are aligned;
// a warp's slots go out 32 consecutive ones per store, beside the other
// arrays (after them, in a pass of their own, they took 710 us for 110M
// children; 543 so).  The search counts in 32 bits (children number below
// 2^32).  A search per child, in 64 bits, took 83 us for 16.4M children of 1M
// parents without lineage state (8 bytes each); one per thread 39 us, and
// 36 us in 32 bits.
__device__ __forceinline__ void fill_tiles(const FillIo& a, FillShared& sh) {
  const uint64_t n_tiles = ceil_div(a.N, FILL_TILE);
  const bool vec = (((uintptr_t)a.child_parent | (uintptr_t)a.child_ordinal) & 15u) == 0;
  for (uint64_t t = blockIdx.x; t < n_tiles; t += gridDim.x) {
    const uint64_t c0 = t * FILL_TILE, c1 = min(c0 + FILL_TILE, a.N);
    const uint64_t p_lo = a.tfp[t];
    const uint64_t p_hi = (t + 1 < n_tiles) ? a.tfp[t + 1] : a.P - 1;
    const uint64_t R = p_hi - p_lo + 2;   // offsets[p_lo .. p_hi+1]
    const bool staged = R <= FILL_SMEM_CAP;
    if (staged)
      for (uint32_t k = threadIdx.x; k < (uint32_t)R; k += FILL_THREADS) sh.off[k] = (uint32_t)a.offsets[p_lo + k];
    __syncthreads();
    for (uint64_t cc = c0 + (threadIdx.x & ~31u) * 4; cc < c1; cc += 4 * FILL_THREADS) {   // 128 children a warp
      const uint64_t c = cc + 4 * (threadIdx.x & 31);
      const int n = c >= c1 ? 0 : c1 - c < 4 ? (int)(c1 - c) : 4;
      uint32_t p[4], o[4];
      if (staged && n) {
        const uint32_t last = (uint32_t)R - 1u;   // offsets[p_hi + 1] is past every child of the tile
        const uint32_t c32 = (uint32_t)c;
        uint32_t k = last_le(sh.off, 0u, last, c32);
        uint32_t base = sh.off[k], next = sh.off[k + 1];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (j < n && c32 + j >= next) {
            ++k;
            if (k + 1 < last && sh.off[k + 1] <= c32 + j) k = last_le(sh.off, k + 1, last, c32 + j);
            base = sh.off[k];
            next = sh.off[k + 1];
          }
          p[j] = (uint32_t)p_lo + k;
          o[j] = c32 + j - base;
        }
      } else if (n) {   // many empty parents inside one tile: search the global offsets
        for (int j = 0; j < 4; ++j) {
          const uint64_t q = j < n ? last_le(a.offsets, p_lo, p_hi + 1, c + j) : p_lo;
          p[j] = (uint32_t)q;
          o[j] = (uint32_t)(c + j - a.offsets[q]);
        }
      }
      if (a.slot) {   // the warp's 128 slots, 32 consecutive ones per store
        uint32_t calls = 0;   // of this thread's children, a byte each
        if (a.parent_call)
          for (int j = 0; j < n; ++j) calls |= (uint32_t)a.parent_call[p[j]] << (8 * j);
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint32_t x = (uint32_t)j * 32 + (threadIdx.x & 31);
          const uint32_t call = (__shfl_sync(0xffffffffu, calls, x >> 2) >> (8 * (x & 3))) & 255u;
          if (cc + x < c1)
            *reinterpret_cast<uint4*>(a.slot + cc + x) = make_uint4(WAIT_UNCLAIMED, 0u, 0u, call << (W_CALL_SHIFT - 32));
        }
      }
      if (n == 4 && vec) {
        *reinterpret_cast<uint4*>(a.child_parent + c) = make_uint4(p[0], p[1], p[2], p[3]);
        *reinterpret_cast<uint4*>(a.child_ordinal + c) = make_uint4(o[0], o[1], o[2], o[3]);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (j < n) {
            a.child_parent[c + j] = p[j];
            a.child_ordinal[c + j] = o[j];
          }
      }
      if (a.par) {   // (the context's array is aligned)
        if (n == 4) {
          *reinterpret_cast<uint4*>(a.par + c) = make_uint4(p[0], p[1], p[2], p[3]);
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (j < n) a.par[c + j] = p[j];
        }
      }
    }
    __syncthreads();
  }
}

}  // namespace ro
