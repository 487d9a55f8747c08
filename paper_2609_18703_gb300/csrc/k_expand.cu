// k_expand.cu — ro_expand kernels (Section 4.2; Table 2 child key; Eq. 1).
//
// expand_scan: single-pass exclusive scan of the child counts with
//   decoupled look-back (ro_expand.cuh).  Alongside the offsets it
//   initialises each parent's terminal counter (remaining = count), lists
//   the empty parents (a second prefix sum carried in the same scan), and
//   records for every fill tile (4096 children) the parent of its first child,
//   so that the fill needs no search in global memory.
// expand_fill: one CTA per 4096-child tile stages the offsets of the parents
//   that tile touches in shared memory and gives every child its parent and
//   ordinal (ro_expand.cuh); it also initialises the child's Grain phase
//   (WAITING, unclaimed) and result record.  Work per CTA is bounded by the
//   tile, so one 100k-child parent spreads over 25 tiles instead of
//   serialising a warp.
#include <algorithm>

#include "ro_expand.cuh"

namespace ro {

// The last CTA's totals, straight to the host (which waits for seq instead of
// for a copy and the stream); n_heavy starts the next scan at zero.
__device__ __forceinline__ void report(const ExpandScanArgs& a) {
  DevScalars* ds = a.ds;
  volatile ExpandReport* h = a.report;
  h->n_children = __ldcg(&ds->n_children);
  h->n_empty = __ldcg(&ds->n_empty);
  h->n_heavy = __ldcg(&ds->n_heavy);
  h->err = __ldcg(&ds->err);
  ds->n_heavy = 0;
  __threadfence_system();
  h->seq = a.seq;
}

template <int ITEMS>
__global__ void __launch_bounds__(EXP_THREADS, 3) expand_scan_kernel(ExpandScanArgs a) {
  wait_predecessor();
  __shared__ ScanShared<ITEMS> sh;
  const uint64_t n_tiles = ceil_div(a.P, (uint64_t)EXP_THREADS * ITEMS);
  DevScalars* ds = a.ds;
  if (n_tiles == 0) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      a.offsets_user[0] = 0;
      a.offsets[0] = 0;
      ds->n_children = 0;
      ds->n_empty = 0;
      report(a);
    }
    return;
  }
  const uint32_t n_part = participants(n_tiles);
  if (blockIdx.x >= n_part) return;
  ScanIo io{};
  io.counts = a.counts;
  io.P = a.P;
  io.offsets = a.offsets_user;
  io.offsets2 = a.offsets;
  io.pw = a.pw;
  io.empty_out = a.empty_out;
  io.tfp = a.tfp;
  io.tfp_cap = a.tfp_cap;
  io.ts = a.ts;
  io.epoch = ds->epoch[TS_EXPAND];
  io.tile_ctr = &ds->tile_ctr[TS_EXPAND];
  io.err = &ds->err;
  io.n_children = &ds->n_children;
  io.n_empty = &ds->n_empty;
  io.n_heavy = &ds->n_heavy;
  io.gb = a.gb;
  io.bitmap = a.bitmap;
  scan_tiles<ITEMS>(io, sh);
  if (threadIdx.x == 0 && retire_cta(ds, TS_EXPAND, n_part)) report(a);
}

__global__ void __launch_bounds__(FILL_THREADS, 5) expand_fill_kernel(ExpandFillArgs a) {
  wait_predecessor();
  __shared__ FillShared sh;
  fill_tiles(FillIo{a.offsets, a.P, a.N, a.tfp, a.parent_call, a.child_parent, a.child_ordinal, a.slot, a.par}, sh);
}

void launch_expand_scan(const LaunchCfg& L, const ExpandScanArgs& a) {
  const uint64_t tiles = std::max<uint64_t>(1, ceil_div(a.P, scan_tile(a.P)));
  launch_k(L, K_EXPAND_SCAN, a.P <= SCAN_SMALL ? expand_scan_kernel<4> : expand_scan_kernel<EXP_ITEMS>,
           (int)std::min<uint64_t>(tiles, (uint64_t)L.grid_expand_scan), EXP_THREADS, 0, a);
}

void launch_expand_fill(const LaunchCfg& L, const ExpandFillArgs& a) {
  const uint64_t n_tiles = ceil_div(a.N, FILL_TILE);
  if (n_tiles == 0) return;
  const int grid = (int)std::min<uint64_t>(n_tiles, (uint64_t)L.grid_fill);
  launch_k(L, K_FILL, expand_fill_kernel, grid, FILL_THREADS, 0, a);
}

uint64_t expand_scan_tiles(uint64_t P) { return ceil_div(P, scan_tile(P)); }

const void* kernel_ptr_expand(int which) {
  return which == K_EXPAND_SCAN ? (const void*)expand_scan_kernel<EXP_ITEMS> : (const void*)expand_fill_kernel;
}

}  // namespace ro
