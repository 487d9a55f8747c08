// k_parent.cu — parent-bound reservation (Section 4.3): each reservation
// takes up to B queued siblings of the parent of the queue's first entry and
// leaves the other entries in order.
//
// Repeated reservations have a closed form, which these kernels compute in
// parallel: rank every queued entry among its parent's queued entries (queue
// order) and cut each parent's entries into chunks of B; the reservations
// take exactly these chunks, in increasing queue position of each chunk's
// first entry (without flush, up to the first chunk shorter than B).  The
// ranks come from a stable sort of the window by parent id.
//
//   pb_keys     window copy: child, parent (sort key), position (sort value);
//               clears the per-position chunk sizes and marks; per tile digit
//               counts of the first pass
//   pb_hist     the same counts for a later pass
//   pb_rowscan  per digit, exclusive scan over tiles; digit totals
//   pb_sort     stable scatter of one digit pass (warp match + per-warp counts)
//   pb_bounds   per parent, sorted range of its entries
//   pb_heads    sorted order: each chunk's first entry records the chunk size
//               at its queue position; the first short chunk (no flush)
//   pb_mark     sorted order, no flush only: marks entries of chunks at or
//               after the first short chunk, which stay queued
//   pb_scan     queue order, single-pass scan (decoupled look-back): output
//               offset of each taken chunk, batch boundaries, entries left
//   pb_emit     sorted order: writes each taken chunk's entries contiguously
//               (IN-FLIGHT) and the queue's remainder, or on a refusal
//               (capacity) undoes the admission
// Only chunk heads (about one entry in B) and marked entries are written by
// queue position; everything else moves in sorted order.
// The admission itself (launch_ready with parent_bound set)
// runs first and queues every admitted Grain.
#include <algorithm>

#include "ro_internal.h"

namespace ro {

constexpr int PB_U = 4;   // entries per thread and step of the sorted-order kernels: their dependent loads go out together

__device__ __forceinline__ uint64_t pb_tiles(uint64_t Q) { return ceil_div(Q, (uint64_t)PB_TILE); }

// A tile's digit counts of pass a.pass, from its keys (item k of a thread is
// entry k * PB_THREADS + thread; in: bit k, the entry exists), into its row.
__device__ __forceinline__ void count_digits(const ParentArgs& a, uint64_t t, const uint32_t (&key)[PB_ITEMS],
                                             uint32_t in, uint32_t* s_h) {
  const uint32_t D = 1u << a.dbits;
  const int shift = a.dbits * a.pass;
  for (uint32_t d = threadIdx.x; d < D; d += PB_THREADS) s_h[d] = 0u;
  __syncthreads();
#pragma unroll
  for (int k = 0; k < PB_ITEMS; ++k)
    if ((in >> k) & 1u) atomicAdd(&s_h[(key[k] >> shift) & (D - 1u)], 1u);
  __syncthreads();
  for (uint32_t d = threadIdx.x; d < D; d += PB_THREADS) a.hist[t * D + d] = s_h[d];
  __syncthreads();
}

// Two dependent random loads an entry (queue, parent): a tile's are all in
// flight together.
__global__ void __launch_bounds__(PB_THREADS) pb_keys_kernel(ParentArgs a) {
  wait_predecessor();
  __shared__ uint32_t s_h[PB_DIGITS];
  const DevScalars* ds = a.ds;
  const uint64_t Q = ds->pb_Q, head = ds->pb_head, T = pb_tiles(Q);
  for (uint64_t t = blockIdx.x; t < T; t += gridDim.x) {
    const uint64_t j0 = t * PB_TILE + threadIdx.x;
    uint32_t c[PB_ITEMS], p[PB_ITEMS], in = 0u;
#pragma unroll
    for (int k = 0; k < PB_ITEMS; ++k) {
      const uint64_t j = j0 + (uint64_t)k * PB_THREADS;
      if (j < Q) in |= 1u << k;
      c[k] = j < Q ? a.queue[head + j] : 0u;
    }
#pragma unroll
    for (int k = 0; k < PB_ITEMS; ++k) p[k] = (in >> k) & 1u ? a.par[c[k]] : 0u;
#pragma unroll
    for (int k = 0; k < PB_ITEMS; ++k) {
      if (!((in >> k) & 1u)) continue;
      const uint64_t j = j0 + (uint64_t)k * PB_THREADS;
      a.child[j] = c[k];
      a.key[0][j] = p[k];
      if (a.passes == 0) a.val[0][j] = (uint32_t)j;   // (the first pass makes the positions up)
      a.hsz[j] = 0u;
      a.left[j] = 0u;
    }
    if (a.passes) count_digits(a, t, p, in, s_h);
  }
}

__global__ void __launch_bounds__(PB_THREADS) pb_hist_kernel(ParentArgs a) {
  wait_predecessor();
  __shared__ uint32_t s_h[PB_DIGITS];
  const uint64_t Q = a.ds->pb_Q, T = pb_tiles(Q);
  const uint32_t* key = a.key[a.pass & 1];
  for (uint64_t t = blockIdx.x; t < T; t += gridDim.x) {
    uint32_t kk[PB_ITEMS], in = 0u;
#pragma unroll
    for (int k = 0; k < PB_ITEMS; ++k) {
      const uint64_t i = t * PB_TILE + (uint64_t)k * PB_THREADS + threadIdx.x;
      if (i < Q) in |= 1u << k;
      kk[k] = i < Q ? key[i] : 0u;
    }
    count_digits(a, t, kk, in, s_h);
  }
}

// PB_ROW_DIGITS digits per CTA: exclusive scan of each one's counts over the
// tiles.  A thread owns one digit of a contiguous range of tiles (a sector
// holds the CTA's digits of one tile) and reads it twice, 8 loads in flight.
__global__ void __launch_bounds__(PB_ROW_THREADS) pb_rowscan_kernel(ParentArgs a) {
  wait_predecessor();
  constexpr int NL = PB_ROW_THREADS / PB_ROW_DIGITS, NW = PB_ROW_THREADS / 32;
  static_assert(PB_ROW_DIGITS == 8 && NW == 32, "a warp holds 4 ranges of 8 digits; one warp scans a digit's 32 sums");
  __shared__ uint32_t s_w[NW][PB_ROW_DIGITS];
  const uint64_t T = pb_tiles(a.ds->pb_Q), D = 1ull << a.dbits;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, dl = threadIdx.x % PB_ROW_DIGITS;
  const uint64_t d = (uint64_t)blockIdx.x * PB_ROW_DIGITS + dl;
  const uint64_t per = ceil_div(T, (uint64_t)NL);
  const uint64_t t0 = min((threadIdx.x / PB_ROW_DIGITS) * per, T), t1 = min(t0 + per, T);
  const bool ok = d < D;   // fewer digits than the CTA holds
  constexpr int U = 8;
  uint32_t sum = 0;
  for (uint64_t t = t0; ok && t < t1; t += U) {
#pragma unroll
    for (int u = 0; u < U; ++u) sum += t + u < t1 ? a.hist[(t + u) * D + d] : 0u;
  }
  uint32_t inc = sum;
#pragma unroll
  for (int sh = PB_ROW_DIGITS; sh < 32; sh *= 2) {
    const uint32_t x = __shfl_up_sync(0xffffffffu, inc, sh);
    if (lane >= sh) inc += x;
  }
  if (lane >= 32 - PB_ROW_DIGITS) s_w[w][dl] = inc;
  __syncthreads();
  if (w < PB_ROW_DIGITS) {   // warp w: digit w's sums over the warps
    const uint32_t v = s_w[lane][w];
    uint32_t x = v;
#pragma unroll
    for (int sh = 1; sh < 32; sh <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, sh);
      if (lane >= sh) x += y;
    }
    s_w[lane][w] = x - v;
    const uint64_t dw = (uint64_t)blockIdx.x * PB_ROW_DIGITS + w;
    if (lane == 31 && dw < D) a.dtot[dw] = x;
  }
  __syncthreads();
  uint32_t run = s_w[w][dl] + inc - sum;
  for (uint64_t t = t0; ok && t < t1; t += U) {
    uint32_t v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) v[u] = t + u < t1 ? a.hist[(t + u) * D + d] : 0u;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (t + u >= t1) break;
      a.hist[(t + u) * D + d] = run;
      run += v[u];
    }
  }
}

// Stable scatter of one digit pass.  Warp w of a tile owns entries
// [w*256, (w+1)*256) of the tile and walks them 32 at a time in order; lanes
// holding the same digit find each other with a warp match and take
// consecutive places after the warp's running count of that digit.  The
// warps' counts are then scanned per digit, so places follow tile order,
// warp order, round order and lane order: the original order.
// The tile's entries go out through shared memory in digit order, so that a
// warp's stores are a few runs; 22 KB of it (the counts' room), because other
// contexts' kernels share the SM (with 45 KB: 30 us alone for 2.05M entries
// but three contexts in turn 600 us a pass instead of 420).  Digits of up to
// 10 bits: 250,000 parents take 2 passes of 9 bits at 32 us, where 8-bit
// digits stored straight from registers took 41 + 41 + 21 us and a histogram
// and a scan more.  The positions are loaded after the ranking, for registers.
__global__ void __launch_bounds__(PB_THREADS, 5) pb_sort_kernel(ParentArgs a) {
  wait_predecessor();
  constexpr int NW = PB_THREADS / 32, DT = PB_DIGITS / PB_THREADS;
  __shared__ union {
    uint16_t cnt[NW][PB_DIGITS];              // at most 256 of a digit per warp, 2,048 per tile
    struct {
      uint32_t key[PB_TILE], val[PB_TILE];    // the tile's entries in digit order, once the counts are read
    } out;
  } sh;
  __shared__ uint16_t s_lbase[PB_DIGITS];     // the tile's entries of smaller digits
  __shared__ uint32_t s_gbase[PB_DIGITS];     // output place of a digit's entry less its place in the tile
  __shared__ uint32_t s_scan[33];
  const uint64_t Q = a.ds->pb_Q, T = pb_tiles(Q);
  const uint32_t* kin = a.key[a.pass & 1];
  const uint32_t* vin = a.val[a.pass & 1];
  uint32_t* kout = a.key[(a.pass + 1) & 1];
  uint32_t* vout = a.val[(a.pass + 1) & 1];
  const uint32_t D = 1u << a.dbits;
  const int shift = a.dbits * a.pass;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (blockIdx.x >= T) return;
  uint32_t dbase[DT];   // the window's entries of digits below this thread's DT consecutive ones
  {
    uint32_t v[DT], sum = 0, tot;
#pragma unroll
    for (int k = 0; k < DT; ++k) {
      const uint32_t d = threadIdx.x * DT + k;
      v[k] = d < D ? a.dtot[d] : 0u;
      sum += v[k];
    }
    uint32_t ex = block_excl_scan(sum, s_scan, &tot);
#pragma unroll
    for (int k = 0; k < DT; ++k) {
      dbase[k] = ex;
      ex += v[k];
    }
  }
  for (uint64_t t = blockIdx.x; t < T; t += gridDim.x) {
    const uint64_t base = t * PB_TILE + (uint64_t)w * (32 * PB_ITEMS) + lane;
    uint32_t kk[PB_ITEMS], vv[PB_ITEMS];
    uint32_t lo[PB_ITEMS / 2] = {};   // places among the warp's entries of the digit, two to a register
#pragma unroll
    for (int r = 0; r < PB_ITEMS; ++r) kk[r] = base + r * 32 < Q ? kin[base + r * 32] : 0u;
    for (uint32_t d = lane; d < D; d += 32) sh.cnt[w][d] = 0u;
    __syncwarp();
#pragma unroll
    for (int r = 0; r < PB_ITEMS; ++r) {
      const bool valid = base + r * 32 < Q;
      const uint32_t d = valid ? (kk[r] >> shift) & (D - 1u) : D;
      const uint32_t peers = __match_any_sync(0xffffffffu, d);
      const uint32_t before = __popc(peers & ((1u << lane) - 1u));
      const uint32_t run = valid ? sh.cnt[w][d] : 0u;
      __syncwarp();
      if (valid && before == 0u) sh.cnt[w][d] = (uint16_t)(run + __popc(peers));
      __syncwarp();
      lo[r / 2] |= (run + before) << (16 * (r % 2));
    }
#pragma unroll
    for (int r = 0; r < PB_ITEMS; ++r)
      vv[r] = a.pass == 0 ? (uint32_t)(base + r * 32) : base + r * 32 < Q ? vin[base + r * 32] : 0u;
    __syncthreads();
    // a thread owns DT consecutive digits: the warps' counts become places
    // within the digit, the digits' totals places within the tile
    uint32_t tot[DT] = {}, sum = 0, all;
#pragma unroll
    for (int k = 0; k < DT; ++k) {
      const uint32_t d = threadIdx.x * DT + k;
      if (d >= D) break;
#pragma unroll
      for (int w2 = 0; w2 < NW; ++w2) {
        const uint32_t c = sh.cnt[w2][d];
        sh.cnt[w2][d] = (uint16_t)tot[k];
        tot[k] += c;
      }
      sum += tot[k];
    }
    uint32_t ex = block_excl_scan(sum, s_scan, &all);
#pragma unroll
    for (int k = 0; k < DT; ++k) {
      const uint32_t d = threadIdx.x * DT + k;
      if (d >= D) break;
      s_lbase[d] = (uint16_t)ex;
      s_gbase[d] = dbase[k] + a.hist[t * D + d] - ex;
      ex += tot[k];
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < PB_ITEMS; ++r) {
      if (base + r * 32 >= Q) continue;
      const uint32_t d = (kk[r] >> shift) & (D - 1u);
      lo[r / 2] += (uint32_t)(s_lbase[d] + sh.cnt[w][d]) << (16 * (r % 2));   // places in the tile, below 2,048
    }
    __syncthreads();   // the counts are read
#pragma unroll
    for (int r = 0; r < PB_ITEMS; ++r) {
      if (base + r * 32 >= Q) continue;
      const uint32_t l = (lo[r / 2] >> (16 * (r % 2))) & 0xFFFFu;
      sh.out.key[l] = kk[r];
      sh.out.val[l] = vv[r];
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < PB_ITEMS; ++r) {
      const uint32_t l = r * PB_THREADS + threadIdx.x;
      if (l >= all) break;
      const uint32_t key = sh.out.key[l], o = s_gbase[(key >> shift) & (D - 1u)] + l;
      kout[o] = key;
      vout[o] = sh.out.val[l];
    }
    __syncthreads();
  }
}

__global__ void __launch_bounds__(PB_THREADS) pb_bounds_kernel(ParentArgs a) {
  wait_predecessor();
  const uint64_t Q = a.ds->pb_Q;
  const uint32_t* key = a.key[a.passes & 1];
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t s = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; s < Q; s += stride) {
    const uint32_t p = key[s];
    if (s == 0 || key[s - 1] != p) a.first[p] = (uint32_t)s;
    if (s + 1 == Q || key[s + 1] != p) a.endp[p] = (uint32_t)(s + 1);
  }
}

// Sorted order: the first entry of each chunk (rank a multiple of B among
// its parent's entries) records the chunk's size at its queue position.
__global__ void __launch_bounds__(PB_THREADS) pb_heads_kernel(ParentArgs a) {
  wait_predecessor();
  DevScalars* ds = a.ds;
  const uint64_t Q = ds->pb_Q;
  const uint32_t* key = a.key[a.passes & 1];
  const uint32_t* val = a.val[a.passes & 1];
  const uint32_t B = a.B;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t s0 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; s0 < Q; s0 += PB_U * stride) {
    uint32_t p[PB_U], f[PB_U];
#pragma unroll
    for (int u = 0; u < PB_U; ++u) p[u] = s0 + u * stride < Q ? key[s0 + u * stride] : 0u;
#pragma unroll
    for (int u = 0; u < PB_U; ++u) f[u] = s0 + u * stride < Q ? a.first[p[u]] : 0u;
#pragma unroll
    for (int u = 0; u < PB_U; ++u) {
      const uint64_t s = s0 + u * stride;
      if (s >= Q || ((uint32_t)s - f[u]) % B != 0u) continue;
      const uint32_t i = val[s];
      const uint32_t sz = min(B, a.endp[p[u]] - (uint32_t)s);
      a.hsz[i] = sz;
      if (!a.flush && sz < B) atomicMin(&ds->pb_stop, (unsigned long long)i);
    }
  }
}

// Sorted order, only when a short chunk stops the reservations: entries of
// chunks whose first entry is at or after the stop stay queued.
__global__ void __launch_bounds__(PB_THREADS) pb_mark_kernel(ParentArgs a) {
  wait_predecessor();
  const DevScalars* ds = a.ds;
  const unsigned long long stop = ds->pb_stop;
  if (stop == ~0ull) return;
  const uint64_t Q = ds->pb_Q;
  const uint32_t* key = a.key[a.passes & 1];
  const uint32_t* val = a.val[a.passes & 1];
  const uint32_t B = a.B;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t s = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; s < Q; s += stride) {
    const uint32_t f = a.first[key[s]];
    const uint32_t r = (uint32_t)s - f;
    const uint32_t hw = val[f + (r - r % B)];   // queue position of the chunk's first entry
    if (hw >= stop) a.left[val[s]] = 1u;
  }
}

__global__ void __launch_bounds__(PB_SCAN_THREADS) pb_scan_kernel(ParentArgs a) {
  wait_predecessor();
  __shared__ Pair64 s_scan[33];
  __shared__ uint32_t s_tile;
  __shared__ Pair64 s_prefix;
  DevScalars* ds = a.ds;
  const uint64_t Q = ds->pb_Q;
  const unsigned long long stop = ds->pb_stop;
  const uint32_t B = a.B;
  const uint64_t n_tiles = ceil_div(Q, (uint64_t)PB_SCAN_THREADS * PB_ITEMS);
  if (n_tiles == 0) {   // empty window: nothing taken, nothing left
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      ds->pb_npop = ds->pb_nb = ds->pb_R = 0;
      if (a.batch_off && a.off_cap < 1) {
        ds->pb_err = 1u;
        atomicOr(&ds->err, ERR_CAPACITY);
      } else if (a.batch_off) {
        a.batch_off[0] = 0;
      }
      if (a.n_batched_out) *a.n_batched_out = 0;
      if (a.n_batches_out) *a.n_batches_out = 0;
    }
    return;
  }
  const uint32_t n_part = participants(n_tiles);
  if (blockIdx.x >= n_part) return;
  for (;;) {
    if (threadIdx.x == 0) s_tile = claim_tile(&ds->tile_ctr[TS_PARENT]);
    __syncthreads();
    const uint32_t tile = s_tile;
    __syncthreads();
    if (tile >= n_tiles) break;
    const uint64_t i0 = (uint64_t)tile * (PB_SCAN_THREADS * PB_ITEMS) + (uint64_t)threadIdx.x * PB_ITEMS;
    // a: entries of the taken chunks; b: taken chunks << 32 | entries left
    Pair64 mine{0, 0};
    uint32_t take_head = 0, left = 0, sz[PB_ITEMS], lf[PB_ITEMS / 4] = {};
    static_assert(PB_ITEMS == 8, "a thread's 8 sizes are two 16-byte loads, its marks one of 8 bytes");
    if (i0 + PB_ITEMS <= Q) {
      *reinterpret_cast<uint4*>(sz) = *reinterpret_cast<const uint4*>(a.hsz + i0);
      *reinterpret_cast<uint4*>(sz + 4) = *reinterpret_cast<const uint4*>(a.hsz + i0 + 4);
      *reinterpret_cast<uint2*>(lf) = *reinterpret_cast<const uint2*>(a.left + i0);
    } else {
#pragma unroll
      for (int k = 0; k < PB_ITEMS; ++k) {
        sz[k] = i0 + k < Q ? a.hsz[i0 + k] : 0u;
        lf[k / 4] |= (i0 + k < Q ? (uint32_t)a.left[i0 + k] : 0u) << (8 * (k % 4));
      }
    }
#pragma unroll
    for (int k = 0; k < PB_ITEMS; ++k) {
      const uint64_t i = i0 + k;
      if (i >= Q) continue;
      if ((lf[k / 4] >> (8 * (k % 4))) & 0xFFu) {
        left |= 1u << k;
        mine.b += 1;
      } else if (sz[k] != 0u && i < stop) {
        take_head |= 1u << k;
        mine.a += sz[k];
        mine.b += 1ull << 32;
      }
    }
    Pair64 total;
    const Pair64 excl = block_excl_scan_pair(mine, s_scan, &total);
    if (threadIdx.x < 32) {  // one warp looks back
      const Pair64 pfx = lookback_exclusive(a.ts, tile, total, ds->epoch[TS_PARENT], &ds->err);
      if (threadIdx.x == 0) s_prefix = pfx;
    }
    __syncthreads();
    Pair64 run = s_prefix + excl;
#pragma unroll
    for (int k = 0; k < PB_ITEMS; ++k) {
      const uint64_t i = i0 + k;
      if (take_head & (1u << k)) {
        a.hoff[i] = (uint32_t)run.a;
        const uint64_t b = run.b >> 32;
        if (a.batch_off && b < a.off_cap) a.batch_off[b] = run.a;
        run.a += sz[k];
        run.b += 1ull << 32;
      } else if (left & (1u << k)) {
        a.rem[run.b & 0xFFFFFFFFull] = a.child[i];
        run.b += 1;
      }
    }
    if (tile == n_tiles - 1 && threadIdx.x == PB_SCAN_THREADS - 1) {
      const unsigned long long npop = run.a, nb = run.b >> 32, R = run.b & 0xFFFFFFFFull;
      ds->pb_npop = npop;
      ds->pb_nb = nb;
      ds->pb_R = R;
      if (a.n_batched_out) *a.n_batched_out = npop;
      if (a.n_batches_out) *a.n_batches_out = nb;
      if (npop > a.cap || (a.batch_off && nb + 1 > a.off_cap)) {
        ds->pb_err = 1u;
        atomicOr(&ds->err, ERR_CAPACITY);
      } else if (a.batch_off) {
        a.batch_off[nb] = npop;
      }
    }
  }
  if (threadIdx.x == 0) retire_cta(ds, TS_PARENT, n_part);
}

__global__ void __launch_bounds__(PB_THREADS) pb_emit_kernel(ParentArgs a) {
  wait_predecessor();
  DevScalars* ds = a.ds;
  const uint64_t Q = ds->pb_Q, head = ds->pb_head;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  const uint64_t g = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (ds->pb_err) {
    // refused: the admitted Grains go back to WAITING, the tail back
    const uint64_t t0 = ds->pb_old_tail, t1 = head + Q;
    for (uint64_t t = t0 + g; t < t1; t += stride) a.slot[a.queue[t]].phase = WAIT_UNCLAIMED;
    if (g == 0) a.qstate[1] = t0;
    return;
  }
  const unsigned long long stop = ds->pb_stop, npop = ds->pb_npop, R = ds->pb_R;
  const uint32_t* key = a.key[a.passes & 1];
  const uint32_t* val = a.val[a.passes & 1];
  const uint32_t B = a.B;
  // sorted order: a taken chunk's entries are consecutive here and in the
  // output, so the writes to the batches are contiguous
  for (uint64_t s = g; s < Q; s += stride) {
    const uint32_t f = a.first[key[s]];
    const uint32_t r = (uint32_t)s - f, k = r % B;
    const uint32_t hw = val[f + (r - k)];   // queue position of the chunk's first entry
    if (hw >= stop) continue;
    const uint32_t c = a.child[val[s]];
    a.batched[a.hoff[hw] + k] = c;
    a.slot[c].phase = (a.slot[c].phase & ~3u) | PH_INFLIGHT;
  }
  for (uint64_t j = g; j < R; j += stride) a.queue[head + npop + j] = a.rem[j];
  if (g == 0) {
    a.qstate[0] = head + npop;
    ds->stats[5] += ds->pb_bad;
  }
}

void launch_parent(const LaunchCfg& L, const ParentArgs& a) {
  const uint64_t tiles = std::max<uint64_t>(1, ceil_div(a.N, (uint64_t)PB_TILE));
  const int g_scan = (int)std::max<uint64_t>(
      1, std::min<uint64_t>(ceil_div(a.N, (uint64_t)PB_SCAN_THREADS * PB_ITEMS), (uint64_t)L.grid_pb_scan));
  const int g_rows = (int)ceil_div(1ull << a.dbits, (uint64_t)PB_ROW_DIGITS);
  const int g_elem = (int)std::max<uint64_t>(
      1, std::min<uint64_t>(ceil_div(a.N, (uint64_t)PB_THREADS), (uint64_t)L.grid_pb));
  const int g_tile = (int)std::min<uint64_t>(tiles, (uint64_t)L.grid_pb_sort);
  launch_k(L, K_PB_KEYS, pb_keys_kernel, g_tile, PB_THREADS, 0, a);
  for (int p = 0; p < a.passes; ++p) {
    ParentArgs b = a;
    b.pass = p;
    if (p) launch_k(L, K_PB_HIST, pb_hist_kernel, g_tile, PB_THREADS, 0, b);
    launch_k(L, K_PB_ROWSCAN, pb_rowscan_kernel, g_rows, PB_ROW_THREADS, 0, b);
    launch_k(L, K_PB_SORT, pb_sort_kernel, g_tile, PB_THREADS, 0, b);
  }
  launch_k(L, K_PB_BOUNDS, pb_bounds_kernel, g_elem, PB_THREADS, 0, a);
  launch_k(L, K_PB_HEADS, pb_heads_kernel, g_elem, PB_THREADS, 0, a);
  if (!a.flush) launch_k(L, K_PB_MARK, pb_mark_kernel, g_elem, PB_THREADS, 0, a);
  launch_k(L, K_PB_SCAN, pb_scan_kernel, g_scan, PB_SCAN_THREADS, 0, a);
  launch_k(L, K_PB_EMIT, pb_emit_kernel, g_elem, PB_THREADS, 0, a);
}

const void* kernel_ptr_parent(int which) {
  switch (which) {
    case K_PB_SORT: return (const void*)pb_sort_kernel;
    case K_PB_SCAN: return (const void*)pb_scan_kernel;
    default: return (const void*)pb_heads_kernel;
  }
}

}  // namespace ro
