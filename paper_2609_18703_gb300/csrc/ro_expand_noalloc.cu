// ro_expand_noalloc.cu — expansion lineage (offsets, parent and ordinal of
// every child) for callers that cannot allocate device memory.
//
// Some callers cannot call cudaMalloc: code running inside a memory budget
// that a framework's caching allocator owns, code paths that must not
// synchronise the device the way cudaMalloc/cudaFree can, or embedders that
// forbid allocation after start-up.  This entry point needs no context and
// allocates nothing: its scratch (the scan's per-tile look-back status, the
// per-fill-tile parent table and a few counters) lives in one file-scope
// __device__ array of fixed size, which every GPU that loads the library
// holds until the process exits.
//
// Its kernels are variants of expand_scan / expand_fill that write only the
// caller's outputs (no lineage state is kept, so nothing later can commit or
// assemble against this expansion).
#include <cstddef>
#include <mutex>

#include "../../include/rayorch_gpu.h"
#include "ro_expand.cuh"

namespace ro {
namespace {

constexpr uint64_t NA_MAX_PARENTS = 1ull << 24;    // 16,777,216
constexpr uint64_t NA_MAX_CHILDREN = 1ull << 27;   // 134,217,728
constexpr uint64_t NA_SCAN_TILE = (uint64_t)EXP_THREADS * EXP_ITEMS;
constexpr uint64_t NA_TILES = NA_MAX_PARENTS / NA_SCAN_TILE;        // 4096
constexpr uint64_t NA_TFP = NA_MAX_CHILDREN / FILL_TILE + 1;         // 32769

// Layout of the static scratch.  A scan leaves the header's counters at zero
// for the next one; they are cleared before a scan only where the call before
// did not get that far.  The epoch goes on (it keeps stale tile flags from
// looking current).
struct NaHeader {
  uint32_t tile_ctr, exit_ctr, err, pad;
  unsigned long long n_children, n_empty, epoch;
};
constexpr size_t NA_OFF_FLAGS = 256;
constexpr size_t NA_OFF_AGG = NA_OFF_FLAGS + NA_TILES * sizeof(unsigned long long);
constexpr size_t NA_OFF_INC = NA_OFF_AGG + NA_TILES * sizeof(Pair64);
constexpr size_t NA_OFF_TFP = NA_OFF_INC + NA_TILES * sizeof(Pair64);
constexpr size_t NA_BYTES = NA_OFF_TFP + NA_TFP * sizeof(uint32_t);   // ~292 KB

static __device__ __align__(256) unsigned char g_expand_scratch[NA_BYTES];

template <int ITEMS>
__global__ void __launch_bounds__(EXP_THREADS, 3)
expand_scan_noalloc_kernel(const uint32_t* counts, uint64_t P, uint64_t* offsets,
                           uint32_t* empty_out, unsigned char* scratch) {
  __shared__ ScanShared<ITEMS> sh;
  NaHeader* h = reinterpret_cast<NaHeader*>(scratch);
  ScanIo io{};
  io.counts = counts;
  io.P = P;
  io.offsets = offsets;
  io.empty_out = empty_out;
  io.tfp = reinterpret_cast<uint32_t*>(scratch + NA_OFF_TFP);
  io.tfp_cap = NA_TFP;
  io.ts = TileStatus<Pair64>{reinterpret_cast<unsigned long long*>(scratch + NA_OFF_FLAGS),
                             reinterpret_cast<Pair64*>(scratch + NA_OFF_AGG),
                             reinterpret_cast<Pair64*>(scratch + NA_OFF_INC)};
  io.epoch = h->epoch;
  io.tile_ctr = &h->tile_ctr;
  io.err = &h->err;
  io.n_children = &h->n_children;
  io.n_empty = &h->n_empty;
  scan_tiles<ITEMS>(io, sh);
  if (threadIdx.x == 0) {
    if (P == 0 && blockIdx.x == 0) {
      offsets[0] = 0;
      h->n_children = 0;
      h->n_empty = 0;
    }
    if (ticket(&h->exit_ctr) == gridDim.x - 1) {
      h->tile_ctr = 0u;
      h->exit_ctr = 0u;
      h->epoch = io.epoch + 1ull;
    }
  }
}

__global__ void __launch_bounds__(FILL_THREADS)
expand_fill_noalloc_kernel(const uint64_t* offsets, uint64_t P, uint64_t N, uint32_t* child_parent,
                           uint32_t* child_ordinal, const unsigned char* scratch) {
  __shared__ FillShared sh;
  FillIo io{};
  io.offsets = offsets;
  io.P = P;
  io.N = N;
  io.tfp = reinterpret_cast<const uint32_t*>(scratch + NA_OFF_TFP);
  io.child_parent = child_parent;
  io.child_ordinal = child_ordinal;
  fill_tiles(io, sh);
}

// Device address of the static scratch, looked up once per device.
constexpr int NA_MAX_DEVICES = 64;
std::mutex g_na_mu;
unsigned char* g_na_ptr[NA_MAX_DEVICES] = {};
int g_na_sms[NA_MAX_DEVICES] = {};
bool g_na_clean[NA_MAX_DEVICES] = {};

// *clean: whether the scratch's counters are zero; they count as used until
// na_clean says that a scan has put them back.
ro_status na_setup(int dev, unsigned char** ptr, int* sms, bool* clean) {
  if (dev < 0 || dev >= NA_MAX_DEVICES) return RO_E_CUDA;
  std::lock_guard<std::mutex> lock(g_na_mu);
  if (!g_na_ptr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_expand_scratch) != cudaSuccess || !p) {
      cudaGetLastError();
      return RO_E_CUDA;
    }
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) {
      cudaGetLastError();
      return RO_E_CUDA;
    }
    g_na_ptr[dev] = static_cast<unsigned char*>(p);
    g_na_sms[dev] = n;
  }
  *ptr = g_na_ptr[dev];
  *sms = g_na_sms[dev];
  *clean = g_na_clean[dev];
  g_na_clean[dev] = false;
  return RO_OK;
}
void na_clean(int dev) {
  std::lock_guard<std::mutex> lock(g_na_mu);
  g_na_clean[dev] = true;
}

}  // namespace
}  // namespace ro

extern "C" ro_status ro_expand_noalloc(const uint32_t* d_counts, uint64_t n_parents,
                                       uint64_t* d_offsets, uint32_t* d_child_parent,
                                       uint32_t* d_child_ordinal, uint64_t child_cap,
                                       uint32_t* d_empty_parents, void* stream,
                                       uint64_t* h_n_children, uint64_t* h_n_empty) {
  using namespace ro;
  if (!h_n_children || !d_offsets || (n_parents && !d_counts)) return RO_E_INVAL;
  if (n_parents > NA_MAX_PARENTS) return RO_E_CAPACITY;   // beyond the static scratch
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return RO_E_CUDA;
  }
  unsigned char* scratch = nullptr;
  int sms = 0;
  bool clean = false;
  ro_status st = na_setup(dev, &scratch, &sms, &clean);
  if (st != RO_OK) return st;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  // counters must start at zero (the epoch is kept): the scan's last CTA leaves
  // them so, unless a call on this device did not get that far or met an error
  if (!clean && cudaMemsetAsync(scratch, 0, offsetof(NaHeader, n_children), s) != cudaSuccess) {
    cudaGetLastError();
    return RO_E_CUDA;
  }
  const uint64_t tiles = ceil_div(n_parents, scan_tile(n_parents));
  const int scan_grid = (int)(tiles < (uint64_t)sms * 4 ? (tiles ? tiles : 1) : (uint64_t)sms * 4);
  auto* scan = n_parents <= SCAN_SMALL ? expand_scan_noalloc_kernel<4> : expand_scan_noalloc_kernel<EXP_ITEMS>;
  scan<<<scan_grid, EXP_THREADS, 0, s>>>(d_counts, n_parents, d_offsets, d_empty_parents, scratch);
  if (cudaGetLastError() != cudaSuccess) return RO_E_CUDA;   // not launched: the header is stale
  NaHeader hh{};
  cudaError_t e = cudaMemcpyAsync(&hh, scratch, sizeof(NaHeader), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return RO_E_CUDA;
  }
  *h_n_children = hh.n_children;
  if (h_n_empty) *h_n_empty = hh.n_empty;
  if (hh.err & ERR_TIMEOUT) return RO_E_TIMEOUT;
  if (!hh.err) na_clean(dev);
  const uint64_t N = hh.n_children;
  if (N >= (1ull << 32)) return RO_E_OVERFLOW;
  if (N > NA_MAX_CHILDREN) return RO_E_CAPACITY;   // beyond the static scratch
  if (N > child_cap) return RO_E_CAPACITY;
  if (N == 0) return RO_OK;
  if (!d_child_parent || !d_child_ordinal) return RO_E_INVAL;
  const uint64_t n_tiles = ceil_div(N, FILL_TILE);
  const int grid = (int)(n_tiles < (uint64_t)sms * 8 ? n_tiles : (uint64_t)sms * 8);
  expand_fill_noalloc_kernel<<<grid, FILL_THREADS, 0, s>>>(d_offsets, n_parents, N, d_child_parent,
                                                          d_child_ordinal, scratch);
  if (cudaGetLastError() != cudaSuccess) return RO_E_CUDA;
  // The fill reads the shared scratch (its per-tile parent table): return
  // only once it is done, so that a caller who takes the return as
  // completion may start the next call from any stream or thread.
  if (cudaStreamSynchronize(s) != cudaSuccess) {
    cudaGetLastError();
    return RO_E_CUDA;
  }
  return RO_OK;
}
