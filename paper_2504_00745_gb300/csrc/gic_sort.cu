// gic_sort.cu -- a1: stable Morton sort of granules by contact cell.
//
// LSD radix sort over the Morton key of the packed contact cell, 8-bit digits,
// reduce-then-scan per pass (upsweep histograms, per-digit scan over tiles,
// downsweep ranking + scatter).  No kernel here waits on another block, so
// nothing can spin.  The first pass computes keys from the cells on the fly;
// the last pass writes the permutation, and a final kernel gathers the granule
// state (cell, pos, vel, id) and writes the epoch-tagged cell table
// {start, count, epoch} of the occupied cells.
#include "gic_sort.cuh"

namespace gic {

constexpr int kSortThreads = 256;

static int key_bits(const DGrid& G) {
  int m = G.nc[0];
  if (G.nc[1] > m) m = G.nc[1];
  if (G.nc[2] > m) m = G.nc[2];
  int b = 0;
  while ((1 << b) < m) ++b;
  if (b < 1) b = 1;
  return 3 * b;
}

static size_t align_up(size_t v) { return (v + 255) & ~(size_t)255; }

SortLayout sort_layout(const DGrid& G, int64_t n) {
  SortLayout L;
  L.n = n;
  L.tiles = (int)((n + kTile - 1) / kTile);
  if (L.tiles < 1) L.tiles = 1;
  L.passes = (key_bits(G) + 7) / 8;
  size_t a = align_up(sizeof(uint32_t) * (size_t)(n > 0 ? n : 1));
  size_t off = 0;
  L.off_keys_a = off;
  off += a;
  L.off_vals_a = off;
  off += a;
  L.off_keys_b = off;
  off += a;
  L.off_vals_b = off;
  off += a;
  L.off_counts = off;
  off += align_up(sizeof(uint32_t) * (size_t)kRadix * L.tiles);
  L.off_totals = off;
  off += align_up(sizeof(uint32_t) * kRadix);
  L.total = off;
  return L;
}

__global__ void __launch_bounds__(kSortThreads) k_upsweep(int64_t n, int shift, const int32_t* __restrict__ cell,
                                                          const uint32_t* keys, uint32_t* counts, int tiles) {
  __shared__ SortShared<kSortThreads> sh;
  sort_upsweep<kSortThreads>(sh, n, shift, keys == nullptr, cell, keys, counts, tiles);
}

// CTA 0 of the first pass also advances the cell-table epoch.
__global__ void __launch_bounds__(kSortThreads) k_scan_tiles(uint32_t* counts, int tiles, uint32_t* totals,
                                                             uint4* table_head) {
  __shared__ SortShared<kSortThreads> sh;
  sort_scan<kSortThreads>(sh, counts, tiles, totals, table_head);
}

template <bool kFirst, bool kLast>
__global__ void __launch_bounds__(kSortThreads) k_downsweep(int64_t n, int shift, const int32_t* __restrict__ cell,
                                                            const uint32_t* keys_in, const uint32_t* vals_in,
                                                            uint32_t* keys_out, uint32_t* vals_out,
                                                            const uint32_t* counts, const uint32_t* totals, int tiles,
                                                            int32_t* perm) {
  __shared__ SortShared<kSortThreads> sh;
  sort_downsweep<kSortThreads>(sh, n, shift, kFirst, kLast, cell, keys_in, vals_in, keys_out, vals_out, counts, totals, tiles, perm);
}

template <typename T>
__global__ void __launch_bounds__(256) k_permute_table(DGrid G, int64_t n, const uint32_t* keys, ScatterState S,
                                                       uint4* table, uint32_t* status) {
  int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k < n) sort_gather<T>(G, n, k, keys, S, table, status);
}

template <typename T>
static int launch_sort(const DGrid& G, const GicGranules* in, GicGranules* out, int32_t* perm, uint4* table,
                       char* ws, const SortLayout& L, cudaStream_t st) {
  int64_t n = in->n;
  uint32_t* keys_a = (uint32_t*)(ws + L.off_keys_a);
  uint32_t* vals_a = (uint32_t*)(ws + L.off_vals_a);
  uint32_t* keys_b = (uint32_t*)(ws + L.off_keys_b);
  uint32_t* vals_b = (uint32_t*)(ws + L.off_vals_b);
  uint32_t* counts = (uint32_t*)(ws + L.off_counts);
  uint32_t* totals = (uint32_t*)(ws + L.off_totals);
  ScatterState S{in->cell, in->pos,  in->vel, in->id, out->cell,
                 out->pos, out->vel, out->id, perm, sizeof(T) == 4 ? (float4*)out->posf : nullptr};
  const uint32_t* kin = nullptr;
  const uint32_t* vin = nullptr;
  uint32_t* kout = keys_a;
  uint32_t* vout = vals_a;
  int launches = 0;
  for (int p = 0; p < L.passes; ++p) {
    const int shift = 8 * p;
    const bool first = p == 0, last = p == L.passes - 1;
    k_upsweep<<<L.tiles, kSortThreads, 0, st>>>(n, shift, in->cell, kin, counts, L.tiles);
    k_scan_tiles<<<L.tiles <= kWarpScanTiles ? 32 * kRadix / kSortThreads : kRadix, kSortThreads, 0, st>>>(
        counts, L.tiles, totals, first ? table : nullptr);
    auto down = first ? (last ? k_downsweep<true, true> : k_downsweep<true, false>)
                      : (last ? k_downsweep<false, true> : k_downsweep<false, false>);
    down<<<L.tiles, kSortThreads, 0, st>>>(n, shift, in->cell, kin, vin, kout, vout, counts, totals, L.tiles, perm);
    launches += 3;
    kin = kout;
    vin = vout;
    kout = (kout == keys_a) ? keys_b : keys_a;
    vout = (vout == vals_a) ? vals_b : vals_a;
  }
  // kin now holds the sorted keys
  k_permute_table<T><<<grid_blocks(n, 256), 256, 0, st>>>(G, n, kin, S, table, status_word());
  launches += 1;
  count_launches(launches);
  GIC_CHECK_LAUNCH("gic_sort");
  return GIC_OK;
}

}  // namespace gic

using namespace gic;

extern "C" int gic_workspace_size(const GicGrid* grid, int64_t n, int32_t precision, size_t* bytes) {
  GIC_RANGE("gic_workspace_size");
  DGrid G;
  int rc = make_grid(grid, &G);
  if (rc) return rc;
  if (!bytes) return set_error(GIC_ERR_INVALID, "bytes is NULL");
  if (n < 0) return set_error(GIC_ERR_INVALID, "n < 0");
  if (precision != GIC_FP32 && precision != GIC_FP64) return set_error(GIC_ERR_INVALID, "bad precision");
  *bytes = sort_layout(G, n).total;
  return GIC_OK;
}

extern "C" int gic_sort(const GicGrid* grid, const GicGranules* in, GicGranules* out, int32_t* perm, void* cell_table,
                        void* ws, size_t ws_bytes, gic_stream_t stream) {
  GIC_RANGE("gic_sort");
  DGrid G;
  int rc = make_grid(grid, &G);
  if (rc) return rc;
  if ((rc = check_granules(in, "gic_sort in"))) return rc;
  if ((rc = check_granules(out, "gic_sort out"))) return rc;
  if (in->n != out->n || in->precision != out->precision)
    return set_error(GIC_ERR_INVALID, "gic_sort: in/out size or precision differ");
  if (!cell_table) return set_error(GIC_ERR_INVALID, "gic_sort: cell_table is NULL");
  if ((uintptr_t)cell_table % 16) return set_error(GIC_ERR_ALIGN, "gic_sort: cell_table must be 16-byte aligned");
  int64_t n = in->n;
  if (n == 0) return GIC_OK;
  if (!perm) return set_error(GIC_ERR_INVALID, "gic_sort: perm is NULL");
  if (in->cell == out->cell || in->pos == out->pos || in->vel == out->vel)
    return set_error(GIC_ERR_INVALID, "gic_sort: in and out must not alias");
  SortLayout L = sort_layout(G, n);
  if (!ws || ws_bytes < L.total)
    return set_error(GIC_ERR_WORKSPACE, "gic_sort: workspace of %zu bytes needed, %zu given", L.total, ws_bytes);
  if ((uintptr_t)ws % 256) return set_error(GIC_ERR_ALIGN, "gic_sort: workspace must be 256-byte aligned");
  if (in->precision == GIC_FP32)
    return launch_sort<float>(G, in, out, perm, (uint4*)cell_table, (char*)ws, L, (cudaStream_t)stream);
  return launch_sort<double>(G, in, out, perm, (uint4*)cell_table, (char*)ws, L, (cudaStream_t)stream);
}

// ----------------------------------------------------------------- adjoint

namespace gic {
template <typename T>
__global__ void k_sort_adj(int64_t n, const int32_t* __restrict__ perm, const vec_t<T>* __restrict__ gpo,
                           const vec_t<T>* __restrict__ gvo, vec_t<T>* __restrict__ gpi, vec_t<T>* __restrict__ gvi) {
  int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= n) return;
  int32_t s = perm[k];
  if (gpi) gpi[s] = gpo[k];
  if (gvi) gvi[s] = gvo[k];
}
}  // namespace gic

extern "C" int gic_sort_adj(int64_t n, int32_t precision, const int32_t* perm, const void* g_pos_out,
                            const void* g_vel_out, void* g_pos_in, void* g_vel_in, gic_stream_t stream) {
  GIC_RANGE("gic_sort_adj");
  if (n < 0) return set_error(GIC_ERR_INVALID, "gic_sort_adj: n < 0");
  if (n == 0) return GIC_OK;
  if (!perm) return set_error(GIC_ERR_INVALID, "gic_sort_adj: perm is NULL");
  if ((g_pos_in && !g_pos_out) || (g_vel_in && !g_vel_out))
    return set_error(GIC_ERR_INVALID, "gic_sort_adj: missing upstream gradient");
  if (precision == GIC_FP32 || precision == GIC_FP64) {
    int rc = check_vecs(precision, "gic_sort_adj", {g_pos_out, g_vel_out, g_pos_in, g_vel_in});
    if (rc) return rc;
  }
  if (precision == GIC_FP32)
    k_sort_adj<float><<<grid_blocks(n, 256), 256, 0, stream>>>(n, perm, (const float4*)g_pos_out,
                                                                (const float4*)g_vel_out, (float4*)g_pos_in,
                                                                (float4*)g_vel_in);
  else if (precision == GIC_FP64)
    k_sort_adj<double><<<grid_blocks(n, 256), 256, 0, stream>>>(n, perm, (const d4*)g_pos_out, (const d4*)g_vel_out,
                                                                 (d4*)g_pos_in, (d4*)g_vel_in);
  else
    return set_error(GIC_ERR_INVALID, "gic_sort_adj: bad precision");
  count_launches(1);
  GIC_CHECK_LAUNCH("gic_sort_adj");
  return GIC_OK;
}

// ----------------------------------------------------------------- sort without a caller workspace
//
// For callers that cannot allocate device memory themselves -- code running
// where a cudaMalloc would be unsafe or unavailable, such as inside a host
// callback, a signal-free real-time loop, or a host that hands the library
// only pre-registered buffers -- this variant takes its radix-sort scratch
// from a fixed array compiled into the library instead of a workspace
// argument.  The array exists once per device that loads the library and
// lives until the process exits.

namespace gic {

// Largest granule count the static scratch holds.
constexpr int64_t kStaticSortMaxN = 1 << 18;  // 262,144 granules
constexpr int kStaticSortTiles = (int)((kStaticSortMaxN + kTile - 1) / kTile);
// keys and values ping-pong (4 x n x 4 B) + per-tile digit counts + digit totals
constexpr size_t kStaticSortBytes =
    4 * ((sizeof(uint32_t) * kStaticSortMaxN + 255) & ~(size_t)255) +
    ((sizeof(uint32_t) * (size_t)kRadix * kStaticSortTiles + 255) & ~(size_t)255) +
    ((sizeof(uint32_t) * kRadix + 255) & ~(size_t)255);

static __device__ __align__(256) unsigned char g_static_sort_scratch[kStaticSortBytes];

// Device address of the static scratch on the current device (host code may
// not use the symbol's name as an address).  It is looked up on every call
// rather than cached: a cudaDeviceReset in the same process reloads the
// module, after which a cached address would point at freed memory.  The
// lookup allocates nothing; the first one on a device loads the module
// (lazy loading), which is why that first call must precede any stream
// capture.
static int static_scratch(void** out) {
  void* p = nullptr;
  const cudaError_t e = cudaGetSymbolAddress(&p, g_static_sort_scratch);
  if (e != cudaSuccess || !p)
    return set_error(GIC_ERR_CUDA, "gic_sort_static: cudaGetSymbolAddress failed: %s", cudaGetErrorString(e));
  *out = p;
  return GIC_OK;
}

}  // namespace gic

extern "C" int64_t gic_sort_static_max_n(void) { return gic::kStaticSortMaxN; }

extern "C" int gic_sort_static(const GicGrid* grid, const GicGranules* in, GicGranules* out, int32_t* perm,
                               void* cell_table, gic_stream_t stream) {
  GIC_RANGE("gic_sort_static");
  DGrid G;
  int rc = make_grid(grid, &G);
  if (rc) return rc;
  if ((rc = check_granules(in, "gic_sort_static in"))) return rc;
  if ((rc = check_granules(out, "gic_sort_static out"))) return rc;
  if (in->n != out->n || in->precision != out->precision)
    return set_error(GIC_ERR_INVALID, "gic_sort_static: in/out size or precision differ");
  if (in->n > kStaticSortMaxN)
    return set_error(GIC_ERR_INVALID, "gic_sort_static: %lld granules exceed the static scratch limit of %lld",
                     (long long)in->n, (long long)kStaticSortMaxN);
  if (!cell_table) return set_error(GIC_ERR_INVALID, "gic_sort_static: cell_table is NULL");
  if ((uintptr_t)cell_table % 16) return set_error(GIC_ERR_ALIGN, "gic_sort_static: cell_table must be 16-byte aligned");
  int64_t n = in->n;
  if (n == 0) return GIC_OK;
  if (!perm) return set_error(GIC_ERR_INVALID, "gic_sort_static: perm is NULL");
  if (in->cell == out->cell || in->pos == out->pos || in->vel == out->vel)
    return set_error(GIC_ERR_INVALID, "gic_sort_static: in and out must not alias");
  void* scratch = nullptr;
  if ((rc = static_scratch(&scratch))) return rc;
  // Every pass writes the scratch regions it later reads (all tile counts in
  // the upsweep, keys and values in the downsweep), so the previous call's
  // contents need no clearing.
  SortLayout L = sort_layout(G, n);
  if (L.total > kStaticSortBytes) return set_error(GIC_ERR_INVALID, "gic_sort_static: scratch layout too large");
  if (in->precision == GIC_FP32)
    return launch_sort<float>(G, in, out, perm, (uint4*)cell_table, (char*)scratch, L, (cudaStream_t)stream);
  return launch_sort<double>(G, in, out, perm, (uint4*)cell_table, (char*)scratch, L, (cudaStream_t)stream);
}
