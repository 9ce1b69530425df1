// gic_step_sort.cu -- gic_step's sort: when the previous call left a granule
// beyond skin / 2 of its reference, or a rebuild was requested, the state is
// sorted (a1), and the substep kernel that follows builds the Verlet rows;
// otherwise the kernel returns at once.  The decision is on the device, the
// launches are the same either way, and nothing is instantiated or kept between
// calls.
//
// One cooperative launch (every CTA resident, a grid barrier between the
// passes), so that a call that does not rebuild pays for one idle launch (2.6
// us), not for the ten of gic_sort.  16M granules (30-bit keys, four passes):
// 1018 us, the ten launches together 1046 us.  Before, a conditional CUDA graph
// per set of buffers chose the branch: 200-300 us to instantiate (three graphs
// per simulator), and about 14 us per call on the device (1M dam break, a
// list-keeping call: 93.2 -> 78.1 us; 8k granules FP64, a 10-substep window:
// 1003 -> 566 us).
#include <cuda.h>

#include <mutex>

#include "gic_contact.cuh"
#include "gic_sort.cuh"

namespace gic {

// Grid barrier of a cooperative launch: the CTAs' arrivals counted in a word of
// the lists' flags, target = barriers so far x CTAs.  Waits at most `polls` looks;
// past that the launch cannot be complete: the CTA flags the status word, marks
// the lists as stalled and returns.  The others run out in the same way: one that
// arrives late may still pass this barrier (everyone arrived at it, so what it reads
// is complete), but not the next.
__device__ __forceinline__ bool grid_barrier(uint32_t* flags, uint32_t target, int polls, uint32_t* status) {
  __shared__ int s_ok;
  uint32_t* cnt = &flags[kNbBarrier];
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(cnt, 1u);
    int ok = 0;
    for (int k = 0; k < polls; ++k) {
      uint32_t v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(cnt) : "memory");
      if (v >= target) {
        ok = 1;
        break;
      }
      __nanosleep(40);
    }
    __threadfence();
    if (!ok) {
      flags[kNbSorted] = kNbStalled;
      raise_status(status, GIC_STATUS_STALL);
    }
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

constexpr int kStepSortThreads = 256;
constexpr int kStepSortCtas = 6;  // per SM: 40 registers, 9 KB of shared memory each

template <typename T>
struct StepSortArgs {
  DGrid G;
  int64_t n;
  ScatterState S;
  uint32_t *keys_a, *vals_a, *keys_b, *vals_b, *counts, *totals;
  int tiles, passes, polls;
  uint4* table;
  uint32_t* flags;  // of the lists
  uint32_t* status;
};

template <typename T>
__global__ void __launch_bounds__(kStepSortThreads, kStepSortCtas)
    k_step_sort(const __grid_constant__ StepSortArgs<T> A) {
  __shared__ SortShared<kStepSortThreads> sh;
  const bool stalled = A.flags[kNbSorted] == kNbStalled;  // by an earlier call
  if (stalled || !step_rebuilds(A.flags)) {  // uniform: the words change only in the substep kernels
    if (stalled && blockIdx.x == 0 && threadIdx.x == 0) raise_status(A.status, GIC_STATUS_STALL);
    asm volatile("griddepcontrol.launch_dependents;");  // the substep kernel may start
    return;
  }
  uint32_t arrived = 0;
  auto barrier = [&]() { return grid_barrier(A.flags, arrived += gridDim.x, A.polls, A.status); };
  // the radix passes, ping-ponging between the two key / value buffers
  for (int p = 0; p < A.passes; ++p) {
    const bool first = p == 0, last = p == A.passes - 1;
    const uint32_t* kin = p & 1 ? A.keys_a : A.keys_b;
    const uint32_t* vin = p & 1 ? A.vals_a : A.vals_b;
    uint32_t* kout = p & 1 ? A.keys_b : A.keys_a;
    uint32_t* vout = p & 1 ? A.vals_b : A.vals_a;
    sort_upsweep<kStepSortThreads>(sh, A.n, 8 * p, first, A.S.in_cell, kin, A.counts, A.tiles);
    if (!barrier()) return;
    sort_scan<kStepSortThreads>(sh, A.counts, A.tiles, A.totals, first ? A.table : nullptr);
    if (!barrier()) return;
    sort_downsweep<kStepSortThreads>(sh, A.n, 8 * p, first, last, A.S.in_cell, kin, vin, kout, vout, A.counts,
                                     A.totals, A.tiles, A.S.perm);
    if (!barrier()) return;
  }
  const uint32_t* keys = A.passes & 1 ? A.keys_a : A.keys_b;
  for (int64_t k = blockIdx.x * (int64_t)kStepSortThreads + threadIdx.x; k < A.n;
       k += (int64_t)gridDim.x * kStepSortThreads)
    sort_gather<T>(A.G, A.n, k, keys, A.S, A.table, A.status);
  // past the last barrier: the last CTA (of all: one that gave up there does not
  // arrive here) clears the count of arrivals and tells the substep kernel
  if (threadIdx.x == 0 && atomicAdd(&A.flags[kNbBarrier], 1u) == arrived + gridDim.x - 1) {
    A.flags[kNbBarrier] = 0u;
    A.flags[kNbSorted] = 1u;
  }
}

// SMs of a stream that owns a part of the device's (a green context's), 0 for any
// other.
static int partition_sms(cudaStream_t st) {
  using StreamGetCtx = CUresult (*)(CUstream, CUcontext*, CUgreenCtx*);
  using GetDevResource = CUresult (*)(CUgreenCtx, CUdevResource*, CUdevResourceType);
  static const auto entry = [](const char* name, unsigned version) {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult found;
    return cudaGetDriverEntryPointByVersion(name, &f, version, cudaEnableDefault, &found) == cudaSuccess &&
                   found == cudaDriverEntryPointSuccess
               ? f
               : nullptr;
  };
  static const StreamGetCtx get_ctx = (StreamGetCtx)entry("cuStreamGetCtx", 12050);
  static const GetDevResource get_resource = (GetDevResource)entry("cuGreenCtxGetDevResource", 12040);
  if (!get_ctx || !get_resource) return 0;
  CUcontext ctx = nullptr;
  CUgreenCtx green = nullptr;
  CUdevResource r;
  if (get_ctx((CUstream)st, &ctx, &green) != CUDA_SUCCESS || !green ||
      get_resource(green, &r, CU_DEV_RESOURCE_TYPE_SM) != CUDA_SUCCESS)
    return 0;
  return (int)r.sm.smCount;
}

// CTAs of the cooperative launch that are resident at once on the SMs the stream
// has: more would wait at a barrier for CTAs that cannot start.
template <typename T>
static int resident_ctas(cudaStream_t st) {
  static std::mutex mu;
  static int sms[64] = {0}, per[64] = {0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  const int part = partition_sms(st);
  std::lock_guard<std::mutex> lock(mu);
  if (!sms[dev]) {
    int m = 0, p = 0;
    if (cudaDeviceGetAttribute(&m, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&p, k_step_sort<T>, kStepSortThreads, 0) != cudaSuccess)
      return 0;
    sms[dev] = m;
    per[dev] = p < kStepSortCtas ? p : kStepSortCtas;
  }
  return (part > 0 && part < sms[dev] ? part : sms[dev]) * per[dev];
}

template <typename T>
static int launch(const DGrid& G, const GicGranules* in, const GicGranules* out, int32_t* perm, void* table, char* ws,
                  uint32_t* flags, int polls, cudaStream_t st) {
  const SortLayout L = sort_layout(G, in->n);
  StepSortArgs<T> A{G,
                    in->n,
                    ScatterState{in->cell, in->pos, in->vel, in->id, out->cell, out->pos, out->vel, out->id, perm,
                                 sizeof(T) == 4 ? (float4*)out->posf : nullptr},
                    (uint32_t*)(ws + L.off_keys_a),
                    (uint32_t*)(ws + L.off_vals_a),
                    (uint32_t*)(ws + L.off_keys_b),
                    (uint32_t*)(ws + L.off_vals_b),
                    (uint32_t*)(ws + L.off_counts),
                    (uint32_t*)(ws + L.off_totals),
                    L.tiles,
                    L.passes,
                    polls,
                    (uint4*)table,
                    flags,
                    status_word()};
  const int most = resident_ctas<T>(st);
  if (most < 1) return set_error(GIC_ERR_CUDA, "gic_step: no room for the sort kernel on this device");
  const unsigned want = grid_blocks(in->n, kStepSortThreads);
  void* args[] = {&A};
  const cudaError_t e = cudaLaunchCooperativeKernel(k_step_sort<T>, dim3(want < (unsigned)most ? want : most),
                                                    dim3(kStepSortThreads), args, 0, st);
  if (e != cudaSuccess) return set_error(GIC_ERR_CUDA, "gic_step: sort launch: %s", cudaGetErrorString(e));
  count_launches(1);
  return GIC_OK;
}

int launch_step_sort(const DGrid& G, const GicGranules* in, const GicGranules* out, int32_t* perm, void* table,
                     void* ws, uint32_t* flags, int polls, cudaStream_t st) {
  return in->precision == GIC_FP32 ? launch<float>(G, in, out, perm, table, (char*)ws, flags, polls, st)
                                   : launch<double>(G, in, out, perm, table, (char*)ws, flags, polls, st);
}

}  // namespace gic
