// steel_attn_run_noalloc: the attention call for callers that must not allocate device memory.
//
// The regular path keeps its work lists (items, per-CTA ranges, key-tile step lists) and its status
// word in buffers that steel_attn_create obtains from cudaMalloc.  Some callers cannot do that: code
// running inside another framework's memory pool with the allocator locked, code on a latency path
// where cudaMalloc's implicit device synchronisation is not acceptable, or a process whose memory
// budget is fixed up front.  For them the same kernel runs with those lists in a fixed-size array
// that is part of the library image: every GPU that loads the library holds kScratchBytes for it
// until the process exits.  Inputs and outputs are still the caller's.
#include <cuda_runtime.h>

#include <cstring>
#include <mutex>
#include <new>

#include "../../include/steel_attn.h"
#include "steel_kernel.h"
#include "steel_planner.h"

using namespace steel;

namespace {

// In host code this name is only a handle for the symbol, never a device address: the address the
// kernel needs comes from cudaGetSymbolAddress below.
static __device__ __align__(256) unsigned char g_scratch[kNoallocBytes];

constexpr int kMaxDevices = 64;
std::mutex g_mutex;
unsigned char *g_scratch_addr[kMaxDevices] = {};
int g_sm_count[kMaxDevices] = {};

// The step lists of single query tiles, from the bitmap: one warp per item, one lane per key tile, 32 at a time; a vote
// gives each visible tile its place, in ascending order.  Bound by the latency of its few loads.  With the entries
// made and copied by the host the call took 175 us (8 heads x 4096 d64, 64-token blocks), as here 144.  A list that is
// not as long as the planner has counted sets the status word.
constexpr int kListWarps = 8;
constexpr int32_t kListMismatch = STEEL_ERR_CUDA;  // beside STEEL_ERR_TIMEOUT of the attention kernel
__global__ void write_lists(const WorkItem *items, int n_items, const uint32_t *bitmap, BitmapMask mask, StepPair *steps,
                            int32_t *status) {
  const int n = (blockIdx.x * blockDim.x + threadIdx.x) / 32, lane = threadIdx.x % 32;
  if (n >= n_items || items[n].kind != 1) return;
  const WorkItem &w = items[n];
  const uint32_t *rows = bitmap + size_t(w.head[0]) * mask.blocks_q * mask.words;
  ListWriter list{steps + w.j0[0], w.n_steps};
  for (int j0 = 0; j0 < mask.key_tiles(); j0 += 32) {
    const uint32_t e = j0 + lane < mask.key_tiles() ? mask.entry(rows, w.qtile[0], j0 + lane) : 0u;
    list.place(lane, e, __ballot_sync(0xffffffffu, e != 0));
  }
  if (!list.finish(lane) && lane == 0) atomicExch(status, kListMismatch);
}

// Once per device, with that device current: resolve the array's device address, read the SM
// count, load every kernel that a later call may launch (code is loaded lazily, which can allocate device memory and wait
// for the device) and opt the attention kernels in to their shared-memory size.
steel_status_t setup_device(int device, unsigned char **base, int *sm_count) {
  std::lock_guard<std::mutex> lock(g_mutex);
  if (!g_scratch_addr[device]) {
    cudaDeviceProp prop;
    if (cudaGetDeviceProperties(&prop, device) != cudaSuccess) return STEEL_ERR_CUDA;
    if (prop.major != 10) return STEEL_ERR_CUDA;
    void *ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_scratch) != cudaSuccess || !ptr) return STEEL_ERR_CUDA;
    cudaFuncAttributes loaded;
    if (configure_kernels() != cudaSuccess || cudaFuncGetAttributes(&loaded, write_lists) != cudaSuccess)
      return STEEL_ERR_CUDA;
    g_sm_count[device] = prop.multiProcessorCount;
    g_scratch_addr[device] = static_cast<unsigned char *>(ptr);
  }
  *base = g_scratch_addr[device];
  *sm_count = g_sm_count[device];
  return STEEL_OK;
}

}  // namespace

extern "C" steel_status_t steel_attn_run_noalloc(const steel_attn_params_t *params, const void *q, const void *k,
                                                 const void *v, void *o, float *lse, void *cuda_stream) {
  if (!q || !k || !v || !o) return STEEL_ERR_INVALID_ARG;
  const uintptr_t align = reinterpret_cast<uintptr_t>(q) | reinterpret_cast<uintptr_t>(k) |
                          reinterpret_cast<uintptr_t>(v) | reinterpret_cast<uintptr_t>(o);
  if ((align & 15u) || (reinterpret_cast<uintptr_t>(lse) & 3u)) return STEEL_ERR_INVALID_ARG;
  steel_status_t st = validate_params(params);
  if (st != STEEL_OK) return st;

  int device = 0;
  if (cudaGetDevice(&device) != cudaSuccess) {
    cudaGetLastError();
    return STEEL_ERR_CUDA;
  }
  if (device < 0 || device >= kMaxDevices) return STEEL_ERR_UNSUPPORTED;
  unsigned char *base = nullptr;
  int sm_count = 0;
  st = setup_device(device, &base, &sm_count);
  if (st != STEEL_OK) {
    cudaGetLastError();
    return st;
  }

  // Host memory only.
  NoallocPlan np;
  std::vector<unsigned char> lists;  // what is copied: all but the status word's rest and device-written lists
  try {
    st = plan_noalloc(params, sm_count, &np);
    if (st != STEEL_OK) return st;
    lists.resize(np.copy_bytes);
  } catch (const std::bad_alloc &) {
    return STEEL_ERR_ALLOC;
  }
  const Plan &plan = np.plan;
  auto put = [&lists](size_t at, const void *data, size_t bytes) {
    if (bytes) std::memcpy(lists.data() + at, data, bytes);
  };
  put(np.off_cta_begin, plan.cta_begin.data(), plan.cta_begin.size() * sizeof(int32_t));
  put(np.off_items, plan.items.data(), plan.items.size() * sizeof(WorkItem));
  put(np.off_bitmap, params->mask.bitmap, np.bitmap_bytes);
  put(np.off_steps, plan.steps.data(), plan.steps.size() * sizeof(StepPair));

  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  // The array still holds the previous call's lists and status word: overwrite both (the word with 0).
  if (cudaMemcpyAsync(base, lists.data(), lists.size(), cudaMemcpyHostToDevice, stream) != cudaSuccess) {
    cudaGetLastError();
    return STEEL_ERR_CUDA;
  }
  if (np.device_lists) {
    const int n_items = int(plan.items.size());
    write_lists<<<(n_items + kListWarps - 1) / kListWarps, kListWarps * 32, 0, stream>>>(
        reinterpret_cast<const WorkItem *>(base + np.off_items), n_items, reinterpret_cast<const uint32_t *>(base + np.off_bitmap),
        bitmap_mask(*params), reinterpret_cast<StepPair *>(base + np.off_steps), reinterpret_cast<int32_t *>(base));
    if (cudaGetLastError() != cudaSuccess) return STEEL_ERR_CUDA;
  }
  KernelParams kp{};  // no split query tiles: their buffers have no room in the array
  kp.items = reinterpret_cast<const WorkItem *>(base + np.off_items);
  kp.cta_begin = reinterpret_cast<const int32_t *>(base + np.off_cta_begin);
  kp.steps = reinterpret_cast<const StepPair *>(base + np.off_steps);
  kp.status = reinterpret_cast<int32_t *>(base);
  set_query_view(*params, plan.packed, &kp);
  kp.overlap_launch = plan.stats.max_cta_steps <= kOverlapSteps;
  kp.timeout_cycles = kDefaultTimeoutCycles;
  kp.stall_cta = -1;
  st = launch_with_params(*params, kp, plan.grid, q, k, v, o, lse, stream, nullptr);
  if (st != STEEL_OK) return st;
  // Blocking by design: the host lists above must outlive the copy, and the status word has to be read
  // before the next call clears it.  The read on the same stream waits for the kernel.
  int32_t word = 0;
  if (cudaMemcpyAsync(&word, base, sizeof word, cudaMemcpyDeviceToHost, stream) != cudaSuccess ||
      cudaStreamSynchronize(stream) != cudaSuccess) {
    cudaGetLastError();
    return STEEL_ERR_CUDA;
  }
  return static_cast<steel_status_t>(word);  // 0, or set by one of the kernels
}
