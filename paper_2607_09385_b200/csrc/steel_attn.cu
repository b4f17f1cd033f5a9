// C ABI of the library (see include/steel_attn.h): argument checks, plan upload, tensor maps, launch.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <limits>
#include <mutex>
#include <new>
#include <vector>

#include "../../include/steel_attn.h"
#include "steel_kernel.h"
#include "steel_planner.h"

using namespace steel;

static_assert(sizeof(steel_mask_desc_t) == 32 && sizeof(steel_attn_params_t) == 72, "public struct layout");

// Cut plans: the parts of a launch are left in buffers and counted in counters.  Launches that may overlap must
// not share them, so a handle has several sets: one for the stream that it was first run on; one for all its other
// streams, whose launches an event keeps apart; and one for each sequence of captured launches (one stream in one
// capture), because a graph replays them at any time beside anything else.  A launch for which there is no set
// runs the plan without cuts, which leaves nothing on the device.
constexpr int kHomeSet = 0, kRoamingSet = 1, kFirstCapturedSet = 2, kMaxPartSets = 32;
constexpr size_t kCapturedPartBytes = size_t(64) << 20;  // part buffers of all captured sequences of a handle

struct PartSet {
  float *parts = nullptr;
  unsigned long long stream = 0, capture = 0;  // who uses it: a stream's id, or its handle and the capture's id
  bool used = false;
};

struct DeviceLists {  // a plan's lists in device memory
  WorkItem *items = nullptr;
  int32_t *cta_begin = nullptr;
  StepPair *steps = nullptr;
  int grid = 0;
  bool overlap_launch = false;
};

struct steel_attn {
  steel_attn_params_t params;
  steel_attn_stats_t stats;
  int device = -1;
  unsigned char *d_lists = nullptr;  // one allocation: everything below except the part buffers
  DeviceLists plan, whole;           // `whole`: the plan without cuts, where `plan` cuts key ranges
  int32_t *d_status = nullptr;
  SplitTile *d_split_tiles = nullptr;  // null: no query tile is split
  int32_t *d_arrivals = nullptr;       // counters of kMaxPartSets sets, n_split * 4 each
  size_t n_split = 0;
  size_t part_bytes = 0;
  int32_t part_rows = 0;
  bool packed = false;
  std::mutex parts_lock;  // held from the choice of a set to the end of the launch's record
  PartSet sets[kMaxPartSets];
  int n_sets = kFirstCapturedSet;
  cudaEvent_t roaming_done = nullptr;  // after the last launch with the roaming set
  long long *d_clock_probe = nullptr;
  long long timeout_cycles = kDefaultTimeoutCycles;
  int32_t stall_cta = -1;
  TensorMaps maps;  // of the last (q, k, v) triple run on this handle
};

namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// The driver entry point is resolved at run time so that the library loads (and its host-only
// functions work) on machines without the CUDA driver.
EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = [] {
    void *f = nullptr;
    cudaDriverEntryPointQueryResult res;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &res) != cudaSuccess ||
        res != cudaDriverEntryPointSuccess)
      f = nullptr;
    return reinterpret_cast<EncodeTiledFn>(f);
  }();
  return fn;
}

// bf16 [matrices, rows, head_dim] viewed as a 3-D tensor; boxes of 128 rows x 64 columns (128 bytes),
// 128-byte swizzle; rows beyond `rows` read as zero.
bool make_map(CUtensorMap *map, const void *base, int head_dim, int64_t rows, int64_t matrices) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[3] = {cuuint64_t(head_dim), cuuint64_t(rows), cuuint64_t(matrices)};
  cuuint64_t strides[2] = {cuuint64_t(head_dim) * 2, cuuint64_t(head_dim) * 2 * cuuint64_t(rows)};
  cuuint32_t box[3] = {64, cuuint32_t(kTile), 1};
  cuuint32_t elem_strides[3] = {1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box, elem_strides,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

void free_device(steel_attn *h) {
  if (h->d_lists) cudaFree(h->d_lists);
  for (PartSet &set : h->sets)
    if (set.parts) cudaFree(set.parts);
  if (h->roaming_done) cudaEventDestroy(h->roaming_done);
}

constexpr size_t round16(size_t n) { return round_up(n, 16); }

// Append a plan's lists to `image`; `lists` receives offsets, which place_lists makes addresses.
void append_lists(const Plan &plan, std::vector<unsigned char> *image, DeviceLists *lists) {
  auto put = [image](const void *data, size_t bytes, size_t align = 16) {
    const size_t at = round_up(image->size(), align);
    image->resize(at + round16(bytes));
    if (bytes) std::memcpy(image->data() + at, data, bytes);
    return at;
  };
  lists->cta_begin = reinterpret_cast<int32_t *>(put(plan.cta_begin.data(), plan.cta_begin.size() * sizeof(int32_t)));
  lists->items = reinterpret_cast<WorkItem *>(put(plan.items.data(), plan.items.size() * sizeof(WorkItem), 64));
  lists->steps = reinterpret_cast<StepPair *>(put(plan.steps.data(), plan.steps.size() * sizeof(StepPair)));
  lists->grid = plan.grid;
  lists->overlap_launch = plan.stats.max_cta_steps <= kOverlapSteps;
}

template <class T>
void place(T **offset, unsigned char *base) {
  *offset = reinterpret_cast<T *>(base + reinterpret_cast<uintptr_t>(*offset));
}
void place_lists(DeviceLists *lists, unsigned char *base) {
  place(&lists->cta_begin, base);
  place(&lists->items, base);
  place(&lists->steps, base);
}

// cudaMalloc that is also possible while a stream is captured (the allocation is not part of the capture).
bool allocate_parts(steel_attn *h, PartSet *set) {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  if (cudaThreadExchangeStreamCaptureMode(&mode) != cudaSuccess) return false;
  const bool ok = cudaMalloc(&set->parts, h->part_bytes) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    set->parts = nullptr;
  }
  cudaThreadExchangeStreamCaptureMode(&mode);
  return ok;
}

// The set for a launch on `stream`, or -1: none is left, or nothing can be said about the stream.
int take_part_set(steel_attn *h, cudaStream_t stream) {
  unsigned long long id = 0, capture = 0;
  cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
  if (cudaStreamGetCaptureInfo(stream, &status, &capture) != cudaSuccess) {
    cudaGetLastError();
    return -1;
  }
  if (status == cudaStreamCaptureStatusNone) {
    // ids, not handles: the handle of a destroyed stream, whose work may still run, can come back.  (Asking for
    // the id of a stream that is being captured would end the capture.)
    if (cudaStreamGetId(stream, &id) != cudaSuccess) {
      cudaGetLastError();
      return -1;
    }
    PartSet &home = h->sets[kHomeSet], &roaming = h->sets[kRoamingSet];
    if (!home.used) {
      home.used = true;
      home.stream = id;
    }
    if (home.stream == id) return kHomeSet;
    if (!h->roaming_done && cudaEventCreateWithFlags(&h->roaming_done, cudaEventDisableTiming) != cudaSuccess) {
      cudaGetLastError();
      h->roaming_done = nullptr;
      return -1;
    }
    if (!roaming.parts && !allocate_parts(h, &roaming)) return -1;
    if (roaming.used && roaming.stream != id && cudaStreamWaitEvent(stream, h->roaming_done, 0) != cudaSuccess) {
      cudaGetLastError();
      return -1;
    }
    roaming.used = true;
    roaming.stream = id;
    return kRoamingSet;
  }
  if (status != cudaStreamCaptureStatusActive) return -1;
  id = reinterpret_cast<uintptr_t>(stream);  // within one capture the handle says enough
  for (int n = kFirstCapturedSet; n < h->n_sets; ++n)
    if (h->sets[n].capture == capture && h->sets[n].stream == id) return n;
  const size_t captured = size_t(h->n_sets - kFirstCapturedSet) * h->part_bytes;
  if (h->n_sets == kMaxPartSets || captured + h->part_bytes > kCapturedPartBytes) return -1;
  PartSet &set = h->sets[h->n_sets];
  if (!allocate_parts(h, &set)) return -1;
  set.stream = id;
  set.capture = capture;
  return h->n_sets++;
}

}  // namespace

namespace steel {

// Encode the tensor maps for (q, k, v) unless `cache` holds them already, fill the problem fields
// of `kp` (whose list and status pointers and view of Q the caller has set) and enqueue the kernel.
steel_status_t launch_with_params(const steel_attn_params_t &p, KernelParams kp, int grid, const void *q,
                                  const void *k, const void *v, void *o, float *lse, cudaStream_t stream,
                                  TensorMaps *cache) {
  TensorMaps local;
  TensorMaps &m = cache ? *cache : local;
  if (m.q_ptr != q || m.k_ptr != k || m.v_ptr != v) {
    m.q_ptr = m.k_ptr = m.v_ptr = nullptr;
    if (!make_map(&m.q, q, p.head_dim, kp.rows_q, int64_t(p.batch) * kp.heads_q) ||
        !make_map(&m.k, k, p.head_dim, p.seq_kv, int64_t(p.batch) * p.heads_kv) ||
        !make_map(&m.v, v, p.head_dim, p.seq_kv, int64_t(p.batch) * p.heads_kv))
      return STEEL_ERR_CUDA;
    m.q_ptr = q;
    m.k_ptr = k;
    m.v_ptr = v;
  }
  kp.o = o;
  kp.o_aligned32 = (reinterpret_cast<uintptr_t>(o) & 31u) == 0;
  kp.lse = lse;
  kp.heads_kv = p.heads_kv;
  kp.seq_q = p.seq_q;
  kp.seq_kv = p.seq_kv;
  kp.mask_flags = p.mask.flags;
  // a window wider than the key sequence hides nothing: clamp it so that the kernel's 32-bit
  // column arithmetic cannot overflow
  kp.window = int32_t(std::min<int64_t>(p.mask.window, int64_t(std::max(p.seq_q, p.seq_kv)) + kTile));
  kp.scale_log2 = p.scale * 1.4426950408889634f;
  if (launch_attention(p.head_dim, p.exp_emulation, m.q, m.k, m.v, kp, grid, stream) != cudaSuccess)
    return STEEL_ERR_CUDA;
  return STEEL_OK;
}

}  // namespace steel

namespace steel {

steel_status_t create_attention(const steel_attn_params_t *params, Spread most, steel_attn_t **out) {
  if (!out) return STEEL_ERR_INVALID_ARG;
  *out = nullptr;
  steel_status_t st = validate_params(params);
  if (st != STEEL_OK) return st;

  // two attributes: all properties take 2.5 ms, most of what creating a handle took
  int device = 0, major = 0, num_sms = 0;
  if (cudaGetDevice(&device) != cudaSuccess ||
      cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, device) != cudaSuccess ||
      cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) {
    cudaGetLastError();
    return STEEL_ERR_CUDA;
  }
  if (major != 10) return STEEL_ERR_CUDA;  // the kernel is built for sm_100a only

  steel_attn *h = new (std::nothrow) steel_attn();
  if (!h) return STEEL_ERR_ALLOC;
  Plan plan, whole;
  std::vector<unsigned char> image;
  try {
    for (Spread spread : {most, Spread::kTiles}) {  // the second only without memory for the first's part buffers
      whole = Plan();
      st = build_plan(params, num_sms, &plan, /*stats=*/true, spread, &whole);
      if (st != STEEL_OK) {
        delete h;
        return st;
      }
      if (plan.split_tiles.empty()) break;
      // part buffers; without memory for them the key ranges stay whole.  Rows in multiples of four: every
      // part's buffer then starts on a 16-byte boundary.
      h->part_rows = int32_t(std::min<int64_t>((plan_rows_q(*params, plan) + 3) / 4 * 4, kTile));
      h->part_bytes = size_t(plan.n_parts) * size_t(h->part_rows) * size_t(params->head_dim + 2) * sizeof(float);
      if (allocate_parts(h, &h->sets[kHomeSet])) break;
    }
    // one image of status word, counters (both zero) and lists
    h->n_split = plan.split_tiles.size();
    const size_t at_arrivals = 256;
    image.resize(at_arrivals + round16(h->n_split * 4 * sizeof(int32_t) * kMaxPartSets));
    h->d_split_tiles = reinterpret_cast<SplitTile *>(image.size());
    image.resize(image.size() + round16(h->n_split * sizeof(SplitTile)));
    if (h->n_split)
      std::memcpy(image.data() + reinterpret_cast<uintptr_t>(h->d_split_tiles), plan.split_tiles.data(),
                  h->n_split * sizeof(SplitTile));
    append_lists(plan, &image, &h->plan);
    if (h->n_split) append_lists(whole, &image, &h->whole);
    h->d_arrivals = reinterpret_cast<int32_t *>(at_arrivals);
  } catch (const std::bad_alloc &) {
    free_device(h);
    delete h;
    return STEEL_ERR_ALLOC;
  }
  h->params = *params;
  h->params.mask.bitmap = nullptr;  // the caller's bitmap is not referenced after create
  h->stats = plan.stats;
  h->device = device;
  h->packed = plan.packed;
  if (cudaMalloc(&h->d_lists, image.size()) != cudaSuccess) {
    cudaGetLastError();
    h->d_lists = nullptr;
    free_device(h);
    delete h;
    return STEEL_ERR_ALLOC;
  }
  h->d_status = reinterpret_cast<int32_t *>(h->d_lists);
  place(&h->d_arrivals, h->d_lists);
  place(&h->d_split_tiles, h->d_lists);
  if (h->n_split == 0) h->d_split_tiles = nullptr;
  place_lists(&h->plan, h->d_lists);
  place_lists(&h->whole, h->d_lists);
  if (cudaMemcpy(h->d_lists, image.data(), image.size(), cudaMemcpyHostToDevice) != cudaSuccess ||
      configure_kernels(params->head_dim, params->exp_emulation) != cudaSuccess ||
      cudaDeviceSynchronize() != cudaSuccess || !encode_fn()) {
    cudaGetLastError();
    free_device(h);
    delete h;
    return STEEL_ERR_CUDA;
  }
  *out = h;
  return STEEL_OK;
}

}  // namespace steel

extern "C" {

steel_status_t steel_attn_create(const steel_attn_params_t *params, steel_attn_t **out) {
  return create_attention(params, Spread::kCut, out);
}

steel_status_t steel_attn_run(steel_attn_t *h, const void *q, const void *k, const void *v, void *o, float *lse,
                              void *cuda_stream) {
  if (!h || !q || !k || !v || !o) return STEEL_ERR_INVALID_ARG;
  if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(o) || (reinterpret_cast<uintptr_t>(lse) & 3u))
    return STEEL_ERR_INVALID_ARG;
  int device = -1;
  if (cudaGetDevice(&device) != cudaSuccess) return STEEL_ERR_CUDA;
  if (device != h->device) return STEEL_ERR_INVALID_ARG;  // the work lists live on the create-time device
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  KernelParams kp{};
  kp.status = h->d_status;
  set_query_view(h->params, h->packed, &kp);
  kp.clock_probe = h->d_clock_probe;
  kp.timeout_cycles = h->timeout_cycles;
  kp.stall_cta = h->stall_cta;
  auto launch = [&](const DeviceLists &lists) {
    kp.items = lists.items;
    kp.cta_begin = lists.cta_begin;
    kp.steps = lists.steps;
    kp.overlap_launch = lists.overlap_launch;
    return launch_with_params(h->params, kp, lists.grid, q, k, v, o, lse, stream, &h->maps);
  };
  if (!h->d_split_tiles) return launch(h->plan);
  std::lock_guard<std::mutex> lock(h->parts_lock);
  const int set = take_part_set(h, stream);
  if (set < 0) return launch(h->whole);
  kp.split_tiles = h->d_split_tiles;
  kp.parts = h->sets[set].parts;
  kp.part_rows = h->part_rows;
  kp.arrivals = h->d_arrivals + size_t(set) * h->n_split * 4;
  const steel_status_t st = launch(h->plan);
  if (set == kRoamingSet && cudaEventRecord(h->roaming_done, stream) != cudaSuccess) {
    cudaGetLastError();
    cudaStreamSynchronize(stream);  // in place of the event
    return STEEL_ERR_CUDA;
  }
  return st;
}

steel_status_t steel_attn_last_status(steel_attn_t *h, void *cuda_stream) {
  if (!h) return STEEL_ERR_INVALID_ARG;
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  // Read and clear on `stream` alone, and wait for both: on the default stream they would wait for work that is not
  // the handle's, and a clear that nothing orders before the handle's next run could take that run's status away.
  int32_t word = 0;
  if (cudaMemcpyAsync(&word, h->d_status, sizeof word, cudaMemcpyDeviceToHost, stream) != cudaSuccess ||
      cudaStreamSynchronize(stream) != cudaSuccess)
    return STEEL_ERR_CUDA;
  if (word != 0 && (cudaMemsetAsync(h->d_status, 0, sizeof(int32_t), stream) != cudaSuccess ||
                    cudaStreamSynchronize(stream) != cudaSuccess))
    return STEEL_ERR_CUDA;
  return word == 0 ? STEEL_OK : STEEL_ERR_TIMEOUT;
}

steel_status_t steel_attn_destroy(steel_attn_t *h) {
  if (!h) return STEEL_OK;
  free_device(h);
  delete h;
  return STEEL_OK;
}

steel_status_t steel_attn_get_stats(const steel_attn_t *h, steel_attn_stats_t *stats) {
  if (!h || !stats) return STEEL_ERR_INVALID_ARG;
  *stats = h->stats;
  return STEEL_OK;
}

steel_status_t steel_attn_plan_host(const steel_attn_params_t *params, steel_attn_stats_t *stats, int32_t *tiles,
                                    int64_t capacity, int64_t *n_tiles) {
  if (!stats) return STEEL_ERR_INVALID_ARG;
  Plan plan;
  steel_status_t st;
  try {
    st = build_plan(params, kPlanHostCtas, &plan);
  } catch (const std::bad_alloc &) {
    return STEEL_ERR_ALLOC;
  }
  if (st != STEEL_OK) return st;
  *stats = plan.stats;
  int64_t n = 0;
  if (tiles) {
    walk_plan(plan, [&](int item, const WorkItem &w, int slot, int, uint32_t entry, bool shared) {
      if (n < capacity) {
        int32_t *rec = tiles + 6 * n;
        rec[0] = item;
        rec[1] = w.batch;
        rec[2] = w.head[slot];
        rec[3] = w.qtile[slot];
        rec[4] = int32_t(entry & kEntryTileMask);
        rec[5] = int32_t(((entry & kEntryPartial) ? 1 : 0) | (shared ? 2 : 0) |
                         (((entry >> kEntrySubShift) & 0xF) << 4));
        ++n;
      }
    }, params);
  }
  if (n_tiles) *n_tiles = n;
  return STEEL_OK;
}

steel_status_t steel_attn_debug_clock_probe(steel_attn_t *h, int64_t *device_pair) {
  if (!h || (reinterpret_cast<uintptr_t>(device_pair) & 7u)) return STEEL_ERR_INVALID_ARG;
  h->d_clock_probe = reinterpret_cast<long long *>(device_pair);
  return STEEL_OK;
}

steel_status_t steel_attn_debug_stall(steel_attn_t *h, int32_t cta, int64_t timeout_cycles) {
  if (!h || cta >= h->plan.grid) return STEEL_ERR_INVALID_ARG;
  h->stall_cta = cta < 0 ? -1 : cta;
  h->timeout_cycles = timeout_cycles > 0 ? std::min<int64_t>(timeout_cycles, kMaxTimeoutCycles) : kDefaultTimeoutCycles;
  return STEEL_OK;
}

const char *steel_status_string(steel_status_t status) {
  switch (status) {
    case STEEL_OK: return "ok";
    case STEEL_ERR_INVALID_ARG: return "invalid argument";
    case STEEL_ERR_UNSUPPORTED: return "unsupported configuration";
    case STEEL_ERR_ALLOC: return "allocation failed";
    case STEEL_ERR_CUDA: return "CUDA error";
    case STEEL_ERR_TIMEOUT: return "device-side wait timed out";
  }
  return "unknown status";
}

}  // extern "C"
