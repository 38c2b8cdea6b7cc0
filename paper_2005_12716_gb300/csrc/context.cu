// Per-device scratch workspace, twiddle table and error reporting.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <memory>
#include <mutex>
#include <string>
#include <vector>

#include "fft.cuh"
#include "internal.cuh"
#include "mlp.cuh"

namespace swense {

static thread_local std::string g_last_error;
static std::atomic<int64_t> g_launches{0};

void count_launches(int n) { g_launches.fetch_add(n, std::memory_order_relaxed); }

void set_error(const std::string& msg) { g_last_error = msg; }

int fail(int status, const std::string& msg) {
  g_last_error = std::string(swense_strerror(status)) + ": " + msg;
  return status;
}

int cuda_fail(cudaError_t e, const char* what) {
  g_last_error = std::string("SWENSE_ERR_CUDA: ") + what + ": " + cudaGetErrorString(e);
  return SWENSE_ERR_CUDA;
}

namespace {

constexpr int kMaxDevices = 64;

// A workspace and the captured graphs (and graphs instantiated from them) that hold its address: they use
// it at every replay, so it lives as long as they do. Counted by user objects of the graphs.
struct Scratch {
  void* p = nullptr;
  size_t bytes = 0;
  std::shared_ptr<std::atomic<int>> graphs = std::make_shared<std::atomic<int>>(0);
};

struct DeviceState {
  Scratch ws;
  // Outgrown while graphs held them; freed by the growth after the last of these is gone, or
  // swense_release. Each is at most four fifths of the one after it, so together they are at most four times
  // the present one.
  std::vector<Scratch> kept;
  bool tw_ready = false;
  // Smallest optional request that could not be had, and how many more of at least its size are answered
  // so without another try: a failing allocation on every call would cost more than the larger scratch
  // gives, and memory may come free later.
  size_t refused = SIZE_MAX;
  int refusals_left = 0;
  size_t limit = SIZE_MAX;      // self-test: larger allocations fail (swense_selftest_workspace_limit)
};
constexpr int kRefusals = 256;

std::mutex g_mutex;
DeviceState g_dev[kMaxDevices];

// Entry j holds e^{+2 pi i e / SWENSE_MAX_FFT}, e = twiddle_exponent(j): the plain table, then the
// pass-major tables (layout at stk_twp), then the wide passes' tables (wide_exponent). Computed in
// FP64 with sincospi (exact argument scaling) and rounded once, so each pass-major entry equals the
// plain entry of the same e bit for bit.
__device__ float2 g_twiddle[kTwiddleAll];

__global__ void k_fill_twiddles() {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= kTwiddleAll) return;
  const int e = j < kWideTw ? twiddle_exponent(j) : wide_exponent(j);
  double s, c;
  sincospi(2.0 * double(e) / double(SWENSE_MAX_FFT), &s, &c);
  g_twiddle[j] = make_float2(float(c), float(s));
}

int current_device(int* dev) {
  SWENSE_CUDA_TRY(cudaGetDevice(dev));
  if (*dev < 0 || *dev >= kMaxDevices) return fail(SWENSE_ERR_UNSUPPORTED, "device index too large");
  return SWENSE_OK;
}

}  // namespace

namespace {

void free_scratch(Scratch& s) {
  cudaDeviceSynchronize();                       // work in flight may still use it
  cudaFree(s.p);
  s = Scratch{};
}

void free_unheld(DeviceState& d) {
  for (size_t i = 0; i < d.kept.size();) {
    if (d.kept[i].graphs->load() > 0) {
      ++i;
    } else {
      free_scratch(d.kept[i]);
      d.kept.erase(d.kept.begin() + i);
    }
  }
}

// A new workspace in place of the device's own, which is freed (unless a graph holds it) once the new one
// is there.
cudaError_t replace_workspace(DeviceState& d, size_t want) {
  void* p = nullptr;
  const cudaError_t e = want > d.limit ? cudaErrorMemoryAllocation : cudaMalloc(&p, want);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return e;
  }
  if (d.ws.p) {
    if (d.ws.graphs->load() > 0) d.kept.push_back(d.ws);
    else free_scratch(d.ws);
  }
  d.ws = Scratch{};
  d.ws.p = p;
  d.ws.bytes = want;
  if (want >= d.refused) d.refused = SIZE_MAX;
  return cudaSuccess;
}

void CUDART_CB drop_graph(void* held) {
  auto* g = static_cast<std::shared_ptr<std::atomic<int>>*>(held);
  --**g;
  delete g;
}

// The workspace is used by work captured on `stream`: the graph holds it.
int hold_for_capture(DeviceState& d, cudaStream_t stream) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  cudaGraph_t graph = nullptr;
  if (cudaStreamGetCaptureInfo(stream, &cap, nullptr, &graph, nullptr, nullptr, nullptr) != cudaSuccess) {
    cudaGetLastError();                          // (the legacy stream beside a capture: its launch will say so)
    return SWENSE_OK;
  }
  if (cap != cudaStreamCaptureStatusActive) return SWENSE_OK;
  auto* held = new std::shared_ptr<std::atomic<int>>(d.ws.graphs);
  ++**held;
  cudaUserObject_t obj = nullptr;
  cudaError_t e = cudaUserObjectCreate(&obj, held, drop_graph, 1, cudaUserObjectNoDestructorSync);
  if (e != cudaSuccess) {
    drop_graph(held);
    return cuda_fail(e, "cudaUserObjectCreate");
  }
  e = cudaGraphRetainUserObject(graph, obj, 1, cudaGraphUserObjectMove);
  if (e != cudaSuccess) {
    cudaUserObjectRelease(obj, 1);
    return cuda_fail(e, "cudaGraphRetainUserObject");
  }
  return SWENSE_OK;
}

int grow(size_t bytes, cudaStream_t stream, void** out, bool optional) {
  int dev;
  int st = current_device(&dev);
  if (st) return st;
  std::lock_guard<std::mutex> lock(g_mutex);
  DeviceState& d = g_dev[dev];
  bytes = (bytes + 255) & ~size_t(255);
  if (bytes <= d.ws.bytes) {
    *out = d.ws.p;
    return hold_for_capture(d, stream);
  }
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  SWENSE_CUDA_TRY(cudaStreamIsCapturing(stream, &cap));
  const bool capturing = cap != cudaStreamCaptureStatusNone;
  if (optional && (capturing || (bytes >= d.refused && d.refusals_left-- > 0))) return SWENSE_ERR_OOM;
  if (capturing)
    return fail(SWENSE_ERR_ARG, "scratch workspace must grow, which is not allowed during stream "
                                "capture; make one call with the same sizes before capturing");
  free_unheld(d);
  const size_t want = bytes + bytes / 4;         // headroom so small growth does not reallocate
  cudaError_t e = replace_workspace(d, want);
  if (e != cudaSuccess && optional) {
    d.refused = std::min(d.refused, bytes);
    d.refusals_left = kRefusals;
    return SWENSE_ERR_OOM;
  }
  if (e != cudaSuccess && d.ws.p && d.ws.graphs->load() == 0) {   // no room for both: give up the old one first
    free_scratch(d.ws);
    e = replace_workspace(d, want);
  }
  if (e != cudaSuccess)
    return fail(SWENSE_ERR_OOM, "cudaMalloc of the scratch workspace (" + std::to_string(want) + " bytes) failed: " +
                                    cudaGetErrorString(e) +
                                    (d.ws.p || !d.kept.empty() ? "; captured graphs hold the present one" : ""));
  *out = d.ws.p;
  return SWENSE_OK;
}

}  // namespace

int workspace(size_t bytes, cudaStream_t stream, void** out) { return grow(bytes, stream, out, false); }
int workspace_optional(size_t bytes, cudaStream_t stream, void** out) { return grow(bytes, stream, out, true); }

int twiddles(cudaStream_t stream, const float2** out) {
  int dev;
  int st = current_device(&dev);
  if (st) return st;
  {
    std::lock_guard<std::mutex> lock(g_mutex);
    if (!g_dev[dev].tw_ready) {
      // Filled once per device and waited for, so that every later stream sees it.
      cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
      SWENSE_CUDA_TRY(cudaStreamIsCapturing(stream, &cap));
      if (cap != cudaStreamCaptureStatusNone)
        return fail(SWENSE_ERR_ARG, "the first call on a device must not be inside a stream "
                                    "capture (it fills the twiddle table)");
      k_fill_twiddles<<<(kTwiddleAll + 255) / 256, 256, 0, stream>>>();
      SWENSE_CUDA_TRY(cudaGetLastError());
      count_launches(1);
      SWENSE_CUDA_TRY(cudaStreamSynchronize(stream));
      g_dev[dev].tw_ready = true;
    }
  }
  void* p = nullptr;
  SWENSE_CUDA_TRY(cudaGetSymbolAddress(&p, g_twiddle));
  *out = static_cast<const float2*>(p);
  return SWENSE_OK;
}

}  // namespace swense

extern "C" {

int64_t swense_workspace_bytes(void) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= swense::kMaxDevices) return 0;
  std::lock_guard<std::mutex> lock(swense::g_mutex);
  size_t bytes = swense::g_dev[dev].ws.bytes;
  for (const swense::Scratch& s : swense::g_dev[dev].kept) bytes += s.bytes;
  return int64_t(bytes);
}

int swense_release(void) {
  int dev = 0;
  SWENSE_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= swense::kMaxDevices) return SWENSE_OK;
  std::lock_guard<std::mutex> lock(swense::g_mutex);
  swense::DeviceState& d = swense::g_dev[dev];
  if (d.ws.p) SWENSE_CUDA_TRY(cudaDeviceSynchronize());
  if (d.ws.p) swense::free_scratch(d.ws);
  for (swense::Scratch& s : d.kept) swense::free_scratch(s);
  d.kept.clear();
  d.refused = SIZE_MAX;
  d.refusals_left = 0;
  return SWENSE_OK;
}

int swense_selftest_workspace_limit(int64_t bytes) {
  int dev = 0;
  int st = swense::current_device(&dev);
  if (st) return st;
  std::lock_guard<std::mutex> lock(swense::g_mutex);
  swense::g_dev[dev].limit = bytes > 0 ? size_t(bytes) : SIZE_MAX;
  return SWENSE_OK;
}

const char* swense_last_error(void) { return swense::g_last_error.c_str(); }

const char* swense_strerror(int status) {
  switch (status) {
    case SWENSE_OK: return "SWENSE_OK";
    case SWENSE_ERR_ARG: return "SWENSE_ERR_ARG";
    case SWENSE_ERR_SIZE: return "SWENSE_ERR_SIZE";
    case SWENSE_ERR_LEVELS: return "SWENSE_ERR_LEVELS";
    case SWENSE_ERR_OOM: return "SWENSE_ERR_OOM";
    case SWENSE_ERR_CUDA: return "SWENSE_ERR_CUDA";
    case SWENSE_ERR_TIMEOUT: return "SWENSE_ERR_TIMEOUT";
    case SWENSE_ERR_UNSUPPORTED: return "SWENSE_ERR_UNSUPPORTED";
    case SWENSE_ERR_CONVERGENCE: return "SWENSE_ERR_CONVERGENCE";
    default: return "SWENSE_ERR_UNKNOWN";
  }
}

int swense_async_status(int32_t reset, void* stream) {
  SWENSE_CUDA_TRY(cudaStreamSynchronize(static_cast<cudaStream_t>(stream)));
  int grid = 0, direct = 0, learned = 0;
  int st = swense::grid_async_flag(reset != 0, &grid);
  if (!st) st = swense::direct_async_flag(reset != 0, &direct);
  if (!st) st = swense::learned_async_flag(reset != 0, &learned);
  if (st) return st;
  if (grid)
    return swense::fail(SWENSE_ERR_TIMEOUT, "a bounded wait of a staged row pass (k_row_w, k_row_tma) gave "
                                            "up; the grid rows of that block or warp were not written");
  if (direct)
    return swense::fail(SWENSE_ERR_TIMEOUT, "a bounded wait of the tensor-core direct sum "
                                            "(k_direct_tc) gave up; the outputs of that tile were "
                                            "not written");
  if (learned)
    return swense::fail(SWENSE_ERR_TIMEOUT, "a bounded wait of the learned gather (k_interp_learned) gave "
                                            "up; u, v, w, p of those points are NaN");
  return SWENSE_OK;
}

int swense_version(void) { return SWENSE_VERSION; }

int64_t swense_launches(void) { return swense::g_launches.load(std::memory_order_relaxed); }

}  // extern "C"
