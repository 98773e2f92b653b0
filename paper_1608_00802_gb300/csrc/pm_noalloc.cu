// pm_deposit_noalloc: the cloud-in-cell deposit for callers that must not
// allocate device memory.  Some callers cannot call cudaMalloc or cudaFree:
// cudaFree synchronises the whole device and cudaMalloc may block, which a
// latency-critical serving loop or a real-time thread cannot afford, and a
// process that has already handed its whole device-memory budget to fixed
// arenas has nothing left to allocate from.  This entry point therefore keeps
// every temporary (particle records, sort keys, row starts) in one file-scope static device array
// of PM_NOALLOC_SCRATCH_BYTES, which every GPU that loads the library holds
// until the process exits.  It calls no allocating routine, its own or a
// library's.
#include <cuda_runtime.h>
#include <stdio.h>
#include <string.h>

#include <atomic>
#include <mutex>

#include "../../include/pm.h"
#include "pm_internal.h"

using namespace pm;

namespace {

constexpr int64_t kMaxPart = PM_NOALLOC_MAX_PARTICLES;
constexpr int kMaxMesh = PM_NOALLOC_MAX_MESH;
static_assert(kMaxPart <= SORT_SMALL_MAX, "the deposit sorts with the one-kernel sort");

constexpr size_t align256(size_t v) { return (v + 255) & ~size_t(255); }

// offsets inside the static scratch array
constexpr size_t kPos0 = 0;
constexpr size_t kPos1 = kPos0 + align256(kMaxPart * 16);
constexpr size_t kKeys = kPos1 + align256(kMaxPart * 16);
constexpr size_t kRows = kKeys + align256(kMaxPart * 4);
constexpr size_t kErr = kRows + align256((size_t(kMaxMesh) * kMaxMesh + CROWD_WORDS) * 4);
constexpr size_t kTotal = kErr + 256;
static_assert(kTotal <= PM_NOALLOC_SCRATCH_BYTES, "scratch layout exceeds PM_NOALLOC_SCRATCH_BYTES");

static __device__ __align__(256) unsigned char g_scratch[PM_NOALLOC_SCRATCH_BYTES];

// Device address of g_scratch per device, looked up once per device (with
// that device current) by the first call made on it.
std::mutex g_mu;
void* g_addr[64];
bool g_ready[64];
// A call is on its way, or stopped at an error between its launches: the error word may hold bits of positions that
// it placed.  The next call clears them.
std::atomic<bool> g_unfinished[64];

thread_local char g_msg[256];
thread_local int g_fail_after = -1;  // test aid: launches after which this thread's next call "fails"

// hands the call's error bits to the caller's word (device or mapped host
// memory) and clears them for the next call
__global__ void k_copy_error(uint32_t* err, uint32_t* out) {
  *out = *err;
  *err = 0;
}

// the message goes where pm_last_error(NULL) reads it
pm_status nfail(pm_status st, const char* msg) {
  set_global_error(msg);
  return st;
}

pm_status scratch_address(unsigned char** out, int* device) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nfail(PM_ERR_CUDA, "no current device");
  std::lock_guard<std::mutex> lock(g_mu);  // also serialises the message buffer
  if (!g_ready[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_scratch);
    if (e == cudaSuccess) e = deposit_prepare<float>();
    if (e != cudaSuccess || !p) {
      snprintf(g_msg, sizeof g_msg, "static scratch address or deposit preparation: %s", cudaGetErrorString(e));
      return nfail(PM_ERR_CUDA, g_msg);
    }
    g_addr[dev] = p;
    g_ready[dev] = true;
  }
  *out = static_cast<unsigned char*>(g_addr[dev]);
  *device = dev;
  return PM_OK;
}

}  // namespace

extern "C" {

pm_status pm_deposit_noalloc(const double* x_dev, int64_t n_part, int32_t n_mesh, double box, float* rho_dev,
                             uint32_t* err_dev, void* stream) {
  if (n_part < 1 || n_part > kMaxPart) {
    snprintf(g_msg, sizeof g_msg, "n_part = %lld is outside [1, %lld], the static scratch limit", (long long)n_part,
             (long long)kMaxPart);
    return nfail(PM_ERR_INVALID_ARG, g_msg);
  }
  if (n_mesh < 8 || n_mesh > kMaxMesh || (n_mesh & 1)) {
    snprintf(g_msg, sizeof g_msg, "n_mesh = %d must be even and in [8, %d], the static scratch limit", n_mesh,
             kMaxMesh);
    return nfail(PM_ERR_INVALID_ARG, g_msg);
  }
  if (!x_dev || !rho_dev || !(box > 0)) return nfail(PM_ERR_INVALID_ARG, "x, rho must be device pointers, box > 0");
  unsigned char* base = nullptr;
  int dev = 0;
  pm_status st = scratch_address(&base, &dev);
  if (st != PM_OK) return st;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const int64_t n = n_part;
  Mesh m;
  m.n = n_mesh;
  m.log2n = (n_mesh & (n_mesh - 1)) == 0 ? __builtin_ctz(unsigned(n_mesh)) : -1;
  m.n2 = uint32_t(n_mesh) * uint32_t(n_mesh);
  m.n3 = m.n2 * uint32_t(n_mesh);
  int bits = 0;
  while ((uint32_t(1) << bits) < m.n3) ++bits;
  uint32_t* err = reinterpret_cast<uint32_t*>(base + kErr);
  uint32_t* keys = reinterpret_cast<uint32_t*>(base + kKeys);
  uint32_t* rows = reinterpret_cast<uint32_t*>(base + kRows);
  void* pos[2] = {base + kPos0, base + kPos1};

  int fail_after = g_fail_after;
  g_fail_after = -1;
#define NA_CU(expr)                                                                             \
  do {                                                                                          \
    cudaError_t e_ = fail_after-- == 0 ? cudaErrorLaunchFailure : (expr);                       \
    if (e_ != cudaSuccess) {                                                                    \
      snprintf(g_msg, sizeof g_msg, "%s: %s", #expr, cudaGetErrorString(e_));                   \
      return nfail(PM_ERR_CUDA, g_msg);                                                         \
    }                                                                                           \
  } while (0)
  // the array keeps the previous call's contents; every buffer is written before it is read, except the error
  // word, which starts at zero and is zero again after each call that came to its end: cleared as it is handed
  // over, or, with nobody to hand it to, by the sort
  const bool stale = g_unfinished[dev].exchange(true);
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  if (stale) {
    NA_CU(cudaMemsetAsync(err, 0, 4, s));
    NA_CU(cudaStreamIsCapturing(s, &capture));
  }
  // positions to cell + offset as pm_set_particles converts them (1/dx with dx = box/N)
  NA_CU(launch_init_particles<float>(x_dev, nullptr, n, m, 1.0 / (box / n_mesh), pos[0], nullptr, keys, err, s));
  NA_CU(launch_sort_small<float>(keys, n, bits, keys, pos[0], nullptr, pos[1], nullptr, rows, m,
                                 err_dev ? nullptr : err, s));
  NA_CU(launch_deposit<float>(pos[1], rows, n, m, double(m.n3) / double(n), rho_dev, s,
                              default_tuning(n_mesh, n, false).dep_warps));
  if (err_dev) {
    k_copy_error<<<1, 1, 0, s>>>(err, err_dev);
    NA_CU(cudaGetLastError());
  }
#undef NA_CU
  g_unfinished[dev] = stale && capture != cudaStreamCaptureStatusNone;  // (a captured clear has not run yet)
  return PM_OK;
}

pm_status pm_debug_fail_noalloc(int32_t launches) {
  if (launches < -1 || launches > 2) return nfail(PM_ERR_INVALID_ARG, "launches must be in [-1, 2]");
  g_fail_after = launches;
  return PM_OK;
}

}  // extern "C"
