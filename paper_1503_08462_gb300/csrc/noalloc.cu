// Allocation-free variant of the dense symmetric eigensolver entry point.
//
// Some callers cannot allocate device memory at the time they need the
// eigensolver: code running inside a memory pool that forbids outside
// cudaMalloc/cudaFree, callers that must not synchronise the device (cudaFree
// does), or embedded hosts whose allocator is owned by another runtime.  This
// entry point takes device pointers for its input and outputs and keeps all of
// its scratch in one file-scope __device__ array of fixed size, so it calls no
// cudaMalloc, cudaFree or allocating library routine.
//
// The array costs every GPU that loads the library kNoAllocScratchBytes of
// device memory until the process exits.  All calls on a device share it, and
// it keeps the contents of the last call; the eigensolver writes every scratch
// element before reading it, so nothing needs clearing between calls.  Calls
// whose executions overlap on the GPU (different streams, or different host
// threads) race on the array: serialise them.
#include <cuda_runtime.h>

#include <cstring>
#include <mutex>
#include <string>

#include "amgeig.h"
#include "common.cuh"
#include "kernels.cuh"
#include "prof.cuh"

namespace amgeig {
namespace {

constexpr int kNoAllocMaxN = 128;
constexpr int kNoAllocMaxWant = 64;
constexpr size_t kNoAllocScratchBytes = 544 * 1024;  // n = 128, nwant = 64 take 516 KiB

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

constexpr int kMaxDevices = 64;
std::mutex g_mu;
void* g_scratch_ptr[kMaxDevices] = {};

// Device address of the scratch array on the current device (looked up once per device).
int scratch_address(int device, void** out) {
  std::lock_guard<std::mutex> lk(g_mu);
  if (device < 0 || device >= kMaxDevices) return set_last_error(AMGEIG_EINVAL, "device ordinal beyond 63");
  if (!g_scratch_ptr[device]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess)
      return set_last_error(AMGEIG_ECUDA, (std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e)).c_str());
    g_scratch_ptr[device] = p;
  }
  *out = g_scratch_ptr[device];
  return AMGEIG_OK;
}

}  // namespace
}  // namespace amgeig

using namespace amgeig;

extern "C" int amgeig_sym_eigh_noalloc(int n, int nwant, const double* H, double* evals, double* evecs,
                                       void* stream) {
  set_last_error(AMGEIG_OK, nullptr);
  if (!H || !evals || !evecs) return set_last_error(AMGEIG_EINVAL, "NULL pointer");
  if (n < 1 || nwant < 1 || nwant > n) return set_last_error(AMGEIG_EINVAL, "need 1 <= nwant <= n");
  if (n > kNoAllocMaxN || nwant > kNoAllocMaxWant)
    return set_last_error(AMGEIG_EINVAL, "n > 128 or nwant > 64: beyond the fixed scratch array");
  int device = 0;
  cudaError_t ge = cudaGetDevice(&device);
  if (ge != cudaSuccess)
    return set_last_error(AMGEIG_ECUDA, (std::string("cudaGetDevice: ") + cudaGetErrorString(ge)).c_str());
  void* base = nullptr;
  int rc = scratch_address(device, &base);
  if (rc) return rc;
  if (syev_scratch_bytes(n, nwant) > kNoAllocScratchBytes)
    return set_last_error(AMGEIG_EINVAL, "scratch layout exceeds the fixed array");
  launch_syev_df_into(n, nwant, H, evals, evecs, base, static_cast<cudaStream_t>(stream));
  cudaError_t le = cudaGetLastError();
  if (le != cudaSuccess)
    return set_last_error(AMGEIG_ECUDA, (std::string("eigensolver launch: ") + cudaGetErrorString(le)).c_str());
  return AMGEIG_OK;
}
