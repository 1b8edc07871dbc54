// ed_double_occupation_static: the double-occupancy reduction of
// ed_double_occupation with its scratch memory in a fixed device array of
// this library instead of a per-call allocation.  It serves callers that
// must not allocate device memory while they run: code inside a region whose
// device memory is fixed up front (a latency-critical step loop, a memory
// budget enforced by the host application), or hosts that cannot call
// cudaMalloc at that point.
#include <cuda_runtime.h>

#include <mutex>

#include "ctx.h"
#include "kernels.cuh"

namespace ed {

namespace {

constexpr int64_t kStaticMaxElems = 67108864;
constexpr int kStaticMaxDevices = 64;

// Partial sums of every block (1024 rows of 17 doubles) followed by the
// final sums (one row): 139,400 bytes per device.
static_assert(kDoccScratchDoubles * sizeof(double) == 139400, "the documented size");
__device__ __align__(256) double g_docc_scratch[kDoccScratchDoubles];

std::mutex g_scratch_mutex;
double* g_scratch_ptr[kStaticMaxDevices] = {nullptr};

// Device address of the scratch array on the current device, looked up once
// per device.  In host code the array's name is only a host-side stand-in, so
// the address must come from cudaGetSymbolAddress.
cudaError_t scratch_address(double** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kStaticMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_scratch_mutex);
  if (!g_scratch_ptr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_docc_scratch);
    if (e != cudaSuccess) return e;
    g_scratch_ptr[dev] = static_cast<double*>(p);
  }
  *out = g_scratch_ptr[dev];
  return cudaSuccess;
}

}  // namespace
}  // namespace ed

using namespace ed;

extern "C" ed_status ed_double_occupation_static(ed_ctx* ctx, const void* psi, ed_dtype dtype,
                                                 double* d_avg, double* d_site, void* stream) {
  if (!ctx || !psi || !d_avg) return fail(ctx, ED_ERR_ARG, "NULL argument");
  if (dtype != ED_C128 && dtype != ED_C64) return fail(ctx, ED_ERR_ARG, "bad dtype");
  const int64_t D = ctx->dim_up * ctx->dim_dn;
  if (D > kStaticMaxElems)
    return fail(ctx, ED_ERR_UNSUPPORTED,
                "ed_double_occupation_static: sector dimension " + std::to_string(D) +
                    " exceeds its fixed scratch (at most 67,108,864 elements); use "
                    "ed_double_occupation");
  if (!ctx->lattice_set || !ctx->sec.uploaded)
    return fail(ctx, ED_ERR_STATE,
                "ed_double_occupation_static needs the context's tables on the device "
                "already (call any GPU entry point on this context first)");
  if (!is_device_ptr(psi)) return fail(ctx, ED_ERR_ARG, "psi must be a device pointer");
  // the tables and psi must live on the current device, whose scratch array
  // the kernels below use
  if (ed_status e = check_device(ctx, {psi})) return e;
  double* scratch = nullptr;
  CK(ctx, scratch_address(&scratch));
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  CK(ctx, docc_sites(dtype == ED_C128, psi, ctx->sec.dev, ctx->Ns, scratch, d_avg, d_site, s));
  return ED_OK;
}
