// lb_noalloc.cu -- lb_structure_export for callers that cannot allocate device
// memory per call: processes whose host framework's caching allocator has
// reserved the device memory (a cudaMalloc there fails or fragments the pool,
// and a cudaFree synchronizes the whole device, stalling every other stream),
// and real-time or embedded callers that reserve all memory once at start-up
// and may not allocate afterwards.  The export places every row by its closed
// form and needs no scratch; this entry point also keeps its limit on N.  The
// paper has no counterpart: it is a deployment concern of this library.
#include "lb_internal.h"

namespace {

// Largest M this entry point takes: N <= 256 (M = N^2 - 1 = 65535).
constexpr int64_t kNoAllocMaxM = 65535;

}  // namespace

extern "C" {

int lb_structure_export_noalloc(const lb_basis_t* b, int which, int32_t* idx3, double* val, int64_t capacity,
                                int64_t* nnz, void* stream) {
  if (b == nullptr || nnz == nullptr) {
    lbi::set_error("lb_structure_export_noalloc: NULL argument");
    return LB_EINVAL;
  }
  if (which != LB_F && which != LB_D) {
    lbi::set_error("lb_structure_export_noalloc: which = %d", which);
    return LB_EINVAL;
  }
  if (b->M > kNoAllocMaxM) {
    lbi::set_error("lb_structure_export_noalloc: M = %lld (N = %d) exceeds the maximum "
                   "M = %lld (N = 256); use lb_structure_export",
                   (long long)b->M, b->N, (long long)kNoAllocMaxM);
    return LB_EINVAL;
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int64_t total = lbi::structure_total(b->N, which);
  *nnz = total;
  if (idx3 == nullptr || val == nullptr) {
    lbi::set_error("lb_structure_export_noalloc: NULL output buffer");
    return LB_EINVAL;
  }
  if (capacity < total) {
    lbi::set_error("lb_structure_export_noalloc: capacity %lld < %lld triples", (long long)capacity,
                   (long long)total);
    return LB_EINVAL;
  }
  cudaError_t e = lbi::structure_fill(b->view(), which, idx3, val, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return lbi::cuda_fail(e, "lb_structure_export_noalloc: fill");
  return LB_OK;
}

}  // extern "C"
