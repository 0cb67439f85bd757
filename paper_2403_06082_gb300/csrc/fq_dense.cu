// Weight reconstruction (include/framequant_dense.h): W_hat = T_out^T diag(gamma) C_hat T_in
// as the FQ_BF16 forward of the d_in unit vectors.  The forward of unit vector e_j is column j
// of W_hat, and the synthesis writes its output that way round.  The analysis of e_j is column j
// of T_in, exact in bf16, so the chain starts from that transpose and runs only the code product
// and the synthesis on the tensor cores.
#include <cuda_runtime.h>

#include "fq_internal.h"
#include "framequant_dense.h"

namespace fq {
namespace {

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

}  // namespace
}  // namespace fq

using namespace fq;

extern "C" {

size_t fq_reconstruct_workspace_bytes(int d_in, int n_in, int n_out, int d_out) {
  if (d_in <= 0 || n_in <= 0 || n_out <= 0 || d_out <= 0) return 0;
  return tc_workspace_bytes(d_in, d_in, n_in, n_out, d_out, 0);
}

fq_status fq_reconstruct_weight(const void* T_in, const fq_packed* C, const void* T_out_t,
                                int d_in, int d_out, const float* gamma, void* W_hat, void* ws,
                                size_t ws_bytes, fq_stream_t stream) {
  if (!T_in || !C || !T_out_t || !W_hat || d_in <= 0 || d_out <= 0) return FQ_ERR_INVALID_ARG;
  // the checks of the forward this call makes, before anything is launched
  if (const fq_status cs = check_packed(C)) return cs;
  if (d_in % 8 || d_out % 8 || !aligned16(W_hat) || !aligned16(T_in) || !aligned16(T_out_t) ||
      (gamma && !aligned16(gamma)))
    return FQ_ERR_ALIGNMENT;
  if (!ws) return FQ_ERR_WORKSPACE;
  if ((reinterpret_cast<uintptr_t>(ws) & 255u) != 0) return FQ_ERR_ALIGNMENT;
  if (ws_bytes < fq_reconstruct_workspace_bytes(d_in, C->n_in, C->n_out, d_out))
    return FQ_ERR_WORKSPACE;
  {
    int dev = 0, major = 0, minor = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev) != cudaSuccess)
      return FQ_ERR_CUDA;
    if (major * 10 + minor != 103) return FQ_ERR_UNSUPPORTED;
  }
  // every check of the chain passed above (sizes, alignment, workspace, device)
  return launch_tc_unit_forward(T_in, d_in, *C, T_out_t, d_out, gamma, W_hat,
                                static_cast<char*>(ws), ws_bytes,
                                reinterpret_cast<cudaStream_t>(stream));
}

}  // extern "C"
