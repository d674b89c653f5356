// fock_build_jk_noalloc: the J/K build with its per-call scratch in a fixed
// device array owned by the library instead of memory obtained per call.
//
// Who needs this: callers that must not allocate device memory while they
// run, such as services that reserve their whole memory budget at start-up,
// applications whose allocator policy forbids the CUDA runtime's
// stream-ordered pool (cudaMallocAsync), and real-time loops where an
// allocation could stall.  fock_build_jk takes its scratch from the pool on
// every call; this variant takes it from g_noalloc_scratch below and calls no
// allocation routine at all.  It launches the same kernels with the same
// arguments as fock_build_jk, in both precisions.
#include "fock_impl.h"

namespace fk {
namespace {

// Per-call scratch of fock_build_jk_noalloc, laid out as in fock_build_jk
// (scratch_layout): the shell-block density maxima (nshell^2 doubles), kCounters
// work counters per tier and the bits of max|D|, the FP32 copy of D (N^2 floats, mixed
// precision only), the FP32 shell-block maxima (nshell^2 floats) and, in the
// decay-bound exchange mode, the bounds (nshell^2 floats), distance bins and
// fit, each part 256-byte aligned.  Every GPU that loads the library keeps
// this array for the life of the process.
constexpr size_t kNoallocBytes = 4u << 20;  // 4 MiB: FP64 handles up to 591 shells
// The counters of f-shell handles take up to 1280 bytes (100 ordered class
// pairs); what they take beyond the first 256 lies in a tail of the array, so
// that they do not move the limit of nshell and N.
constexpr size_t kNoallocTail = 1024;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoallocBytes + kNoallocTail];

}  // namespace
}  // namespace fk

using namespace fk;

extern "C" fock_status fock_build_jk_noalloc(const fock_shellpairs *sp, const double *D, double schwarz_thresh,
                                             double *J, double *K, cudaStream_t stream) {
  const fock_status s = check_build_args(sp, D, schwarz_thresh, J, K);
  if (s != FOCK_OK) return s;
  const ScratchLayout L = scratch_layout(sp);
  const size_t cnt = L.df_off - L.cnt_off;  // counters, a multiple of 256
  if (L.total > kNoallocBytes + (cnt - 256) || L.total > kNoallocBytes + kNoallocTail)
    return FOCK_ERR_INVALID_ARG;  // basis too large for the fixed array
  RelaxedCaptureMode relaxed;
  // In host code g_noalloc_scratch names a host-side stand-in; the device
  // address comes from cudaGetSymbolAddress with the device current.  It is
  // looked up on every call: the array belongs to the library's module in
  // the device's current context, and a context torn down and created again
  // (cudaDeviceReset) may place it elsewhere.  The lookup is cheap once the
  // module is loaded; the first call on a device loads it.
  void *scratch = nullptr;
  const cudaError_t e = cudaGetSymbolAddress(&scratch, g_noalloc_scratch);
  if (e != cudaSuccess) return cuda_status(e, "cudaGetSymbolAddress");
  return enqueue_build(sp, D, schwarz_thresh, J, K, (char *)scratch, stream, nullptr);
}
