// ada_ldlp_eval_static: the length predictor (class-logit form) for callers that cannot allocate.
//
// Every other entry point works inside a workspace the caller allocated.  Some callers have no way
// to get one: code that runs after the process has handed all device memory to another allocator,
// plugins called from inside a host framework that forbids cudaMalloc on its threads, or anything
// running where an allocation would synchronise the device at a bad moment.  For them this one
// call keeps its scratch (the predictor's hidden activations) in a fixed array that is part of the
// library image: ADA_STATIC_MAX_HIDDEN floats (16 KiB) on every GPU that loads the library, held
// until the process exits.
//
// The array is shared by all calls on a device and keeps what the last call wrote.  Nothing in it has
// to start at zero: a call overwrites every entry it later reads.  Two calls that overlap on the
// GPU (different streams, or threads racing on one device) use the same array and corrupt each
// other; callers must order them.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <atomic>

#include "ada.h"
#include "ada_ldlp.cuh"

namespace {

static __device__ __align__(256) float g_ldlp_hidden[ADA_STATIC_MAX_HIDDEN];

// In host code the name above is only a handle; the device address is looked up once per device.
constexpr int kMaxDevices = 64;
std::atomic<float *> g_scratch_addr[kMaxDevices];   // (zero-initialised; threads racing on the first call store the same address)

using ada::kLdlpThreads;
using ada::kLdlpUnits;

// hidden = ReLU(W1 [e ; f] + b1); the kernel after this one may start its own loads meanwhile.  Launched plainly: the call
// is ordered behind all that was enqueued before it.  7B widths, whole call: 30.7 us with one warp and element-wise loads per
// hidden unit; now 8.2 us back to back with the weights in level 2, 13.3 us for one call with them in HBM.  (One launch whose last
// block takes the outputs: 10.3 and 14.3 us.  With programmatic serialization 7.8 and 14.3, but behind a kernel of the caller's
// that was itself launched so and ends without waiting, that would start before the kernels in front of it have completed.)
template <bool VEC>
__global__ void __launch_bounds__(kLdlpThreads) k_static_hidden(const __nv_bfloat16 *w1, const __nv_bfloat16 *b1,
                                                                const __nv_bfloat16 *e, const float *f, int d, int hid,
                                                                float *hidden) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  ada::ldlp_hidden_block<VEC>(w1, b1, e, f, d, hid, blockIdx.x * kLdlpUnits, hidden);
}

// z = W2 hidden + b2, one warp per output; n = argmax + 1, lowest index among equals.  Launched with programmatic
// serialization behind the kernel above: the weights are requested before it waits for the hidden activations.
template <bool VEC>
__global__ void __launch_bounds__(32 * ADA_MAX_NMAX) k_static_out(const float *hidden, const __nv_bfloat16 *w2,
                                                                  const __nv_bfloat16 *b2, int hid, int nmax, int *n_out,
                                                                  float *z_out) {
  __shared__ float zs[ADA_MAX_NMAX];
  const int c = threadIdx.x >> 5, lane = threadIdx.x & 31;
  ada::LdlpRow row;
  const __nv_bfloat16 *w = w2 + (size_t)c * hid;
  ada::ldlp_out_ahead<VEC>(w, hid, row);
  const float bias = __bfloat162float(b2[c]);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const float z = ada::ldlp_out_dot<VEC>(w, hidden, hid, row) + bias;
  if (lane == 0) {
    zs[c] = z;
    if (z_out) z_out[c] = z;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    float best = -INFINITY;
    int bi = 0;
    for (int i = 0; i < nmax; ++i)
      if (zs[i] > best) { best = zs[i]; bi = i; }
    *n_out = bi + 1;
  }
}

template <bool VEC>
cudaError_t launch(const __nv_bfloat16 *w1, const __nv_bfloat16 *b1, const __nv_bfloat16 *w2, const __nv_bfloat16 *b2,
                   const __nv_bfloat16 *e, const float *f, int d, int hid, int nmax, int *n, float *z, float *hidden, cudaStream_t st) {
  k_static_hidden<VEC><<<(hid + kLdlpUnits - 1) / kLdlpUnits, kLdlpThreads, 0, st>>>(w1, b1, e, f, d, hid, hidden);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(1); cfg.blockDim = dim3(32 * nmax); cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_static_out<VEC>, (const float *)hidden, w2, b2, hid, nmax, n, z);
}

}  // namespace

extern "C" int ada_ldlp_eval_static(const void *d_w1, const void *d_b1, const void *d_w2, const void *d_b2,
                                    const void *d_embed_row, const float *d_feature, int32_t d_model, int32_t hidden,
                                    int32_t n_max, int32_t *d_n, float *d_z, void *cuda_stream) {
  if (!d_w1 || !d_b1 || !d_w2 || !d_b2 || !d_embed_row || !d_feature || !d_n) return ADA_ERR_NULL;
  if (hidden > ADA_STATIC_MAX_HIDDEN) return ADA_ERR_TOO_LARGE;
  if (d_model < 1 || hidden < 1 || n_max < 1 || n_max > ADA_MAX_NMAX) return ADA_ERR_RANGE;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return ADA_ERR_CUDA;
  float *scratch = g_scratch_addr[dev].load(std::memory_order_acquire);
  if (!scratch) {  // first call on this device (it is the current one): look the array up
    if (cudaGetSymbolAddress((void **)&scratch, g_ldlp_hidden) != cudaSuccess || !scratch) return ADA_ERR_CUDA;
    g_scratch_addr[dev].store(scratch, std::memory_order_release);
  }
  cudaStream_t st = (cudaStream_t)cuda_stream;
  const __nv_bfloat16 *w1 = (const __nv_bfloat16 *)d_w1, *b1 = (const __nv_bfloat16 *)d_b1, *w2 = (const __nv_bfloat16 *)d_w2,
                      *b2 = (const __nv_bfloat16 *)d_b2, *e = (const __nv_bfloat16 *)d_embed_row;
  // 16-byte loads where every row starts on 16 bytes (the caller's pointers need no more than their type's alignment)
  const bool vec = d_model % 8 == 0 && hidden % 8 == 0 &&
                   (((uintptr_t)d_w1 | (uintptr_t)d_w2 | (uintptr_t)d_embed_row | (uintptr_t)d_feature) & 15) == 0;
  const cudaError_t err = vec ? launch<true>(w1, b1, w2, b2, e, d_feature, d_model, hidden, n_max, d_n, d_z, scratch, st)
                              : launch<false>(w1, b1, w2, b2, e, d_feature, d_model, hidden, n_max, d_n, d_z, scratch, st);
  if (err != cudaSuccess) { cudaGetLastError(); return ADA_ERR_CUDA; }
  return cudaGetLastError() == cudaSuccess ? ADA_OK : ADA_ERR_CUDA;
}
