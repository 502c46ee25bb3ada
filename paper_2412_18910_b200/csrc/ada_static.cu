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
// to start at zero: a call overwrites every entry it later reads (the counts beside it do, see g_ldlp_done).  Two calls that overlap on the
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

// Blocks that have left their hidden activations, by the number of blocks of a call: a count wraps to zero with the call's last
// block, and it is whole again even after calls that overlapped, for those that share it add as much each.
static __device__ unsigned g_ldlp_done[(ADA_STATIC_MAX_HIDDEN + ada::kLdlpUnits - 1) / ada::kLdlpUnits];

// One launch: hidden = ReLU(W1 [e ; f] + b1), four units a block; the block that comes last takes z = W2 hidden + b2, a warp per
// output, and n = argmax + 1, lowest index among equals.  Bound by the latency of its chain (launch, W1 from HBM, count, hidden
// from level 2), not by its bytes.  7B widths, calls back to back: 30.7 us with one warp and element-wise loads per hidden unit,
// 9.1 us with a second launch for the outputs behind this one, 7.5 us so.  Launched with programmatic serialization: the blocks
// are in place, waiting, when the kernel before them ends (nothing is read or written before that).
template <bool VEC>
__global__ void __launch_bounds__(kLdlpThreads) k_static_predict(const __nv_bfloat16 *w1, const __nv_bfloat16 *b1,
                                                                 const __nv_bfloat16 *w2, const __nv_bfloat16 *b2,
                                                                 const __nv_bfloat16 *e, const float *f, int d, int hid, int nmax,
                                                                 float *hidden, int *n_out, float *z_out) {
  constexpr int kWarps = kLdlpThreads / 32;
  __shared__ float zs[ADA_MAX_NMAX];
  __shared__ int last_s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (blockIdx.x == 0)   // the last block finds W2 in level 2
    for (int i = threadIdx.x * 64; i < nmax * hid; i += kLdlpThreads * 64) asm volatile("prefetch.global.L2 [%0];" ::"l"(w2 + i));
  ada::ldlp_hidden_block<VEC>(w1, b1, e, f, d, hid, blockIdx.x * kLdlpUnits, hidden);   // (its first threads store)
  if (warp == 0) {
    __syncwarp();
    if (lane == 0) {
      unsigned old;
      asm volatile("atom.acq_rel.gpu.global.inc.u32 %0, [%1], %2;" : "=r"(old) : "l"(g_ldlp_done + (gridDim.x - 1)), "r"(gridDim.x - 1) : "memory");
      last_s = old == gridDim.x - 1;
    }
  }
  __syncthreads();
  if (!last_s) return;
  for (int c = warp; c < nmax; c += kWarps) {
    ada::LdlpRow row;
    const __nv_bfloat16 *w = w2 + (size_t)c * hid;
    ada::ldlp_out_ahead<VEC>(w, hid, row);
    const float z = ada::ldlp_out_dot<VEC>(w, hidden, hid, row) + __bfloat162float(b2[c]);
    if (lane == 0) {
      zs[c] = z;
      if (z_out) z_out[c] = z;
    }
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
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((hid + kLdlpUnits - 1) / kLdlpUnits); cfg.blockDim = dim3(kLdlpThreads); cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_static_predict<VEC>, w1, b1, w2, b2, e, f, d, hid, nmax, hidden, n, z);
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
