// Library-wide pieces of the C ABI: status strings, launch accounting, device queries and the
// whole-step entry point that moves a step's inputs and results across PCIe around the two
// kernels (Alg. 1, blocks "Sparse Attention Mask Creation" and "Verification with Sparse
// Attention").
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <mutex>
#include <new>

#include "specattn.h"
#include "nvtx_range.h"

namespace specattn {

std::atomic<long long> g_launch_count{0};

// Number of SMs of the current device (cached per device ordinal); <= 0 on failure.
int device_sm_count() {
  static std::mutex mu;
  static int cache[64] = {0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return -1;
  }
  if (dev < 0 || dev >= 64) return -1;
  std::lock_guard<std::mutex> lock(mu);
  if (cache[dev] == 0) {
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
      cudaGetLastError();
      return -1;
    }
    cache[dev] = n;
  }
  return cache[dev];
}

}  // namespace specattn

extern "C" const char* specattn_status_string(int code) {
  switch (code) {
    case SPECATTN_OK: return "ok";
    case SPECATTN_ERR_NULL: return "a required pointer is NULL";
    case SPECATTN_ERR_STRUCT_SIZE: return "struct_size does not match this library";
    case SPECATTN_ERR_RANGE: return "a scalar argument is out of range";
    case SPECATTN_ERR_ALIGN: return "a pointer or stride breaks the 16-byte alignment rules";
    case SPECATTN_ERR_WORKSPACE: return "workspace missing or too small";
    case SPECATTN_ERR_UNSUPPORTED: return "shape outside what the kernels support";
    case SPECATTN_ERR_CUDA: return "the CUDA runtime reported an error";
    case SPECATTN_ERR_STATIC_SCRATCH:
      return "the shape needs more scratch than the library's built-in static buffer holds";
    default: return "unknown status code";
  }
}

extern "C" int64_t specattn_kernel_launch_count(void) {
  return static_cast<int64_t>(specattn::g_launch_count.load(std::memory_order_relaxed));
}

namespace specattn {
namespace {

// Copy streams and events of the whole-step call, created on first use per device and kept
// until the process exits.  One call at a time per device enqueues through them (the mutex is
// held while enqueueing, which never blocks on the GPU).
struct HostPipe {
  cudaStream_t h2d = nullptr, d2h = nullptr;
  cudaEvent_t start = nullptr, q_in = nullptr, done = nullptr;
  cudaEvent_t layer_in[SPECATTN_MAX_DRAFT_LAYERS] = {nullptr};
  cudaEvent_t* layer_out = nullptr;  // one per target layer
  int n_layer_out = 0;
  std::mutex mu;
};
HostPipe g_pipe[64];

// Copies small blocks from or to host memory that the GPU can address (pinned or registered) in one launch: grid
// row y copies block y with 16-byte accesses over the bus.  A copy-engine transfer of ~100 KB takes 7 us of which
// 2 are transfer, and an engine serves one at a time: eight layers' queries delayed the draft rows by 57 us, their
// outputs (two transfers a layer) came in 16 us apart.
constexpr int kGatherBlocks = 64;
constexpr size_t kGatherMost = 4u << 20;  // larger blocks are left to the copy engine
struct HostBlocks {
  const uint4* src[kGatherBlocks];
  uint4* dst[kGatherBlocks];
  unsigned int n16[kGatherBlocks];
};
__global__ void __launch_bounds__(256) copy_host_blocks(const __grid_constant__ HostBlocks B) {
  const uint4* const src = B.src[blockIdx.y];
  uint4* const dst = B.dst[blockIdx.y];
  const unsigned int n = B.n16[blockIdx.y], step = gridDim.x * 256;
  for (unsigned int i = blockIdx.x * 256 + threadIdx.x; i < n; i += 4 * step) {
    uint4 v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (i + k * step < n) v[k] = src[i + k * step];
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (i + k * step < n) dst[i + k * step] = v[k];
  }
}

// The address at which the current device sees host memory `p`, or nullptr if it does not see the whole block
// (pageable memory, a block that reaches beyond its pinned allocation or registered range) or if 16-byte accesses to
// the block, or its size, do not suit the kernel above.  The driver's query is looked up through the runtime (no
// link-time dependency on the driver library).
uint4* device_view(const void* p, const void* device_side, size_t bytes) {
  if (bytes % 16 != 0 || bytes > kGatherMost || reinterpret_cast<uintptr_t>(device_side) % 16 != 0) return nullptr;
  typedef CUresult (*query_fn)(unsigned int, CUpointer_attribute*, void**, CUdeviceptr);
  static std::atomic<query_fn> cached{nullptr};
  query_fn fn = cached.load(std::memory_order_acquire);
  if (fn == nullptr) {
    void* sym = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuPointerGetAttributes", &sym, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || sym == nullptr) {
      cudaGetLastError();
      return nullptr;
    }
    fn = reinterpret_cast<query_fn>(sym);
    cached.store(fn, std::memory_order_release);
  }
  unsigned int type = 0, managed = 0;
  CUdeviceptr seen = 0, start = 0;
  size_t size = 0;
  CUpointer_attribute what[5] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_IS_MANAGED, CU_POINTER_ATTRIBUTE_DEVICE_POINTER,
                                 CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, CU_POINTER_ATTRIBUTE_RANGE_SIZE};
  void* into[5] = {&type, &managed, &seen, &start, &size};
  if (fn(5, what, into, static_cast<CUdeviceptr>(reinterpret_cast<uintptr_t>(p))) != CUDA_SUCCESS) return nullptr;
  if (type != CU_MEMORYTYPE_HOST || managed != 0 || seen == 0 || seen % 16 != 0) return nullptr;
  if (seen < start || seen - start > size || size - (seen - start) < bytes) return nullptr;
  return reinterpret_cast<uint4*>(static_cast<uintptr_t>(seen));
}

bool make_event(cudaEvent_t* e) {
  if (*e != nullptr) return true;
  if (cudaEventCreateWithFlags(e, cudaEventDisableTiming) != cudaSuccess) {
    cudaGetLastError();
    *e = nullptr;
    return false;
  }
  return true;
}

// Called with pipe.mu held.
bool prepare_pipe(HostPipe& pipe, int n_target_layers) {
  if (pipe.h2d == nullptr && cudaStreamCreateWithFlags(&pipe.h2d, cudaStreamNonBlocking) != cudaSuccess) {
    cudaGetLastError();
    pipe.h2d = nullptr;
    return false;
  }
  if (pipe.d2h == nullptr && cudaStreamCreateWithFlags(&pipe.d2h, cudaStreamNonBlocking) != cudaSuccess) {
    cudaGetLastError();
    pipe.d2h = nullptr;
    return false;
  }
  if (!make_event(&pipe.start) || !make_event(&pipe.q_in) || !make_event(&pipe.done)) return false;
  for (int u = 0; u < SPECATTN_MAX_DRAFT_LAYERS; ++u)
    if (!make_event(&pipe.layer_in[u])) return false;
  if (pipe.n_layer_out < n_target_layers) {
    cudaEvent_t* grown = new (std::nothrow) cudaEvent_t[n_target_layers];
    if (grown == nullptr) return false;
    for (int j = 0; j < n_target_layers; ++j) grown[j] = (j < pipe.n_layer_out) ? pipe.layer_out[j] : nullptr;
    delete[] pipe.layer_out;
    pipe.layer_out = grown;
    const int old = pipe.n_layer_out;
    pipe.n_layer_out = n_target_layers;
    for (int j = old; j < n_target_layers; ++j)
      if (!make_event(&pipe.layer_out[j])) return false;
  }
  return true;
}

}  // namespace
}  // namespace specattn

// The step as a three-lane pipeline.  Lane "in" (a copy stream) uploads the draft rows one mapped draft layer
// at a time while a kernel fetches the query blocks; the caller's stream runs the selection of a
// draft layer as soon as its rows have landed and then the verify launches of the target layers
// mapped to it, while the next draft layer is still crossing PCIe; lane "out" (a second copy
// stream) downloads a layer's results while later layers compute and later inputs upload.  The
// call returns with everything enqueued; the caller's stream has been made to wait for the last
// download, so stream order is what it would be had everything run on that stream.
extern "C" int specattn_verify_step_host(const specattn_step_host_args* args, void* cuda_stream) {
  specattn::NvtxRange nvtx_range("specattn_verify_step_host");
  if (args == nullptr) return SPECATTN_ERR_NULL;
  if (args->struct_size != sizeof(specattn_step_host_args)) return SPECATTN_ERR_STRUCT_SIZE;
  const specattn_step_host_args& S = *args;
  if (!S.select || !S.draft_probs_host || S.n_target_layers < 0) return SPECATTN_ERR_NULL;
  if (S.n_target_layers > 0 && (!S.verify || !S.q_host || !S.out_host || !S.lse_host)) return SPECATTN_ERR_NULL;
  const specattn_select_args& sel = *S.select;
  if (sel.struct_size != sizeof(specattn_select_args)) return SPECATTN_ERR_STRUCT_SIZE;
  if (!sel.draft_probs || !sel.layer_map) return SPECATTN_ERR_NULL;
  if (sel.n_draft_layers < 1 || sel.n_draft_layers > SPECATTN_MAX_DRAFT_LAYERS) return SPECATTN_ERR_RANGE;
  if (sel.n_target_layers != S.n_target_layers) return SPECATTN_ERR_RANGE;
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);

  bool used[SPECATTN_MAX_DRAFT_LAYERS] = {false};
  for (int j = 0; j < sel.n_target_layers; ++j) {
    const int u = sel.layer_map[j];
    if (u < -1 || u >= sel.n_draft_layers) return SPECATTN_ERR_RANGE;
    if (u >= 0) used[u] = true;
  }
  for (int u = 0; u < sel.n_draft_layers; ++u)
    if (used[u] && (!S.draft_probs_host[u] || !sel.draft_probs[u])) return SPECATTN_ERR_NULL;
  for (int j = 0; j < S.n_target_layers; ++j) {
    const specattn_verify_args& v = S.verify[j];
    if (v.struct_size != sizeof(specattn_verify_args)) return SPECATTN_ERR_STRUCT_SIZE;
    if (!S.q_host[j] || !S.out_host[j] || !S.lse_host[j] || !v.q || !v.out || !v.lse) return SPECATTN_ERR_NULL;
  }

  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    cudaGetLastError();
    return SPECATTN_ERR_CUDA;
  }
  specattn::HostPipe& pipe = specattn::g_pipe[dev];
  std::lock_guard<std::mutex> lock(pipe.mu);
  if (!specattn::prepare_pipe(pipe, S.n_target_layers)) return SPECATTN_ERR_CUDA;
  auto ok = [](cudaError_t e) {
    if (e == cudaSuccess) return true;
    cudaGetLastError();
    return false;
  };

  // the copy lanes start after whatever the caller's stream already holds
  if (!ok(cudaEventRecord(pipe.start, stream)) || !ok(cudaStreamWaitEvent(pipe.h2d, pipe.start, 0)) ||
      !ok(cudaStreamWaitEvent(pipe.d2h, pipe.start, 0)))
    return SPECATTN_ERR_CUDA;

  // The query blocks: one kernel on the caller's stream, which has nothing else to do until the first
  // draft layer is in, reads those that the GPU can read.  The others (pageable, unaligned, large) go by the copy
  // engine ahead of the draft rows: behind them they would hold up the first layer until the last one's rows are in.
  bool q_copied = false;  // by the copy engine: the first verify call waits for it
  specattn::HostBlocks blocks;
  int n_blocks = 0;
  auto fetch_blocks = [&]() {
    if (n_blocks == 0) return true;
    specattn::copy_host_blocks<<<dim3(8, static_cast<unsigned>(n_blocks)), 256, 0, stream>>>(blocks);
    n_blocks = 0;
    specattn::g_launch_count.fetch_add(1, std::memory_order_relaxed);
    return ok(cudaGetLastError());
  };
  for (int j = 0; j < S.n_target_layers; ++j) {
    const specattn_verify_args& v = S.verify[j];
    const size_t bytes = static_cast<size_t>(v.batch) * v.n_q * v.n_q_heads * v.head_dim * 2;
    if (bytes == 0) continue;
    const uint4* src = specattn::device_view(S.q_host[j], v.q, bytes);
    if (src != nullptr) {
      if (n_blocks == specattn::kGatherBlocks && !fetch_blocks()) return SPECATTN_ERR_CUDA;
      blocks.src[n_blocks] = src;
      blocks.dst[n_blocks] = static_cast<uint4*>(const_cast<void*>(v.q));
      blocks.n16[n_blocks] = static_cast<unsigned int>(bytes / 16);
      ++n_blocks;
    } else {
      q_copied = true;
      if (!ok(cudaMemcpyAsync(const_cast<void*>(v.q), S.q_host[j], bytes, cudaMemcpyHostToDevice, pipe.h2d)))
        return SPECATTN_ERR_CUDA;
    }
  }
  if (q_copied && !ok(cudaEventRecord(pipe.q_in, pipe.h2d))) return SPECATTN_ERR_CUDA;

  // lane "in": the draft rows in the order the layers need them.  They bound the step (a PCIe link's ~53 GB/s).
  const size_t layer_bytes = static_cast<size_t>(sel.batch) * sel.n_draft_heads * sel.gamma *
                             static_cast<size_t>(sel.L_stride) * sizeof(float);
  bool uploaded[SPECATTN_MAX_DRAFT_LAYERS] = {false};
  auto upload = [&](int u) {
    if (uploaded[u]) return true;
    uploaded[u] = true;
    return ok(cudaMemcpyAsync(const_cast<float*>(sel.draft_probs[u]), S.draft_probs_host[u], layer_bytes,
                              cudaMemcpyHostToDevice, pipe.h2d)) &&
           ok(cudaEventRecord(pipe.layer_in[u], pipe.h2d));
  };
  for (int j = 0; j < S.n_target_layers; ++j)
    if (sel.layer_map[j] >= 0 && !upload(sel.layer_map[j])) return SPECATTN_ERR_CUDA;
  if (!fetch_blocks()) return SPECATTN_ERR_CUDA;

  // the caller's stream: selection per draft layer when first needed, then the verify launches
  bool selected[SPECATTN_MAX_DRAFT_LAYERS] = {false};
  int to_select = 0;  // draft layers whose selection is still to be enqueued
  for (int u = 0; u < sel.n_draft_layers; ++u) to_select += used[u] ? 1 : 0;
  const void* planned[SPECATTN_MAX_DRAFT_LAYERS + 1];
  int n_planned = 0;
  // A verify launch may skip its wait for the preceding kernel (SPECATTN_VERIFY_LISTS_STABLE)
  // only when that kernel is another verify launch: the first one after a selection or a plan
  // launch enqueued here reads what those kernels wrote, so the flag is dropped for it.
  bool fresh = true;
  for (int j = 0; j < S.n_target_layers; ++j) {
    const int u = sel.layer_map[j];
    if (u >= 0 && !selected[u]) {
      selected[u] = true;
      --to_select;
      fresh = true;
      if (!ok(cudaStreamWaitEvent(stream, pipe.layer_in[u], 0))) return SPECATTN_ERR_CUDA;
      specattn_select_args one = sel;  // the lists of draft layer u only
      const int32_t only = u;
      one.n_target_layers = 1;
      one.layer_map = &only;
      const int rc = specattn_select_topp(&one, cuda_stream);
      if (rc != SPECATTN_OK) return rc;
    }
    const specattn_verify_args& v = S.verify[j];
    // a work partition that several layers share is computed before its first user
    if (v.plan != nullptr) {
      bool done = false;
      for (int k = 0; k < n_planned && !done; ++k) done = planned[k] == v.plan;
      if (!done) {
        const int prc = specattn_verify_plan(&v, const_cast<void*>(v.plan), specattn_verify_plan_bytes(&v), cuda_stream);
        if (prc != SPECATTN_OK) return prc;
        if (n_planned < SPECATTN_MAX_DRAFT_LAYERS + 1) planned[n_planned++] = v.plan;
        fresh = true;
      }
    }
    if (q_copied) {
      q_copied = false;
      if (!ok(cudaStreamWaitEvent(stream, pipe.q_in, 0))) return SPECATTN_ERR_CUDA;
    }
    specattn_verify_args call = v;
    if (fresh) call.flags &= ~SPECATTN_VERIFY_LISTS_STABLE;
    fresh = false;
    const int rc = specattn_sparse_verify(&call, cuda_stream);
    if (rc != SPECATTN_OK) return rc;
    // lane "out"
    const size_t rows = static_cast<size_t>(v.batch) * v.n_q * v.n_q_heads;
    if (!ok(cudaEventRecord(pipe.layer_out[j], stream)) || !ok(cudaStreamWaitEvent(pipe.d2h, pipe.layer_out[j], 0)))
      return SPECATTN_ERR_CUDA;
    if (rows == 0) continue;
    const size_t out_bytes = rows * v.head_dim * sizeof(float), lse_bytes = rows * sizeof(float);
    // The kernel, whose stores crawl while draft rows still come in (27 us instead of 7, and its CTAs hold up
    // the attention's), serves the layers after the last selection; the copy engine's way is hidden before it.
    uint4* const out_view = (to_select == 0) ? specattn::device_view(S.out_host[j], v.out, out_bytes) : nullptr;
    uint4* const lse_view = (to_select == 0) ? specattn::device_view(S.lse_host[j], v.lse, lse_bytes) : nullptr;
    if (out_view != nullptr && lse_view != nullptr) {
      blocks.src[0] = reinterpret_cast<const uint4*>(v.out);
      blocks.dst[0] = out_view;
      blocks.n16[0] = static_cast<unsigned int>(out_bytes / 16);
      blocks.src[1] = reinterpret_cast<const uint4*>(v.lse);
      blocks.dst[1] = lse_view;
      blocks.n16[1] = static_cast<unsigned int>(lse_bytes / 16);
      specattn::copy_host_blocks<<<dim3(8, 2), 256, 0, pipe.d2h>>>(blocks);
      specattn::g_launch_count.fetch_add(1, std::memory_order_relaxed);
      if (!ok(cudaGetLastError())) return SPECATTN_ERR_CUDA;
    } else if (!ok(cudaMemcpyAsync(S.out_host[j], v.out, out_bytes, cudaMemcpyDeviceToHost, pipe.d2h)) ||
               !ok(cudaMemcpyAsync(S.lse_host[j], v.lse, lse_bytes, cudaMemcpyDeviceToHost, pipe.d2h))) {
      return SPECATTN_ERR_CUDA;
    }
  }
  // join: later work on the caller's stream sees the inputs consumed and the results delivered
  if (!ok(cudaEventRecord(pipe.done, pipe.d2h)) || !ok(cudaStreamWaitEvent(stream, pipe.done, 0)))
    return SPECATTN_ERR_CUDA;
  if (!ok(cudaEventRecord(pipe.done, pipe.h2d)) || !ok(cudaStreamWaitEvent(stream, pipe.done, 0)))
    return SPECATTN_ERR_CUDA;
  return SPECATTN_OK;
}
