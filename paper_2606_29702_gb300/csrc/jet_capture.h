// Descriptors of batched calls under stream capture.
//
// An eager call uploads its descriptors through the batch's staging buffers, on
// the stream.  A captured call runs later and repeatedly, with other calls in
// between: an upload captured from the staging would replay with the arguments of
// whichever call wrote it last, on a work list of another length.  So a captured
// call's descriptors go to device memory of their own, filled at once (nothing of
// the upload is in the graph).  The graph holds a reference: when the last graph
// of a block is gone, a later captured call takes it over.
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <memory>
#include <vector>

namespace jet {

class CaptureStore {
  struct Block {
    char* dev = nullptr;
    size_t bytes = 0;
    std::atomic<bool> in_graph{false};
  };
  std::vector<std::shared_ptr<Block>> blocks;

  // destructor of the graph's reference (may run on a thread of the driver)
  static void CUDART_CB release(void* p) {
    auto* ref = static_cast<std::shared_ptr<Block>*>(p);
    (*ref)->in_graph = false;
    delete ref;
  }

  cudaError_t take(size_t bytes, std::shared_ptr<Block>* out) {
    for (const auto& b : blocks)
      if (!b->in_graph && b->bytes >= bytes) {
        *out = b;
        return cudaSuccess;
      }
    auto b = std::make_shared<Block>();
    const cudaError_t e = cudaMalloc((void**)&b->dev, bytes);
    if (e != cudaSuccess) return e;
    b->bytes = bytes;
    blocks.push_back(b);
    *out = b;
    return cudaSuccess;
  }

  // copies the parts on a stream of its own and waits for them
  static cudaError_t fill(char* dev, const void* const* src, const size_t* bytes, const size_t* off, int n) {
    cudaStream_t up;
    cudaError_t e = cudaStreamCreateWithFlags(&up, cudaStreamNonBlocking);
    if (e != cudaSuccess) return e;
    for (int i = 0; i < n && e == cudaSuccess; ++i)
      if (bytes[i] > 0) e = cudaMemcpyAsync(dev + off[i], src[i], bytes[i], cudaMemcpyHostToDevice, up);
    if (e == cudaSuccess) e = cudaStreamSynchronize(up);
    cudaStreamDestroy(up);
    return e;
  }

 public:
  static constexpr int kMaxParts = 4;

  // Device copies dst[i] of the n parts for the call being captured on s
  // (256-byte aligned).
  cudaError_t put(cudaStream_t s, int n, const void* const* src, const size_t* bytes, char** dst) {
    size_t off[kMaxParts], total = 0;
    for (int i = 0; i < n; ++i) {
      off[i] = total;
      total += (bytes[i] + 255) / 256 * 256;
    }
    // an allocation and a copy on another stream are no part of the capture
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaError_t e = cudaThreadExchangeStreamCaptureMode(&mode);
    if (e != cudaSuccess) return e;
    std::shared_ptr<Block> b;
    e = take(total > 0 ? total : 256, &b);
    if (e == cudaSuccess) e = fill(b->dev, src, bytes, off, n);
    cudaThreadExchangeStreamCaptureMode(&mode);
    if (e != cudaSuccess) return e;
    cudaStreamCaptureStatus st;
    cudaGraph_t graph = nullptr;
    e = cudaStreamGetCaptureInfo(s, &st, nullptr, &graph);
    if (e != cudaSuccess) return e;
    if (st != cudaStreamCaptureStatusActive) return cudaErrorStreamCaptureInvalidated;
    cudaUserObject_t ref;
    auto* own = new std::shared_ptr<Block>(b);
    e = cudaUserObjectCreate(&ref, own, release, 1, cudaUserObjectNoDestructorSync);
    if (e != cudaSuccess) {
      delete own;
      return e;
    }
    b->in_graph = true;
    e = cudaGraphRetainUserObject(graph, ref, 1, cudaGraphUserObjectMove);
    if (e != cudaSuccess) {
      cudaUserObjectRelease(ref, 1);
      return e;
    }
    for (int i = 0; i < n; ++i) dst[i] = b->dev + off[i];
    return cudaSuccess;
  }

  ~CaptureStore() {
    for (const auto& b : blocks) cudaFree(b->dev);
  }
};

inline bool stream_is_capturing(cudaStream_t s) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  return cudaStreamIsCapturing(s, &cs) == cudaSuccess && cs != cudaStreamCaptureStatusNone;
}

}  // namespace jet
