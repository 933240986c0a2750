// Device memory that captured calls use.
//
// A captured call runs later and repeatedly, with other calls in between, on the
// memory that its graph's nodes name.  GraphUse tells whether a graph that uses a
// piece of memory is still there: the graph, its clones and its executables hold a
// reference each, which goes with them.
//
// CaptureStore keeps the descriptors of captured batch calls.  An eager call
// uploads its descriptors through the batch's staging buffers, on the stream; an
// upload captured from the staging would replay with the arguments of whichever
// call wrote it last, on a work list of another length.  So a captured call's
// descriptors go to device memory of their own, filled at once (nothing of the
// upload is in the graph); when no graph uses a block, a later captured call takes
// it over.
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <memory>
#include <vector>

namespace jet {

inline bool stream_is_capturing(cudaStream_t s) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  return cudaStreamIsCapturing(s, &cs) == cudaSuccess && cs != cudaStreamCaptureStatusNone;
}

// the capture that s is part of (never 0), 0: none
inline unsigned long long stream_capture_id(cudaStream_t s) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  unsigned long long id = 0;
  if (cudaStreamGetCaptureInfo(s, &cs, &id) != cudaSuccess || cs == cudaStreamCaptureStatusNone) return 0;
  return id;
}

class GraphUse {
  using Count = std::shared_ptr<std::atomic<int>>;
  Count n = std::make_shared<std::atomic<int>>(0);

  // a graph's reference goes (may run on a thread of the driver, after the plan or batch)
  static void CUDART_CB release(void* p) {
    auto* ref = static_cast<Count*>(p);
    --**ref;
    delete ref;
  }

 public:
  bool live() const { return *n > 0; }

  // the graph that is being captured on s uses the memory
  cudaError_t add(cudaStream_t s) {
    cudaStreamCaptureStatus st;
    cudaGraph_t graph = nullptr;
    cudaError_t e = cudaStreamGetCaptureInfo(s, &st, nullptr, &graph);
    if (e != cudaSuccess) return e;
    if (st != cudaStreamCaptureStatusActive) return cudaErrorStreamCaptureInvalidated;
    auto* own = new Count(n);
    ++*n;
    cudaUserObject_t ref;
    e = cudaUserObjectCreate(&ref, own, release, 1, cudaUserObjectNoDestructorSync);
    if (e != cudaSuccess) {
      release(own);
      return e;
    }
    e = cudaGraphRetainUserObject(graph, ref, 1, cudaGraphUserObjectMove);
    if (e != cudaSuccess) cudaUserObjectRelease(ref, 1);
    return e;
  }
};

class CaptureStore {
  struct Block {
    char* dev = nullptr;
    size_t bytes = 0;
    GraphUse use;
  };
  std::vector<Block> blocks;

  cudaError_t take(size_t bytes, Block** out) {
    for (Block& b : blocks)
      if (!b.use.live() && b.bytes >= bytes) {
        *out = &b;
        return cudaSuccess;
      }
    Block b;
    const cudaError_t e = cudaMalloc((void**)&b.dev, bytes);
    if (e != cudaSuccess) return e;
    b.bytes = bytes;
    blocks.push_back(b);
    *out = &blocks.back();
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
    Block* b = nullptr;
    e = take(total > 0 ? total : 256, &b);
    if (e == cudaSuccess) e = fill(b->dev, src, bytes, off, n);
    cudaThreadExchangeStreamCaptureMode(&mode);
    if (e == cudaSuccess) e = b->use.add(s);
    if (e != cudaSuccess) return e;
    for (int i = 0; i < n; ++i) dst[i] = b->dev + off[i];
    return cudaSuccess;
  }

  ~CaptureStore() {
    for (const Block& b : blocks) cudaFree(b.dev);
  }
};

}  // namespace jet
