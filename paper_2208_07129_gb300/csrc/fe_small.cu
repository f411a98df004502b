// Ownership of the small meshes' product scratch (fe_small.h).
#include "fe_small.h"

#include <mutex>
#include <new>

namespace fe {

struct SmallScratch::Captures {
  std::mutex lock;
  struct Slot {
    bool taken = false;
    unsigned long long capture = 0;
    cudaStream_t stream = nullptr;
  } slot[kCaptures];
};

SmallScratch::~SmallScratch() {
  cudaFree(mem_);
  for (char* m : captured_mem_) cudaFree(m);
  if (done_) cudaEventDestroy(done_);
}

cudaError_t SmallScratch::create(size_t block_bytes) {
  captures_ = std::make_shared<Captures>();
  cudaError_t e = cudaMalloc(&mem_, block_bytes);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&done_, cudaEventDisableTiming);
  if (e == cudaSuccess) bytes_ = block_bytes;
  return e;
}

namespace {
// The calls below (a query, an allocation, user objects) are allowed while a thread captures a stream (this one or
// another, in the global mode) only in the relaxed mode: otherwise they
// invalidate its capture.
struct RelaxedCapture {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
  ~RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};
}  // namespace

void* SmallScratch::block(cudaStream_t s) {
  if (bytes_ == 0) return nullptr;
  const RelaxedCapture relaxed;
  cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
  unsigned long long capture = 0, stream = 0;
  cudaGraph_t graph = nullptr;
  cudaError_t e = cudaStreamGetCaptureInfo(s, &status, &capture, &graph);
  if (e == cudaSuccess && status == cudaStreamCaptureStatusActive) return captured_block(capture, s, graph);
  // (asking a capturing stream for its id would end its capture)
  if (e == cudaSuccess && status == cudaStreamCaptureStatusNone) e = cudaStreamGetId(s, &stream);
  if (e != cudaSuccess || status != cudaStreamCaptureStatusNone) {
    cudaGetLastError();   // e.g. the legacy stream while another thread captures: the launches report it
    return nullptr;
  }
  if (used_ && stream != stream_) {
    if (cudaEventQuery(done_) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
  }
  used_ = true;
  captured_ = false;
  stream_ = stream;
  return mem_;
}

cudaError_t SmallScratch::enqueued(cudaStream_t s) { return captured_ ? cudaSuccess : cudaEventRecord(done_, s); }

void* SmallScratch::captured_block(unsigned long long capture, cudaStream_t stream, cudaGraph_t graph) {
  struct Hold {   // what the graph's user object gives back
    std::shared_ptr<Captures> of;
    int slot;
    static void release(void* p) {
      Hold* h = static_cast<Hold*>(p);
      {
        std::lock_guard<std::mutex> hold(h->of->lock);
        h->of->slot[h->slot].taken = false;
      }
      delete h;
    }
  };
  int k = 0;
  {
    std::lock_guard<std::mutex> hold(captures_->lock);
    int free_slot = kCaptures;
    for (k = 0; k < kCaptures; ++k) {
      const Captures::Slot& t = captures_->slot[k];
      if (t.taken && t.capture == capture && t.stream == stream) {
        captured_ = true;
        return captured_mem_[k];
      }
      if (!t.taken && free_slot == kCaptures) free_slot = k;
    }
    k = free_slot;
    if (k == kCaptures) return nullptr;
    if (!captured_mem_[k] && cudaMalloc(&captured_mem_[k], bytes_) != cudaSuccess) {
      cudaGetLastError();
      captured_mem_[k] = nullptr;
      return nullptr;
    }
    captures_->slot[k].taken = true;
    captures_->slot[k].capture = capture;
    captures_->slot[k].stream = stream;
  }
  Hold* h = new (std::nothrow) Hold{captures_, k};
  cudaUserObject_t object = nullptr;
  cudaError_t e = h ? cudaUserObjectCreate(&object, h, Hold::release, 1, cudaUserObjectNoDestructorSync)
                    : cudaErrorMemoryAllocation;
  if (e != cudaSuccess) {
    cudaGetLastError();
    std::lock_guard<std::mutex> hold(captures_->lock);
    captures_->slot[k].taken = false;
    delete h;
    return nullptr;
  }
  if (cudaGraphRetainUserObject(graph, object, 1, cudaGraphUserObjectMove) != cudaSuccess) {
    cudaGetLastError();
    cudaUserObjectRelease(object, 1);   // gives the slot back
    return nullptr;
  }
  captured_ = true;
  return captured_mem_[k];
}

}  // namespace fe
