// Scratch of small meshes' products (see launch_box), and who may use it when.
//
// Such a product is two launches: the cells write their results to a block of
// scratch, a gather adds them up into Y.  Between the two the block belongs to
// that product.  Products of one context may come from several host threads,
// on several streams and inside stream captures, and none of them has to know
// of the others:
//  * one stream: fe_apply holds the context's lock while it enqueues a
//    product, so the two launches of two threads' products do not interleave;
//  * several streams: one block, which a product takes when it comes on the
//    same stream as the last one (streams are compared by their id, which is
//    never used again, not by their handle) or when the last one has
//    completed; otherwise it takes the colour-ordered launches, whose result
//    is the same bit for bit.  Nothing ever waits for another stream;
//  * captures: a captured product may run again at any time, so every pair of
//    (capture, stream) has a block of its own, held until the graph and all
//    that was instantiated from it are destroyed (a user object of the graph
//    gives it back).  The blocks are allocated when captures first ask for
//    them, kCaptures at most, and kept for later captures; past these, or
//    without memory, captured products take the colour-ordered launches.
#pragma once

#include <cuda_runtime.h>
#include <cstddef>
#include <memory>

namespace fe {

class SmallScratch {
 public:
  SmallScratch() = default;
  SmallScratch(const SmallScratch&) = delete;
  SmallScratch& operator=(const SmallScratch&) = delete;
  ~SmallScratch();
  cudaError_t create(size_t block_bytes);
  size_t bytes() const { return bytes_; }   // of one block, 0 without scratch
  // The block for a product on s, or null: colour-ordered launches.  The
  // caller holds the context's lock until it has called enqueued().
  void* block(cudaStream_t s);
  cudaError_t enqueued(cudaStream_t s);

 private:
  static constexpr int kCaptures = 16;
  struct Captures;
  void* captured_block(unsigned long long capture, cudaStream_t stream, cudaGraph_t graph);
  char* mem_ = nullptr;                 // outside captures
  char* captured_mem_[kCaptures] = {};
  size_t bytes_ = 0;
  cudaEvent_t done_ = nullptr;          // after the last product outside captures
  bool used_ = false, captured_ = false;
  unsigned long long stream_ = 0;       // its stream
  std::shared_ptr<Captures> captures_;  // also held by the graphs' user objects
};

}  // namespace fe
