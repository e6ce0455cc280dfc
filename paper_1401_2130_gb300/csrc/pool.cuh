// pool.cuh -- scratch of the calls that is kept between them (pool.cu).
#pragma once

#include "common.cuh"

namespace pc {

// Stream-ordered device scratch from the library's own memory pool of the
// current device.  Freed with cudaFreeAsync.
cudaError_t scratch_alloc(void** p, size_t bytes, cudaStream_t st);

// A pinned host buffer for one copy back, borrowed for the length of a call.
// data() is null when the copy is too large for it (the caller then copies to
// its own buffers).
class HostStage {
 public:
  explicit HostStage(size_t bytes);
  ~HostStage();
  HostStage(const HostStage&) = delete;
  HostStage& operator=(const HostStage&) = delete;
  char* data() const { return p_; }

 private:
  char* p_ = nullptr;
};

// Takes an executable graph launched on st, to be destroyed later (pool.cu).
void retire_graph(cudaGraphExec_t ex, cudaStream_t st);

// A word of pinned memory that a kernel answers a call in: it writes tag << 32 |
// answer.  Nobody waits for it, and the word is another call's kMails calls
// later: an answer with another tag is no answer.
struct Mail {
  unsigned long long* at = nullptr;  // null: no pinned memory
  unsigned tag = 0;
  bool answer(unsigned* v) const;    // (host) true if it has come
};
Mail take_mail();

void release_pools();  // pc_shutdown

}  // namespace pc
