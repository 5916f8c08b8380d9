// overlap.h -- what a plan owns to run its band chain next to its column pass.
#pragma once

#include <cuda_runtime.h>

namespace dsnu {

// One of the two runs on `side` (a low-priority stream): the band chain, or with
// col_side the column pass, whose persistent grid leaves `reserve` SMs free.
struct Overlap {
  cudaStream_t side;
  cudaEvent_t fork, join;
  int reserve;
  int col_side;
  bool on;  // false: both in line on the caller's stream
};

// The runtime's calls (a test puts failing ones in their place).
struct OverlapCuda {
  static cudaError_t priorities(int* least, int* greatest) { return cudaDeviceGetStreamPriorityRange(least, greatest); }
  static cudaError_t stream(cudaStream_t* s, int priority) {
    return cudaStreamCreateWithPriority(s, cudaStreamNonBlocking, priority);
  }
  static cudaError_t event(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, cudaEventDisableTiming); }
  static void drop(cudaStream_t s) {
    cudaStreamSynchronize(s);
    cudaStreamDestroy(s);
  }
  static void drop(cudaEvent_t e) { cudaEventDestroy(e); }
  static void clear_error() { cudaGetLastError(); }
};

template <typename Api = OverlapCuda>
void overlap_close(Overlap& ov) {
  if (ov.side) Api::drop(ov.side);
  if (ov.fork) Api::drop(ov.fork);
  if (ov.join) Api::drop(ov.join);
  ov.side = nullptr;
  ov.fork = ov.join = nullptr;
  ov.on = false;
}

// Creates the stream and the events of a zeroed `ov`.  Where one of them cannot
// be had, none is kept, and neither is the error (the next launch would report
// it): the plan runs both in line.
template <typename Api = OverlapCuda>
void overlap_open(Overlap& ov) {
  int least = 0, greatest = 0;
  cudaError_t e = Api::priorities(&least, &greatest);
  if (e == cudaSuccess) e = Api::stream(&ov.side, least);
  if (e == cudaSuccess) e = Api::event(&ov.fork);
  if (e == cudaSuccess) e = Api::event(&ov.join);
  ov.on = (e == cudaSuccess);
  if (ov.on) return;
  overlap_close<Api>(ov);
  Api::clear_error();
}

}  // namespace dsnu
