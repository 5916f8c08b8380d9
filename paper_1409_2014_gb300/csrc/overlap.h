// overlap.h -- what a plan owns to run its band chain next to its column pass.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>

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

// SMs that the column pass leaves free on a device of `sms`; 0: in line.
//
// On large grids the column pass is the longer of the two: the band chain runs
// on the side stream, the column pass leaving it 16 of every 152 SMs, in mixed
// plans a share growing as 1/sqrt(nx ny) below 4096^2, since the band chain's
// node work does not shrink with the grid (mixed 4096^2 507 us with 16 SMs, 525
// with 32, 521 in line; 2048^2 131 with 32, 139 with 16, 150 in line; FP64, whose
// column pass is heavier, 4096^2 2041 us, with 24 SMs 2093, in line 2057; 2048^2
// 499, with 32 SMs 516, in line 541).  Below 2048^2 the band chain is the longer
// one: it stays on the caller's stream, where its launches overlap, and the
// column pass fills the rest of the GPU from the side stream (FP64 512^2 74 us;
// 1024^2 156, in line 166; mixed 256^2 41 against 47).  There the mixed share is
// capped at 48 SMs (1024^2 55.6 us with 48, 63.3 with 16; 2048 x 512 53.6 and
// 59.7).  All measured with 16384 nodes of the default widths: node count and
// width do not enter.  With few nodes a smaller share would do (2048 x 1024 with
// 288 nodes: 76 us, with 16 SMs 70, in line 84; with 16384 nodes 82, 84 and 94).
//
// `env` (DSNU_BAND_SMS) sets the number.  One that leaves the column pass no SM
// runs both in line: its grid would be a single CTA.
inline bool overlap_col_side(int nx, int ny) { return nx < 2048 || ny < 2048; }
inline int overlap_reserve(int nx, int ny, bool mixed, int sms, const char* env) {
  double share = 16.0 / 152.0;
  if (mixed) share *= 4096.0 / std::sqrt(double(nx) * ny);
  if (overlap_col_side(nx, ny)) share = std::min(share, 48.0 / 152.0);
  const int n = env ? std::atoi(env) : std::max(1, int(std::lround(sms * share)));
  return (n > 0 && n < sms) ? n : 0;
}

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
