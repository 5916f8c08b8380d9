// Host-only check of overlap.h with a fake of the runtime's calls: whichever
// creation fails, nothing of the stream and the events is left, the error is
// cleared and the plan is told to run in line; on success everything is
// dropped once by the close.  And the rule for the SMs left free.  Prints "OK" or the failing checks.
#include <cstdio>

#include "overlap.h"

static int failures = 0, live = 0, calls = 0, fail_at = 0, cleared = 0, next_handle = 0;
static void expect(bool c, const char* what, int at) {
  if (!c) {
    std::printf("FAIL (call %d fails) %s\n", at, what);
    ++failures;
  }
}

struct Fake {
  static cudaError_t result() { return ++calls == fail_at ? cudaErrorMemoryAllocation : cudaSuccess; }
  template <typename H>
  static cudaError_t make(H* h) {
    const cudaError_t e = result();
    if (e != cudaSuccess) return e;
    ++live;
    *h = reinterpret_cast<H>(static_cast<size_t>(++next_handle));
    return e;
  }
  static cudaError_t priorities(int* least, int* greatest) {
    *least = 0;
    *greatest = -5;
    return result();
  }
  static cudaError_t stream(cudaStream_t* s, int priority) {
    expect(priority == 0, "lowest priority", fail_at);
    return make(s);
  }
  static cudaError_t event(cudaEvent_t* e) { return make(e); }
  static void drop(cudaStream_t) { --live; }
  static void drop(cudaEvent_t) { --live; }
  static void clear_error() { ++cleared; }
};

int main() {
  for (fail_at = 0; fail_at <= 4; ++fail_at) {
    calls = cleared = 0;
    dsnu::Overlap ov{};
    ov.reserve = 16;
    ov.col_side = 1;
    dsnu::overlap_open<Fake>(ov);
    const bool want = fail_at == 0;
    expect(ov.on == want, "on", fail_at);
    expect(live == (want ? 3 : 0), "objects left after opening", fail_at);
    expect(cleared == (want ? 0 : 1), "error cleared", fail_at);
    expect(ov.reserve == 16 && ov.col_side == 1, "settings kept", fail_at);
    dsnu::overlap_close<Fake>(ov);
    expect(live == 0 && !ov.on, "objects left after closing", fail_at);
    dsnu::overlap_close<Fake>(ov);
    expect(live == 0, "closed twice", fail_at);
  }
  // the reserve: the measured shares of 152 SMs, scaled to other devices; a wish
  // that leaves the column pass no SM, or none, runs in line
  struct { int nx, ny, mixed, sms; const char* env; int want; } rule[] = {
      {4096, 4096, 1, 152, nullptr, 16}, {2048, 2048, 1, 152, nullptr, 32}, {4096, 2048, 1, 152, nullptr, 23},
      {1024, 1024, 1, 152, nullptr, 48}, {128, 16, 1, 152, nullptr, 48},    {2048, 512, 1, 152, nullptr, 48},
      {4096, 4096, 0, 152, nullptr, 16}, {64, 64, 0, 152, nullptr, 16},     {64, 64, 0, 4, nullptr, 1},
      {64, 64, 0, 1, nullptr, 0},        {512, 512, 1, 152, "24", 24},      {512, 512, 1, 152, "151", 151},
      {512, 512, 1, 152, "152", 0},      {512, 512, 0, 152, "1000", 0},     {4096, 4096, 1, 152, "0", 0},
      {4096, 4096, 0, 152, "-3", 0},     {4096, 4096, 0, 152, "", 0}};
  for (auto& r : rule)
    expect(dsnu::overlap_reserve(r.nx, r.ny, r.mixed != 0, r.sms, r.env) == r.want, "reserve", r.nx * 10000 + r.ny);
  if (failures == 0) std::printf("OK\n");
  return failures == 0 ? 0 : 1;
}
