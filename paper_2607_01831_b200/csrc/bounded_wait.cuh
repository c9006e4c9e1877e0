// The loop of every bounded wait on the chip, over whatever is waited for: probe() looks once (and may park its thread for
// some 20 us), now_ns() is a clock.  Plain C++, so that its behaviour can be checked on the host.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define LYNX_HD __host__ __device__ __forceinline__
#else
#define LYNX_HD inline
#endif

namespace lynx {

constexpr uint64_t kWaitLimitNs = 2000000000ull;

// Waits until probe() succeeds.  Gives up after about two seconds, or within 16 probes once another thread of the CTA has given
// up (the abort word is set): then it sets the abort word and returns false.
// (Inlined at some forty places of a kernel whose roles compete for the instruction caches: one test behind every 16th probe
// and nothing else.  32-column verification of 131072 tokens takes 97.2 us this way -- the same with a test per 256 probes --
// and 100.4 us with the abort word looked at in front of the probes and apart from the clock, 64 columns 217 and 228 us.)
template <class Probe, class Clock>
LYNX_HD bool bounded_wait(Probe probe, Clock now_ns, volatile int* abort_word) {
  uint64_t t0 = 0;
  for (uint32_t i = 1; !probe(); ++i) {
    if ((i & 15u) != 0) continue;
    const uint64_t now = now_ns();
    if (t0 == 0) t0 = now;
    if (*abort_word || now - t0 > kWaitLimitNs) {
      *abort_word = 1;
      return false;
    }
  }
  return true;
}

// Whether `first` came before `second`, for a warp whose next steps depend on it.  wait(probe) is the bounded wait; every lane waits
// for itself, and lanes that look at a barrier while its phase ends may leave by different conditions, so that the answer is one
// vote: any(x) is true in every lane if x is in one.  (What one lane has seen complete stays so for the others' waits.)
template <class Wait, class First, class Second, class Any>
LYNX_HD bool first_of(Wait wait, First first, Second second, Any any) {
  bool seen = false;
  wait([&] { seen = first(); return seen || second(); });
  return any(seen);
}

// What follows a wait that gave up, behind the last copy and product of the CTA and before it gives back the memory that they
// write to: a millisecond, a thousand times what one of them takes.
constexpr uint64_t kLandNs = 1000000ull;
template <class Clock>
LYNX_HD void land_after_abort(Clock now_ns, volatile int* abort_word) {
  if (!*abort_word) return;
  for (const uint64_t t0 = now_ns(); now_ns() - t0 < kLandNs;) {}
}

}  // namespace lynx
