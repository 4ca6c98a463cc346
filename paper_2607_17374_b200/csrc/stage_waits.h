// A ring of operand stages guarded by mbarriers: use number `it` falls on stage it % stages and is phase it / stages of that
// stage's barrier.  Plain C++, so that the rules below can be run against model barriers on the host.
#pragma once

#ifdef __CUDACC__
#define TAURUS_HD __host__ __device__ __forceinline__
#else
#define TAURUS_HD inline
#endif

// Parity of the last phase begun on stage s after `begun` uses of the ring, -1: the stage has not been used.
TAURUS_HD int last_phase_parity(int begun, int stages, int s) { return begun <= s ? -1 : ((begun - 1 - s) / stages) & 1; }

// Waits until the last phase begun on every stage is complete, at most `limit` polls per stage; false: one was not.
// try_wait(s, parity) is mbarrier.try_wait.parity on the barrier of stage s: true when the phase of that parity is over, that is,
// when the phase now running has the other one.  (Asking for either parity says nothing: one of the two is always over.)
template <class TryWait>
TAURUS_HD bool wait_last_phases(int begun, int stages, unsigned limit, TryWait try_wait) {
  bool all = true;
  for (int s = 0; s < stages; ++s) {
    const int parity = last_phase_parity(begun, stages, s);
    if (parity < 0) continue;
    unsigned i = 0;
    while (i < limit && !try_wait(s, (unsigned)parity)) ++i;
    all = all && i < limit;
  }
  return all;
}
