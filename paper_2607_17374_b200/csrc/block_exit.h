// How a block that meets at barriers which count a fixed number of threads leaves early: all of them or none.  Plain C++, so that it can be run by
// host threads.
#pragma once

#include "stage_waits.h"

// Whether the block goes on, the same answer in every thread: an error flag that other blocks and kernels may raise meanwhile is read by one of
// them.  (Read by each for itself, some threads may see it and leave, and those that do not would wait for them for good.)  go: memory of
// the block, written here alone.  sync(): the block's barrier.
template <class Sync>
TAURUS_HD bool block_goes_on(int thread, const volatile int* error, volatile int* go, Sync sync) {
  if (thread == 0) *go = *error == 0;
  sync();
  return *go != 0;
}
