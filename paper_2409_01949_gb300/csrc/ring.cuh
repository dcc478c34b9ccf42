// The producer's side of a shared-memory ring of copies, separate from the
// instructions it drives so that its order can be checked on the host.
#pragma once

#if defined(__CUDACC__)
#define RING_FN __device__ __forceinline__
#else
#define RING_FN inline
#endif

// Issues copies 0 .. n - 1 into `stages` stages in turn: copy b goes to stage
// b mod stages once copy b - stages has been released.  io.wait_empty(stage,
// parity) and io.wait_full(stage, parity) are bounded and return whether the
// phase completed; io.issue(b, stage) starts a copy that completes the stage's
// full barrier.  After a wait that gave up no copy is issued; in either case the
// last copies have landed, or a bounded wait for each has given up, on return,
// so that none is in flight when the block's shared memory goes to another.
// Returns whether every wait completed.
template <class Io>
RING_FN bool ring_produce(int n, int stages, Io& io) {
  bool ok = true;
  int issued = 0;
  for (int st = 0, ph = 1; issued < n; ++issued) {
    ok = io.wait_empty(st, ph);   // the first round passes at once
    if (!ok) break;
    io.issue(issued, st);
    if (++st == stages) {
      st = 0;
      ph ^= 1;
    }
  }
  for (int b = issued > stages ? issued - stages : 0; b < issued; ++b)
    if (!io.wait_full(b % stages, (b / stages) & 1)) ok = false;
  return ok;
}
