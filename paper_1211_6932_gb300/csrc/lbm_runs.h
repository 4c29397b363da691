// How the steps of one call are queued (host only): runs of kGraphSteps and of the lower powers
// of two are replayed from a graph once a run of that length comes back (36 launches of a
// 100-step call kept the host busy for 80 us, more than the steps of a small lattice take); a
// persistent run of any length is one launch.  The first run is launched: the GPU steps while
// the host queues the launches, but waits for a capture (the first 100 steps of 193 x 147
// with their transfers: 670 us with the capture, 381 without), and a batch that retires
// instances would wait at every retirement.  The second run captures; from the third on a run
// is a replay.  A caller's own capture of a short run gets its launches; of 64 steps and more it
// fails, as no graph can be launched into a capture.
#pragma once

namespace lbm {

constexpr int kGraphLog = 6;
constexpr int kGraphSteps = 1 << kGraphLog;  // even, so a replay returns to the same slab

// Ops (a run starts from the current slab): int& uses(k), how often 2^k steps were launched;
// bool captured(k); int capture(k), replay(k) and launch(steps), which return 0 or an error;
// long long& firsts(), counts the runs that were not queued as the next such run will be.
template <typename Ops>
int queue_runs(long long n, bool persist, bool capturing, Ops& ops) {
  const bool replay = !persist && !capturing;
  while (n > 0) {
    int k = kGraphLog;
    while (k > 0 && (1LL << k) > n) --k;
    int rc = 0, m = 1 << k;
    if (replay ? k > 0 && ops.uses(k) > 0 : k == kGraphLog) {
      if (!ops.captured(k)) {
        ++ops.firsts();
        rc = ops.capture(k);
      }
      if (rc == 0) rc = ops.replay(k);
    } else {
      if (persist) m = (int)n;
      if (replay && k > 0) ++ops.firsts();
      int& uses = ops.uses(k);
      rc = ops.launch(m);
      if (rc == 0) ++uses;
    }
    if (rc) return rc;
    n -= m;
  }
  return 0;
}

// Run n steps until a run of them is queued as the next one will be (before timing it).
template <typename Run, typename Ops>
int warm_up(const Run& run, Ops& ops) {
  for (;;) {
    const long long before = ops.firsts();
    if (int rc = run()) return rc;
    if (ops.firsts() == before) return 0;
  }
}

}  // namespace lbm
