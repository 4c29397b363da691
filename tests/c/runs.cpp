// Prints how the steps of repeated calls are queued (csrc/lbm_runs.h), one line a call: L<steps>
// for a run queued launch by launch, C<k> for the capture of 2^k steps, R<k> for a replay.
// Arguments: persistent (0 or 1), capturing (0 or 1), steps, calls; a call count of 0 warms up
// as the autotuner does, then prints the two calls that it times.
#include <cstdio>
#include <cstdlib>

#include "lbm_runs.h"

struct Log {
  int cur = 0;
  int n[lbm::kGraphLog + 1][2] = {};
  bool graph[lbm::kGraphLog + 1][2] = {};
  long long first = 0;
  bool quiet = false;
  void say(char c, int v) {
    if (!quiet) std::printf("%c%d ", c, v);
  }
  int& uses(int k) { return n[k][cur]; }
  bool captured(int k) { return graph[k][cur]; }
  long long& firsts() { return first; }
  int capture(int k) {
    graph[k][cur] = true;
    say('C', k);
    return 0;
  }
  int replay(int k) {
    say('R', k);
    return 0;
  }
  int launch(int steps) {
    say('L', steps);
    cur ^= steps & 1;
    return 0;
  }
};

int main(int argc, char** argv) {
  if (argc != 5) return 2;
  const bool persist = std::atoi(argv[1]) != 0, capturing = std::atoi(argv[2]) != 0;
  const long long steps = std::atoll(argv[3]);
  int calls = std::atoi(argv[4]);
  Log log;
  auto run = [&] { return lbm::queue_runs(steps, persist, capturing, log); };
  if (calls == 0) {
    log.quiet = true;
    if (lbm::warm_up(run, log)) return 1;
    log.quiet = false;
    calls = 2;
  }
  for (int k = 0; k < calls; ++k) {
    if (run()) return 1;
    std::printf("\n");
  }
  return 0;
}
