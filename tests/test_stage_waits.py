"""What a CTA of the projection waits for before it gives its shared memory back after a wait of its own has run out: the phases that
its copies and MMAs have begun.  The header that the kernel uses, against model barriers on the host."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_17374_b200", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "stage_waits.h"

struct Barrier { int phase = 0; };   // phases completed; a parity wait succeeds when the running phase has the other parity
static bool over(const Barrier& b, unsigned parity) { return ((unsigned)b.phase & 1u) != parity; }

int main() {
  long long states = 0;
  for (int stages = 1; stages <= 8; ++stages)
    for (int begun = 0; begun <= 4 * stages + 1; ++begun) {
      const int live = begun < stages ? begun : stages;   // a stage is begun anew only when its use before is over
      for (unsigned open = 0; open < (1u << live); ++open) {   // which of the last uses are still on their way
        std::vector<Barrier> bar(stages);
        for (int it = 0; it < begun; ++it) bar[it % stages].phase++;
        for (int k = 0; k < live; ++k)
          if (open >> k & 1u) bar[(begun - 1 - k) % stages].phase--;
        const bool got = wait_last_phases(begun, stages, 4u, [&](int s, unsigned p) { return over(bar[s], p); });
        if (got != (open == 0)) { printf("stages %d begun %d open %x: %d\n", stages, begun, open, (int)got); return 1; }
        int polls = 0;   // one lands with every poll: the wait sees all of them through
        const bool all = wait_last_phases(begun, stages, 64u, [&](int s, unsigned p) {
          ++polls;
          if (over(bar[s], p)) return true;
          bar[s].phase++;
          return false;
        });
        int left = 0;
        for (int it = 0; it < begun; ++it) left++;
        for (auto& b : bar) left -= b.phase;
        if (!all || left != 0) { printf("stages %d begun %d open %x: %d left after %d polls\n", stages, begun, open, left, polls); return 1; }
        ++states;
      }
    }
  printf("%lld states\n", states);
  return 0;
}
"""


def test_every_state_of_rings_of_one_to_eight_stages(tmp_path):
    src, exe = tmp_path / "waits.cc", tmp_path / "waits"
    src.write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", CSRC, "-o", str(exe), str(src)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert int(r.stdout.split()[0]) > 3_000
