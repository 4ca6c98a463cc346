"""Blocks of the accounting meet at barriers that count a fixed number of threads, so they go on or leave as one, whatever becomes of the error flag
meanwhile: the header that the kernels use, run by host threads against a flag that others raise; and no way out of such a block but that."""
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_17374_b200", "csrc")

PROGRAM = r"""
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
#include "block_exit.h"

int main() {
  const int threads = 8, rounds = 2000;
  int left = 0, stayed = 0;
  for (int r = 0; r < rounds; ++r) {
    volatile int error = 0, go = -1;
    std::atomic<int> arrived{0}, on{0}, start{0};
    std::vector<std::thread> block;
    for (int t = 0; t < threads; ++t)
      block.emplace_back([&, t] {
        while (!start) {}
        for (int k = 0; k < (t * 37 + r) % 200; ++k) if (error > 1) return;   // threads come late by different spans
        if (block_goes_on(t, &error, &go, [&] { ++arrived; while (arrived < threads) std::this_thread::yield(); })) ++on;
      });
    std::thread other([&] { while (!start) {} for (int k = 0; k < r % 400; ++k) if (error > 1) return; error = 1; });
    start = 1;
    for (auto& t : block) t.join();
    other.join();
    if (on != 0 && on != threads) { printf("%d of %d went on\n", (int)on, threads); return 1; }
    if (on) ++stayed; else ++left;
  }
  printf("%d %d\n", left, stayed);
  return left + stayed == rounds ? 0 : 1;
}
"""


def test_all_threads_or_none(tmp_path):
    src, exe = tmp_path / "exit.cc", tmp_path / "exit"
    src.write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, "-o", str(exe), str(src)])
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout


def test_no_thread_leaves_such_a_block_by_itself():
    text = open(os.path.join(CSRC, "account.cuh")).read()
    bodies = re.split(r"\n(?=template <|__device__ |static |struct )", text)
    counted = [b for b in bodies if "account_sync<THREADS>" in b]
    assert len(counted) == 2
    for body in counted:
        exits = re.findall(r"[^;{}]*\breturn\b[^;]*;", body)
        assert len(exits) == 1 and "block_goes_on" in exits[0], exits
        assert body.index("block_goes_on") < body.index("account_sync<THREADS>()")
    elsewhere = [f for f in os.listdir(CSRC) if "bar.sync" in open(os.path.join(CSRC, f)).read()]
    assert elsewhere == ["account.cuh"]
