"""The context's host threads (csrc/hostpool.h), compiled here on their own:
every task runs exactly once, from one caller and from several at the same
time, for any number of tasks and wanted threads, and the threads are joined."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1010_1386_gb300", "csrc")

PROGRAM = r"""
#include <stdio.h>
#include "hostpool.h"
static int check(RsHostPool &pool, int n, int want) {
  std::vector<std::atomic<int>> hits(n + 1);
  for (auto &h : hits) h = 0;
  std::vector<long> out(n + 1, 0);
  pool.run(n, want, [&](int i) { hits[i]++; out[i] = 3L * i + 1; });
  for (int i = 0; i < n; ++i)
    if (hits[i] != 1 || out[i] != 3L * i + 1) return 1;
  return hits[n] != 0;
}
int main() {
  int bad = 0;
  { RsHostPool idle; }
  for (int r = 0; r < 50; ++r) {
    RsHostPool pool;
    for (int n : {0, 1, 2, 3, 15, 16, 17, 1000})
      for (int want : {-1, 0, 1, 2, 5, 16, 100}) bad += check(pool, n, want);
    std::atomic<int> fails{0};
    std::vector<std::thread> callers;
    for (int t = 0; t < 4; ++t)
      callers.emplace_back([&] { for (int k = 0; k < 40; ++k) fails += check(pool, 20 + k, 16); });
    for (auto &t : callers) t.join();
    bad += fails;
  }
  printf("bad %d\n", bad);
  return bad != 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
@pytest.mark.parametrize("flags", [["-O2"], ["-O1", "-g", "-fsanitize=thread"]])
def test_every_task_once(tmp_path, flags):
    src, exe = tmp_path / "pool.cpp", tmp_path / "pool"
    src.write_text(PROGRAM)
    build = subprocess.run(["g++", "-std=c++17", "-pthread", *flags, "-I", CSRC, str(src), "-o", str(exe)],
                           capture_output=True, text=True)
    if build.returncode != 0 and "-fsanitize=thread" in flags:
        pytest.skip("no thread sanitizer here")
    assert build.returncode == 0, build.stderr
    run = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    if "FATAL: ThreadSanitizer" in run.stderr:
        pytest.skip("the thread sanitizer cannot run here")
    assert run.returncode == 0, run.stdout + run.stderr[-2000:]
