"""The planner's loop over host threads: every index runs once, for one caller, several at a
time, loops inside loops, a loop that throws, and in a forked child, which has none of its
parent's threads.  Compiled with g++ against the planner sources, plain and with the thread
sanitizer: no CUDA, no GPU."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2001_04890_gb300", "csrc")

PROG = r"""
#include "plan.hpp"
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <stdexcept>
#include <sys/wait.h>
#include <unistd.h>
using namespace dmrg;

static bool sums(size_t n) {  // plain writes, read here after the loop
  std::vector<int> hit(n, 0);
  parallel_for(n, [&](size_t i) { ++hit[i]; });
  for (int h : hit)
    if (h != 1) return false;
  return true;
}
static bool nested(size_t n) {
  std::vector<std::vector<int>> hit(n, std::vector<int>(n, 0));
  parallel_for(n, [&](size_t i) { parallel_for(n, [&](size_t j) { ++hit[i][j]; }); });
  for (auto &r : hit)
    for (int h : r)
      if (h != 1) return false;
  return true;
}
static bool throws(size_t n) {
  std::atomic<int> ran{0};
  try {
    parallel_for(n, [&](size_t i) {
      if (i == n / 2) throw std::runtime_error("x");
      ++ran;
    });
  } catch (const std::runtime_error &e) {
    return !std::strcmp(e.what(), "x") && ran < (int)n;
  }
  return false;
}
static bool all() {
  bool ok = true;
  for (int rep = 0; rep < 5; ++rep)
    for (size_t n : {0, 1, 2, 15, 16, 17, 1000}) ok = sums(n) && ok;
  for (size_t n : {1, 2, 17}) ok = nested(n) && ok;
  for (size_t n : {1, 2, 40}) ok = throws(n) && ok;
  return ok && sums(100);
}

int main(int argc, char **) {
  bool ok = all();
  std::vector<std::thread> t;
  std::atomic<int> bad{0};
  for (int k = 0; k < 4; ++k) t.emplace_back([&] { bad += !all(); });
  for (auto &x : t) x.join();
  ok = ok && bad == 0;
  if (argc > 1) {
    const pid_t pid = fork();
    if (pid == 0) _exit(all() ? 0 : 1);
    int st = 1;
    waitpid(pid, &st, 0);
    ok = ok && WIFEXITED(st) && WEXITSTATUS(st) == 0;
  }
  std::printf("%s\n", ok ? "ok" : "FAILED");
  return ok ? 0 : 1;
}
"""


@pytest.mark.parametrize("flags,args", [([], ["fork"]), (["-fsanitize=thread", "-g"], [])])
def test_loops_over_helper_threads(tmp_path, flags, args):
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROG)
    cmd = ["g++", "-O1", "-std=c++17", "-pthread", *flags, "-I", CSRC, str(src), os.path.join(CSRC, "plan.cpp"), "-o", str(exe)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode and flags:
        pytest.skip("no thread sanitizer")
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe), *args], capture_output=True, text=True, timeout=120)
    if "unexpected memory mapping" in r.stderr:
        pytest.skip("the thread sanitizer does not run on this machine")
    assert r.returncode == 0, r.stdout + r.stderr
