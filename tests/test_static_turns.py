"""The order in which calls of the static entry point take the parts of its scratch (csrc/static_turns.h), compiled with the host compiler:
every call that is launched finds its part emptied by the one launched before it, with several threads and calls that fail."""
import ctypes as C
import shutil
import subprocess

import pytest

from paper_2511_22972_b200 import build

N = 4


@pytest.fixture(scope="module")
def turns(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("turns")
    (d / "turns.cpp").write_text("""
#include "static_turns.h"
#include <thread>
#include <vector>
// `threads` threads make `calls` calls each; every `fail`-th of them is not launched.  Returns the calls that were launched and did not find
// their part emptied by the call launched before them, or -1 if another number of calls was launched than should have been.
extern "C" int stale(int threads, int calls, int fail) {
  fly::Turns<%d> turns;
  unsigned emptied = 0;  // by the call that was launched last
  int wrong = 0, launched = 0;
  auto work = [&](int t) {
    for (int i = 0; i < calls; ++i) {
      const bool ok = fail == 0 || (i + t) %% fail != 0;
      const bool got = turns.take([&](unsigned part, unsigned next) {
        const unsigned before = emptied;
        std::this_thread::yield();  // (another launch would come between)
        if (!ok) return false;
        wrong += part != before || next == part || next >= %d;
        ++launched;
        emptied = next;
        return true;
      });
      if (got != ok) wrong += 1000000;
    }
  };
  std::vector<std::thread> all;
  for (int t = 0; t < threads; ++t) all.emplace_back(work, t);
  for (auto& t : all) t.join();
  int want = 0;
  for (int t = 0; t < threads; ++t)
    for (int i = 0; i < calls; ++i) want += fail == 0 || (i + t) %% fail != 0;
  return launched == want ? wrong : -1;
}
""" % (N, N))
    subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-Wextra", "-Werror", "-pthread", "-shared", "-fPIC", "-I", build.CSRC, "-o",
                    str(d / "turns.so"), str(d / "turns.cpp")], check=True)
    return C.CDLL(str(d / "turns.so")).stale


@pytest.mark.parametrize("threads,calls,fail", [(1, 100, 0), (1, 100, 3), (2, 20000, 0), (4, 20000, 3), (8, 5000, 2)])
def test_a_call_finds_its_part_emptied_by_the_one_before(turns, threads, calls, fail):
    assert turns(threads, calls, fail) == 0
