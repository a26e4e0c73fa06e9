"""The host side of the generation loop (csrc/cs_loop_host.h) against a device that is played on the
CPU: steps finish at the worst moments, between any two looks of the host at the progress word.  No
step may be sent that nobody needs, none may be missing, and at most two may be ahead of the reports."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2502_08923_b200", "csrc")

PROGRAM = r"""
#include <stdio.h>
#include <stdlib.h>
#include "cs_loop_host.h"

// argv: max_new k seed eager; accepted lengths per step come from the seed
int main(int argc, char** argv) {
  const int max_new = atoi(argv[1]), k = atoi(argv[2]), eager = atoi(argv[4]);
  unsigned rnd = 2654435761u * (unsigned)(atoi(argv[3]) + 1);
  auto next = [&] { rnd = rnd * 1664525u + 1013904223u; return rnd >> 8; };
  int sent = 0, done = 0, emitted = 0, looks = 0, useless = 0, ahead = 0, most[4096];
  most[0] = max_new;                                   // most[n]: tokens wanted after n steps
  for (int n = 1; n < 4096; ++n) {
    const int left = most[n - 1] - 1 - (int)(next() % (unsigned)(k + 1));
    most[n] = left > 0 ? left : 0;
  }
  auto finish = [&] { if (done < sent) { ++done; emitted = max_new - most[done]; } };
  // the device may finish one step before and one after every look
  auto word = [&]() -> unsigned long long {
    ++looks;
    if (eager == 0 || (eager == 2 && (next() & 1))) finish();
    const unsigned long long w = (unsigned long long)(unsigned)done << 32 | (unsigned)most[done];
    if (eager == 1 || (eager == 2 && (next() & 1))) finish();
    return w;
  };
  auto send = [&](int n, int) {
    if (n != sent + 1) return 2;
    if (most[sent] == 0) ++useless;                    // what is in flight already ends every sequence
    ++sent;
    if (sent - done > ahead) ahead = sent - done;
    return 0;
  };
  auto wait = [&](LoopProgress* at, int n) {
    if (n != sent) return 4;
    if (k == 0 && likely_last(*at, n, max_new) != (at->wanted <= n - at->steps && at->steps > 0)) return 5;   // certain where a step brings one token
    for (int i = 0; i < 64; ++i)
      if (newer_report(word, at)) return 0;
    return 3;                                          // waited for a report that cannot come
  };
  const int status = drive_loop(max_new, k, send, wait);
  while (done < sent) finish();
  printf("%d %d %d %d %d\n", status, useless, emitted, ahead, sent);
  return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    gxx = shutil.which("g++")
    assert gxx, "g++ is part of the toolchain"
    d = tmp_path_factory.mktemp("loop_host")
    (d / "main.cpp").write_text(PROGRAM)
    subprocess.run([gxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-I", CSRC, "-o", str(d / "main"), str(d / "main.cpp")], check=True)
    return str(d / "main")


@pytest.mark.parametrize("k", [0, 1, 10])
@pytest.mark.parametrize("eager", [0, 1, 2])     # a step finishes before the look, behind it, at random
def test_every_step_is_needed(program, k, eager):
    for max_new in (0, 1, 2, 11, 12, 23, 60, 200):
        for seed in range(12):
            out = subprocess.run([program, str(max_new), str(k), str(seed), str(eager)], check=True, capture_output=True, text=True, timeout=20)
            status, useless, emitted, ahead, sent = map(int, out.stdout.split())
            assert (status, useless, emitted) == (0, 0, max_new), (max_new, seed)
            assert ahead <= 2 and sent <= max_new
