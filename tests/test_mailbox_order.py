"""The order in which the loop reads the host's words: blink_start promises that everything submitted before it is
visible to the first iteration.  The reading function is plain C++; here it runs against a host whose stores (publish the
entries, then set start) fall between any two of its loads."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_07609_b200", "csrc")

PROGRAM = r"""
#include <stdio.h>
#include "mailbox.h"
struct Host {                       // the host's two stores happen before load number `tail_at` and `start_at`
  int load = 0, tail_at, start_at;
  uint32_t stop_relaxed() { ++load; return 0; }
  uint32_t start_acquire() { return load++ >= start_at; }
  uint64_t sub_tail_acquire() { return load++ >= tail_at ? 8 : 5; }
};
int main() {
  int bad = 0, paused = 0;
  for (int tail_at = 0; tail_at <= 4; ++tail_at)
    for (int start_at = tail_at; start_at <= 4; ++start_at) {   // submit before start
      Host h;
      h.tail_at = tail_at; h.start_at = start_at;
      const blink::MailboxView v = blink::read_mailbox(h, true);
      if (v.started && v.tail != 8) { printf("started with %d of 8 entries: stores before loads %d and %d\n", (int)v.tail, tail_at, start_at); bad = 1; }
      paused += !v.started;
      Host g;
      g.tail_at = tail_at; g.start_at = 99;
      if (!blink::read_mailbox(g, false).started || g.load != 2) { printf("an open loop read the start word\n"); bad = 1; }
    }
  if (!paused) { printf("the gate never held\n"); bad = 1; }
  return bad;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_a_started_loop_sees_everything_submitted_before_the_start(tmp_path):
    src, exe = tmp_path / "order.cpp", tmp_path / "order"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
