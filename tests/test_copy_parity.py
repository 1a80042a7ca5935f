"""The wait of a warp for its copy, when it gives up: the copy is still in flight, and what then drains it must wait for it."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1910_05124_b200", "csrc")

# A barrier with one arrival per phase: a wait on a parity succeeds once the phase of that parity has completed.
PROGRAM = r"""
#include <cstdio>
#include "pm_copy_parity.cuh"
struct Barrier { unsigned phase = 0; bool passed(unsigned parity) const { return (phase & 1u) != parity; } };
int main() {
  // `before` copies have landed and been seen; the next is in flight when the wait gives up, and lands after `late` polls
  for (int before = 0; before < 5; ++before)
    for (int late = 0; late < 4; ++late) {
      Barrier bar;
      pm::CopyParity copy;
      for (int i = 0; i < before; ++i) { ++bar.phase; if (!copy.await([&](unsigned p) { return bar.passed(p); })) return 1; }
      if (copy.await([&](unsigned p) { return bar.passed(p); })) return 2;        // in flight: must not count as landed
      int polls = 0;
      copy.drain([&](unsigned p) { if (polls++ == late) ++bar.phase; return bar.passed(p); }, [&] { return polls < 100; });
      if (bar.phase != before + 1u || polls != late + 1) { std::printf("before %d late %d: %d polls\n", before, late, polls); return 3; }
      polls = 0;                                                                  // a copy that never lands: the bound ends the wait
      copy.parity ^= 1u;
      copy.drain([&](unsigned p) { ++polls; return bar.passed(p); }, [&] { return polls < 7; });
      if (polls != 7) return 4;
    }
  return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_wait_that_gives_up_leaves_the_copy_to_drain(tmp_path):
    src = tmp_path / "parity.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "parity"
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-x", "c++", str(src), "-o", str(exe)], check=True)
    run = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert run.returncode == 0, (run.returncode, run.stdout)


def test_the_epilogue_keeps_its_parity_there():
    text = open(os.path.join(CSRC, "pm_umma.cu")).read()
    stage = text[text.index("struct EpiStage"):]
    stage = stage[:stage.index("\n};")]
    assert "copy.await(" in stage and "copy.drain(" in stage and "^= 1u" not in stage
