"""The end flag of a chi block with a helper warp (csrc/pair_end.h), compiled for
the host: every interleaving of the two warps' steps -- barrier, question,
work -- over several batches ends with both warps gone and none left waiting
at a barrier.  A single flag, asked and announced the same way, does not."""
import os
import subprocess

from paper_1806_10889_gb300.build import CSRC

SOURCE = r"""
#include <cstdio>
#include <set>
#include <tuple>
#include "pair_end.h"

struct OneFlag {  // the form that ends a batch early
  int done;
  void clear() { done = 0; }
  void announce(uint32_t) { done = 1; }
  bool reached(uint32_t) const { return done != 0; }
};

// One warp's place: 0 before the barrier of `batch`, 1 waiting at it, 2 past it,
// 3 gone.
struct Warp {
  int at;
  uint32_t batch;
};

template <class Flag>
bool ends(Warp run, Warp help, Flag f, uint32_t batches) {
  // the barrier opens once both wait at it
  if (run.at == 1 && help.at == 1) return run.at = help.at = 2, ends(run, help, f, batches);
  if (run.at == 3 && help.at == 3) return true;
  bool moved = false, ok = true;
  if (run.at == 0 || run.at == 2) {
    Warp r = run;
    Flag g = f;
    if (r.at == 0) {
      if (r.batch == batches) g.announce(r.batch & 1u);  // all cells are done
      r.at = 1;
    } else if (r.batch == batches) {
      r.at = 3;
    } else {
      r.at = 0, ++r.batch;  // this batch's events
    }
    moved = true;
    ok = ok && ends(r, help, g, batches);
  }
  if (help.at == 0 || help.at == 2) {
    Warp h = help;
    if (h.at == 0) h.at = 1;
    else if (f.reached(h.batch & 1u)) h.at = 3;
    else h.at = 0, ++h.batch;  // the next batch's draws
    moved = true;
    ok = ok && ends(run, h, f, batches);
  }
  return moved && ok;
}

template <class Flag>
bool all(uint32_t batches) {
  Flag f;
  f.clear();
  return ends(Warp{0, 0}, Warp{0, 0}, f, batches);
}

int main() {
  for (uint32_t b = 0; b < 7; ++b) std::printf("%d %d\n", all<tsg::PairEnd>(b), all<OneFlag>(b));
}
"""


def test_both_warps_reach_every_barrier_in_every_interleaving(tmp_path):
    src, exe = tmp_path / "pair.cpp", tmp_path / "pair"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", f"-I{CSRC}", str(src), "-o", str(exe)], check=True)
    rows = [tuple(map(int, ln.split())) for ln in
            subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split("\n")
            if ln]
    assert [r[0] for r in rows] == [1] * 7
    assert [r[1] for r in rows] == [1] + [0] * 6  # with a batch before the last barrier it fails


def test_the_kernel_asks_and_announces_through_it():
    with open(os.path.join(CSRC, "chi_lane.cuh")) as fh:
        code = fh.read()
    assert "ex->end.reached(ph)" in code and "ex->end.announce(phase)" in code
    assert "ex->done" not in code
