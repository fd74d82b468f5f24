"""The byte-counted exchange of the table-driven selection, from the geometry that its kernel uses
(csrc/select_slices.h, compiled for the host): no CTA of a cluster can overrun another's key buffers."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_13804_gb300", "csrc")
C = 8  # CTAs of a cluster
N_MAX = 1016

PROGRAM = r"""
#include <cstdio>
#include "select_slices.h"
int main() {
  for (int n = 1; n <= %d; ++n) {
    std::printf("%%d", sp::words_of_round(n, %d));
    for (int r = 0; r < %d; ++r) {
      const sp::Slice s = sp::slice_of(n, %d, r);
      std::printf(" %%d %%d %%d %%d", s.n_loc, s.j0, s.nl, s.words);
    }
    std::printf("\n");
  }
}
""" % (N_MAX, C, C, C)


@pytest.fixture(scope="module")
def slices(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("slices")
    (d / "main.cc").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(d / "main.cc"), "-o", str(d / "main")], check=True)
    lines = subprocess.run([str(d / "main")], check=True, capture_output=True, text=True).stdout.split("\n")[:N_MAX]
    rows = [[int(x) for x in line.split()] for line in lines]
    return {n + 1: (r[0], [tuple(r[1 + 4 * i:5 + 4 * i]) for i in range(C)]) for n, r in enumerate(rows)}


def test_every_slot_is_sent_once(slices):
    for n, (total, ranks) in slices.items():
        sent = [j0 + i for _, j0, _, words in ranks for i in range(words)]
        assert len(sent) == len(set(sent)) == total, n
        assert set(range(n)) <= set(sent) and max(sent) < C * ranks[0][0], n  # (the key buffer's C n_loc slots)
        assert sum(nl for _, _, nl, _ in ranks) == n


def test_no_cta_runs_two_rounds_ahead_of_a_delayed_one(slices):
    """One CTA stands still before its wait of round 0, the others run as far as the counts let them: none may
    send for round 2, which goes to the buffers of round 0."""
    for n, (total, ranks) in slices.items():
        words = [w for _, _, _, w in ranks]
        for slow in range(C):
            sent = [1] * C  # rounds sent; round 0 is out
            while max(sent) < 4:
                # a CTA sends for round q + 1 once it has everybody's words of round q
                ready = [r for r in range(C) if r != slow and
                         sum(w for w, s in zip(words, sent) if s >= sent[r]) == total]
                if not ready:
                    break
                for r in ready:
                    sent[r] += 1
            assert max(sent) <= 2, (n, slow)
