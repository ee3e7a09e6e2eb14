"""The order of the activations' rows (csrc/rows.h), run on the host: every row of every sequence has one place, and the
rows that a layer has are the first ones."""
import ctypes
import itertools
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_20488_b200", "csrc")

SHIM = r"""
#include "rows.h"
using namespace firp;
static Rows rows(int n_seq, int T, int kc, int chains, int by_step) {
  const int k = chains ? T * kc : kc;
  return Rows{n_seq, T, k, T + k, n_seq * (T + k), 0, chains, kc, 0, 0, by_step};
}
extern "C" {
int place(int n_seq, int T, int kc, int chains, int by_step, int s, int v) { return act_row(rows(n_seq, T, kc, chains, by_step), s, v); }
int word(int s, int v) { const uint16_t w = seq_row(s, v); return row_seq(w) << 16 | row_in_seq(w); }
}
"""


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    d = tmp_path_factory.mktemp("rows")
    src = d / "shim.cpp"
    src.write_text(SHIM)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "shim.so"), str(src)])
    return ctypes.CDLL(str(d / "shim.so"))


@pytest.mark.parametrize("chains", [0, 1])
@pytest.mark.parametrize("by_step", [0, 1])
def test_rows_have_one_place_each_and_a_layers_rows_come_first(rows, chains, by_step):
    for n_seq, T, kc in itertools.product((1, 2, 3, 16), (1, 2, 7, 36), (0, 1, 3)):
        Ms = T + (T * kc if chains else kc)
        case = (n_seq, T, kc, chains, by_step)
        places = {(s, v): rows.place(*case, s, v) for s in range(n_seq) for v in range(Ms)}
        assert sorted(places.values()) == list(range(n_seq * Ms))
        for s, v in places:
            assert rows.word(s, v) == s << 16 | v
        if by_step or n_seq == 1:
            for steps in range(kc + 1):
                alive = T + steps * (T if chains else 1)      # rows of a sequence once that many steps are inserted
                assert sorted(places[s, v] for s in range(n_seq) for v in range(alive)) == list(range(n_seq * alive))
