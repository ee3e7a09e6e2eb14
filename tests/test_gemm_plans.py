"""The GEMMs' plans (csrc/gemm_plan.h), run on the host: the sums of a call are no longer than they were first fixed to be
(golden/gemm_additions.txt, the additions in a row that an accumulator sees), whatever rows a layer has and whatever plan is the fastest."""
import ctypes
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2410_20488_b200", "csrc")

SHIM = r"""
#include "gemm_plan.h"
using namespace firp;
using namespace firp::gemm;
// CTAs that can run at once in clusters of n on a B200
static const int kCtas[9] = {0, 148, 148, 135, 132, 130, 132, 105, 120};
extern "C" void plan(int epi, int N, int K, int F, int dh, int planes, int rows, int call_rows, int *o) {
  const Plan p = make_plan({(GemmEpilogue)epi, N, K, F, dh, planes}, rows, call_rows, kCtas);
  const int whole = p.cf.tp >= 1 && p.cf.sw >= 1 && p.cf.sx >= 1 && (p.cf.by_tile || p.cf.issuers == 1 || !((p.cf.sw | p.cf.sx | p.cf.sets) & 1));
  const int v[9] = {p.adds, p.tm, p.sc.split, p.cf.sets, p.sc.n_tiles, p.sc.jobs, p.smem, (int)p.cf.tmem_cols, whole};
  for (int i = 0; i < 9; ++i) o[i] = v[i];
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plans")
    src = d / "shim.cpp"
    src.write_text(SHIM)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "shim.so"), str(src)])
    lib = ctypes.CDLL(str(d / "shim.so"))

    def of(shape, rows, call_rows):
        o = (ctypes.c_int * 9)()
        lib.plan(*shape, rows, call_rows, o)
        return dict(zip(("adds", "tm", "split", "sets", "tiles", "jobs", "smem", "tmem", "whole"), o))
    return of


def golden():
    with open(os.path.join(HERE, "golden", "gemm_additions.txt")) as f:
        for line in f:
            if line.startswith("#"):
                continue
            words = line.split()
            fixed = {}
            for w in (w for w in words[6:] if ":" in w):
                row, adds = map(int, w.split(":"))
                fixed.update({r: adds for r in range(row, 145)})
            fixed.update({int(w.split("=")[0]): int(w.split("=")[1]) for w in words[6:] if "=" in w})
            yield tuple(map(int, words[:6])), fixed


@pytest.mark.parametrize("shape,fixed", list(golden()), ids=lambda x: "-".join(map(str, x)) if isinstance(x, tuple) else "")
def test_no_sum_of_a_call_becomes_longer(plan, shape, fixed):
    for call_rows, adds in fixed.items():
        # the layers below the insertions: 1 to 8 pseudo rows fewer (one chain), 12 sequences' three, or half and a quarter (a chain under every node)
        below = {call_rows, call_rows - 1, call_rows - 3, call_rows - 8, call_rows - 36, call_rows // 2, call_rows // 4}
        for rows in sorted(r for r in below if r >= 1):
            p = plan(shape, rows, call_rows)
            assert p["tm"] >= 1 and 0 < p["adds"] <= adds, (rows, call_rows, p, adds)
            assert p["jobs"] * p["tm"] >= p["tiles"] and p["smem"] <= 227 * 1024 and p["tmem"] <= 512 and p["split"] <= 8 and p["whole"], (rows, call_rows, p)
