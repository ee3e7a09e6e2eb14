"""The GEMMs' epilogues at the row counts where their passes change: 8 token rows at a time up to 48 rows and 16 above, a last pass of 1 row and of all
of them, operands of an odd multiple of 8 columns (a pass of 16 reads past them), one or two planes to an operand; with rows that
a layer does not have yet (pseudo rows inserted at the second layer) and matrices that end inside a tile, a group of 8 gate and up rows among
them.  Matrices of this size take single tiles and no cluster; test_gemm_variants.py has the kernels of large ones.  Lock-step against the oracle,
the bounds are the harness's own."""
import pytest

import synth_inputs as si
from test_gemm_edges import _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [47, 48, 49, 56, 57, 64, 88, 104, 120, 121, 128, 129])
def test_rows_of_a_step(rows):
    shape = si.scaled(si.CONFIGS["c1"], d=384, H=3, Hkv=1, dh=128, F=1544, V=1001, l=1)
    _run(shape, 20, T=rows - shape.k, steps=1, forced_steps=(0,))
