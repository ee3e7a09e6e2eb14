"""The GEMM kernels that large matrices take around the row counts where the plans change: passes of 8 and of 16 rows, jobs of one to three
tiles, k slices over a cluster, up to four accumulator sets, planes side by side or one after the other.  One layer at the width of the 7B and
of the 34B shape, a step on 200 cached tokens against the oracle: logits and cache rows, the bounds are the harness's own.  Which kernels
those are is asked of the planner, on the host."""
import pytest

import synth_inputs as si
from test_gemm_plans import plan  # noqa: F401

# rows of a step -> of the QKV, O, gate/up and down projection: tiles per job, k slices, more than two accumulator sets, rows of a pass
D1, D4, U3 = (1, 1, True), (1, 4, True), (3, 4, False)
WIDE = {
    "c2": {47: (D1 + (8,), D4 + (8,), (2, 1, False, 8), D4 + (8,)),
           48: (D1 + (8,), D4 + (8,), (2, 1, False, 8), D4 + (8,)),
           49: ((2, 2, False, 16), (1, 4, False, 16), (2, 1, False, 16), D4 + (16,)),
           67: ((2, 2, False, 16), (1, 4, False, 16), (2, 1, False, 16), (1, 4, False, 16)),
           108: (U3 + (16,), (1, 4, False, 16), (3, 2, False, 16), (1, 4, False, 16)),
           131: (U3 + (16,), D4 + (16,), (2, 3, False, 16), D4 + (16,))},
    "c5": {35: ((2, 3, False, 8), (1, 2, True, 8), (3, 1, False, 8), (1, 2, True, 8)),
           41: (D1 + (8,), (1, 2, True, 8), (3, 2, False, 8), (1, 2, True, 8)),
           49: ((2, 3, False, 16), (2, 4, False, 16), (3, 2, False, 16), (2, 4, False, 16)),
           80: ((2, 3, False, 16), (2, 4, False, 16), (3, 2, False, 16), (2, 4, False, 16)),
           131: (U3 + (16,), (3, 6, False, 16), (2, 3, False, 16), (3, 6, False, 16))},
}


def _shape(name):
    return si.scaled(si.CONFIGS[name], L=1, l=0, V=32000 if name == "c2" else 1000, name=name + "-width-1-layer")


@pytest.mark.parametrize("name", sorted(WIDE))
def test_the_sizes_take_these_kernels(plan, name):  # noqa: F811
    s = _shape(name)
    for rows, want in WIDE[name].items():
        for (epi, N, K), kernel in zip(((1, (s.H + 2 * s.Hkv) * s.dh, s.d), (0, s.d, s.H * s.dh), (2, 2 * s.F, s.d), (0, s.d, s.F)), want):
            p = plan((epi, N, K, s.F, s.dh, 2), rows, rows)
            assert (p["tm"], p["split"], p["sets"] > 2, 8 if rows <= 48 else 16) == kernel, (rows, epi, N, K, p)


@pytest.fixture(scope="module")
def weights():
    made = {}

    def of(name):
        if name not in made:
            made.clear()
            made[name] = si.all_weights(_shape(name), gains=True)
        return made[name]
    return of


@pytest.mark.gpu
@pytest.mark.parametrize("name,rows", [(n, r) for n in sorted(WIDE) for r in WIDE[n]])
def test_a_layer_at_full_width(weights, name, rows):
    import oracle
    from lockstep import lockstep_steps, seed_prefix
    from paper_2410_20488_b200 import FirpEngine
    shape, T = _shape(name), rows - 3
    eng = FirpEngine(shape, weights(name), max_ctx=512, max_tree=T)
    orc = oracle.Oracle(shape, weights(name), max_ctx=512)
    seed_prefix(eng, orc, shape, 0, 200)
    st = lockstep_steps(eng, orc, shape, si.tree_template(T, (4, 4, 8)) if T > 8 else si.tree_template(T), si.random_tokens(shape, T, 5), 1, k=3, l=0)
    assert st.steps == 1
    eng.close()
