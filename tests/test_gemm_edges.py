"""The GEMMs with their fused epilogues, prompts that run in one stretch, and the attention's blocks of many query rows, at the
sizes where a tile, a block of rows or a stretch ends: lock-step against the oracle (prefill logits, cache rows, two steps; the bounds are the harness's own)."""
import pytest

import synth_inputs as si
from lockstep import lockstep_run

pytestmark = pytest.mark.gpu

SMALL = si.scaled(si.CONFIGS["c1"], d=256, H=2, Hkv=2, dh=128, F=512)


def _run(shape, P, steps=2, T=8, forced_steps=(), masked=False):
    import oracle
    from paper_2410_20488_b200 import FirpEngine
    weights = si.all_weights(shape, gains=True)
    parents = si.tree_template(T, (4, 4, 8))
    max_ctx = (P + 8 * T + 63) // 64 * 64
    eng = FirpEngine(shape, weights, max_ctx=max_ctx, max_tree=T)
    orc = oracle.Oracle(shape, weights, max_ctx=max_ctx, masked=masked)
    if masked:
        eng.set_pseudo_masked(True)
    lockstep_run(eng, orc, shape, parents, si.prompt(shape, length=P), steps, forced_steps=forced_steps)
    eng.close()


# 144 rows: what a step may have; 256: a block of token rows; 2047 rows: a stretch (3 of them pseudo rows)
@pytest.mark.parametrize("P", [1, 15, 125, 141, 142, 145, 253, 254, 257, 500, 1021, 2044, 2045, 2100])
def test_prompt_lengths(P):
    _run(SMALL, P, forced_steps=(1,))


@pytest.mark.parametrize("l", [0, 1])
def test_prompt_with_masked_pseudo_rows(l):
    _run(si.scaled(SMALL, l=l), 300, masked=True)


# rows of the matrices that end inside a tile: odd vocabularies, FFN widths, head counts
@pytest.mark.parametrize("kw", [dict(d=384, H=3, Hkv=1, dh=128, F=1000, V=1001), dict(d=128, H=1, Hkv=1, dh=128, F=8, V=9),
                                dict(d=384, H=5, Hkv=1, dh=64, F=136, V=2050), dict(d=1152, H=9, Hkv=3, dh=128, F=1544, V=1031)])
def test_ragged_matrices(kw):
    _run(si.scaled(si.CONFIGS["c1"], **kw), 200)


# more than 48 query rows on more than six tiles of context: one block of 128 rows, or two; clusters of five to eight splits of one or two tiles
# (many tiles per block, lone blocks: test_rows_attention.py)
@pytest.mark.parametrize("T,H,Hkv,P,masked", [(46, 2, 2, 764, False), (61, 2, 2, 1023, True), (125, 2, 2, 893, False), (126, 2, 1, 1150, False),
                                              (8, 16, 2, 800, False), (32, 8, 1, 1021, False)])
def test_many_query_rows(T, H, Hkv, P, masked):
    _run(si.scaled(SMALL, d=H * 128, H=H, Hkv=Hkv), P, T=T, forced_steps=(1,), masked=masked)


def test_a_limit_shorter_than_a_kernel_is_no_time_out():
    """Waits are for single tiles and start when the kernel before has completed: launches of several hundred microseconds, of blocks
    that work 60 us each, pass under a limit of 50 us."""
    import torch
    from paper_2410_20488_b200 import FirpEngine
    shape = si.scaled(si.CONFIGS["c1"], L=1, l=0, d=4096, H=32, Hkv=32, dh=128, F=11008)
    P = 2044
    eng = FirpEngine(shape, si.all_weights(shape), max_ctx=2112)
    prompt = torch.from_numpy(si.prompt(shape, length=P)).cuda()
    parents = si.tree_template(shape.T)
    first, second = (eng.new_out(1, 1, shape.k, T_next=shape.T) for _ in range(2))
    eng.prefill(0, prompt, shape.k, shape.l, parents, first)
    assert eng.context_len(0) == P
    eng.set_wait_limit_us(50)
    eng.prefill(0, prompt, shape.k, shape.l, parents, second)
    assert eng.context_len(0) == P                 # raises on a time-out
    assert torch.equal(first.logits, second.logits)
    eng.close()


@pytest.mark.parametrize("T,Hkv", [(32, 64), (128, 8)])
def test_a_limit_shorter_than_the_projection_before_the_attention_is_no_time_out(T, Hkv):
    """The attention's blocks start under the QKV projection (403 MB of weights or 131 rows: more than 40 us) and load the first tiles of
    the cached context, which has many for each; their waits for what the projection ends do not count it: a limit of 25 us is no time-out.
    Both tcgen05 kernels: 35 query rows on 64 kv heads, 1048 on 8."""
    import numpy as np
    import torch
    from paper_2410_20488_b200 import FirpEngine
    n = 4000
    shape = si.scaled(si.CONFIGS["c1"], L=1, l=0, d=8192, H=64, Hkv=Hkv, dh=128, F=1024)
    eng = FirpEngine(shape, si.all_weights(shape), max_ctx=4352, max_tree=T)
    eng.kv.view(torch.bfloat16).normal_(0.0, 1.8)
    tokens = torch.from_numpy(si.random_tokens(shape, T, 3)).cuda()
    first, second = eng.new_out(1, T, shape.k), eng.new_out(1, T, shape.k)
    for out, limit in ((first, 0), (second, 25)):
        eng.set_wait_limit_us(limit)
        for _ in range(4):
            eng.set_context_len(0, n)
            eng.step(tokens, np.asarray(si.tree_template(T)), shape.k, shape.l, out)
            assert eng.context_len(0) == n         # raises on a time-out
    assert torch.equal(first.logits, second.logits)
    eng.close()


@pytest.mark.parametrize("d,H,Hkv,F,V", [(4096, 32, 32, 11008, 32000), (5120, 40, 40, 13824, 32000), (8192, 64, 8, 22016, 32000)])
def test_sums_of_a_step_are_no_longer_than_equal_shares_make_them(d, H, Hkv, F, V):
    """The tensor core truncates on every addition: no accumulator of a step sees more in a row than if every SM had an equal share
    of the matrix (pairs of 128-row tiles; both planes in the same columns from 49 rows on), or 96 (1.6e-6, below the planes' own 2.4e-6)."""
    import ctypes
    from paper_2410_20488_b200 import binding
    additions = binding.load_library()._ZN4firp14gemm_additionsENS_12GemmEpilogueEiiiiii
    additions.restype, additions.argtypes = ctypes.c_int, [ctypes.c_int] * 7
    for rows in (1, 4, 11, 18, 35, 48, 49, 67, 72, 96, 108, 128, 129, 131, 140, 144):
        for epi, N, K in ((0, d, H * 128), (0, d, F), (1, (H + 2 * Hkv) * 128, d), (2, 2 * F, d), (3, V, d), (4, 3 * d, d)):
            blocks, pairs = -(-K // 64), -(-(-(-N // 128)) // 2)
            share = 4 * min(blocks, -(-pairs * blocks // 148)) * (1 if rows <= 48 else 2)
            assert 0 < additions(epi, N, K, F, 128, rows, 2) <= max(96, share), (rows, epi, N, K)
