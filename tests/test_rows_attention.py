"""The attention with 128 query rows to a block (more than 48 query rows on more than six tiles of context) where a block goes
through many tiles: buffers and barriers used again and again, the running maximum handed back and forth, a lone block or a
cluster, blocks without tiles, pages, chains, trees of different sizes, one plane; against the oracle, on the plan the test wants."""
import ctypes

import numpy as np
import pytest

import synth_inputs as si
from lockstep import Stats, compare_step, gpu_outputs, lockstep_steps, own_tree_view, seed_prefix

pytestmark = pytest.mark.gpu

BASE = si.scaled(si.CONFIGS["c1"], d=256, H=2, Hkv=2, dh=128, F=512)


class Plan(ctypes.Structure):      # firp::AttnTcPlan
    _fields_ = [("rows", ctypes.c_bool), ("qblocks", ctypes.c_int), ("qper", ctypes.c_int), ("splits", ctypes.c_int)]


def check_plan(qrows, seq_heads, positions, qblocks, splits, tiles):
    """The blocks, splits and tiles per block (of the longest context) that the case is about."""
    from paper_2410_20488_b200 import binding
    plan = binding.load_library()._ZN4firp17attention_tc_planEiiibi
    plan.restype, plan.argtypes = Plan, [ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.c_bool, ctypes.c_int]
    kv_tiles = (positions + 127) // 128
    p = plan(qrows, seq_heads, kv_tiles, False, 148)
    assert (p.rows, p.qblocks, p.splits, -(-kv_tiles // p.splits)) == (True, qblocks, splits, tiles)


def pair(shape, max_ctx, T, k, n_seq=1, max_rows=0, masked=False):
    import oracle
    from paper_2410_20488_b200 import FirpEngine
    weights = si.all_weights(shape, gains=True)
    eng = FirpEngine(shape, weights, max_ctx=max_ctx, max_batch=n_seq, max_tree=T, max_k=k, max_depth=3, max_rows=max_rows)
    eng.set_pseudo_masked(masked)
    return eng, oracle.Oracle(shape, weights, max_ctx=max_ctx, n_seq=n_seq, masked=masked)


def steps_with_trees(eng, orc, shape, trees, T, k, contexts, steps):
    """Sequences with trees of their own on seeded contexts; both sides commit the oracle's path."""
    import torch
    n_seq, rng = len(trees), np.random.default_rng(3)
    sizes = np.array([len(t) for t in trees], np.int32)
    parents = np.full((n_seq, T), 1, np.int32)
    tokens = rng.integers(0, shape.V, (n_seq, T)).astype(np.int32)
    for i, t in enumerate(trees):
        parents[i, :len(t)] = t
        seed_prefix(eng, orc, shape, i, contexts[i])
    out, st = eng.new_out(n_seq, T, k), Stats()
    for _ in range(steps):
        eng.step_trees(torch.from_numpy(tokens).cuda(), parents, sizes, k, 1, out, seq_ids=list(range(n_seq)))
        paths = []
        for i in range(n_seq):
            ref = orc.step(tokens[i, :sizes[i]], trees[i], k, 1, seq=i)
            compare_step(shape, trees[i], tokens[i, :sizes[i]], k, own_tree_view(gpu_outputs(out, i, T, k), int(sizes[i]), T, k), ref, st)
            orc.commit(ref["path"], seq=i)
            paths.append(ref["path"])
            tokens[i, :sizes[i]] = ref["next_tokens"]
        eng.commit(n_seq, seq_ids=list(range(n_seq)), path=paths)
    assert st.steps == steps * n_seq


@pytest.mark.parametrize("contexts,splits,tiles", [((1150, 700), 1, 10), ((2000, 900), 3, 6)])
def test_lone_blocks_and_clusters_on_a_paged_cache(contexts, splits, tiles):
    shape, T, k = si.scaled(BASE, H=40, Hkv=40), 60, 3
    check_plan(T + k, 2 * 40, max(contexts) + T + k, 1, splits, tiles)
    eng, orc = pair(shape, 2304, T, k, n_seq=2)
    eng.set_kv_pages(np.random.default_rng(1).permutation(2 * 2304 // 64).astype(np.int32).reshape(2, -1))
    tree = si.random_tree(4, T, 3, 1)
    steps_with_trees(eng, orc, shape, [tree, tree], T, k, contexts, 1)
    eng.close()


def test_grouped_heads_and_a_tree_per_sequence():
    """Three contexts under one plan: six tiles for every block of the longest, at most one for a block of the shortest."""
    shape, T, k = si.scaled(BASE, H=32, Hkv=8), 16, 3
    contexts = (4000, 1200, 130)
    check_plan((T + k) * 4, 3 * 8, max(contexts) + T + k, 1, 6, 6)
    eng, orc = pair(shape, 4096, T, k, n_seq=3)
    steps_with_trees(eng, orc, shape, [si.random_tree(8, 16, 3, 1), si.random_tree(8, 11, 3, 2), si.chain_template(3)], T, k, contexts, 2)
    eng.close()


@pytest.mark.parametrize("masked", [False, True])
def test_a_chain_under_every_node(masked):
    shape, T, k, n = si.scaled(BASE, H=16, Hkv=8), 36, 3, 4000
    check_plan(T * (1 + k) * 2, 8, n + T * (1 + k), 3, 6, 6)
    eng, orc = pair(shape, 4352, T, k, max_rows=T * (1 + k), masked=masked)
    seed_prefix(eng, orc, shape, 0, n)
    st = lockstep_steps(eng, orc, shape, si.random_tree(9, T, 3, 3), np.arange(T) * 7 % shape.V, 1, k=k, l=[0, 1, 1], chains=True)
    assert st.steps == 1
    eng.close()


def test_planes_and_repeats():
    """One plane of the queries and the probabilities stays inside the bound and is coarser than two; a step repeats bit for bit."""
    import torch
    shape, T, k, n = si.scaled(BASE, H=40, Hkv=40), 60, 3, 2000
    check_plan(T + k, 40, n + T + k, 1, 3, 6)
    parents, tokens, dev = si.random_tree(4, T, 3, 1), np.arange(T, dtype=np.int32) * 5 % shape.V, {}
    eng, orc = pair(shape, 2304, T, k)
    for planes in (2, 1):
        eng.set_attention_planes(planes, planes)
        seed_prefix(eng, orc, shape, 0, n)
        dev[planes] = lockstep_steps(eng, orc, shape, parents, tokens, 1, k=k, l=1, check_cache_rows=False).max_abs
    assert dev[1] > 2 * dev[2], dev
    eng.set_attention_planes(2, 2)
    d_tokens, runs = torch.from_numpy(tokens).cuda(), []
    for _ in range(20):
        eng.set_context_len(0, n)
        out = eng.new_out(1, T, k)
        eng.step(d_tokens, parents, k, 1, out)
        runs.append(out.logits)
    assert all(torch.equal(r, runs[0]) for r in runs)
    eng.close()
