"""Several sequences in one step with pseudo rows inserted at layers of their own: the rows of the activations then go by prediction step
(csrc/rows.h) and the layers run on 24, 27, ... of them.  One chain and a chain under every node, Eq. 3 on the raw and on the normalised
state, pseudo rows that do not see one another, trees of different sizes; contexts of their own, both head dimensions.  Lock-step against the
oracle, sequence by sequence: logits, walks, candidates, committed cache rows; the bounds are the harness's own."""
import numpy as np
import pytest

import synth_inputs as si
from lockstep import Stats, check_cache, compare_step, gpu_outputs, lockstep_run_batch, own_tree_view
from test_gpu_parity import dh128_shape, make_pair, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu

LENGTHS = (45, 9, 131)


def _pair(c1, head_dim, **kw):
    shape = si.scaled(c1, Hkv=2) if head_dim == 64 else dh128_shape(c1, 4, 2)
    shape = si.scaled(shape, L=4, l=1)
    weights = si.all_weights(shape, gains=True)
    weights["pred_b"] = si.normal_bf16(shape.seed, si.stream_id("pred_w", 9), shape.k * shape.d, 0.5).reshape(shape.k, shape.d)
    eng, orc = make_pair(shape, weights, 256, max_batch=3, max_tree=12, max_k=3, max_depth=3, **kw)
    return shape, eng, orc


def _prefill(eng, orc, shape, trees, layers):
    import torch
    tokens = []
    for s, n in enumerate(LENGTHS):
        prompt = si.prompt(shape, seq=s, length=n)
        eng.prefill(s, torch.from_numpy(prompt).cuda(), 3, layers, trees[s], eng.new_out(1, 1, 3, T_next=len(trees[s])))
        tokens.append(orc.prefill(prompt, 3, layers, trees[s], seq=s)["next_tokens"].copy())
    return tokens


def _commit(eng, orc, shape, refs):
    n0 = [orc.context_len(s) for s in range(3)]
    eng.commit(3, path=[r["path"] for r in refs])
    for s in range(3):
        orc.commit(refs[s]["path"], seq=s)
        assert eng.context_len(s) == orc.context_len(s)
        check_cache(eng, orc, s, range(n0[s], orc.context_len(s)), range(shape.L))


@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("layers,kw", [([0, 1, 3], {}), ([1, 2, 2], dict(prenorm=True)), ([0, 2, 3], dict(masked=True))])
def test_one_chain_with_a_layer_for_each_step(torch_cuda, c1, head_dim, layers, kw):  # noqa: F811
    shape, eng, orc = _pair(c1, head_dim, **kw)
    parents = si.random_tree(5, 8, 3, 6)
    st = lockstep_run_batch(eng, orc, shape, parents, [si.prompt(shape, seq=s, length=n) for s, n in enumerate(LENGTHS)], 3, l=layers)
    assert st.steps == 9
    eng.close()


@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("T,layers,kw", [(12, [0, 1, 3], {}), (12, [1, 2, 2], dict(prenorm=True)), (11, 2, dict(prenorm=True)), (5, [0, 0, 2], dict(masked=True))])
def test_a_chain_under_every_node(torch_cuda, c1, head_dim, T, layers, kw):  # noqa: F811
    import torch
    shape, eng, orc = _pair(c1, head_dim, max_rows=3 * 12 * 4, **kw)
    parents = si.random_tree(6, T, 3, 3)
    tokens = _prefill(eng, orc, shape, [parents] * 3, layers)
    out, st = eng.new_out(3, T, 3, chains=True), Stats()
    for _ in range(2):
        eng.step_chains(torch.from_numpy(np.stack(tokens)).cuda(), parents, 3, layers, out, n_seq=3)
        refs = [orc.step_chains(tokens[s], parents, 3, layers, seq=s) for s in range(3)]
        for s in range(3):
            compare_step(shape, parents, tokens[s], 3, gpu_outputs(out, s, T, 3), refs[s], st, chains=True)
            tokens[s] = refs[s]["next_tokens"].copy()
        _commit(eng, orc, shape, refs)
    assert st.steps == 6
    eng.close()


@pytest.mark.parametrize("head_dim", [64, 128])
def test_trees_of_different_sizes(torch_cuda, c1, head_dim):  # noqa: F811
    import torch
    shape, eng, orc = _pair(c1, head_dim, prenorm=True)
    T, layers, trees = 8, [0, 1, 3], [si.tree_template(8), si.random_tree(8, 5, 3, 1), si.chain_template(3)]
    sizes = np.array([len(t) for t in trees], np.int32)
    parents = np.zeros((3, T), np.int32)
    for s, t in enumerate(trees):
        parents[s, : len(t)] = t
    tokens = _prefill(eng, orc, shape, trees, layers)
    out, st = eng.new_out(3, T, 3), Stats()
    for _ in range(2):
        padded = np.stack([np.pad(t, (0, T - len(t))) for t in tokens]).astype(np.int32)
        eng.step_trees(torch.from_numpy(padded).cuda(), parents, sizes, 3, layers, out)
        refs = [orc.step(tokens[s], trees[s], 3, layers, seq=s) for s in range(3)]
        for s in range(3):
            compare_step(shape, trees[s], tokens[s], 3, own_tree_view(gpu_outputs(out, s, T, 3), int(sizes[s]), T, 3), refs[s], st)
            tokens[s] = refs[s]["next_tokens"].copy()
        _commit(eng, orc, shape, refs)
    assert st.steps == 6
    eng.close()
