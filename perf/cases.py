"""The work that a user of this package has it do, as measurable cases.

A serving loop prefills a prompt once per request and then runs draft+verify rounds (firp_step*, firp_kv_commit)
until the reply ends; a host with its own sampler calls the stand-alone top-B.  `listed()` holds one case for each
regime of that use, `draw()` gives others of the same ranges.

A round is measured as the loop runs it: the step, then the commit of the path the step found, read on the device.
Every kROUNDS rounds the context is rewound to the prompt, as when a reply ends and the next one starts from the
same cached prompt (otherwise a state that is run thousands of times would outgrow its cache).  The draft tokens
of a state are fixed: random weights accept practically no draft, and feeding a round's own candidates back would make
the second round's inputs hang on near-ties of the first.

Weights, cached prefix rows, prompts and tokens are seeded and made on the GPU: matrices N(0, 0.02), prediction maps
N(0, 1/d), gains 1 + 0.25 N(0, 1), cache rows N(0, (0.02 sqrt(d))^2), the spread that the projections of a unit-RMS row
have.

What is compared: the logits of every row, the values of the candidates of every pseudo row, the cache rows that the
round or the prompt wrote, the accepted path with its length, depth and visibility of every row.  The ids of the
candidates (and the next tree's tokens, taken from them) are left out where logits are computed and not given: with
random weights the eighth and ninth best of 32000 logits are often closer than two correct sums of them.  The top-B cases,
whose logits are given, return the ids.
"""
import itertools
import math

import numpy as np
import torch

import paper_2410_20488_b200 as firp

kROUNDS = 32         # rounds until a state's context is rewound to its prompt
kMAX_ROWS = 144      # rows that one step may carry

# Decoder shapes of the package's benchmark configurations: layers, width, query heads, kv heads, head dimension, FFN
# width, vocabulary.  The 34B shape is cut to 12 of its 48 layers so that three states fit one GPU; a layer costs the same.
MODELS = {
    "tiny": (2, 256, 4, 4, 64, 688, 1024),
    "7b": (32, 4096, 32, 32, 128, 11008, 32000),
    "13b": (40, 5120, 40, 40, 128, 13824, 32000),
    "34b-gqa": (12, 8192, 64, 8, 128, 22016, 32000),
}
# Insertion layers of the prediction steps: one for all of them, or one for each (the published 7B and 13B settings).
SINGLE = {"tiny": 1, "7b": 16, "13b": 20, "34b-gqa": 6}
SPREAD = {"tiny": (0, 1, 1), "7b": (15, 20, 25), "13b": (25, 30, 35), "34b-gqa": (4, 6, 9)}


def _round(model, T, k, context, batch=1, chains=False, spread=False, trees=False, paged=False):
    return {"op": "round", "model": model, "T": T, "k": k, "context": context, "batch": batch, "chains": chains, "spread": spread,
            "trees": trees, "paged": paged}


def listed():
    return [
        # Selection alone, for a host that samples by itself: 35 rows of a 32000-word vocabulary.  The smallest call.
        dict({"op": "topb", "rows": 35, "vocab": 32000, "b": 8}, name="topb-35x32000"),
        # The same for one row of an odd vocabulary.
        dict({"op": "topb", "rows": 1, "vocab": 50257, "b": 5}, name="topb-1x50257"),
        # A tiny draft model on a short context: launches and host work are all there is.
        dict(_round("tiny", 8, 3, 32), name="tiny-round"),
        # Plain decoding, one row and no draft: the first token of a reply, or a user who turned the drafts off.
        dict(_round("7b", 1, 0, 128), name="7b-plain"),
        # The ordinary round: 32 tree rows, 3 pseudo rows, half a thousand committed tokens.
        dict(_round("7b", 32, 3, 512), name="7b-round"),
        # A long conversation: the cache is a third of the bytes.
        dict(_round("7b", 32, 3, 8192), name="7b-long"),
        # The widest tree, at an odd context: rows rather than weights bound the contractions.
        dict(_round("7b", 128, 3, 2047), name="7b-wide"),
        # A chain of pseudo rows under every node, one insertion layer for each prediction step.
        dict(_round("7b", 32, 3, 512, chains=True, spread=True), name="7b-chains"),
        # Several requests at once, each with its own tree and its own context, on a paged cache.
        dict(_round("7b", 16, 2, 1024, batch=6, trees=True, paged=True), name="7b-batch"),
        # The 13B shape with 64 tree rows and the published insertion layers.
        dict(_round("13b", 64, 3, 1024, spread=True), name="13b-round"),
        # Grouped-query attention, four requests with contexts from a few hundred to four thousand tokens.
        dict(_round("34b-gqa", 32, 3, 4096, batch=4), name="34b-batch"),
        # A long prompt, ragged against every chunk size.  The largest call.
        dict({"op": "prefill", "model": "7b", "k": 3, "spread": False, "tokens": 1999, "T": 32}, name="7b-prompt-1999"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(("topb", "tiny", "round", "batch", "chains", "prompt"), (1, 1, 5, 2, 1, 2))[0]
    if kind == "topb":
        vocab = _log_uniform(rng, 1000, 130000)
        return {"op": "topb", "rows": min(_log_uniform(rng, 1, kMAX_ROWS), 4096 // -(-vocab // 2048)), "vocab": vocab, "b": rng.randint(1, 8)}
    model = rng.choices(("7b", "13b", "34b-gqa"), (4, 1, 1))[0]
    spread = rng.random() < 0.4
    if kind == "prompt":
        return {"op": "prefill", "model": "7b", "k": rng.randint(0, 3), "spread": spread, "tokens": _log_uniform(rng, 16, 1999), "T": 32}
    if kind == "tiny":
        return _round("tiny", _log_uniform(rng, 1, 64), 3, _log_uniform(rng, 8, 2000), spread=spread, paged=rng.random() < 0.3)
    k = rng.randint(1, 3)
    if kind == "batch":
        batch = rng.randint(2, 12)
        T = _log_uniform(rng, 1, kMAX_ROWS // batch - k)
        return _round(model, T, k, _log_uniform(rng, 64, min(4096, 12288 // batch)), batch=batch, spread=spread, trees=rng.random() < 0.5, paged=rng.random() < 0.5)
    if kind == "chains":
        return _round(model, _log_uniform(rng, 2, kMAX_ROWS // (1 + k)), k, _log_uniform(rng, 32, 4096), chains=True, spread=spread)
    T = _log_uniform(rng, 1, 128)
    return _round(model, T, 0 if T == 1 else k, _log_uniform(rng, 32, 8192), spread=spread, paged=rng.random() < 0.3)


# ---- trees ---------------------------------------------------------------------------------------------------------
def _tree(T, depth):
    """Parents of a draft tree of T nodes, at most 8 children each and at most `depth` deep: the first T nodes, by sum of
    sibling ranks, of the smallest per-depth-width product tree that holds so many."""
    if T == 1:
        return [-1]
    for top in range(1, 9):
        widths = [max(1, top - j) for j in range(depth)]
        nodes = [n for d in range(depth + 1) for n in itertools.product(*(range(w) for w in widths[:d]))]
        if len(nodes) >= T:
            break
    else:
        nodes = [n for d in range(depth + 1) for n in itertools.product(*(range(8) for _ in range(d)))]
    nodes.sort(key=lambda n: (sum(n), len(n), n))
    nodes = nodes[:T]
    at = {n: i for i, n in enumerate(nodes)}
    return [-1] + [at[n[:-1]] for n in nodes[1:]]


def _most_nodes(T, k):
    """The largest tree that k prediction steps can fill with 8 candidates each, at most T."""
    return min(T, sum(8 ** j for j in range(k + 1)))


# ---- states --------------------------------------------------------------------------------------------------------
class _Engine(firp.FirpEngine):
    """The package's engine on weights that are on the GPU already."""

    def _dev(self, bits):
        return bits


class _Shape:
    """The fields of a decoder shape that the engine reads."""

    def __init__(self, model, T, k):
        self.L, self.d, self.H, self.Hkv, self.dh, self.F, self.V = MODELS[model]
        self.T, self.k, self.eps, self.theta = T, k, 1e-5, 1e4


def _weights(s, n_maps, gen, device):
    def normal(std, *shape):
        return torch.empty(shape, dtype=torch.bfloat16, device=device).normal_(0.0, std, generator=gen)

    def gain():
        return 1.0 + normal(0.25, s.d)

    n_qkv = (s.H + 2 * s.Hkv) * s.dh
    w = {"embed": normal(0.02, s.V, s.d), "lm_head": normal(0.02, s.V, s.d), "g_final": gain()}
    if n_maps:
        w["pred_w"] = normal(s.d ** -0.5, n_maps, s.d, s.d)
        w["pred_b"] = normal(0.02, n_maps, s.d)
    w["layers"] = [{"wqkv": normal(0.02, n_qkv, s.d), "wo": normal(0.02, s.d, s.H * s.dh), "wgu": normal(0.02, 2 * s.F, s.d),
                    "wd": normal(0.02, s.d, s.F), "g_attn": gain(), "g_mlp": gain()} for _ in range(s.L)]
    return w


def _layers(case):
    return list(SPREAD[case["model"]][:case["k"]]) if case["spread"] else SINGLE[case["model"]]


def _contexts(case):
    """Committed tokens of each sequence: the case's own for one, from an eighth of it up to it for several."""
    n, batch = case["context"], case["batch"]
    return [n] if batch == 1 else [max(1, n - (n - n // 8) * i // (batch - 1)) for i in range(batch)]


def _rows(case):
    return case["T"] * (1 + case["k"]) if case.get("chains") else case["T"] + case["k"]


class _TopB:
    def __init__(self, case, seed):
        gen = torch.Generator("cuda").manual_seed(seed)
        self.rows, self.vocab, self.b = case["rows"], case["vocab"], case["b"]
        self.logits = torch.empty(self.rows, self.vocab, device="cuda").normal_(0.0, 1.3, generator=gen)
        self.ids = torch.empty(self.rows, self.b, dtype=torch.int32, device="cuda")
        self.vals = torch.empty(self.rows, self.b, device="cuda")

    def run(self):
        firp.firp_topb_static(self.logits.data_ptr(), self.rows, self.vocab, self.b, self.ids.data_ptr(), self.vals.data_ptr(),
                              torch.cuda.current_stream().cuda_stream)
        return self.ids, self.vals


class _Prompt:
    def __init__(self, case, seed):
        gen = torch.Generator("cuda").manual_seed(seed)
        self.k, self.T, self.P, self.l = case["k"], case["T"] if case["k"] else 1, case["tokens"], _layers(case)
        self.T = min(self.T, _most_nodes(self.T, self.k)) if self.k else 1
        s = _Shape(case["model"], self.T, self.k)
        self.eng = _Engine(s, _weights(s, self.k, gen, "cuda"), max_ctx=-(-(self.P + self.k + 128) // 64) * 64, max_tree=self.T, max_k=self.k)
        self.prompt = torch.randint(0, s.V, (self.P,), dtype=torch.int32, device="cuda", generator=gen)
        self.parents = np.array(_tree(self.T, self.k), np.int32) if self.k else None
        out = self.out = self.eng.new_out(1, 1, self.k, T_next=self.T)
        cache = self.eng.kv.view(torch.bfloat16).view(s.L, 2, -1, s.Hkv * s.dh)
        self.result = {"logits": out.logits, "n_accepted": out.n_accepted, "cache": cache[:, :, :self.P]}
        if self.k:
            self.result["topb_vals"] = out.topb_vals

    def run(self):
        self.eng.prefill(0, self.prompt, self.k, self.l, self.parents, self.out)
        return self.result


class _Round:
    def __init__(self, case, seed):
        gen = torch.Generator("cuda").manual_seed(seed)
        k, batch, chains = case["k"], case["batch"], case["chains"]
        T = _most_nodes(case["T"], k) if k else 1
        s = _Shape(case["model"], T, k)
        rows = T * (1 + k) if chains else T + k
        self.k, self.batch, self.l, self.contexts = k, batch, _layers(case), _contexts(case)
        depth = max(k, 1)
        max_ctx = -(-(max(self.contexts) + kROUNDS * (depth + 1) + rows) // 64) * 64
        self.eng = _Engine(s, _weights(s, k, gen, "cuda"), max_ctx=max_ctx, max_batch=batch, max_tree=T, max_k=k, max_rows=batch * rows)
        # the committed prefix (and stale rows after it, as in any cache that has been used)
        self.eng.kv.view(torch.bfloat16).normal_(0.0, 0.02 * math.sqrt(s.d), generator=gen)
        self.tokens = torch.randint(0, s.V, (batch, T), dtype=torch.int32, device="cuda", generator=gen)
        self.parents = np.array(_tree(T, k), np.int32)
        self.trees = None
        if case["trees"] and k:            # every sequence another size of tree, from the whole one down to a quarter
            self.sizes = np.array([max(1, T - (3 * T // 4) * i // max(1, batch - 1)) for i in range(batch)], np.int32)
            self.trees = np.stack([self.parents] * batch)
        written = [(n, n + kROUNDS * (depth + 1) + rows) for n in self.contexts]
        cache = self.eng.kv.view(torch.bfloat16).view(s.L, 2, batch * max_ctx, s.Hkv * s.dh)
        if case["paged"]:                  # pages in random order, those that rounds write in the upper part of the cache
            pps = max_ctx // 64
            late = [[a // 64 <= p < -(-b // 64) for p in range(pps)] for a, b in written]
            order = np.random.RandomState(seed & 0x7fffffff)
            early_n, table = sum(not x for r in late for x in r), np.empty((batch, pps), np.int32)
            late_np = np.array(late)
            table[~late_np] = order.permutation(early_n)
            table[late_np] = early_n + order.permutation(batch * pps - early_n)
            self.eng.set_kv_pages(table)
            new_rows = [cache[:, :, early_n * 64:]]
        else:
            new_rows = [cache[:, :, i * max_ctx + a:i * max_ctx + b] for i, (a, b) in enumerate(written)]
        for i, n in enumerate(self.contexts):
            self.eng.set_context_len(i, n)
        self.step = self.eng.step_chains if chains else self.eng.step
        self.rounds = 0
        out = self.out = self.eng.new_out(batch, T, k, chains=chains)
        self.result = {"logits": out.logits, "n_accepted": out.n_accepted, "path": out.path, "depth": out.depth, "mask": out.mask, "cache": new_rows}
        if k and not chains:
            self.result["topb_vals"] = out.topb_vals
        if self.trees is not None:         # rows beyond a sequence's own tree are padding: what the outputs hold for them is unspecified
            keep = [slice(0, int(n)) for n in self.sizes]
            self.result["logits"] = [x for i in range(batch) for x in (out.logits[i, keep[i]], out.logits[i, T:])]
            self.result["depth"] = [out.depth[i, keep[i]] for i in range(batch)]
            self.result["mask"] = [out.mask[i, keep[i]] for i in range(batch)]

    def run(self):
        eng = self.eng
        if self.rounds == kROUNDS:
            for i, n in enumerate(self.contexts):
                eng.set_context_len(i, n)
            self.rounds = 0
        if self.trees is not None:
            eng.step_trees(self.tokens, self.trees, self.sizes, self.k, self.l, self.out)
        else:
            self.step(self.tokens, self.parents, self.k, self.l, self.out, n_seq=self.batch)
        eng.commit(self.batch)
        self.rounds += 1
        return self.result


def prepare(case, seed):
    return {"topb": _TopB, "prefill": _Prompt, "round": _Round}[case["op"]](case, seed)


def run(state):
    return state.run()


# ---- what a pass cannot do without ----------------------------------------------------------------------------------
def work(case):
    if case["op"] == "topb":
        return {"bytes": 4 * case["rows"] * case["vocab"] + 8 * case["rows"] * case["b"], "flops": 0}
    L, d, H, Hkv, dh, F, V = MODELS[case["model"]]
    k = case["k"]
    per_layer = (H + 2 * Hkv) * dh * d + d * H * dh + 3 * d * F
    weights = L * per_layer + V * d + k * d * d
    if case["op"] == "prefill":
        T, P = 1, case["tokens"]
        read, tree_rows, chain_rows, sources = 0, P, k, 1
        attended = P * (P + 1) // 2 + k * P
        head_rows = 1 + k
    else:
        T, batch = (_most_nodes(case["T"], k) if k else 1), case["batch"]
        read = sum(_contexts(case))
        tree_rows, chain_rows = batch * T, batch * (T * k if case["chains"] else k)
        sources = batch * (T if case["chains"] else 1)
        attended = (T + chain_rows // batch) * read
        head_rows = tree_rows + chain_rows
    first = SPREAD[case["model"]][:k] if case["spread"] else (SINGLE[case["model"]],) * k
    row_layers = tree_rows * L + sum(L - t for t in first) * (chain_rows // k if k else 0)      # rows of all layers together
    kv_row = 2 * 2 * Hkv * dh
    bytes_ = 2 * weights + kv_row * (L * read + row_layers) + 2 * d * tree_rows + 4 * V * head_rows
    flops = 2 * per_layer * row_layers + 2 * V * d * head_rows + 2 * k * d * d * sources + 4 * H * dh * attended * L
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    if case["op"] == "topb":
        return "exact"
    # Measured between the package's own orders of summation (a third activation plane on the QKV projection, the other
    # attention kernel, the persistent kernel): up to 2.7e-4 (rounds) and 1.3e-3 (prompts, whose cache rows feed one another) in
    # the 2-norm, and single cache values one or two bf16 steps apart (0.008, 0.012).  Plain bf16 activations give 7e-3 to 3e-2.
    return {"rel": 5e-3, "max": 0.05} if case["op"] == "prefill" else {"rel": 1.2e-3, "max": 0.03}
