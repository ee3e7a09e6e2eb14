"""Top-B selection at the sizes and orders where its threshold and its passes can go wrong: around one thread's, one
CTA's and one cluster's share of a row, rows in ascending and descending order (every element of a lane qualifies, or one),
ties, infinities, NaN and signed zeros; exact against a host sort by (value descending, id ascending)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _rows(vocab, rng):
    normal = rng.standard_normal(vocab).astype(np.float32)
    special = normal.copy()
    special[rng.integers(0, vocab, vocab // 3 + 1)] = np.nan
    special[rng.integers(0, vocab, vocab // 3 + 1)] = -np.inf
    special[rng.integers(0, vocab, 2)] = np.inf
    zeros = np.where(rng.random(vocab) < 0.5, np.float32(0.0), np.float32(-0.0))
    return np.stack([normal, np.sort(normal), np.sort(normal)[::-1], np.round(normal), special, zeros, np.full(vocab, -np.inf, np.float32)])


@pytest.mark.parametrize("vocab,b", [(1, 8), (7, 8), (8, 8), (9, 3), (512, 8), (513, 8), (4095, 8), (4096, 1), (4097, 8), (32767, 8),
                                     (32768, 5), (32769, 8), (50257, 5), (130001, 8),
                                     (32, 8), (33, 8), (1023, 8), (1028, 8), (8192, 8), (8193, 8), (32772, 8), (65536, 3), (65537, 8), (262144, 8),
                                     (262149, 8), (524296, 5)])
def test_topb_edges(vocab, b):
    import torch
    from paper_2410_20488_b200 import firp_topb_static
    logits = np.ascontiguousarray(_rows(vocab, np.random.default_rng(vocab)))
    n = len(logits)
    d = torch.from_numpy(logits).cuda()
    ids, vals = torch.full((n, b), -1, dtype=torch.int32, device="cuda"), torch.zeros(n, b, device="cuda")
    firp_topb_static(d.data_ptr(), n, vocab, b, ids.data_ptr(), vals.data_ptr(), torch.cuda.current_stream().cuda_stream)
    got_ids, got_vals = ids.cpu().numpy(), vals.cpu().numpy()
    for r, row in enumerate(logits):
        order = np.lexsort((np.arange(vocab), -row))
        order = order[~np.isnan(row[order])][:b]
        m = len(order)
        assert np.array_equal(got_ids[r, :m], order), "row %d" % r
        assert np.array_equal(got_vals[r, :m].view(np.int32), row[order].view(np.int32)), "row %d" % r       # bit for bit, the sign of zeros too
        assert (got_ids[r, m:] == 0x7fffffff).all() and (got_vals[r, m:] == -np.inf).all(), "row %d" % r
