"""The giant-shot BP launch that keeps its tables on chip, against the oracle where its split has
edges: fewer variables than threads, one more than a block's threads, rows shorter than the
widest, columns of degree 1 to 4, a check of degree 1, no iteration and one iteration."""
import numpy as np
import pytest
import torch

import oracle
from paper_2406_18655_gb300 import inputs as I
from tests.gpu_cases import code

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_2406_18655_gb300 import build, lsd
    build.build()
    lsd.lib()
    return lsd


def _chain(n):
    h = np.zeros((n, n), np.uint8)
    h[np.arange(n), np.arange(n)] = 1
    h[np.arange(1, n), np.arange(n - 1)] = 1
    return h


@pytest.mark.parametrize("name", ["chain_5", "chain_129", "chain_3000", "irreg_37x61", "st_bb144_d12", "hgp"])
@pytest.mark.parametrize("iters", [0, 1, 2, 17])
def test_posteriors_and_decisions(L, name, iters):
    h = _chain(int(name[6:])) if name.startswith("chain") else code(name)
    p = 0.02 if h.shape[1] > 1000 else 0.1
    probs = (p * (0.5 + np.random.default_rng(1).random(h.shape[1]))).astype(np.float32)
    e = I.sample_errors(23, 5, probs.astype(np.float64))
    s = I.syndromes(h, e)
    gd = L.GiantDecoder.from_dense(h, probs, iters)
    llr, hard, used, conv = oracle.bp(h, probs.astype(np.float64), s, iters, precision=1)
    post = torch.empty(h.shape[1], dtype=torch.float32, device="cuda")
    for k in range(s.shape[0]):
        corr, info = gd.decode(torch.from_numpy(s[k]).cuda(), posteriors=post)
        assert np.array_equal(post.cpu().numpy(), llr[k].astype(np.float32))
        assert info["bp_iterations"] == used[k]
        assert (info["status"] == 1) == bool(conv[k])
