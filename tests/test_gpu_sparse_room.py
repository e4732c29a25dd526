"""Shots that outgrow the small instance of the CTA-per-shot LSD kernel, or change from many
growing clusters to one, thousands at a time so that every CTA meets them one after another: all
its threads have to take each turn at the same barrier, or the CTA's later shots are decoded
wrongly.  Every output is compared with the oracle's."""
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


def _columns(m, n, weight, seed):
    """n columns of the given weight, spread evenly over the rows (no row beyond 32 edges)."""
    rng = np.random.default_rng(seed)
    while True:
        h = np.zeros((m, n), np.uint8)
        for j in range(n):
            p = 1.0 / (1.0 + h.sum(1)) ** 4
            h[rng.choice(m, weight, replace=False, p=p / p.sum()), j] = 1
        if h.sum(1).max() <= 32:
            return h


def _compare(L, h, s, order, cs, seed, copies=20):
    """The shots of s, each `copies` times in one batch."""
    n, shots = h.shape[1], s.shape[0]
    llr = np.random.default_rng(seed).normal(1.5, 2.0, (shots, n)).astype(np.float32)
    probs = np.full(n, 0.05, np.float32)
    d = L.Decoder(h, probs, 5, order, osd_cs=cs, lsd_kernel=2)
    corr, status, info = (x.cpu().numpy().reshape((copies, shots) + x.shape[1:]) for x in d.postprocess(
        torch.from_numpy(llr).cuda().repeat(copies, 1), torch.from_numpy(s).cuda().repeat(copies, 1)))
    kw = {} if cs is None else {"osd_cs": cs}
    r = oracle.lsd(h, s, llr.astype(np.float64), order=order, probs=probs.astype(np.float64), **kw)
    assert (r["status"] == 2).all()
    assert (status == r["status"]).all()
    assert (corr == r["corrections"]).all()
    for k, key in enumerate(("nu", "kappa", "steps")):
        assert (info[..., k] == r[key]).all()


@pytest.mark.parametrize("order,cs", [(0, None), (3, 2)])
def test_list_of_a_single_cluster(L, order, cs):
    """One seed, columns of weight 3: its cluster lists more than 1536 faults before it is
    valid."""
    h = _columns(512, 2048, 3, 1)
    s = np.zeros((200, 512), np.uint8)
    s[np.arange(200), np.random.default_rng(2).integers(0, 512, 200)] = 1
    _compare(L, h, s, order, cs, 3)


def test_dependent_columns_of_a_single_cluster(L):
    """One seed and columns of even weight: no solution, and 1201 dependent columns on the way."""
    h = _columns(300, 1500, 4, 4)
    rng = np.random.default_rng(5)
    s = np.zeros((2000, 300), np.uint8)
    s[np.arange(2000), rng.integers(0, 300, 2000)] = 1
    llr = rng.normal(1.5, 2.0, (2000, 1500)).astype(np.float32)
    d = L.Decoder(h, np.full(1500, 0.05, np.float32), 5, 2, lsd_kernel=2)
    corr, status, info = d.postprocess(torch.from_numpy(llr).cuda(), torch.from_numpy(s).cuda())
    assert (status == 3).all() and not corr.any()
    # one cluster, which took every column before it found no candidate
    assert (info == torch.tensor([1, 1500, 1500], device="cuda", dtype=info.dtype)).all()


@pytest.mark.parametrize("order,cs", [(0, None), (3, 2)])
def test_list_of_many_clusters(L, order, cs):
    """30 seeds list some 350 faults, and more than 1536 after four steps of all of them."""
    h = _columns(512, 2048, 3, 1)
    rng = np.random.default_rng(7)
    s = np.zeros((200, 512), np.uint8)
    for row in s:
        row[rng.choice(512, 30, replace=False)] = 1
    _compare(L, h, s, order, cs, 8)


@pytest.mark.parametrize("rows", [8, 33])
def test_dependent_columns_of_many_clusters(L, rows):
    """A direct sum of blocks with a seed in each, grown until all its columns are in: 960 (of
    clusters that a warp takes) or 924 dependent columns (of clusters that the CTA takes)."""
    b = _columns(rows, 3 * rows, 3, 9)
    blocks = 480 // rows
    h = np.kron(np.eye(blocks, dtype=np.uint8), b)
    s = np.zeros((100, h.shape[0]), np.uint8)
    for k in range(blocks):
        s[np.arange(100), k * rows + np.random.default_rng(k).integers(0, rows, 100)] = 1
    _compare(L, h, s, 3 * rows, 4, 10)


@pytest.mark.parametrize("order,cs", [(0, None), (2, None)])
@pytest.mark.parametrize("name,p", [("bb72", 0.04), ("bb144", 0.04), ("rep_boundary", 0.15)])
def test_several_clusters_then_one(L, name, p, order, cs):
    """Small shots that go on with their last invalid cluster alone: the count of growing
    clusters is read by every thread before it is cleared."""
    h = code(name)
    e = I.sample_errors(13, 2000, np.full(h.shape[1], p))
    _compare(L, h, I.syndromes(h, e), order, cs, 14, copies=40)
