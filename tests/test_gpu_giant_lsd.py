"""P-LSD of the giant shot in one launch, against the oracle where its ways part: more changed
clusters than warps (a lane each), few clusters (one block, candidates from the clusters' side),
the step between the two, and clusters beyond 1024 detectors (eight words per lane)."""
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


@pytest.mark.parametrize("name,p,copies,order", [
    ("bb72", 0.08, 12000, 0), ("bb72", 0.08, 3000, 0), ("bb72", 0.08, 20, 0), ("bb72", 0.08, 2, 0), ("bb72", 0.06, 900, 3),
    ("irreg_37x61", 0.1, 2500, 0), ("ldpc_96x192", 0.06, 400, 0)])
def test_direct_sum(L, name, p, copies, order):
    """A direct sum of blocks with a shot of the batch in each: clusters never leave their block,
    so the blocks' results are the oracle's, the largest kappa and the most steps of any block."""
    h = code(name)
    mb, nb = h.shape
    probs = np.full(nb, p, np.float32)
    e = I.sample_errors(29, copies, probs.astype(np.float64))
    s = I.syndromes(h, e)
    g = I.Xoshiro256ss(31, np.arange(copies * nb, dtype=np.uint64))
    llr = np.round(g.uniform() * 5 - 0.5, 1).astype(np.float32).reshape(copies, nb)  # (ties)
    r = oracle.lsd(h, s, llr.astype(np.float64), order=order, probs=probs.astype(np.float64))
    rb, cb = np.nonzero(h)
    k = np.arange(copies)[:, None]
    rows, cols = (rb + mb * k).ravel(), (cb + nb * k).ravel()
    gd = L.GiantDecoder(mb * copies, nb * copies, rows, cols, np.tile(probs, copies), 10, order)
    corr, info = gd.postprocess(torch.from_numpy(llr.ravel()).cuda(),
                                torch.from_numpy(s.ravel()).cuda())
    assert info["status"] == 2 and (r["status"] == 2).all()
    assert np.array_equal(corr.cpu().numpy().reshape(copies, nb), r["corrections"])
    assert info["nu"] == r["nu"].sum()
    assert (info["kappa"], info["steps"]) == (r["kappa"].max(), r["steps"].max())


def test_cluster_beyond_1024_detectors(L):
    """One seed at the end of a chain whose only other end is 1400 faults away."""
    n = 1400
    h = np.zeros((n, n), np.uint8)
    h[np.arange(n), np.arange(n)] = 1
    h[np.arange(1, n), np.arange(n - 1)] = 1
    probs = np.full(n, 0.1, np.float32)
    s = np.zeros((1, n), np.uint8)
    s[0, 0] = 1
    llr = np.round(np.random.default_rng(2).random((1, n)) * 4, 1).astype(np.float32)
    r = oracle.lsd(h, s, llr.astype(np.float64), order=0, probs=probs.astype(np.float64))
    gd = L.GiantDecoder.from_dense(h, probs, 10)
    corr, info = gd.postprocess(torch.from_numpy(llr[0]).cuda(), torch.from_numpy(s[0]).cuda())
    assert info["status"] == r["status"][0] == 2
    assert np.array_equal(corr.cpu().numpy(), r["corrections"][0])
    assert (info["nu"], info["kappa"], info["steps"]) == (r["nu"][0], r["kappa"][0], r["steps"][0])


def _chain(L, n, blocks):
    """`blocks` chains of n faults, a seed at the end of the first: n growth steps of one cluster,
    by one block while the others wait."""
    i = np.arange(n * blocks)
    j = i[i % n != n - 1]
    rows, cols = np.concatenate([i, j + 1]), np.concatenate([i, j])
    gd = L.GiantDecoder(n * blocks, n * blocks, rows, cols, np.full(n * blocks, 0.1, np.float32), 5)
    s = torch.zeros(n * blocks, dtype=torch.uint8, device="cuda")
    s[0] = 1
    return gd, torch.ones(n * blocks, device="cuda"), s


def test_bound_starts_again_with_every_step(L):
    """The blocks that wait out the last clusters' steps wait for longer than their bound in all,
    but not for any one step."""
    gd, llr, s = _chain(L, 1400, 8)
    gd.postprocess(llr, s)  # (the first call also loads the kernel)
    want, info = gd.postprocess(llr, s)
    assert info["status"] == 2 and info["steps"] == 1400 and int(want.sum()) == 1400
    limit = int(info["ms_lsd"] * 1e6 / 4)   # a step takes 1/1400 of it
    gd.test_lsd_bound(limit_ns=limit)
    got, again = gd.postprocess(llr, s)
    assert again["ms_lsd"] * 1e6 > 2 * limit
    assert again["status"] == 2 and torch.equal(got, want)


def test_lsd_timeout_leaves_the_device_usable(L):
    """A P-LSD barrier whose wait runs out (block 0 withholds its first arrival) makes the call
    return LSD_ERR_TIMEOUT; the next call, with the hold lifted, decodes."""
    gd, llr, s = _chain(L, 40, 100)
    gd.test_lsd_bound(True, limit_ns=20_000_000)
    with pytest.raises(L.LsdError) as err:
        gd.postprocess(llr, s)
    assert err.value.code == L.LSD_ERR_TIMEOUT
    gd.test_lsd_bound()
    corr, info = gd.postprocess(llr, s)
    assert info["status"] == 2 and int(corr.sum()) == 40
