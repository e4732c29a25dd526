"""The CTA-per-shot LSD kernel where its layout has edges: against the dense kernel on small
matrices (columns of more than four detectors, tied LLRs, every reprocessing), and against the
oracle on a graph whose labels lie in global scratch and on shots that change instance."""
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


def _heavy_columns(m, n, top, seed):
    """Column j has weight 1 + j % top."""
    rng = np.random.default_rng(seed)
    h = np.zeros((m, n), np.uint8)
    for j in range(n):
        h[rng.choice(m, 1 + j % top, replace=False), j] = 1
    return h


def _llrs(shots, n, ties, seed):
    rng = np.random.default_rng(seed)
    x = rng.normal(1.5, 2.0, (shots, n)).astype(np.float32)
    return np.round(x) if ties else x  # rounded: many equal keys, +0 and -0 among them


@pytest.mark.parametrize("name", ["bb72", "bb144", "rep_boundary", "heavy4", "heavy5", "heavy9"])
@pytest.mark.parametrize("order,cs", [(0, None), (3, None), (6, None), (5, 0), (9, 4)])
@pytest.mark.parametrize("ties", [False, True])
def test_equals_dense_kernel(L, name, order, cs, ties):
    h = _heavy_columns(50, 90, int(name[5:]), 3) if name.startswith("heavy") else code(name)
    n, shots = h.shape[1], 400
    probs = np.full(n, 0.07, np.float32)
    s = torch.from_numpy(I.syndromes(h, I.sample_errors(11, shots, probs.astype(np.float64)))).cuda()
    llr = torch.from_numpy(_llrs(shots, n, ties, 5)).cuda()
    got, want = (L.Decoder(h, probs, 5, order, osd_cs=cs, lsd_kernel=k).postprocess(llr, s)
                 for k in (2, 1))
    for a, b in zip(got, want):
        assert torch.equal(a, b)


@pytest.mark.parametrize("name", ["bb72", "bb144", "bb288", "ldpc_96x192", "irreg_37x61"])
@pytest.mark.parametrize("kind", ["close", "infinite", "constant"])
def test_order_of_close_llrs(L, name, kind):
    """LLRs that a coarse key cannot tell apart (an outlier stretches their range, neighbours
    differ in the last bits, in falling order), infinities, and all equal."""
    h = code(name)
    n, shots = h.shape[1], 200
    probs = np.full(n, 0.06, np.float32)
    s = torch.from_numpy(I.syndromes(h, I.sample_errors(12, shots, probs.astype(np.float64)))).cuda()
    x = np.ones((shots, n), np.float32)
    if kind != "constant":
        steps = np.random.default_rng(6).integers(0, 40, (shots, n)) + 40 * (n - np.arange(n))
        x += (steps * 2.0 ** -23).astype(np.float32)
        x[:, 3] = 1e9 if kind == "close" else np.inf
        x[::2, 5] = -1e9 if kind == "close" else -np.inf
    llr = torch.from_numpy(x).cuda()
    got, want = (L.Decoder(h, probs, 5, 2, lsd_kernel=k).postprocess(llr, s) for k in (1, 2))
    for a, b in zip(got, want):
        assert torch.equal(a, b)


def test_syndromes_outside_the_image(L):
    """Unsolvable shots among solvable ones: the same statuses as the dense kernel."""
    h = code("rep_boundary")[1:]           # a chain without boundary and an isolated row
    h = np.concatenate([h, np.zeros((1, h.shape[1]), np.uint8)])
    rng = np.random.default_rng(1)
    s = torch.from_numpy((rng.random((300, h.shape[0])) < 0.2).astype(np.uint8)).cuda()
    llr = torch.from_numpy(_llrs(300, h.shape[1], False, 2)).cuda()
    probs = np.full(h.shape[1], 0.1, np.float32)
    got, want = (L.Decoder(h, probs, 5, lsd_kernel=k).postprocess(llr, s) for k in (2, 1))
    assert set(want[1].cpu().numpy()) == {2, 3}
    for a, b in zip(got[:2], want[:2]):
        assert torch.equal(a, b)


@pytest.mark.parametrize("order", [0, 4])
def test_many_empty_rows(L, order):
    """BB144 spread over 34 000 rows (more labels than shared memory holds) decodes as BB144."""
    h = code("bb144")
    at = np.arange(72) * 472 + 5
    wide = np.zeros((34000, 144), np.uint8)
    wide[at] = h
    probs = np.full(144, 0.06, np.float32)
    s = I.syndromes(h, I.sample_errors(3, 200, probs.astype(np.float64)))
    sw = np.zeros((200, 34000), np.uint8)
    sw[:, at] = s
    llr = torch.from_numpy(_llrs(200, 144, False, 4)).cuda()
    got = L.Decoder(wide, probs, 5, order).postprocess(llr, torch.from_numpy(sw).cuda())
    want = L.Decoder(h, probs, 5, order).postprocess(llr, torch.from_numpy(s).cuda())
    for a, b in zip(got, want):
        assert torch.equal(a, b)


@pytest.mark.parametrize("base,p,order,cs,shots", [
    (66, 0.035, 0, None, 4), (66, 0.02, 2, 4, 3),       # 5808 x 12100: labels in global scratch
    (48, 0.05, 0, None, 4), (48, 0.02, 4, None, 3),     # 3072 x 6400: the large instance
    (48, 0.012, 0, None, 6)])                           # ... and the small one
def test_large_graphs_against_oracle(L, base, p, order, cs, shots):
    h = I.hgp(I.random_regular_ldpc(base, base // 3 * 4, 3, 4, seed=7 + base))[0]
    n = h.shape[1]
    probs = np.full(n, p, np.float32)
    s = I.syndromes(h, I.sample_errors(19, shots, probs.astype(np.float64)))
    d = L.Decoder(h, probs, 6, order, osd_cs=cs)
    llr, _, _ = d.bp(torch.from_numpy(s).cuda())
    corr, st, info = d.postprocess(llr, torch.from_numpy(s).cuda())
    kw = {} if cs is None else {"osd_cs": cs}
    r = oracle.lsd(h, s, llr.cpu().numpy().astype(np.float64), order=order,
                   probs=probs.astype(np.float64), **kw)
    assert np.array_equal(st.cpu().numpy(), r["status"])
    assert np.array_equal(corr.cpu().numpy(), r["corrections"])
    got = info.cpu().numpy()
    for k, key in enumerate(("nu", "kappa", "steps")):
        assert np.array_equal(got[:, k], r[key])


@pytest.mark.parametrize("order", [0, 6])
def test_autotune_times_both_kernels(L, order):
    """A matrix that both kernels take: the report has the dense kernel's shapes and the sparse
    kernel, and the decoder's results stay, whichever it kept."""
    h = code("st_bb72_d6")
    probs = np.full(h.shape[1], 0.02, np.float32)
    s = torch.from_numpy(I.syndromes(h, I.sample_errors(4, 3000, probs.astype(np.float64)))).cuda()
    d = L.Decoder(h, probs, 10, order)
    want = d.decode(s)
    rep = d.autotune(s)
    dense = L.Decoder(h, probs, 10, order, lsd_kernel=1).autotune(s)
    assert rep["lsd_candidates"] == 1 + dense["lsd_candidates"]
    assert 0 < rep["ms_lsd_best"] <= rep["ms_lsd_first"]
    for a, b in zip(d.decode(s), want):
        assert torch.equal(a, b)
