"""The register BP kernels against the generic kernel (itself pinned to the oracle elsewhere):
bit-identical posteriors, iteration counts and convergence where the layouts have their edges
(batch sizes around the number of groups, idle lanes, padded rows, long growing messages)."""
import numpy as np
import pytest
import torch

from tests.gpu_cases import code
from paper_2406_18655_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_2406_18655_gb300 import build, lsd
    build.build()
    lsd.lib()
    return lsd


def _matrix(name):
    if name == "hooks_bb72_d6":
        return I.space_time_hooks(code("bb72"), 6, seed=6)[0]
    if name == "hooks_bb144_d6":
        return I.space_time_hooks(code("bb144"), 6, seed=6)[0]
    if name == "bb60":  # l = 5, m = 6: 30 checks and 60 variables, idle lanes in every slot
        return I.bb_code(5, 6, [("x", 3), ("y", 1), ("y", 2)], [("y", 3), ("x", 1), ("x", 2)])[0]
    return code(name)


def _compare(L, h, p, shots, iters, kernel, seed, **kw):
    probs = np.full(h.shape[1], p, np.float32)
    e = I.sample_errors(seed, shots, probs.astype(np.float64))
    s = torch.from_numpy(I.syndromes(h, e)).cuda()
    got = L.Decoder(h, probs, iters, bp_kernel=kernel, **kw).bp(s)
    ref = L.Decoder(h, probs, iters, bp_kernel=1, **kw).bp(s)
    for a, b in zip(got, ref):  # bit patterns, so that -0 and 0 differ
        a, b = a.cpu().numpy(), b.cpu().numpy()
        assert np.array_equal(a.view(np.uint8), b.view(np.uint8))


@pytest.mark.parametrize("name", ["bb60", "bb72", "bb144", "bb288"])
@pytest.mark.parametrize("shots", [1, 3, 3647, 3649, 9001])
def test_warp_group_kernel_batch_sizes(L, name, shots):
    """3648 = 152 SMs x 3 CTAs x 8 groups: one group more or less than a batch has shots."""
    _compare(L, _matrix(name), 0.06, shots, 20, 2, seed=shots)


@pytest.mark.parametrize("name", ["st_bb72_d6", "st_bb144_d12", "st_bb288_d18", "hgp",
                                  "hooks_bb72_d6", "hooks_bb144_d6"])
@pytest.mark.parametrize("kernel,shots", [(2, 1), (2, 153), (2, 1301), (3, 1), (3, 777)])
def test_cta_kernel_batch_sizes(L, name, kernel, shots):
    """Fewer shots than CTAs, one more than a CTA per SM, and enough that shots are taken ahead
    and then one at a time."""
    _compare(L, _matrix(name), 0.004 if name != "hgp" else 0.03, shots, 12, kernel, seed=shots)


@pytest.mark.parametrize("name", ["bb144", "st_bb72_d6", "hooks_bb72_d6", "rep_boundary", "hgp"])
@pytest.mark.parametrize("alpha,early", [(1.0, False), (3.0, False), (1.0, True)])
def test_messages_that_outgrow_the_empty_minimum(L, name, alpha, early):
    """300 iterations of unscaled (or amplified) min-sum on hard syndromes: message magnitudes
    pass 2^100, where every minimum starts, and have to be clamped as by the generic kernel."""
    h = _matrix(name)
    _compare(L, h, 0.12, 60, 300, 2, seed=9, ms_scaling=alpha, no_early_exit=not early)


@pytest.mark.parametrize("name", ["st_bb72_d3", "st_bb72_d8", "st_bb144_d2", "st_bb144_d10", "st_bb288_d15",
                                  "hooks_bb72_d3", "hooks_bb144_d4", "ldpc_512", "ldpc_600", "ldpc_1100",
                                  "hgp_24", "hgp_30"])
@pytest.mark.parametrize("kernel", [2, 3])
def test_graphs_that_leave_slots_idle(L, name, kernel):
    """Graphs well below the bounds of their shape, whose idle slots are left out."""
    if name.startswith("st_"):
        _, c, d = name.split("_")
        h = I.space_time(code(c), int(d[1:]))
    elif name.startswith("hooks"):
        _, c, d = name.split("_")
        h = I.space_time_hooks(code(c), int(d[1:]), seed=6)[0]
    elif name.startswith("ldpc"):
        m = int(name[5:])
        h = I.random_regular_ldpc(m, 2 * m, 3, 6, seed=3)
    else:
        b = int(name[4:])
        h = I.hgp(I.random_regular_ldpc(b, b // 3 * 4, 3, 4, seed=7 + b))[0]
    _compare(L, h, 0.01, 401, 12, kernel, seed=5)
