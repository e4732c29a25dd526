"""The training kernel's shapes on the GPU against the CPU oracle: sizes off the 16-row tiles
(the padding rows take part in the matrix products), fewer row tiles than warps, and the graph
staged in shared memory, staged up to the last kilobyte, or too large to be staged.

Tolerance: as for the kernel elsewhere, BF16 operands (unit roundoff 2^-9) and FP32 sums over
thousands of edges: 1e-2 of the gradient's L2 norm, cosine 0.9999, the loss within 1 %.
"""
import numpy as np
import pytest
import torch

import oracle.prior as P
from paper_2406_18655_gb300 import inputs as I
from tests.gpu_cases import code
from tests.test_gpu_prior import L, params_case  # noqa: F401  (L: fixture)

pytestmark = pytest.mark.gpu


def graph(name):
    if name == "irreg_37x61":
        return code(name)
    m, n, weight = {"near_limit": (96, 192, 4), "not_staged": (96, 192, 6), "tiny": (3, 5, 2)}[name]
    rng = np.random.default_rng(7)
    h = np.zeros((m, n), np.uint8)
    for j in range(n):
        h[rng.choice(m, weight, replace=False), j] = 1
    return h


@pytest.mark.parametrize("name", ["tiny", "irreg_37x61", "near_limit", "not_staged"])
@pytest.mark.parametrize("rounds", [1, 3])
def test_gradient_shapes(L, name, rounds):  # noqa: F811
    h = graph(name)
    probs = np.full(h.shape[1], 0.06, np.float32)
    shots = 200  # more than one shot for some of the blocks
    e = I.sample_errors(21, shots, probs.astype(np.float64))
    s = I.syndromes(h, e)
    theta = params_case(6).astype(np.float32).astype(np.float64)
    d = L.Decoder(h, probs, 10)
    pr = L.Prior(d, rounds=rounds, params=theta.astype(np.float32))
    loss, g = pr.gradient(torch.from_numpy(s).cuda(), torch.from_numpy(e).cuda())
    lam = np.log((1 - probs.astype(np.float64)) / probs.astype(np.float64))
    ref_loss, ref_g, _ = P.loss_and_grad(h, theta, s, e, lam, rounds=rounds)
    g = g.astype(np.float64)
    assert abs(loss - ref_loss) <= 0.01 * abs(ref_loss)
    assert np.linalg.norm(g - ref_g) <= 1e-2 * np.linalg.norm(ref_g)
    assert g @ ref_g >= 0.9999 * np.linalg.norm(g) * np.linalg.norm(ref_g)


def test_initial_state_gradients_in_one_order(L):  # noqa: F811
    """One pair is one block: the gradients of the initial states (the first 128 values) are sums
    in a fixed order, the same bits in every run."""
    h = code("bb144")
    probs = np.full(h.shape[1], 0.06, np.float32)
    e = I.sample_errors(22, 1, probs.astype(np.float64))
    s = torch.from_numpy(I.syndromes(h, e)).cuda()
    pr = L.Prior(L.Decoder(h, probs, 10), rounds=3, params=params_case(6).astype(np.float32))
    runs = {pr.gradient(s, torch.from_numpy(e).cuda())[1][:128].tobytes() for _ in range(200)}
    assert len(runs) == 1
