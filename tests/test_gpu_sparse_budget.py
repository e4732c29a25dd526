"""The CTA-per-shot LSD kernel's device memory under a budget: what it holds after a call that found
no room, and the calls that are accepted all the same."""
import numpy as np
import pytest
import torch

from paper_2406_18655_gb300 import inputs as I
from tests.gpu_cases import code

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_2406_18655_gb300 import build, lsd
    build.build()
    lsd.lib()
    return lsd


def _case(h, p, shots, seed):
    probs = np.full(h.shape[1], p, np.float32)
    e = I.sample_errors(seed, shots, probs.astype(np.float64))
    return probs, torch.from_numpy(I.syndromes(h, e)).cuda()


def test_retries_hold_no_more(L):
    """A budget with room for the small instance's scratch alone: refused each time, and the second
    and third time hold what the first did."""
    h = np.zeros((34000, 144), np.uint8)  # (labels in global scratch: the small instance has some)
    h[np.arange(72) * 472 + 5] = code("bb144")
    probs, s = _case(h, 0.05, 64, 1)
    llr = torch.ones((64, 144), device="cuda")
    free = L.Decoder(h, probs, 5, 4)
    start = free.workspace_bytes()
    free.postprocess(llr, s)
    full = free.workspace_bytes()  # the last of it: the queue of the shots that change instance
    d = L.Decoder(h, probs, 5, 4, mem_budget=full - 64 * 4 - 1)
    assert d.workspace_bytes() == start
    held = []
    for _ in range(3):
        with pytest.raises(L.LsdError) as err:
            d.postprocess(llr, s)
        assert err.value.code == L.LSD_ERR_ADMISSION
        held.append(d.workspace_bytes())
    assert held[0] == held[1] == held[2] < full
