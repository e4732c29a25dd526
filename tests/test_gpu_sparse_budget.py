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


@pytest.mark.parametrize("order", [0, 6])
@pytest.mark.parametrize("host", [False, True])
def test_budget_of_the_dense_kernel_is_enough(L, order, host):
    """A matrix that both kernels take decodes within what the dense kernel alone needs, from the
    first call, and when a larger batch finds the scratch of earlier small ones in its way."""
    probs, s = _case(code("st_bb72_d6"), 0.02, 20000, 2)
    h = code("st_bb72_d6")

    def call(d, k):
        out = d.decode_host(s[:k].cpu()) if host else d.decode(s[:k])
        return [torch.as_tensor(x).cpu() for x in out[:2]]

    ref = L.Decoder(h, probs, 10, order, lsd_kernel=1)
    want = call(ref, 20000)
    assert (want[1] == 2).sum() > 1000
    first = L.Decoder(h, probs, 10, order, mem_budget=ref.workspace_bytes())
    later = L.Decoder(h, probs, 10, order, mem_budget=ref.workspace_bytes())
    for a, b in zip(call(later, 50), want):
        assert torch.equal(a, b[:50])
    for d in (first, later):
        for _ in range(2):
            for a, b in zip(call(d, 20000), want):
                assert torch.equal(a, b)
        assert d.workspace_bytes() <= ref.workspace_bytes()


def test_belief_propagation_within_the_graphs_own_size(L):
    """A large matrix under a budget that the tables of its LSD pass: BP runs, LSD is refused."""
    h = code("st_bb144_d12")
    m, n = h.shape
    probs, s = _case(h, 0.003, 200, 3)
    d = L.Decoder(h, probs, 10)
    tables = 2 * ((m * int(h.sum(1).max()) + 3) // 4 * 4 + 4 * n)
    tight = L.Decoder(h, probs, 10, mem_budget=d.workspace_bytes() - tables)
    for a, b in zip(tight.bp(s), d.bp(s)):
        assert torch.equal(a, b)
    with pytest.raises(L.LsdError) as err:
        tight.postprocess(torch.ones((200, n), device="cuda"), s)
    assert err.value.code == L.LSD_ERR_ADMISSION
