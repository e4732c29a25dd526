"""The calls that the decoder's speed is judged by: what users of this library have it do.

``listed()`` gives the fixed cases, ``draw(rng)`` one more of the same ranges, and for either
``prepare`` makes what a program holds before the call, ``run`` makes the call, ``work`` says
what the call cannot do without and ``exact`` what it returns in 64 bits.

Codes, noise strengths, iteration counts and orders are those of the benchmark and the tests:
bivariate bicycle (BB) codes, the hypergraph product (HGP) of a (3,4)-regular matrix, their
space-time matrices with and without hook faults, the learned prior, and one giant HGP shot.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2406_18655_gb300 import inputs as I
from paper_2406_18655_gb300 import learned
from paper_2406_18655_gb300.lsd import Decoder, GiantDecoder, Prior, WindowDecoder, pack_bits

HID = 32


def listed():
    return [
        # One small batch of a real-time decoder: 16 logical blocks hand in their space-time
        # syndromes at once.  Latency and launches count.
        {"name": "space_time_bb72_16", "kind": "decode", "code": "bb72", "rounds": 6, "p": 0.003,
         "iters": 30, "order": 0, "sweep": -1, "io": "bytes", "shots": 16},
        # The benchmark's headline: 10^6 code-capacity shots of BB [[144,12,12]] on the device.
        {"name": "bb144_million", "kind": "decode", "code": "bb144", "rounds": 0, "p": 0.05,
         "iters": 50, "order": 0, "sweep": -1, "io": "bytes", "shots": 1000000},
        # The same from bit-packed page-locked host memory and back: a simulation on the host.
        {"name": "bb144_million_host", "kind": "decode", "code": "bb144", "rounds": 0, "p": 0.05,
         "iters": 50, "order": 0, "sweep": -1, "io": "host", "shots": 1000000},
        # The BB experiment of LSD-mu: mu = 0.1 n growth steps, then OSD-CS-4 in each cluster.
        {"name": "bb144_mu14_cs4", "kind": "decode", "code": "bb144", "rounds": 0, "p": 0.06,
         "iters": 50, "order": 14, "sweep": 4, "io": "packed", "shots": 100003},
        # A large code below its threshold, with LSD-10 (OSD-E): BP carries the work.
        {"name": "hgp_p002_mu10", "kind": "decode", "code": "hgp", "rounds": 0, "p": 0.02,
         "iters": 100, "order": 10, "sweep": -1, "io": "bytes", "shots": 50000},
        # The same code where its clusters percolate: long eliminations carry the work.
        {"name": "hgp_p005", "kind": "decode", "code": "hgp", "rounds": 0, "p": 0.05,
         "iters": 100, "order": 0, "sweep": -1, "io": "bytes", "shots": 5000},
        # A memory experiment decoded as a whole: 18 noisy rounds of BB [[288,12,18]].
        {"name": "space_time_bb288", "kind": "decode", "code": "bb288", "rounds": 18, "p": 0.003,
         "iters": 30, "order": 0, "sweep": -1, "io": "bytes", "shots": 20000},
        # Circuit-like noise: hook faults in mid-round, rows of unequal degree, unequal priors.
        {"name": "hooks_bb144", "kind": "decode", "code": "bb144_hooks", "rounds": 6, "p": 0.004,
         "iters": 50, "order": 0, "sweep": -1, "io": "bytes", "shots": 99991},
        # The memory experiment in (3, 1) overlapping windows.
        {"name": "windows_bb144", "kind": "windows", "code": "bb144", "rounds": 12, "window": 3,
         "commit": 1, "p": 0.003, "iters": 30, "shots": 50000},
        # Inference of the learned prior on a large batch.
        {"name": "prior_forward_bb144", "kind": "prior_forward", "code": "bb144", "layers": 4,
         "p": 0.05, "shots": 200000},
        # One batch of its training: loss and gradient.
        {"name": "prior_gradient_bb144", "kind": "prior_gradient", "code": "bb144", "layers": 4,
         "p": 0.05, "shots": 4096},
        # One shot of a code with 640 000 faults, the whole GPU on it.
        {"name": "giant_640k", "kind": "giant", "base_rows": 480, "p": 0.03, "iters": 100},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["bb", "bb", "cs", "hgp", "space_time", "space_time", "hooks", "windows",
                       "prior_forward", "prior_gradient", "giant"])
    if kind == "bb":
        code = rng.choice(["bb72", "bb144", "bb288"])
        order = rng.choice([0, 0, 6])
        top = 1000000 if code != "bb288" and order == 0 else 100000
        return {"kind": "decode", "code": code, "rounds": 0, "p": round(rng.uniform(0.01, 0.08), 4),
                "iters": rng.choice([10, 30, 50]), "order": order, "sweep": -1,
                "io": rng.choice(["bytes", "packed", "host"]), "shots": _log_int(rng, 16, top)}
    if kind == "cs":
        return {"kind": "decode", "code": rng.choice(["bb72", "bb144"]), "rounds": 0,
                "p": round(rng.uniform(0.03, 0.07), 4), "iters": 50, "order": rng.randint(1, 29),
                "sweep": rng.choice([0, 2, 4]), "io": rng.choice(["bytes", "packed"]),
                "shots": _log_int(rng, 100, 100003)}
    if kind == "hgp":
        p = round(rng.uniform(0.01, 0.05), 4)
        return {"kind": "decode", "code": "hgp", "rounds": 0, "p": p, "iters": 100,
                "order": 0 if p > 0.025 else rng.choice([0, 10]), "sweep": -1,
                "io": rng.choice(["bytes", "packed"]),
                "shots": _log_int(rng, 16, 50000 if p <= 0.025 else 3000)}
    if kind == "space_time":
        code, rounds, top = rng.choice([("bb72", 6, 200000), ("bb144", 12, 100000),
                                        ("bb288", 18, 20000)])
        return {"kind": "decode", "code": code, "rounds": rng.randint(rounds // 2, rounds),
                "p": round(rng.uniform(0.001, 0.004), 5), "iters": 30, "order": 0, "sweep": -1,
                "io": rng.choice(["bytes", "packed", "host"]), "shots": _log_int(rng, 1, top)}
    if kind == "hooks":
        return {"kind": "decode", "code": rng.choice(["bb72_hooks", "bb144_hooks"]),
                "rounds": rng.randint(2, 6), "p": round(rng.uniform(0.002, 0.006), 5), "iters": 50,
                "order": 0, "sweep": -1, "io": "bytes", "shots": _log_int(rng, 16, 100000)}
    if kind == "windows":
        w = rng.randint(2, 4)
        return {"kind": "windows", "code": rng.choice(["bb72", "bb144"]),
                "rounds": rng.randint(4, 12), "window": w, "commit": rng.randint(1, w - 1),
                "p": round(rng.uniform(0.001, 0.004), 5), "iters": 30,
                "shots": _log_int(rng, 16, 50000)}
    if kind == "prior_forward":
        return {"kind": kind, "code": rng.choice(["bb72", "bb144", "bb288"]),
                "layers": rng.randint(2, 4), "p": round(rng.uniform(0.02, 0.08), 4),
                "shots": _log_int(rng, 16, 100000)}
    if kind == "prior_gradient":
        return {"kind": kind, "code": rng.choice(["bb72", "bb144"]), "layers": rng.randint(2, 4),
                "p": round(rng.uniform(0.02, 0.08), 4), "shots": _log_int(rng, 64, 4096)}
    return {"kind": "giant", "base_rows": 3 * rng.randint(32, 160),
            "p": round(rng.uniform(0.01, 0.03), 4), "iters": 100}


# ---- codes and samples -----------------------------------------------------------------

@functools.lru_cache(maxsize=None)
def _base(code):
    return {"bb72": I.bb72, "bb144": I.bb144, "bb288": I.bb288, "hgp": I.hgp_48x64}[code]()[0]


@functools.lru_cache(maxsize=8)
def _matrix(code, rounds, p):
    """Check matrix and fault probabilities of a decode case."""
    if code.endswith("_hooks"):
        base = _base(code[:-6])
        h, _ = I.space_time_hooks(base, rounds, seed=rounds + 1)
        probs = I.space_time_hooks_probs(base.shape[1], base.shape[0], rounds, p, seed=rounds + 1)
    elif rounds:
        base = _base(code)
        h = I.space_time(base, rounds)
        probs = I.space_time_probs(base.shape[1], base.shape[0], rounds, p, p)
    else:
        h = _base(code)
        probs = np.full(h.shape[1], p)
    return h, probs.astype(np.float32)


@functools.lru_cache(maxsize=4)
def _giant_matrix(base_rows):
    base = I.random_regular_ldpc(base_rows, base_rows // 3 * 4, 3, 4, seed=2406 + base_rows)
    return I.hgp_coo(base)


def _sample(h, probs, shots, seed):
    """Errors [shots][n] and syndromes [shots][m] (uint8, on the GPU) of the seed alone."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    p = torch.from_numpy(np.asarray(probs, np.float32)).cuda()
    ht = torch.from_numpy(h.T.astype(np.float32)).cuda().half()     # counts are small integers
    m, n = h.shape
    e = torch.empty((shots, n), dtype=torch.uint8, device="cuda")
    s = torch.empty((shots, m), dtype=torch.uint8, device="cuda")
    step = max(1, (1 << 27) // n)
    for a in range(0, shots, step):
        k = min(step, shots - a)
        part = torch.rand((k, n), generator=gen, device="cuda") < p
        e[a:a + k] = part
        s[a:a + k] = ((part.half() @ ht).to(torch.int32) & 1).to(torch.uint8)
    return e, s


def _params():
    """Weights of the learned prior: the library's initialisation and a drawn output layer."""
    theta = learned.init_params(5)
    theta[-33:] = np.random.default_rng(5).normal(0.0, 0.3, 33)
    return theta


# ---- prepare, run ----------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind == "decode":
        h, probs = _matrix(case["code"], case["rounds"], case["p"])
        dec = Decoder(h, probs, case["iters"], case["order"],
                      osd_cs=None if case["sweep"] < 0 else case["sweep"])
        shots = case["shots"]
        _, s = _sample(h, probs, shots, seed)
        if case["io"] == "bytes":
            return {"call": dec.decode, "args": (s,)}
        words = torch.from_numpy(pack_bits(s.cpu().numpy()).view(np.int32))
        if case["io"] == "packed":
            return {"call": dec.decode_packed, "args": (words.cuda(),)}
        out = torch.empty((shots, (h.shape[1] + 31) // 32), dtype=torch.int32).pin_memory()
        status = torch.empty(shots, dtype=torch.uint8).pin_memory()
        return {"call": dec.decode_host_packed, "args": (words.pin_memory(), out, status)}
    if kind == "windows":
        h = _base(case["code"])
        full, probs = _matrix(case["code"], case["rounds"], case["p"])
        win = WindowDecoder(h, case["p"], case["p"], case["rounds"], case["window"],
                            case["commit"], case["iters"])
        _, s = _sample(full, probs, case["shots"], seed)
        return {"call": win.decode, "args": (s,)}
    if kind == "giant":
        m, n, rows, cols = _giant_matrix(case["base_rows"])
        dec = GiantDecoder(m, n, rows, cols, np.float32(case["p"]), case["iters"])
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed)
        e = torch.rand(n, generator=gen, device="cuda") < case["p"]
        hits = torch.from_numpy(rows).cuda().long()[e[torch.from_numpy(cols).cuda().long()]]
        s = (torch.bincount(hits, minlength=m) & 1).to(torch.uint8)
        return {"call": functools.partial(_giant, dec), "args": (s,)}
    h, probs = _matrix(case["code"], 0, case["p"])
    prior = Prior(Decoder(h, probs, 50), rounds=case["layers"], params=_params())
    e, s = _sample(h, probs, case["shots"], seed)
    if kind == "prior_forward":
        return {"call": prior.forward, "args": (s,)}
    return {"call": prior.gradient, "args": (s, e)}


def _giant(dec, s):
    correction, info = dec.decode(s)
    return correction, [info[k] for k in ("status", "bp_iterations", "nu", "kappa", "steps")]


def run(state):
    return state["call"](*state["args"])


# ---- work ------------------------------------------------------------------------------

# Mean BP iterations of a shot by code and noise strength (limit 50; HGP 100, rounds 30), a
# property of the min-sum schedule and not of its implementation; the nearest entry is taken.
_ITERATIONS = {
    "bb72": [(0.01, 1.1), (0.02, 1.9), (0.03, 3.5), (0.04, 6.1), (0.05, 9.7), (0.06, 14), (0.08, 23)],
    "bb144": [(0.01, 1.2), (0.02, 1.8), (0.03, 3.3), (0.04, 6.2), (0.05, 10.8), (0.06, 17), (0.08, 31)],
    "bb288": [(0.01, 1.3), (0.02, 2.5), (0.03, 4.6), (0.04, 8.0), (0.05, 13), (0.06, 21), (0.08, 38)],
    "hgp": [(0.01, 2.8), (0.02, 6.4), (0.03, 13), (0.04, 24), (0.05, 45)],
    "bb72_hooks": [(0.002, 1.3), (0.004, 2.2), (0.006, 3.6)],
    "bb144_hooks": [(0.002, 1.6), (0.004, 3.2), (0.006, 5.5)],
    "bb72_rounds": [(0.001, 1.0), (0.002, 1.1), (0.003, 1.2), (0.004, 1.2)],
    "bb144_rounds": [(0.001, 1.1), (0.002, 1.2), (0.003, 1.5), (0.004, 1.8)],
    "bb288_rounds": [(0.001, 1.2), (0.002, 1.6), (0.003, 2.0), (0.004, 2.5)],
    "giant": [(0.01, 7.0), (0.02, 100.0), (0.03, 100.0)],
}


def _iterations(key, p):
    return min(_ITERATIONS[key], key=lambda entry: abs(math.log(entry[0] / p)))[1]


def work(case):
    """Inputs read once and outputs written once; ten operations for each edge and iteration
    of BP (two minima, signs, scaling, the two sums), or the learned prior's products."""
    kind = case["kind"]
    if kind == "giant":
        m, n, rows, _ = _giant_matrix(case["base_rows"])
        return {"bytes": m + n, "flops": 10 * rows.size * _iterations("giant", case["p"])}
    shots = case["shots"]
    if kind in ("decode", "windows"):
        h, _ = _matrix(case["code"], case["rounds"], case["p"])
        m, n = h.shape
        if kind == "decode" and case["io"] != "bytes":
            m, n = 4 * ((m + 31) // 32), 4 * ((n + 31) // 32)
        key = case["code"]
        if case["rounds"] and not key.endswith("_hooks"):
            key += "_rounds"
        iters = min(case["iters"], _iterations(key, case["p"]))
        return {"bytes": shots * (m + n + 1), "flops": 10 * int(h.sum()) * iters * shots}
    h = _base(case["code"])
    m, n = h.shape
    # a round: two 32 x 32 products and the two projections of the new state for every fault
    # and every check, and a sum of 32 rectified features over each edge in both directions
    forward = shots * case["layers"] * (2 * 3 * HID * HID * (m + n) + 2 * 3 * HID * int(h.sum()))
    params = 4 * 6497
    if kind == "prior_forward":
        return {"bytes": shots * (m + 4 * n) + params, "flops": forward}
    return {"bytes": shots * (m + n) + 2 * params, "flops": 3 * forward}


# ---- 64-bit results --------------------------------------------------------------------

def exact(case, seed):
    """The learned prior in 64 bits; decodings are whole bits and have no rounded value."""
    kind = case["kind"]
    if kind not in ("prior_forward", "prior_gradient"):
        return None
    h, probs = _matrix(case["code"], 0, case["p"])
    e, s = _sample(h, probs, case["shots"], seed)
    theta = torch.from_numpy(_params().astype(np.float64)).cuda()
    lam = torch.log((1.0 - torch.from_numpy(probs.astype(np.float64)))
                    / torch.from_numpy(probs.astype(np.float64))).cuda()
    chk, var = (torch.from_numpy(a).cuda() for a in np.nonzero(h))
    step = max(1, (1 << 25) // (chk.numel() * HID))
    if kind == "prior_forward":
        out = torch.empty((case["shots"], h.shape[1]), dtype=torch.float64, device="cuda")
        with torch.no_grad():
            for a in range(0, case["shots"], step):
                out[a:a + step] = _prior64(theta, s[a:a + step], lam, chk, var, case["layers"])
        return out
    theta.requires_grad_(True)
    loss = 0.0
    for a in range(0, case["shots"], step):
        llr = _prior64(theta, s[a:a + step], lam, chk, var, case["layers"])
        part = (torch.nn.functional.softplus(llr)
                - (1.0 - e[a:a + step].double()) * llr).sum() / e.numel()
        part.backward()
        loss += part.item()
    return loss, theta.grad.cpu().numpy()


def _prior64(theta, s, lam, chk, var, layers):
    part, at = {}, 0
    for name, shape in learned.PARAM_SHAPES:
        size = int(np.prod(shape))
        part[name] = theta[at:at + size].reshape(shape)
        at += size
    sigma = (1.0 - 2.0 * (s != 0).double())[..., None]
    hv = torch.relu(lam[:, None] * part["a0"] + part["a1"]).expand(s.shape[0], -1, -1)
    hc = sigma * part["u0"] + part["u1"]

    def messages(w1, b1, w2, b2, first, second, i_first, i_second, count, i_out):
        z = (first @ w1[:, :HID].T)[:, i_first] + (second @ w1[:, HID:2 * HID].T)[:, i_second]
        z = torch.relu(z + sigma[:, chk] * w1[:, -1] + b1)
        total = torch.zeros((s.shape[0], count, HID), dtype=z.dtype, device=z.device)
        total = total.index_add(1, i_out, z)
        degree = torch.bincount(i_out, minlength=count).to(z.dtype)
        return total @ w2.T + degree[:, None] * b2

    for _ in range(layers):
        hv = hv + messages(part["W1_cv"], part["b1_cv"], part["W2_cv"], part["b2_cv"],
                           hc, hv, chk, var, hv.shape[1], var)
        hc = hc + messages(part["W1_vc"], part["b1_vc"], part["W2_vc"], part["b2_vc"],
                           hv, hc, var, chk, hc.shape[1], chk)
    return lam + hv @ part["w_o"] + part["b_o"]
