"""The default kernels are as exact as the general ones, which run the textbook
recursions in body frames in one thread per environment: the error against 64
bits, as a relative 2-norm over a batch. The bar, 1.2 times the general
kernel's error: both sides are sums of some ten thousand independent roundings
whose largest terms come from the few states with the worst-conditioned mass
matrices, which leaves the ratio of two such norms uncertain by about a tenth."""
import numpy as np
import pytest

from oracle import derivs, rbd
from paper_2605_31481_gb300 import workloads as w
from tests._helpers import from_soa, to_soa_cuda

pytestmark = pytest.mark.gpu

TREES = {"chain7": lambda: w.chain(7, seed=0), "quadruped11": lambda: w.spined_quadruped(seed=0),
         "legged18": lambda: w.legged(6, seed=0), "humanoid29": lambda: w.humanoid(seed=0)}
BAR = 1.2


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_31481_gb300 import build
    build.build(quiet=True)
    return torch


def _setup(name, B, torch, seed=7):
    """A tree, its states rounded to 32 bits (so that both sides start from the same numbers), and on the GPU."""
    tree = TREES[name]()
    s = {k: v.astype(np.float32).astype(np.float64) for k, v in w.random_state(tree, B, seed=seed).items()}
    return tree, s, {k: to_soa_cuda(v, torch) for k, v in s.items()}


def _errors(m, kind, call, ref):
    """Of the general kernel's and of the default's outputs."""
    out = []
    for form in ("generic", "auto"):
        m.set_launch([kind], 0, form)
        got = call()
        out.append({k: np.linalg.norm(from_soa(got[k]) - ref[k]) / np.linalg.norm(ref[k]) for k in ref})
    return out


def _no_further_off(general, default):
    for k in general:
        assert default[k] <= BAR * general[k], (k, default[k], general[k])


@pytest.mark.parametrize("name", list(TREES))
def test_aba_adjoint(torch_cuda, name):
    from paper_2605_31481_gb300 import api
    tree, s, x = _setup(name, 1000, torch_cuda)
    bar = s["qdd"]
    ref = dict(zip(("q", "qd", "tau"), derivs.aba_vjp(tree, s["q"], s["qd"], s["tau"], bar)[:3]))
    m = api.Model(tree)
    m.set_launch(["aba"], 0, "generic")
    qdd = api.aba(m, x["q"], x["qd"], x["tau"])
    _no_further_off(*_errors(m, "aba_vjp", lambda: api.aba_vjp(m, x["q"], x["qd"], qdd, x["qdd"]), ref))
