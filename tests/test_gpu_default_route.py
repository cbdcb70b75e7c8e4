"""The default form of a call is no slower than the form it is chosen over, at
sizes where a rule has to part the two. The bar: 8 %, twice the spread of
either side's minimum over repeated replays of a graph of the call."""
import pytest

from paper_2605_31481_gb300 import workloads as w
from tests._helpers import to_soa_cuda

pytestmark = pytest.mark.gpu
BAR = 1.08

TREES = {"chain7": lambda: w.chain(7, seed=0), "chain10": lambda: w.chain(10, seed=0),
         "chain12": lambda: w.chain(12, seed=0), "chain16": lambda: w.chain(16, seed=0),
         "quadruped11": lambda: w.spined_quadruped(seed=0), "legged18": lambda: w.legged(6, seed=0),
         "humanoid29": lambda: w.humanoid(seed=0)}


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_31481_gb300 import build
    build.build(quiet=True)
    return torch


def _calls(api, torch, m, tree, B):
    s = w.random_state(tree, B, seed=5)
    q, qd, qdd, tau = (to_soa_cuda(s[k], torch) for k in ("q", "qd", "qdd", "tau"))
    ee = list(tree.ee)
    new = lambda *shape: torch.empty(*shape, device="cuda")  # noqa: E731
    o = {"poses": new(m.n_bodies, 12, B).normal_(), "J": new(len(ee), 6, m.nv, B), "tau": new(m.nv, B), "M": new(m.nv, m.nv, B),
         "qdd": new(m.nv, B)}
    return {"jacobian": lambda: api.jacobian(m, q, ee, out=o["J"]),
            "rnea": lambda: api.rnea(m, q, qd, qdd, out=o["tau"]),
            "crba": lambda: api.crba(m, q, out=o["M"]), "aba": lambda: api.aba(m, q, qd, tau, out=o["qdd"]),
            "rnea_store": lambda: api.rnea_store(m, q, qd, qdd, out=o["tau"]), "fk": lambda: api.fk(m, q, out=o["poses"]),
            "fk_vjp": lambda: api.fk_vjp(m, q, o["poses"]),
            "aba_vjp": lambda: api.aba_vjp(m, q, qd, qdd, tau, theta_bar=False),
            "eval": lambda: api.eval(m, q, fk=True, links=ee, out=o)}


def _times(api, torch, name, B, kind, specialize, forms):
    from paper_2605_31481_gb300.autotune import graph_time_us
    tree = TREES[name]()
    m = api.Model(tree, specialize=[kind] if specialize else None)
    call = _calls(api, torch, m, tree, B)[kind]
    best = [float("inf")] * len(forms)
    for n in range(20):  # the forms in turn; longer where another program disturbs the first measurements
        for k, (variant, block) in enumerate(forms):
            m.set_launch([kind], block, variant)
            best[k] = min(best[k], graph_time_us(call))
        if n >= 4 and best[0] <= BAR * min(best[1:]):
            break
    return best


@pytest.mark.parametrize("name,B,kind,specialize", [
    ("chain7", 4096, "rnea", False), ("chain7", 1024, "rnea_store", False), ("chain7", 2048, "aba", False),
    ("chain16", 4096, "rnea_store", False), ("quadruped11", 8192, "jacobian", True),
    ("legged18", 12288, "jacobian", True), ("legged18", 32768, "crba", True), ("legged18", 20480, "rnea", True),
    ("chain7", 4096, "eval", True), ("chain12", 1024, "rnea", True), ("chain10", 6000, "fk", True),
    ("chain10", 4096, "aba", True), ("chain12", 4096, "fk_vjp", True), ("chain7", 22000, "aba_vjp", True),
    ("quadruped11", 22000, "aba_vjp", True), ("chain16", 20000, "aba_vjp", False)])
def test_default_is_not_slower_than_the_form_it_replaces(torch_cuda, name, B, kind, specialize):
    from paper_2605_31481_gb300 import api
    other = "specialized" if specialize else "generic"
    default, other = _times(api, torch_cuda, name, B, kind, specialize,
                            [("auto", 0), (other, 32 if kind == "eval" else 0)])
    assert default <= BAR * other, (default, other)


@pytest.mark.parametrize("name,B,kind", [("humanoid29", 64, "rnea"), ("quadruped11", 4096, "rnea_store"),
                                         ("quadruped11", 64, "aba")])
def test_a_block_set_with_the_default_variant_does_not_slow_the_tiles(torch_cuda, name, B, kind):
    """A block is one of environments, one per thread: 32 of them are one warp, and a tile wants eight."""
    from paper_2605_31481_gb300 import api
    default, other = _times(api, torch_cuda, name, B, kind, False, [("auto", 32), ("generic", 32)])
    assert default <= BAR * other, (default, other)
