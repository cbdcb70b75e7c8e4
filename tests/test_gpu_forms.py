"""One call, one result: an operator gives the same bits as tiles of 32
environments whose warps share the bodies and as one environment per thread,
so that the rules which pick a form by tree, batch and entry point never show
in a result."""
import numpy as np
import pytest

from paper_2605_31481_gb300 import workloads as w
from tests._helpers import to_soa_cuda
from tests.test_gpu_random_trees import random_tree

pytestmark = pytest.mark.gpu

OPS = ("fk", "jacobian", "rnea", "crba", "aba")
TREES = {**{f"random{k}": (lambda k=k: random_tree(k)) for k in range(9)},
         "chain7": lambda: w.chain(7, seed=0), "quadruped11": lambda: w.spined_quadruped(seed=0),
         "humanoid23": lambda: w.humanoid(seed=0, floating=False), "humanoid29": lambda: w.humanoid(seed=0)}


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_31481_gb300 import build
    build.build(quiet=True)
    return torch


def _inputs(tree, B, torch, seed=3):
    s = w.random_state(tree, B, seed=seed)
    return [to_soa_cuda(s[k], torch) for k in ("q", "qd", "qdd", "tau")]


def _run(api, m, x, ee):
    q, qd, qdd, tau = x
    return {"poses": api.fk(m, q), "J": api.jacobian(m, q, ee), "tau": api.rnea(m, q, qd, qdd), "M": api.crba(m, q),
            "qdd": api.aba(m, q, qd, tau)}


def _ee(tree):
    return list(tree.ee) if tree.ee else [tree.n_bodies - 1]


@pytest.mark.parametrize("name", list(TREES))
def test_every_form_gives_the_same_bits(torch_cuda, name):
    torch = torch_cuda
    from paper_2605_31481_gb300 import api
    tree = TREES[name]()
    ee = _ee(tree)
    m = api.Model(tree)
    x = _inputs(tree, 197, torch)
    m.set_launch(None, 64, "generic")
    want = _run(api, m, x, ee)
    for fwd, lean in (("level", "level"), ("level", "levellean"), ("auto", "auto")):
        block = 0 if fwd == "auto" else 128
        m.set_launch(["fk", "jacobian", "rnea"], block, fwd)
        m.set_launch(["crba", "aba"], block, lean)
        got = _run(api, m, x, ee)
        for k in want:
            assert torch.equal(got[k], want[k]), (name, fwd, lean, k)
    m.set_launch(None, 0, "auto")
    got = api.eval(m, *x, fk=True, links=ee, rnea=True, crba=True, aba=True)
    for k in want:
        assert torch.equal(got[k], want[k]), (name, "eval", k)


@pytest.mark.parametrize("counts", [(12000, 4096, 2048), (9728, 64, 33), (9729, 0, 4000)])
def test_mixed_batches_give_the_single_calls_bits(torch_cuda, counts):
    """A chain whose own calls leave the tiles as its batch grows, beside trees whose calls do not."""
    torch = torch_cuda
    from paper_2605_31481_gb300 import api
    trees = [w.chain(7, seed=0), w.humanoid(seed=0, floating=True), w.spined_quadruped(seed=0)]
    _compare_mixed(torch, api, trees, counts)


def test_mixed_batch_of_a_tree_near_the_body_limit(torch_cuda):
    """60 bodies in three levels: the state of some operators fits a tile only in its lean form."""
    torch = torch_cuda
    from paper_2605_31481_gb300 import api
    parent = [-1] + [0] * 9 + [1 + k % 9 for k in range(50)]
    wide = w.random_tree(parent, [w.REVOLUTE] * 60, seed=4, name="wide60")
    _compare_mixed(torch, api, [wide, w.legged(4, seed=0)], (300, 500))


@pytest.mark.parametrize("name", list(TREES))
def test_specialised_kernels_give_the_same_bits(torch_cuda, name):
    """The operators whose own call and fused evaluation may take different forms at one batch size."""
    torch = torch_cuda
    from paper_2605_31481_gb300 import api
    tree = TREES[name]()
    ee = _ee(tree)
    m = api.Model(tree, specialize=["fk", "jacobian", "rnea", "crba"])
    q, qd, qdd, _ = _inputs(tree, 197, torch)
    out = {}
    for form in ("generic", "specialized"):
        m.set_launch(["fk", "jacobian", "rnea", "crba"], 0, form)
        out[form] = {"poses": api.fk(m, q), "J": api.jacobian(m, q, ee), "tau": api.rnea(m, q, qd, qdd),
                     "M": api.crba(m, q)}
    for k, want in out["generic"].items():
        assert torch.equal(out["specialized"][k], want), (name, k)


@pytest.mark.parametrize("name", list(TREES))
def test_the_aba_adjoint_solves_with_m_in_every_form_alike(torch_cuda, name):
    """tau_bar = M^-1 qdd_bar: the adjoint's sweep at rest rounds as the general kernel's does, no worse."""
    torch = torch_cuda
    from paper_2605_31481_gb300 import api
    tree = TREES[name]()
    m = api.Model(tree)
    q, qd, qdd, bar = _inputs(tree, 197, torch)
    out = {}
    for form in ("generic", "auto"):
        m.set_launch(["aba_vjp"], 0, form)
        out[form] = api.aba_vjp(m, q, qd, qdd, bar)["tau"]
    assert torch.equal(out["auto"], out["generic"]), name


LIGHT = ("fk", "jacobian", "rnea", "crba")  # a large tree's fused kernel is not picked: no need to compile it


@pytest.mark.parametrize("name,B,specialize", [
    ("chain7", 4000, None), ("chain7", 6000, None), ("chain12", 2000, None), ("quadruped11", 40000, None),
    ("chain7", 4000, LIGHT + ("aba", "eval")), ("quadruped11", 6000, LIGHT + ("aba", "eval")),
    ("quadruped11", 12000, LIGHT + ("aba", "eval")), ("humanoid29", 26000, LIGHT)])
def test_fused_evaluation_gives_the_calls_bits_where_their_forms_differ(torch_cuda, name, B, specialize):
    torch = torch_cuda
    from paper_2605_31481_gb300 import api
    tree = w.chain(12, seed=0) if name == "chain12" else TREES[name]()
    ee = _ee(tree)
    m = api.Model(tree, specialize=list(specialize) if specialize else None)
    x = _inputs(tree, B, torch)
    want = _run(api, m, x, ee)
    got = api.eval(m, *x, fk=True, links=ee, rnea=True, crba=True, aba=True)
    alone = api.eval(m, x[0], fk=True, links=ee)
    for k in want:
        assert torch.equal(got[k], want[k]), (name, k)
        assert k not in alone or torch.equal(alone[k], want[k]), (name, k, "alone")


def _compare_mixed(torch, api, trees, counts):
    models = [api.Model(t) for t in trees]
    xs = [_inputs(t, B, torch, seed=20 + k) for k, (t, B) in enumerate(zip(trees, counts))]
    items = [{"q": q, "qd": qd, "qdd": qdd, "tau": tau, "fk": True, "rnea": True, "crba": True, "aba": True}
             for q, qd, qdd, tau in xs]
    res = api.MultiBatch(models).eval(items)
    for t, m, r, x in zip(trees, models, res, xs):
        want = _run(api, m, x, _ee(t))
        for k in r:
            assert torch.equal(r[k], want[k]), (t.name, k)
