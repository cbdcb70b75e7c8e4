"""The aligned-frame kernels (csrc/aligned.cuh: adjoints and dense
derivatives) where they can go wrong: random trees with every joint type,
forests beside a floating root, a wide star, a chain whose state just fits in
shared memory (one that does not fit runs the general kernels),
batches of one environment and of one more than a tile; and the general
kernels themselves, which the default no longer reaches for small trees.
Tolerances are those of the adjoint and derivative tests."""
import numpy as np
import pytest

from oracle import derivs, rbd
from paper_2605_31481_gb300 import workloads as w
from tests._helpers import env_err, from_soa, solve_backward_err, to_soa_cuda
from tests.test_gpu_adjoints import BWD_BAR, GTOL, THTOL, _check_aba_vjp, _th_err
from tests.test_gpu_derivatives import DTOL, _err, _mat
from tests.test_gpu_random_trees import random_tree

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_31481_gb300 import build
    build.build(quiet=True)
    return torch


def _floating_forest():
    """A floating root with an arm, beside two fixed roots (one of them a lone body)."""
    R, P = w.REVOLUTE, w.PRISMATIC
    return w.random_tree([-1, 0, 1, 2, -1, 4, 5, -1], [w.FREE, R, P, R, R, w.FIXED, R, P], 9)


TREES = {f"random{s}": (lambda s=s: random_tree(s)) for s in range(5)}
TREES.update({
    "one": lambda: w.chain(1, seed=2),
    "star": lambda: w.random_tree([-1] + [0] * 13, [w.REVOLUTE] * 14, 4),   # one level of 13 bodies
    "floating_forest": _floating_forest,
    "chain30": lambda: w.chain(30, seed=3),                                 # the state nearly fills shared memory
})


def _inputs(torch, tree, B, seed):
    s = w.random_state(tree, B, seed=seed)
    rng = np.random.default_rng(seed + 1)
    bar = rng.standard_normal((B, tree.nv))
    th = rbd.Model(tree).theta() * (1 + rng.uniform(-0.2, 0.2, (tree.n_bodies, 10)))
    x = {k: to_soa_cuda(v, torch) for k, v in s.items()}
    x["bar"] = to_soa_cuda(bar, torch)
    x["th"] = torch.from_numpy(th.astype(np.float32)).cuda()
    return s, bar, th, x


def _check_adjoints(torch, m, tree, B, label):
    from paper_2605_31481_gb300 import api
    s, bar, th, x = _inputs(torch, tree, B, 71)
    res = api.rnea_vjp(m, x["q"], x["qd"], x["qdd"], x["bar"], theta=x["th"])
    L, gth, qb, qdb = api.rnea_loss_grad(m, x["q"], x["qd"], x["qdd"], x["tau"], theta=x["th"], q_bar=True, qd_bar=True)
    torch.cuda.synchronize()
    rq, rqd, rqdd, rth = derivs.rnea_vjp(tree, s["q"], s["qd"], s["qdd"], bar, theta=th)
    for k, ref in (("q", rq), ("qd", rqd), ("qdd", rqdd)):
        assert env_err(from_soa(res[k]), ref).max() <= GTOL, f"{label} {k}"
    # the parameter gradient and the loss against the oracle's with the same override
    r = rbd.rnea(tree, s["q"], s["qd"], s["qdd"], theta=th) - s["tau"]
    lq, lqd, _, lth = derivs.rnea_vjp(tree, s["q"], s["qd"], s["qdd"], 2 * r, theta=th)
    assert _th_err(res["theta"].cpu().numpy(), rth) <= THTOL, label
    assert _th_err(gth.cpu().numpy(), lth) <= THTOL, label
    assert abs(float(L) - (r ** 2).sum()) <= GTOL * (r ** 2).sum(), label
    assert env_err(from_soa(qb), lq).max() <= GTOL and env_err(from_soa(qdb), lqd).max() <= GTOL, label


def _check_forward(torch, m, tree, B, label):
    """ABA's adjoint and derivatives: backward errors (see _check_aba_vjp)."""
    from paper_2605_31481_gb300 import api
    s, bar, _, x = _inputs(torch, tree, B, 73)
    qdd = api.aba(m, x["q"], x["qd"], x["tau"])
    res = api.aba_vjp(m, x["q"], x["qd"], qdd, x["bar"])
    d = api.aba_derivatives(m, x["q"], x["qd"], x["tau"], qdd=True)
    no = api.aba_derivatives(m, x["q"], x["qd"], x["tau"], dq=False)
    torch.cuda.synchronize()
    _check_aba_vjp(tree, s, from_soa(qdd), bar, res, label)
    M = rbd.crba(tree, s["q"])
    Dq, Dqd = derivs.rnea_derivatives(tree, s["q"], s["qd"], from_soa(d["qdd"]))
    for key, rhs in (("q", -Dq), ("qd", -Dqd), ("tau", np.broadcast_to(np.eye(tree.nv), M.shape))):
        if np.abs(rhs).max() < 1e-12:  # identically zero (a lone revolute joint's d tau / d qd): no scale to be relative to
            assert np.abs(_mat(d[key])).max() <= DTOL, f"{label} d qdd / d {key}"
            continue
        bwd = solve_backward_err(M, _mat(d[key]), rhs)
        assert bwd.max() <= BWD_BAR, f"{label} d qdd / d {key}: {bwd.max():.3e}"
    assert torch.equal(no["qd"], d["qd"]) and torch.equal(no["tau"], d["tau"]), label


def _check_derivatives(torch, m, tree, B, label):
    from paper_2605_31481_gb300 import api
    s, _, _, x = _inputs(torch, tree, B, 75)
    res = api.rnea_derivatives(m, x["q"], x["qd"], x["qdd"])
    torch.cuda.synchronize()
    for k, ref in zip(("q", "qd"), derivs.rnea_derivatives(tree, s["q"], s["qd"], s["qdd"])):
        assert _err(_mat(res[k]), ref).max() <= DTOL, f"{label} d tau / d {k}"


@pytest.mark.parametrize("B", [1, 33])
@pytest.mark.parametrize("name", list(TREES))
def test_default_kernels_match_oracle(torch_cuda, name, B):
    from paper_2605_31481_gb300 import api
    tree = TREES[name]()
    m = api.Model(tree)
    if tree.nv == 0:
        pytest.skip("no degree of freedom")
    _check_adjoints(torch_cuda, m, tree, B, name)
    _check_derivatives(torch_cuda, m, tree, B, name)
    _check_forward(torch_cuda, m, tree, B, name)


def test_tree_that_does_not_fit_runs_the_general_kernels(torch_cuda):
    """A 36-body chain's state exceeds shared memory: every default call must
    give the general kernels' results, bit for bit."""
    torch = torch_cuda
    from paper_2605_31481_gb300 import api
    tree = w.chain(36, seed=3)
    m, g = api.Model(tree), api.Model(tree)
    g.set_launch(["rnea_vjp", "aba_vjp", "loss_grad", "rnea_derivatives", "aba_derivatives"], 0, "generic")
    _, _, _, x = _inputs(torch, tree, 33, 71)
    args = x["q"], x["qd"], x["qdd"]
    for call in (lambda k: api.rnea_vjp(k, *args, x["bar"]), lambda k: api.aba_vjp(k, *args, x["bar"]),
                 lambda k: dict(enumerate(api.rnea_loss_grad(k, *args, x["tau"])[:2])),
                 lambda k: api.rnea_derivatives(k, *args), lambda k: api.aba_derivatives(k, *args, qdd=True)):
        a, b = call(m), call(g)
        torch.cuda.synchronize()
        for key in b:
            assert torch.equal(a[key], b[key]), key


@pytest.mark.parametrize("variant", ["generic", "specialized"])
@pytest.mark.parametrize("name", ["random0", "floating_forest"])
def test_general_kernels_match_oracle(torch_cuda, name, variant):
    from paper_2605_31481_gb300 import api
    kinds = ["rnea_vjp", "aba_vjp", "loss_grad", "rnea_derivatives", "aba_derivatives"]
    tree = TREES[name]()
    m = api.Model(tree, specialize=kinds if variant == "specialized" else False)
    m.set_launch(kinds, 0, variant)
    _check_adjoints(torch_cuda, m, tree, 33, name)
    _check_derivatives(torch_cuda, m, tree, 33, name)
    _check_forward(torch_cuda, m, tree, 33, name)


@pytest.mark.parametrize("B", [152 * 64 + 1, 152 * 64 + 65])
@pytest.mark.parametrize("name", ["random1", "random2", "floating_forest", "star"])
def test_lean_forms_give_the_same_bits(torch_cuda, name, B):
    """Past two tiles per SM the default keeps less state per tile (the RNEA
    adjoint, RNEA, the fused evaluation's CRBA): the same arithmetic, so the
    same bits as the small-batch forms give on the environments at both ends
    (a tile and a tail of one; an odd number of tiles)."""
    torch = torch_cuda
    from paper_2605_31481_gb300 import api
    tree = TREES[name]()
    m = api.Model(tree)
    _, _, _, x = _inputs(torch, tree, B, 77)
    part = lambda lo, hi: {k: v[:, lo:hi].contiguous() for k, v in x.items() if k != "th"}  # noqa: E731
    links = list(tree.ee) or [tree.n_bodies - 1]
    run = lambda y: {**api.rnea_vjp(m, y["q"], y["qd"], y["qdd"], y["bar"], theta_bar=False),  # noqa: E731
                     "tau": api.rnea(m, y["q"], y["qd"], y["qdd"]),
                     **{"ev_" + k: v for k, v in api.eval(m, y["q"], y["qd"], y["qdd"], y["tau"], fk=True, links=links,
                                                          rnea=True, crba=True, aba=True).items()}}
    full = run(part(0, B))
    for lo, hi in ((0, 33), (B - 34, B)):
        few = run(part(lo, hi))
        torch.cuda.synchronize()
        for k in few:
            assert torch.equal(full[k][..., lo:hi], few[k]), (name, B, k)


@pytest.mark.parametrize("name,B,specialize", [
    ("chain7", 9728, False), ("chain7", 9729, False),      # RNEA leaves the tiles before its adjoint does
    ("chain12", 4865, False), ("chain30", 40, False), ("wide36", 40, False),  # wide36: only the adjoint does not fit
    ("quadruped11", 8191, True), ("quadruped11", 8192, True), ("quadruped11", 9728, True), ("quadruped11", 9729, True),
])
def test_fused_evaluation_equals_separate_calls_at_the_rules_edges(torch_cuda, name, B, specialize):
    torch = torch_cuda
    from paper_2605_31481_gb300 import api
    tree = {"quadruped11": w.spined_quadruped, "wide36": lambda: w.random_tree([-1] + [i // 3 for i in range(35)],
                                                                          [w.REVOLUTE] * 36, 6),
            }.get(name, lambda: w.chain(int(name[5:]), seed=5))()
    m = api.Model(tree, specialize=specialize)
    _, _, _, x = _inputs(torch, tree, B, 83)
    q, qd, qdd, tau = (x[k] for k in ("q", "qd", "qdd", "tau"))
    links = [tree.n_bodies - 1]
    want = {"poses": api.fk(m, q), "J": api.jacobian(m, q, links), "tau": api.rnea(m, q, qd, qdd),
            "M": api.crba(m, q), "qdd": api.aba(m, q, qd, tau)}
    for bar in ("tau", x["bar"]):
        res = api.eval(m, q, qd, qdd, tau, fk=True, links=links, rnea=True, crba=True, aba=True, tau_bar=bar,
                       q_bar=True, qd_bar=True, qdd_bar=True)
        vjp = api.rnea_vjp(m, q, qd, qdd, want["tau"] if isinstance(bar, str) else bar, theta_bar=False)
        torch.cuda.synchronize()
        for k, v in want.items():
            assert torch.equal(res[k], v), (name, B, k)
        for k in ("q", "qd", "qdd"):
            assert torch.equal(res[k + "_bar"], vjp[k]), (name, B, k + "_bar")
