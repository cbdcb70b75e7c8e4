"""The kernels that the default no longer picks at small sizes, by name: the
checks of the other files that were written for the specialised kernels, the
one-environment-per-thread kernels and the mixed-tree launch's persistent form,
with that form set on every model and group that they make."""
import pytest

from tests import test_gpu_adjoints, test_gpu_derivatives, test_gpu_fused_step, test_gpu_multi, test_gpu_specialized

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_31481_gb300 import build
    build.build(quiet=True)
    return torch


@pytest.fixture
def one_per_thread(monkeypatch):
    """Models run what was specialised for them specialised and the rest generic; groups run the persistent kernel."""
    from paper_2605_31481_gb300 import _ffi, api

    class Model(api.Model):
        def __init__(self, *args, **kw):
            super().__init__(*args, **kw)
            spec = self.specialized()
            for kind in _ffi.SPEC_KINDS:
                self.set_launch([kind], 0, "specialized" if kind in spec and kind != "eval_mixed" else "generic")

    class MultiBatch(api.MultiBatch):
        def __init__(self, models):
            super().__init__(models)
            self.set_launch(64, "generic")

    monkeypatch.setattr(api, "Model", Model)
    monkeypatch.setattr(api, "MultiBatch", MultiBatch)


SP, FS, DV, AD = test_gpu_specialized, test_gpu_fused_step, test_gpu_derivatives, test_gpu_adjoints
CASES = (
    [(SP.test_specialized_forward_ops_match_oracle, (n,)) for n in ("chain7", "quadruped11", "humanoid29", "general8")]
    + [(SP.test_specialized_adjoints_match_oracle, (n,)) for n in ("chain7", "humanoid29", "general8")]
    + [(SP.test_specialized_theta_override, ())]
    + [(FS.test_packed_layout_holds_the_full_layouts_entries, (n, s)) for n in ("quadruped11", "humanoid29", "general8")
       for s in (False, True)]
    + [(FS.test_fused_step_matches_separate_calls_and_oracle, (n, True)) for n in ("quadruped11", "humanoid29")]
    + [(DV.test_rnea_derivatives_match_oracle, (n, s)) for n in ("chain7", "humanoid29", "general8")
       for s in (False, True)]
    + [(DV.test_aba_derivatives_match_oracle, (n, s)) for n in ("quadruped11", "urdf_arm6_tool") for s in (False, True)]
    + [(AD.test_rnea_vjp_matches_oracle, (n,)) for n in ("quadruped11", "humanoid29")]
    + [(AD.test_aba_vjp_matches_oracle, (n,)) for n in ("quadruped11", "humanoid29")]
    + [(AD.test_rnea_store_variant_matches_oracle_and_recompute, (n, s)) for n in ("quadruped11", "general8")
       for s in (False, True)]
)


@pytest.mark.parametrize("check,args", CASES, ids=[f"{f.__name__[5:]}-{'-'.join(map(str, a))}" for f, a in CASES])
def test_by_name(torch_cuda, one_per_thread, check, args):
    check(torch_cuda, *args)


@pytest.mark.parametrize("check", [test_gpu_multi.test_mixed_batch_equals_per_tree_calls_and_oracle,
                                   test_gpu_multi.test_mixed_batch_subsets_and_empty_members,
                                   test_gpu_multi.test_mixed_batch_replays_from_a_cuda_graph])
def test_persistent_mixed_launch(torch_cuda, one_per_thread, check):
    """The atomic work counter is reset between calls and between replays."""
    check(torch_cuda)
