"""The tuner's candidates and its cache on the host, with the model, the timer
and the kernels replaced by fakes (no GPU)."""
import os
import shutil

import pytest

from paper_2605_31481_gb300 import autotune, build

KINDS = ("rnea", "eval", "fk_vjp", "rnea_vjp", "loss_grad", "aba_vjp", "rnea_store")


class FakeModel:
    device = "cpu"
    ee = (1,)
    n_bodies = 2
    name = fingerprint = "fake"

    def __init__(self, specialized=()):
        self.spec, self.launch = specialized, {}

    def specialized(self):
        return self.spec

    def set_launch(self, kinds, block, variant):
        for k in kinds:
            self.launch[k] = (variant, block)


@pytest.fixture
def fakes(monkeypatch, tmp_path):
    monkeypatch.setenv("FST_TUNE_CACHE", str(tmp_path / "tune.json"))
    monkeypatch.setattr(autotune, "Buffers", lambda *a: type("B", (), {"__getattr__": lambda self, k: None})())
    monkeypatch.setattr(autotune, "_op", lambda model, kind, buf: lambda: (model, kind))
    for f in ("aba", "rnea_store"):
        monkeypatch.setattr(autotune.api, f, lambda *a, **k: None)
    monkeypatch.setattr(autotune.torch.cuda, "get_device_name", lambda d: "fake GPU", raising=False)
    monkeypatch.setattr(autotune, "sm_count", lambda d: 152)
    times = {}

    def timer(fn):
        model, kind = fn()
        return times.get(model.launch[kind], 20.0)

    monkeypatch.setattr(autotune, "graph_time_us", timer)
    return times


@pytest.mark.parametrize("specialized", [(), KINDS])
def test_the_untuned_form_is_a_candidate_where_no_other_candidate_names_it(fakes, specialized):
    model = FakeModel(specialized)
    fakes[("auto", 0)] = 5.0
    tuned = autotune.tune(model, 16384, kinds=KINDS, use_cache=False)
    for kind in KINDS:
        assert tuned[kind]["candidates"]["auto/0"] == 5.0
        assert (tuned[kind]["variant"], tuned[kind]["block"]) == ("auto", 0) == model.launch[kind]


def test_a_faster_explicit_form_is_still_chosen(fakes):
    model = FakeModel()
    fakes[("auto", 0)], fakes[("level", 128)] = 5.0, 4.0
    tuned = autotune.tune(model, 16384, kinds=("rnea", "rnea_vjp"), use_cache=False)
    assert model.launch == {"rnea": ("level", 128), "rnea_vjp": ("auto", 0)}
    assert all(t["us"] <= t["candidates"]["auto/0"] for t in tuned.values())


def test_a_choice_among_other_kernels_is_not_read_back(fakes, monkeypatch, tmp_path):
    """The cache's key follows the sources that the library is built from."""
    model = FakeModel()
    csrc = tmp_path / "csrc"
    shutil.copytree(build.CSRC, csrc)
    monkeypatch.setattr(build, "CSRC", str(csrc))

    def choice():
        autotune._code.cache_clear()
        return autotune.tune(model, 64, kinds=("rnea_vjp",))["rnea_vjp"]["variant"]

    fakes[("generic", 64)] = 4.0
    assert choice() == "generic"
    fakes[("auto", 0)] = 3.0
    assert choice() == "generic"                # nothing changed: from the cache
    with open(os.path.join(csrc, "level.cuh"), "a") as fh:
        fh.write("// changed\n")
    assert choice() == "auto"
    autotune._code.cache_clear()
