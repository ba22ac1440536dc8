"""The autotuner times only the launches that a pipeline names as different (no
GPU: timings are replaced by a table), and SplatPipeline names those that its
kernels have."""
import types

import pytest

from paper_2504_13339_gb300 import _lib, autotune as AT
from paper_2504_13339_gb300.render import SplatPipeline


class Pipeline:
    n, V, W, H, capacity, device = 1000, 2, 64, 48, 1 << 22, "cpu"

    def __init__(self, choices):
        self.tf_group = self.tf_group_bwd = self.tile_batch = self.tile_batch_bwd = 0
        self.choices, self.runs = choices, []

    def launch_choices(self, luts):
        return self.choices

    def composite(self, luts):
        self.runs.append(("fwd", self.tf_group, self.tile_batch))

    def backward_2d(self, dout):
        self.runs.append(("bwd", self.tf_group_bwd, self.tile_batch_bwd))


LUTS = types.SimpleNamespace(shape=(4, 256, 4))


@pytest.fixture
def timed(monkeypatch, tmp_path):
    monkeypatch.setenv("XDG_CACHE_HOME", str(tmp_path))
    monkeypatch.setattr(AT.torch.cuda, "get_device_name", lambda d=None: "FakeGPU")
    ms = {("fwd", 0, 128): 2.0, ("fwd", 0, 256): 1.0, ("fwd", 0, 512): 3.0, ("bwd", 1, 0): 5.0,
          ("bwd", 4, 0): 4.0}

    def use(p):
        monkeypatch.setattr(AT, "_time", lambda fn, reps: (fn(), ms[p.runs[-1]])[1])
        return p
    return use


def test_only_the_named_launches_are_timed(timed, monkeypatch):
    choices = {"fwd": [(0, 128), (0, 256), (0, 512)], "bwd": [(1, 0), (4, 0)]}
    p = timed(Pipeline(choices))
    res = AT.tune(p, LUTS, dout=object())
    assert set(res["times"]) == {"fwd0x128", "fwd0x256", "fwd0x512", "bwd1x0", "bwd4x0"}
    assert (res["fwd"], res["fwd_batch"], res["bwd"], res["bwd_batch"]) == (0, 256, 4, 0)
    assert (p.tf_group, p.tile_batch, p.tf_group_bwd, p.tile_batch_bwd) == (0, 256, 4, 0)
    monkeypatch.setattr(AT, "_time", lambda fn, reps: pytest.fail("timed despite the cache"))
    assert AT.tune(Pipeline(choices), LUTS, dout=object()) == res


def test_a_single_launch_is_not_timed(timed, monkeypatch):
    p = timed(Pipeline({"fwd": [(0, 0)], "bwd": [(0, 0)]}))
    monkeypatch.setattr(AT, "_time", lambda fn, reps: pytest.fail("timed a single launch"))
    res = AT.tune(p, LUTS, dout=object(), use_cache=False)
    assert res["times"] == {} and (res["fwd_batch"], res["bwd"]) == (0, 0)
    assert AT.tune(p, LUTS, use_cache=False)["bwd"] == 0


@pytest.mark.parametrize("staged,n_tf,fwd,bwd", [(256, 4, 3, 2), (0, 4, 1, 2), (256, 2, 3, 1),
                                                 (0, 1, 1, 1)])
def test_the_pipelines_launches(monkeypatch, staged, n_tf, fwd, bwd):
    monkeypatch.setattr(_lib, "veg_composite_fwd_batch", lambda *a: staged)
    monkeypatch.setattr(_lib, "tf_desc", lambda luts: None)
    p = types.SimpleNamespace(c_cams=None, n=5)
    got = SplatPipeline.launch_choices(p, types.SimpleNamespace(shape=(n_tf, 256, 4)))
    assert (len(set(got["fwd"])), len(set(got["bwd"]))) == (fwd, bwd)
