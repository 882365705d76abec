"""sort_footprints without a capacity sizes its buffers by gftorf_footprint_bound: a
status other than OK is raised as it is, before anything is sized or launched by it."""
import pytest
import torch

from paper_2505_05356_gb300 import gftorf


class _Failing:
    """Stands for the library: the bound fails, and nothing else may be called."""

    def __init__(self, code):
        self.code = code

    def gftorf_footprint_bound(self, *args):
        return self.code

    def __getattr__(self, name):
        raise AssertionError("%s called after the bound had failed" % name)


@pytest.mark.parametrize("code", [gftorf.ERR_CUDA, gftorf.ERR_ARG])
def test_a_failing_bound_is_reported_as_it_is(monkeypatch, code):
    lib = _Failing(code)
    monkeypatch.setattr(gftorf, "_require_cuda", lambda: None)
    monkeypatch.setattr(gftorf, "load", lambda *a, **k: lib)
    monkeypatch.setattr(gftorf, "_ptr", lambda t: 0)
    monkeypatch.setattr(gftorf, "_stream", lambda: 0)
    u = torch.zeros((1, 4))
    with pytest.raises(gftorf.GftorfError) as e:
        gftorf.sort_footprints(u, u, u.int(), u, 64, 64)
    assert e.value.code == code
