"""Which Gaussians the tile culling drops for their opacity: exactly those with
opacity below alpha_min, whose alpha = o G reaches it nowhere.  Instance counts are
whole numbers, so an opacity one unit in the last place below alpha_min leaves no
instance, one at or above it the instances of the Gaussians around it."""
import numpy as np
import pytest
import torch

from paper_2505_05356_gb300 import gftorf, scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_opacity_at_the_alpha_floor(dtype):
    floor = np.float32(1.0 / 255.0)  # as the C struct holds it
    real = np.float32 if dtype == torch.float32 else np.float64
    o = {"below": np.nextafter(real(floor), real(0)), "a little below": real(floor) * real(1 - 4e-5),
         "at": real(floor), "above": np.nextafter(real(floor), real(1))}
    counts = {}
    for k, v in o.items():
        sc = scenes.make_scene("batch_300k", 5, n=2000, width=64, height=64, frames=1)
        sc.opacity = np.full(sc.n, v, np.float64)
        r = gftorf.Renderer(sc.n, 1, 64, 64, dtype=dtype)
        p = gftorf.params_from_scene(sc, dtype=dtype)
        assert np.all(p["opacity"].cpu().numpy() == v)
        bg = torch.as_tensor(sc.bg).to("cuda", dtype).contiguous()
        r.preprocess(p, gftorf.frames_from_scene(sc), gftorf.sensor_from_scene(sc),
                     gftorf.consts_from_scene(sc))
        r.render_fwd(bg)
        counts[k] = r.check()
    assert counts["below"] == 0 and counts["a little below"] == 0, counts
    assert counts["above"] >= counts["at"] > 1000, counts  # (a larger ellipse)
