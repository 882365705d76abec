"""Batches of many tiles are composited in 32x16 parts of 128 threads: the
forward and the final transmittances bit for bit as in two half batches, which are
composited in 32x32 parts (the same lists, the same records in the same order per
pixel), the gradients within twice the parity bar of 1e-3 (each side is held to it
against the oracle)."""
import numpy as np
import pytest

from paper_2505_05356_gb300 import scenes
from tests.gpu_helpers import absent_groups, grads_close, run_gpu

pytestmark = pytest.mark.gpu

FREQS = [30e6, 80e6, 50e6, 20e6]
PER_FRAME = ("bg", "delta")


@pytest.mark.parametrize("n_freq,depth", [(1, False), (2, True), (3, False), (4, True)])
@pytest.mark.parametrize("tile,mode", [((32, 32), 0), ((64, 32), 1), ((64, 64), 0)])
def test_narrow_parts_composite_the_same_records(n_freq, depth, tile, mode):
    # 64 frames of 300x230: 5120 parts of 32x32, 2560 in a half
    sc = scenes.make_scene("batch_300k", 37, n=600, width=300, height=230, frames=64, tile=tile,
                           freqs_hz=FREQS[:n_freq], depth=depth)
    dout = scenes.random_dout(sc, 3)
    res = run_gpu(sc, dout, render_mode=mode)
    halves = []
    for f in (slice(0, 32), slice(32, 64)):
        half = scenes.Scene(sc.means, sc.coeffs, sc.scales, sc.quats, sc.opacity, sc.amplitude,
                            sc.times[f], sc.cameras[f], sc.delta[f], sc.sensor, sc.consts,
                            sc.bg[f])
        halves.append(run_gpu(half, dout[f], render_mode=mode))
    for k in ("out", "tfinal", "nlast"):
        assert np.array_equal(res[k], np.concatenate([h[k] for h in halves])), k
    ref = {k: np.concatenate([h["grads"][k] for h in halves]) if k in PER_FRAME
           else halves[0]["grads"][k] + halves[1]["grads"][k] for k in res["grads"]}
    for k, (nrm, elem) in grads_close(res["grads"], ref, absent=absent_groups(sc)).items():
        assert nrm <= 2e-3 and elem <= 2e-3, (k, nrm, elem)
