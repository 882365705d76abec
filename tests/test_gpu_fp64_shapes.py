"""The double instantiation for every number of frequencies at every tile shape
narrower than 32, with the library's choice of pixels per thread and with two and
four of them: forward and gradients against the FP64 oracle at the FP64 bars of
test_gpu_parity (1e-9; 1e-8 by norm, 1e-7 by element)."""
import numpy as np
import pytest
import torch

from oracle import oracle as ora
from paper_2505_05356_gb300 import scenes
from tests.gpu_helpers import absent_groups, forward_close, grads_close, run_gpu

pytestmark = pytest.mark.gpu

FREQS = [30e6, 80e6, 50e6, 20e6]


@pytest.mark.parametrize("n_freq,depth", [(1, False), (2, False), (2, True), (3, False), (4, True)])
@pytest.mark.parametrize("tile,ppt", [((16, 32), 0), ((16, 32), 2), ((16, 32), 4), ((16, 16), 0),
                                      ((16, 16), 4), ((8, 8), 0)])
def test_fp64_matches_the_oracle(n_freq, depth, tile, ppt):
    sc = scenes.make_scene("batch_300k", 41, n=800, width=72, height=70, frames=2, tile=tile,
                           freqs_hz=FREQS[:n_freq], depth=depth)
    eps64 = (1e-9, 1e-10, 1.2e-7, 1e-9)  # depth keys are single precision
    q_ora, _, amb, _ = ora.render(sc, eps64)
    dout = scenes.random_dout(sc, 3)
    dout[np.broadcast_to((amb != 0)[:, None], dout.shape)] = 0.0
    g_ora = ora.backward(sc, dout.astype(np.float64))
    res = run_gpu(sc, dout, dtype=torch.float64, pixels_per_thread=ppt)
    ok, worst, _ = forward_close(res["out"], q_ora, amb, rel=1e-9)
    assert ok, worst
    for k, (nrm, elem) in grads_close(res["grads"], g_ora, absent=absent_groups(sc)).items():
        assert nrm <= 1e-8 and elem <= 1e-7, (k, nrm, elem)
