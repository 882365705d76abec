"""The backward's per-record sums (warp rows in shared memory) against the FP64
oracle for every number of values a record can have: one to four frequencies,
with and without the mean-depth channel (9 to 16 values; three, then two
records fill the 32 rows), with one, two and four pixels per thread.  Bars as
in test_gpu_parity: gradients within 1e-3."""
import numpy as np
import pytest

from oracle import oracle as ora
from paper_2505_05356_gb300 import scenes
from tests.gpu_helpers import absent_groups, grads_close, run_gpu

pytestmark = pytest.mark.gpu

FREQS = [30e6, 80e6, 50e6, 20e6]


@pytest.mark.parametrize("n_freq", [1, 2, 3, 4])
@pytest.mark.parametrize("depth", [False, True])
@pytest.mark.parametrize("tile,ppt", [((16, 16), 1), ((16, 32), 1), ((16, 16), 2), ((16, 32), 4),
                                      ((32, 32), 4)])
def test_gradients_for_every_record_width(n_freq, depth, tile, ppt):
    sc = scenes.make_scene("batch_300k", 31, n=1500, width=56, height=40, frames=2, tile=tile,
                           freqs_hz=FREQS[:n_freq], depth=depth)
    _, _, amb, _ = ora.render(sc, ora.EPS_F32)
    dout = scenes.random_dout(sc, 3)
    dout[np.broadcast_to((amb != 0)[:, None], dout.shape)] = 0.0
    g_ora = ora.backward(sc, dout.astype(np.float64))
    res = run_gpu(sc, dout, pixels_per_thread=ppt)
    for k, (nrm, elem) in grads_close(res["grads"], g_ora, absent=absent_groups(sc)).items():
        assert nrm <= 1e-3 and elem <= 1e-3, (k, nrm, elem)
