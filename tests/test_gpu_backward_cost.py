"""The backward's time per frequency and launch shape, as ratios of medians on the
same device: a kernel whose registers spill, or whose shared memory halves the CTAs
per SM, costs more than its extra work."""
import pytest
import torch

from paper_2505_05356_gb300 import gftorf, scenes

pytestmark = pytest.mark.gpu

FREQS = [30e6, 80e6, 50e6, 20e6]


def _backward_us(n_freq, tile, ppt=0):
    sc = scenes.make_scene("batch_300k", 3, n=60000, width=640, height=480, frames=8, tile=tile,
                           freqs_hz=FREQS[:n_freq])
    r = gftorf.Renderer(sc.n, sc.frames, sc.width, sc.height, n_freq, 4, tile=tile,
                        pixels_per_thread=ppt)
    p = gftorf.params_from_scene(sc)
    cam = (gftorf.frames_from_scene(sc), gftorf.sensor_from_scene(sc),
           gftorf.consts_from_scene(sc))
    bg = torch.as_tensor(sc.bg).to("cuda", torch.float32).contiguous()
    r.fit_capacity(p, *cam, bg)
    r.preprocess(p, *cam)
    out = r.render_fwd(bg)
    r.check()
    dout, grads = torch.randn_like(out), r.alloc_grads(p, bg)
    times = []
    for i in range(12):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        r.composite_bwd(bg, dout, grads)
        e1.record()
        e1.synchronize()
        if i >= 3:
            times.append(e0.elapsed_time(e1) * 1e3)
    return sorted(times)[len(times) // 2]


@pytest.mark.parametrize("tile,ppt", [((32, 32), 0), ((16, 32), 4)])
def test_four_frequencies_cost_little_more_than_three(tile, ppt):
    # 15 sums per record instead of 13 and two more features per pair
    t3, t4 = _backward_us(3, tile, ppt), _backward_us(4, tile, ppt)
    assert t4 <= 1.35 * t3, (t3, t4)


def test_one_pixel_per_thread_on_tall_tiles():
    # the same sums from CTAs of 512 threads instead of 256
    t16, t32 = _backward_us(3, (16, 16), 1), _backward_us(3, (16, 32), 1)
    assert t32 <= 1.2 * t16, (t16, t32)
