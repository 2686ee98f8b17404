"""State that a handle keeps between the calls of a training loop."""
import pytest

from tests.gpu_util import GRAD_TOL, grad_rel, make_renderer

pytestmark = pytest.mark.gpu


def _step(rd, dev, cams, d, stream, grads=None, images=None):
    img = rd.forward(dev, cams, images=images, stream=stream)
    return rd.backward(dev, cams, d, grads, stream=stream), img


@pytest.mark.parametrize("attr_res", [1, 3])
@pytest.mark.parametrize("swapped", ["quat", "log_scale", "sh"])
def test_graph_follows_swapped_attribute_arrays(scenes, attr_res, swapped):
    """A captured step whose rotation, scaling or SH array moves to another buffer with other values,
    every other address unchanged: the gradients are the new array's."""
    import torch
    from paper_2503_13961_gb300 import render as R
    sc, cams = scenes.tiny_scene("ico1", noise=0.04, size=(96, 80), r_b=0.03)
    sc = scenes.with_sh(scenes.with_attribute_maps(sc, attr_res, rot_noise=0.3), 2)
    dev = R.scene_to_device(sc)
    gen = torch.Generator(device="cuda").manual_seed(3)
    d = torch.randn((96 * 80, 3), generator=gen, device="cuda")
    other = dict(dev)
    other[swapped] = dev[swapped] + 0.3 * torch.randn(dev[swapped].shape, generator=gen, device="cuda")
    plain = make_renderer(sc, cams)
    want = [_step(plain, x, cams, d, None)[0] for x in (dev, other)]
    assert grad_rel(want[0]["ctrl"].cpu(), want[1]["ctrl"].cpu()) > 10 * GRAD_TOL  # the swap shows
    rd = make_renderer(sc, cams, graph=True)
    grads = {k: torch.empty_like(v) for k, v in want[0].items()}
    img = torch.empty((96 * 80, 3), device="cuda")
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    for x, w in ((dev, want[0]), (other, want[1]), (dev, want[0])):
        _step(rd, x, cams, d, s, grads, img)
        s.synchronize()
        rd.sync_status(stream=s)
        for k, v in w.items():
            assert grad_rel(grads[k].cpu(), v.cpu()) < GRAD_TOL, k
