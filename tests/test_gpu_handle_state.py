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


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("records", [0, 512])  # default capacity; 512: most blocks re-walk their tile lists
def test_backward_twice_after_one_forward(scenes, graph, records):
    """Two image gradients taken back through one forward: each backward overwrites the gradients with
    its own, as after a forward of its own."""
    import torch
    from paper_2503_13961_gb300 import render as R
    sc, cams = scenes.tiny_scene("ico1", noise=0.04, size=(96, 80), r_b=0.03)
    sc = scenes.with_sh(sc, 1)
    dev = R.scene_to_device(sc)
    gen = torch.Generator(device="cuda").manual_seed(4)
    ds = [torch.randn((96 * 80, 3), generator=gen, device="cuda") for _ in range(2)]
    plain = make_renderer(sc, cams)
    want = [_step(plain, dev, cams, d, None)[0] for d in ds]
    rd = make_renderer(sc, cams, graph=graph, max_blend_pairs=records)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    for _ in range(2):  # graphs: captured, then replayed
        rd.forward(dev, cams, stream=s)
        for d, w in zip(ds + ds[:1], want + want[:1]):
            got = rd.backward(dev, cams, d, stream=s)
            s.synchronize()
            rd.sync_status(stream=s)
            for k, v in w.items():
                assert grad_rel(got[k].cpu(), v.cpu()) < GRAD_TOL, k


def test_autograd_of_a_retained_graph(scenes):
    import torch
    from paper_2503_13961_gb300 import render as R
    sc, cams = scenes.tiny_scene("ico1", noise=0.04, size=(70, 50), r_b=0.03)
    dev = R.scene_to_device(sc)
    dev["ctrl"].requires_grad_(True)
    img = R.render(make_renderer(sc, cams), dev, cams)
    a = torch.autograd.grad(img.square().sum(), dev["ctrl"], retain_graph=True)[0]
    b = torch.autograd.grad(img.square().sum(), dev["ctrl"])[0]
    assert grad_rel(b.cpu(), a.cpu()) < GRAD_TOL


def test_backward_refuses_a_scene_of_another_form(scenes):
    """The pass over the last forward's records reads maps and SH of the forward's sizes: a scene with the
    same control points and another map resolution or SH degree is refused before any launch."""
    import torch
    from paper_2503_13961_gb300 import render as R
    sc, cams = scenes.tiny_scene("ico1", size=(40, 30))
    forms = [R.scene_to_device(sc), R.scene_to_device(scenes.with_attribute_maps(sc, 3)),
             R.scene_to_device(scenes.with_sh(sc, 2))]
    for f in forms:
        f["ctrl"] = forms[0]["ctrl"]
    rd = make_renderer(sc, cams)
    d = torch.ones((40 * 30, 3), device="cuda")
    for i, f in enumerate(forms):
        rd.forward(f, cams)
        want = rd.backward(f, cams, d)
        for j, other in enumerate(forms):
            if j != i:
                with pytest.raises(RuntimeError, match="differ from the forward"):
                    rd.backward(other, cams, d)
        assert grad_rel(rd.backward(f, cams, d)["ctrl"].cpu(), want["ctrl"].cpu()) < GRAD_TOL
    for attr_res in (0, 1):  # both name maps of one texel
        rd.forward(dict(forms[0], attr_res=1 - attr_res), cams)
        rd.backward(dict(forms[0], attr_res=attr_res), cams, d)
    rd.sync_status()


def test_loss_right_behind_the_forward(scenes):
    """The loss starts while the forward that writes its images drains: its gradient is that of the
    finished images, two scenes in turn through one buffer."""
    import torch
    from paper_2503_13961_gb300 import render as R
    sc, cams = scenes.tiny_scene("ico1", noise=0.04, size=(96, 80), r_b=0.03)
    dark = dict(sc, color=sc["color"] * 0.25)
    rd = make_renderer(sc, cams)
    devs = [R.scene_to_device(x) for x in (sc, dark)]
    gt = torch.rand((96 * 80, 3), generator=torch.Generator(device="cuda").manual_seed(5), device="cuda")
    img, d = torch.empty_like(gt), [torch.empty_like(gt) for _ in range(40)]
    want = []
    for dev in devs:
        rd.forward(dev, cams, images=img)
        torch.cuda.synchronize()
        want.append(rd.l2_dssim_loss_grad(img, gt, cams).clone())
    torch.cuda.synchronize()
    for i in range(40):
        rd.forward(devs[i % 2], cams, images=img)
        rd.l2_dssim_loss_grad(img, gt, cams, d_images=d[i])
    torch.cuda.synchronize()
    for i in range(40):
        assert torch.equal(d[i], want[i % 2]), i


def test_autograd_of_two_renders_through_one_renderer(scenes):
    """Two views rendered one after the other, their losses added: every backward takes its own view's
    records, whichever forward came last."""
    import torch
    from paper_2503_13961_gb300 import render as R
    sc, _ = scenes.tiny_scene("ico1", noise=0.04, size=(70, 50), r_b=0.03)
    cams = [[scenes.look_at_camera(eye, (0, 0, 0), 70, 50)] for eye in ((4.0, 0.0, 0.0), (0.0, 3.0, 1.0))]
    dev = R.scene_to_device(sc)
    dev["ctrl"].requires_grad_(True)
    rd = make_renderer(sc, cams[0])
    alone = [torch.autograd.grad(R.render(rd, dev, c).square().sum(), dev["ctrl"])[0].cpu() for c in cams]
    assert grad_rel(alone[0], alone[1]) > 10 * GRAD_TOL
    for order in ((0, 1), (1, 0)):
        imgs = [R.render(rd, dev, c) for c in cams]
        got = [None, None]
        for k in order:
            got[k] = torch.autograd.grad(imgs[k].square().sum(), dev["ctrl"])[0]
        assert all(grad_rel(got[k].cpu(), alone[k]) < GRAD_TOL for k in range(2)), order
    both = torch.autograd.grad(sum(R.render(rd, dev, c).square().sum() for c in cams), dev["ctrl"])[0]
    assert grad_rel(both.cpu(), alone[0] + alone[1]) < GRAD_TOL
    rd.sync_status()
