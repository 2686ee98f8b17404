"""Gradients do not depend on the tile size or on how views are batched, where the records of a call
(Gaussians and boundary points) outnumber what the counting launch takes in one round of its grid or the
per-primitive sums change form."""
import pytest

from tests.gpu_util import GRAD_TOL, grad_rel, make_renderer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("records", [0, 1])  # default capacity; 1: every block re-walks its tile list
def test_gradients_of_a_large_batch_agree(scenes, records):
    import torch
    from paper_2503_13961_gb300 import render as R
    sc = scenes.config_scene(3)[0]
    cams = [scenes.look_at_camera((4.0, 0.3 * k, 0.5), (0, 0, 0), 1024, 1024) for k in range(2)]
    dev = R.scene_to_device(sc)
    d = torch.randn((2 << 20, 3), generator=torch.Generator(device="cuda").manual_seed(6), device="cuda")
    want = None
    for tile in (16, 8, 32):
        rd = make_renderer(sc, cams, tile=tile, max_blend_pairs=records)
        rd.forward(dev, cams)
        got = rd.backward(dev, cams, d)
        rd.sync_status()
        c = rd.counts()
        assert c["F"] + c["Nb"] > 4 * 152 * 768  # a round takes four records per thread
        assert (c["walked_blocks"] > 0) == (records == 1)
        want = want or {k: v.cpu() for k, v in got.items()}
        for k, v in want.items():
            assert grad_rel(got[k].cpu(), v) < GRAD_TOL, (tile, k)
        rd.close()


@pytest.mark.parametrize("degree", [1, 2])
def test_gradients_of_a_batch_are_the_sum_of_its_views(scenes, degree):
    """A batch above the size where the per-primitive sums change form, against its views one at a time."""
    import torch
    from paper_2503_13961_gb300 import render as R
    mesh = scenes._Mesh()
    mesh.add_object(("sphere", (0, 0, 0), 1.0), scenes.icosphere_tris(40))
    sc = scenes.make_scene(mesh, degree, 0.0, 0, gauss_scale=0.004)
    cams = [scenes.look_at_camera((3.0, 0.3 * k, 0.5), (0, 0, 0), 1024, 1024) for k in range(4)]
    px = 1024 * 1024
    assert 36 < 4 * px / len(sc["ctrl"]) < 160 and 4 * px > 3 << 20 > px
    dev = R.scene_to_device(sc)
    d = torch.randn((4 * px, 3), generator=torch.Generator(device="cuda").manual_seed(7), device="cuda")
    rd = make_renderer(sc, cams)
    rd.forward(dev, cams)
    got = rd.backward(dev, cams, d)
    want = None
    for k, c in enumerate(cams):
        rd.forward(dev, [c])
        g = rd.backward(dev, [c], d[k * px:(k + 1) * px])
        want = g if want is None else {n: want[n] + g[n] for n in g}
    rd.sync_status()
    for n, v in want.items():
        assert grad_rel(got[n].cpu(), v.cpu()) < GRAD_TOL, n
    rd.close()
