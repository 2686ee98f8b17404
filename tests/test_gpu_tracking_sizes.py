"""The tracking kernels and the split at the sizes where their work items end: edge magnitudes in strips
of 30 columns and segments of 8 or 32 rows (views of one row or column, more than 200 views per call,
a batch of more than 8 M pixels), the back-projection of edges in groups of 128 pixels, and splits of fewer parents
than a block of 8 takes, into outputs that are not 16-byte aligned. Bounds as in the other split tests:
edges 1e-5 relative + 2e-3 against the FP64 oracle, sums 1e-5, counts and copies exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EDGE_SIZES = [
    [(1, 1), (1, 9), (29, 1), (30, 7), (31, 8), (60, 9), (61, 33)],
    [(5 + k % 7, 3 + k % 4) for k in range(205)],
    [(2900, 2900)],
]


@pytest.mark.parametrize("sizes", EDGE_SIZES, ids=["ragged", "many", "large"])
def test_edge_magnitude_sizes(sizes):
    import torch
    from oracle import split as S
    from paper_2503_13961_gb300 import render as R
    rng = np.random.default_rng(sizes[0][0] + len(sizes))
    imgs = [rng.uniform(0, 1, (h, w, 3)).astype(np.float32) for w, h in sizes]
    flat = torch.as_tensor(np.concatenate([i.reshape(-1, 3) for i in imgs]), device="cuda")
    got = R.edge_magnitude(flat, [{"width": w, "height": h} for w, h in sizes]).cpu().numpy().astype(np.float64)
    off = 0
    for img in imgs:
        want = S.edge_magnitude(img).ravel()
        assert np.all(np.abs(got[off: off + want.size] - want) <= 1e-5 * want + 2e-3)
        off += want.size


@pytest.mark.parametrize("size", [(127, 1), (128, 1), (43, 3), (200, 150)])
def test_edge_prior_and_visibility_of_ragged_views(scenes, size):
    import torch
    from paper_2503_13961_gb300 import render as R
    sc, _ = scenes.tiny_scene("ico1", noise=0.04)
    cams = scenes.make_views(np.random.default_rng(size[0]), [size, (7, 5), size], 2.5, 4.0)
    rd = R.Renderer(degree=2, max_prims=20, max_views=3, max_pixels=2 * size[0] * size[1] + 35, max_pairs=1 << 22,
                    max_boundary_pairs=1 << 22)
    dev = R.scene_to_device(sc)
    rd.forward(dev, cams)
    rd.sync_status()
    ids = rd.stage("id")
    edges = torch.rand(len(ids), device="cuda", generator=torch.Generator(device="cuda").manual_seed(3))
    total, count = rd.edge_prior(edges, 20)
    seen, _ = rd.visibility(20)
    e = edges.cpu().numpy().astype(np.float64)
    fg = ids >= 0
    want = np.bincount(ids[fg], e[fg], 20)
    assert np.array_equal(count.cpu().numpy(), np.bincount(ids[fg], minlength=20))
    assert np.all(np.abs(total.cpu().numpy() - want) <= 1e-5 * want)
    views, off = np.zeros(20, int), 0
    for c in cams:
        n = c["width"] * c["height"]
        v = ids[off: off + n]
        views[np.unique(v[v >= 0])] += 1
        off += n
    assert np.array_equal(seen.cpu().numpy(), views)


@pytest.mark.parametrize("degree", [1, 2, 3, 4])
def test_split_of_few_parents_into_unaligned_outputs(scenes, degree):
    """A block's tail, and scalar stores: the same pieces as into aligned outputs, bit for bit, and the
    selected parent's corners in place."""
    import ctypes
    import torch
    from paper_2503_13961_gb300 import _abi
    from paper_2503_13961_gb300 import render as R
    sc = scenes.mixed_shapes_scene(21, degree)
    dev = R.scene_to_device(sc)
    sel = torch.tensor([20, 3, 3, 0, 7, 11, 19, 1, 2, 5], dtype=torch.int32, device="cuda")
    n = len(sel)
    want = R.subdivide(dev, sel)
    ctrl = dev["ctrl"].cpu().numpy()
    got_c = want["ctrl"].cpu().numpy()
    for k, m in enumerate(sel.tolist()):
        assert np.array_equal(got_c[4 * k, 0], ctrl[m, 0])                       # U corner of the U piece
        assert np.array_equal(got_c[4 * k + 2, -1], ctrl[m, -1])                 # W corner of the W piece
    buf = {k: torch.zeros(want[k].numel() + 1, device="cuda") for k in R.SCENE_KEYS}
    pr = _abi.Prims(*(buf[k].data_ptr() + 4 if k in buf else None for k in _abi.PRIMS_KEYS))
    s = R._scene_struct(dev)
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert _abi.load().bgt_subdivide(degree, ctypes.byref(s), ctypes.c_void_p(sel.data_ptr()), n, ctypes.byref(pr),
                                     st) == 0
    torch.cuda.synchronize()
    for k in R.SCENE_KEYS:
        assert torch.equal(buf[k][1:].view(want[k].shape), want[k]), k
