"""I_id, boundary set and the compaction of the foreground pixels at the sizes where they can go wrong:
pixel totals around the block of 2048 pixels and the warp chunk of 256, views that end inside a chunk,
one-pixel and one-row views, more primitives than pixels, and rects far apart inside a warp (the tile
counts). Everything compared is an integer decision, so it has to be equal: I_id to the oracle's raster,
the Gaussians' and boundary points' pixels to the foreground and the 4-neighbour boundary of that I_id in
pixel order, and the tile counts to the sorted lists' rects."""
import numpy as np
import pytest

from tests.gpu_util import make_renderer

pytestmark = pytest.mark.gpu

SIZES = [
    [(23, 89)],                                   # 2047 pixels
    [(64, 32)],                                   # 2048
    [(683, 3)],                                   # 2049
    [(255, 1), (1, 1), (1, 257), (300, 2)],       # views ending inside a chunk
    [(5, 7)] * 70,                                # many views per chunk
    [(1600, 40)],                                 # rows longer than a chunk; warps that wrap to the next row
    [(17, 240), (240, 17), (33, 62)],
]


@pytest.mark.parametrize("tile", [8, 16, 32])
@pytest.mark.parametrize("sizes", SIZES, ids=lambda s: "+".join(f"{w}x{h}" for w, h in s[:3]))
def test_ids_boundary_and_compaction(oracle, scenes, sizes, tile):
    from paper_2503_13961_gb300 import render as R
    sc, _ = scenes.tiny_scene("ico1", noise=0.04, r_b=0.03)
    rng = np.random.default_rng(len(sizes) * 1000 + sizes[0][0])
    cams = scenes.make_views(rng, sizes, 2.5, 4.0)
    rd = make_renderer(sc, cams, tile=tile, pairs_per_px=256)  # Gaussians of ~100 px in the wide view
    rd.forward(R.scene_to_device(sc), cams)
    rd.sync_status()
    ids, counts = rd.stage("id"), rd.counts()
    uv, gauss, bnd = rd.stage("uv"), rd.stage("gauss"), rd.stage("bnd")
    want_g, want_b, off = [], [], 0
    for c in cams:
        W, H = c["width"], c["height"]
        ref = np.asarray(oracle.raster(sc, c)[0]).reshape(H, W)
        got = ids[off: off + W * H].reshape(H, W)
        assert np.array_equal(got, ref)
        differ = np.zeros((H, W), bool)
        differ[:, 1:] |= got[:, 1:] != got[:, :-1]
        differ[:, :-1] |= got[:, 1:] != got[:, :-1]
        differ[1:] |= got[1:] != got[:-1]
        differ[:-1] |= got[1:] != got[:-1]
        for out, m in ((want_g, got >= 0), (want_b, (got >= 0) & differ)):
            y, x = np.nonzero(m)
            out.append(np.stack([x | (y << 16), got[m], off + y * W + x], 1))
        off += W * H
    want_g, want_b = np.concatenate(want_g), np.concatenate(want_b)
    assert counts["F"] == len(want_g) and counts["Nb"] == len(want_b)
    assert np.array_equal(gauss.view(np.int32)[:, 6:8], want_g[:, :2])
    assert np.array_equal(bnd.view(np.int32)[:, 0], want_b[:, 2])
    assert np.array_equal(bnd.view(np.int32)[:, 1], want_b[:, 1])
    assert not uv[ids < 0].any() and (uv[ids >= 0] >= -1e-3).all() and (uv[ids >= 0].sum(1) <= 1.001).all()
    # every counted (Gaussian, tile) pair was emitted once: the lists hold distinct keys of all Gaussians
    ranges, keys = rd.stage("g_ranges"), rd.stage("g_keys")
    assert ranges[-1] == counts["K"] == len(keys)
    index = (keys & np.uint64((1 << 27) - 1)).astype(np.int64)
    tile_of = np.repeat(np.arange(len(ranges) - 1), np.diff(ranges))
    assert len(np.unique(tile_of * (1 << 27) + index)) == len(keys)
    assert len(np.unique(index)) == len(want_g)


def test_more_primitives_than_pixels(oracle, scenes):
    """The per-primitive work of the I_id pass when the pixels fill one block and the primitives many."""
    from paper_2503_13961_gb300 import render as R
    sc, _ = scenes.config_scene(2)[:2]
    cams = [scenes.look_at_camera((4.0, 0.3, 0.1), (0, 0, 0), 20, 11)]
    rd = make_renderer(sc, cams, pairs_per_px=64)
    img = rd.forward(R.scene_to_device(sc), cams)
    rd.sync_status()
    ref = oracle.render(sc, cams[0])
    stable = (ref["flags"] & oracle.FWD_UNSTABLE) == 0
    err = np.abs(img.view(11, 20, 3).cpu().numpy() - ref["image"])[stable]
    assert err.max() < 1e-4  # the images' bound everywhere
