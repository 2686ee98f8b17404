"""Tile lists that leave the common word form of the sort: depths that tie (exact words while depth and index
ranges fit 31 bits together, full keys beyond), and boundary lists whose primitive and index ranges do
not fit. Keys are integers: every list has to hold its keys once, in ascending order."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [2, 33, 127, 128, 129, 300, 511, 512, 513, 1023, 1024, 1025, 2047, 2048, 2049, 4095, 4096, 4097, 9000]


def _bits(x):
    return int(x).bit_length()


def _depths(kind, n, rng):
    ulps = lambda k: (np.float32(4.25).view(np.int32) + k.astype(np.int32)).view(np.float32)
    if kind == "near":      # a surface at one depth up to rounding
        return ulps(rng.integers(0, 3, n))
    if kind == "far":       # three surfaces far apart: ties, and a range that takes the word
        return rng.choice(np.array([0.5, 4.25, 90.0], np.float32), n)
    # the widest depth range whose exact words fit 31 bits, and one bit more; three depths, so ties either way
    span_bits = 31 - 5 - _bits(n - 1) + (kind == "beyond")
    return ulps(rng.choice(np.array([0, 1, (1 << min(span_bits, 23)) - 1]), n))


@pytest.mark.parametrize("kind", ["near", "far", "widest", "beyond"])
def test_tied_depths_at_every_size(scenes, kind):
    from paper_2503_13961_gb300 import render as R
    cap = max(SIZES)
    rd = R.Renderer(degree=2, max_prims=1, max_views=1, max_pixels=cap, max_pairs=4 * cap, max_boundary_pairs=1024,
                    tile_size=32)
    for n in SIZES:
        g = scenes.random_gaussians(n, 32, 32, n)
        g["depth"] = np.ascontiguousarray(_depths(kind, n, np.random.default_rng(n)), np.float32)
        out = rd.bin_sort(g, 32, 32)
        rd.sync_status()
        want = np.sort((((g["depth"].view(np.uint32).astype(np.uint64) << np.uint64(5)) | np.uint64(16))
                        << np.uint64(27)) | np.arange(n, dtype=np.uint64))
        assert out["ranges"].tolist() == [0, n]
        assert np.array_equal(out["keys"], want), (kind, n)
    rd.close()


def _wall(scenes, n, stride):
    """n x n squares of two triangles at one depth in random order, every stride-th primitive; the others
    lie behind the camera."""
    tris = np.asarray(scenes.grid_quad_tris((0, -2.0, -2.0), (0, 4.0, 0), (0, 0, 4.0), n), np.float32)
    tris = tris[np.random.default_rng(0).permutation(len(tris))]
    M = len(tris) * stride
    ctrl = np.full((M, 3, 3), 50.0, np.float32)
    ctrl[::stride] = tris
    quat = np.zeros((M, 4), np.float32)
    quat[:, 0] = 1.0
    return {"degree": 1, "ctrl": ctrl, "color": np.full((M, 3, 3), 0.5, np.float32),
            "opacity": np.full(M, 0.8, np.float32), "r_b": np.full(M, 0.0, np.float32),
            "log_scale": np.full((M, 3), np.log(0.004), np.float32), "quat": quat, "bg": np.zeros(3, np.float32)}


@pytest.mark.parametrize("r_b", [1e-4, 4e-3, 3e-2])
def test_boundary_lists_of_a_wide_primitive_range(scenes, r_b):
    """The lists of a wall do not depend on how far apart its primitives' numbers are."""
    from paper_2503_13961_gb300 import render as R
    stride, W, H = 256, 600, 400
    cam = scenes.look_at_camera((3.0, 0.0, 0.0), (0, 0, 0), W, H)
    got = []
    for s in (1, stride):
        sc = _wall(scenes, 50, s)
        sc["r_b"][:] = r_b
        rd = R.Renderer(degree=1, max_prims=len(sc["ctrl"]), max_views=1, max_pixels=W * H, max_pairs=16 * W * H,
                        max_boundary_pairs=64 * W * H, tess_level=2, tile_size=16)
        img = rd.forward(R.scene_to_device(sc), [cam])
        rd.sync_status()
        got.append({k: rd.stage(k) for k in ("b_keys", "b_ranges", "g_keys", "g_ranges")} | {"img": img.cpu().numpy()})
        rd.close()
    one, wide = got
    keys, ranges = wide["b_keys"], wide["b_ranges"]
    lists = [keys[a:b] for a, b in zip(ranges[:-1], ranges[1:]) if b > a]
    index = np.uint64(0xffffffff)
    over = sum(_bits((k[-1] >> np.uint64(32)) - (k[0] >> np.uint64(32))) + _bits((k & index).max() - (k & index).min()) > 31
               for k in lists)
    assert over > len(lists) // 2, (over, len(lists))  # what the test is about
    for k in ("b_ranges", "g_ranges", "g_keys", "img"):
        assert np.array_equal(one[k], wide[k]), k
    prim = (one["b_keys"] >> np.uint64(32)) * np.uint64(stride)
    assert np.array_equal((prim << np.uint64(32)) | (one["b_keys"] & index), keys)
    assert all((np.diff(k.astype(np.int64)) > 0).all() for k in lists)
