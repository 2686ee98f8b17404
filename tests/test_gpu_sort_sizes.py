"""The per-tile sort at the sizes where it changes form (runs of 32, 64, 128, 256 and 512 words per
warp, two merged runs, the block's quarters, the block's merged runs beyond 4096 keys, the radix sort
beyond 32768) and on depths that need
each of its forms: spread depths, ties, depths closer than the words resolve, all equal (the index
decides), and a range too wide for 32-bit words. Keys are integers: the list has to hold every Gaussian
once, in ascending key order."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 31, 32, 33, 64, 65, 128, 129, 256, 257, 511, 512, 513, 700, 1023, 1024, 1025, 1500, 2047, 2048, 2049,
         3000, 4095, 4096, 4097, 5000]


def _depths(kind, n, rng):
    if kind == "spread":
        return rng.uniform(0.3, 60.0, n)
    if kind == "ties":
        return rng.choice(rng.uniform(2.0, 6.0, max(1, n // 3)), n)
    if kind == "close":  # neighbouring floats, and one far away that takes the words' upper bits
        d = np.float32(3.0) + np.arange(n, dtype=np.float32) * np.float32(2.4e-7)
        d = rng.permutation(d)
        d[0] = 900.0
        return d
    if kind == "equal":
        return np.full(n, 4.25)
    return 10.0 ** rng.uniform(-20, 20, n)  # "wide"


@pytest.mark.parametrize("kind", ["spread", "ties", "close", "equal", "wide"])
def test_one_tile_lists_of_every_size(scenes, kind):
    from paper_2503_13961_gb300 import render as R
    cap = max(SIZES)
    rd = R.Renderer(degree=2, max_prims=1, max_views=1, max_pixels=cap, max_pairs=4 * cap, max_boundary_pairs=1024,
                    tile_size=32)
    for n in SIZES:
        rng = np.random.default_rng(n)
        g = scenes.random_gaussians(n, 32, 32, n)
        g["depth"] = np.ascontiguousarray(_depths(kind, n, rng), np.float32)
        out = rd.bin_sort(g, 32, 32)
        rd.sync_status()
        keys = out["keys"]
        assert out["ranges"].tolist() == [0, n] and len(keys) == n, n
        want = np.sort((((g["depth"].view(np.uint32).astype(np.uint64) << np.uint64(5)) | np.uint64(16))
                        << np.uint64(27)) | np.arange(n, dtype=np.uint64))
        assert np.array_equal(keys, want), (kind, n)
    rd.close()


# lists of a block's merged runs of up to 4096 words (two to eight runs, one to three merge passes, their edges)
# and the radix sort beyond
LONG = [8191, 8192, 8193, 12289, 16385, 20481, 30000, 32767, 32768, 32769]


@pytest.mark.parametrize("kind", ["spread", "ties", "close", "equal", "wide"])
def test_one_tile_lists_of_merged_runs(scenes, kind):
    from paper_2503_13961_gb300 import render as R
    cap = max(LONG)
    rd = R.Renderer(degree=2, max_prims=1, max_views=1, max_pixels=cap, max_pairs=2 * cap, max_boundary_pairs=1024,
                    tile_size=32)
    for n in LONG:
        g = scenes.random_gaussians(n, 32, 32, n)
        g["depth"] = np.ascontiguousarray(_depths(kind, n, np.random.default_rng(n)), np.float32)
        out = rd.bin_sort(g, 32, 32)
        rd.sync_status()
        want = np.sort((((g["depth"].view(np.uint32).astype(np.uint64) << np.uint64(5)) | np.uint64(16))
                        << np.uint64(27)) | np.arange(n, dtype=np.uint64))
        assert out["ranges"].tolist() == [0, n]
        assert np.array_equal(out["keys"], want), (kind, n)
    rd.close()


@pytest.mark.parametrize("size", [200, 300, 420])
def test_boundary_lists_of_merged_runs(scenes, size):
    """Boundary radii larger than the image: every tile lists every boundary point."""
    from paper_2503_13961_gb300 import render as R
    sc = scenes.config_scene(2, r_b=20.0)[0]
    cam = scenes.look_at_camera((4.0, 0.0, 0.0), (0, 0, 0), size, size)
    rd = R.Renderer(degree=2, max_prims=2000, max_views=1, max_pixels=size * size, max_boundary_pairs=1 << 22,
                    tile_size=32)
    rd.forward(R.scene_to_device(sc), [cam])
    rd.sync_status()
    prim = np.ascontiguousarray(rd.stage("bnd")).view(np.int32).reshape(-1, 8)[:, 1].astype(np.uint64)
    n = len(prim)
    assert n > 4096
    want = np.sort((prim << np.uint64(32)) | np.arange(n, dtype=np.uint64))
    keys, ranges = rd.stage("b_keys"), rd.stage("b_ranges")
    assert np.array_equal(ranges, np.arange(((size + 31) // 32) ** 2 + 1) * n)
    assert np.array_equal(keys.reshape(-1, n), np.broadcast_to(want, (len(ranges) - 1, n)))
    rd.close()
