"""The loss kernel's strips (54 output columns) and segments of rows (12, 20, .. rows by the launch's
size) at their edges, against the FP64 oracle with the bounds of the other loss tests: widths around one
and two strips, views of one row or column, heights around a segment and longer than the longest, and more
views than one launch takes (112)."""
import pytest

from tests.test_gpu_loss import LOSS_TOL, _check_grad, _renderer, _run, _views

pytestmark = pytest.mark.gpu

SIZES = [
    [(53, 11), (54, 12), (55, 13)],
    [(108, 20), (109, 21), (64, 28)],
    [(1, 300), (300, 1), (59, 5)],
    [(20, 1100)],
    [(9 + k % 5, 7 + k % 3) for k in range(115)],
]


@pytest.mark.parametrize("sizes", SIZES, ids=lambda s: "+".join(f"{w}x{h}" for w, h in s[:3]))
def test_strip_and_segment_edges(sizes):
    from oracle import loss as L
    pairs, cams = _views(len(sizes), sizes)
    rd = _renderer()
    grads, total = _run(rd, pairs, cams, 0.2)
    want = 0.0
    for (img, gt), g in zip(pairs, grads):
        want += L.loss(img, gt, 0.2)
        _check_grad(g, L.loss_grad(img, gt, 0.2))
    assert abs(total - want) <= LOSS_TOL * abs(want)
    rd.close()
