"""The loss kernel's strips at the widths where their number changes (64 columns of partials, the first and
the last strip own 5 columns more than the 54 of the others), segments of 4 rows in small calls, rows above
the view that no segment reads, and segments of 100 rows (15 groups, every slot of the ring of image rows)
in a batch that fills the chip: every gradient value against the FP64 oracle, with the bounds of the other loss
tests."""
import pytest

from tests.test_gpu_loss import LOSS_TOL, _check_grad, _renderer, _run, _views

pytestmark = pytest.mark.gpu

SIZES = {
    "one-two-strips": [(59, 9), (63, 40), (64, 41), (65, 43), (66, 5)],
    "two-three-strips": [(117, 30), (118, 31), (119, 29), (172, 10), (173, 11)],
    "short": [(64, h) for h in (1, 2, 3, 4, 5, 8, 9, 10, 11, 14, 15)],
    "small": [(64, 64)],
    "segments-of-36": [(64, 64)] * 60 + [(64, 35), (64, 36), (64, 37), (64, 72)],
    "segments-of-100": [(64, 300)] * 94 + [(64, h) for h in (99, 100, 101, 199, 200, 201)],
}


@pytest.mark.parametrize("name", SIZES)
def test_strips_and_segments(name):
    from oracle import loss as L
    pairs, cams = _views(len(name), SIZES[name])
    rd = _renderer()
    grads, total = _run(rd, pairs, cams, 0.2)
    want = 0.0
    for (img, gt), g in zip(pairs, grads):
        want += L.loss(img, gt, 0.2)
        _check_grad(g, L.loss_grad(img, gt, 0.2))
    assert abs(total - want) <= LOSS_TOL * abs(want)
    rd.close()


def test_black_pair_and_one_bright_pixel():
    """Images that the zero padding continues: equal black images have no gradient beyond rounding."""
    import numpy as np
    from oracle import loss as L
    sizes = [(70, 33), (70, 33)]
    cams = [{"width": w, "height": h} for w, h in sizes]
    pairs = [tuple(np.zeros((h, w, 3), np.float32) for _ in range(2)) for w, h in sizes]
    pairs[1][0][0, 0] = 1.0
    rd = _renderer()
    grads, _ = _run(rd, pairs, cams, 0.2)
    # dl/dx = lam / N (F a + 2 x F b + y F c): a, b, c up to 1 / C2 = 1.1e3, their sum to rounding of 2^-24 each
    assert np.abs(grads[0]).max() <= 0.2 / (3 * 70 * 33) * 1.1e3 * 16 * 2.0 ** -24
    want = L.loss_grad(*pairs[1], 0.2)
    assert np.abs(grads[1] - want).max() <= 1e-3 * np.abs(want).max()
    rd.close()
