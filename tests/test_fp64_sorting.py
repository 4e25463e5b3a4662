"""The FP32 distances that sort out FP64 pairs: the bounds they are compared
with (cut-off and list radius, 2^-18 of the longest box edge to either side) must
hold for every position in the box, or a pair inside its cut-off would be left
out.  A numpy restatement of the device's FP32 arithmetic, on the CPU.
"""
import numpy as np
import pytest


def _float_below(x):
    """A non-negative double with its bits cut off to those of a float."""
    b = np.ascontiguousarray(x, dtype=np.float64).view(np.uint64)
    hi, lo = (b >> np.uint64(32)).astype(np.int64), (b & np.uint64(0xFFFFFFFF)).astype(np.int64)
    h = np.maximum(hi - 0x38000000, 0)
    w = ((h << 3) | (lo >> 29)) & 0xFFFFFFFF
    return w.astype(np.uint32).view(np.float32)


def _float_dist(xi, xj, box):
    r2 = np.zeros(len(xi), dtype=np.float32)
    for c in range(3):
        Lf, iLf = np.float32(box[c]), np.float32(1.0 / box[c])
        dx = _float_below(xj[:, c]) - _float_below(xi[:, c])
        k = np.rint(dx * iLf)
        dx = (dx.astype(np.float64) - np.float64(Lf) * k.astype(np.float64)).astype(np.float32)  # one rounding, as fma
        r2 = (dx.astype(np.float64) ** 2 + r2.astype(np.float64)).astype(np.float32)
    return np.sqrt(r2.astype(np.float64))


@pytest.mark.parametrize("box", [(6.0, 6.0, 6.0), (58.48, 58.48, 58.48), (133.7, 41.3, 9.1), (30000.0, 25000.0, 700.0)])
def test_fp32_distances_stay_within_the_margin(box):
    rng = np.random.default_rng(3)
    box = np.array(box)
    n = 400_000
    xi = rng.random((n, 3)) * box
    # partners at list distances in every direction, many across a face, and some on the faces
    r = rng.uniform(0.3, min(2.2, 0.3 * box.min()), (n, 1))
    u = rng.standard_normal((n, 3))
    xj = np.mod(xi + r * u / np.linalg.norm(u, axis=1, keepdims=True), box)
    xi[:1000] = 0.0
    xj[1000:2000, 0] = np.nextafter(box[0], 0.0)
    xj[xj >= box] = 0.0
    d = xj - xi
    d -= box * np.rint(d / box)
    exact = np.sqrt((d * d).sum(1))
    err = np.abs(_float_dist(xi, xj, box) - exact)
    near = exact < 0.4 * box.min()
    assert near.sum() > 0.9 * n
    # margin 2^-18 of the longest edge; the arithmetic stays well inside it
    assert err[near].max() < 0.5 * 2.0 ** -18 * box.max()

