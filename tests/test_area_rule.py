"""The FP32 area test of a face (the triangle of three of its vertices, against a bound on every rounding),
restated in numpy: whatever it calls clear of the smallest kept area, the FP64 rule keeps."""
import numpy as np
import pytest

F = np.float32
U = F(5.9604645e-8)


def clear(p, q, r, box):
    """am_block.cuh's area_clear on (n, 3) FP64 vertices rounded to FP32."""
    p, q, r = (np.asarray(v, dtype=np.float32) for v in (p, q, r))
    a, b = q - p, r - p
    c = np.abs(np.stack([a[:, (i + 1) % 3] * b[:, (i + 2) % 3] - a[:, (i + 2) % 3] * b[:, (i + 1) % 3] for i in range(3)])).max(0)
    s = np.abs(a).sum(1, dtype=np.float32) + np.abs(b).sum(1, dtype=np.float32)
    X = np.abs(np.stack([p, q, r])).max((0, 2))
    amin = np.maximum(F(2e-24) * F(box) * F(box) * F(1.0001), F(1e-30))
    return c > F(12.0) * U * X * s + amin


@pytest.mark.parametrize("box", [1e-4, 1.5, 1e3, 1e6])
def test_clear_faces_are_kept(box):
    rng = np.random.default_rng(5)
    n = 200_000
    p = rng.uniform(-1.0, 1.0, (n, 3)) * box * 10.0 ** rng.uniform(-6, 0, (n, 1))
    a = rng.normal(size=(n, 3)) * box * 10.0 ** rng.uniform(-13, 0, (n, 1))
    # slivers: the third vertex near the first side's line, at every distance down to rounding
    b = a * rng.uniform(-2, 2, (n, 1)) + rng.normal(size=(n, 3)) * box * 10.0 ** rng.uniform(-16, 0, (n, 1))
    q, r = p + a, p + b
    twice = np.linalg.norm(np.cross(q - p, r - p), axis=1)
    ok = clear(p, q, r, box)
    assert np.all(twice[ok] > 2e-24 * box * box)
    # and it is of use: a triangle of a thousandth of the box, a tenth as high as long, is clear
    t = np.array([[0.3, 0.2, 0.1]]) * box
    assert clear(t, t + [[1e-3 * box, 0, 0]], t + [[5e-4 * box, 1e-4 * box, 0]], box).all()
