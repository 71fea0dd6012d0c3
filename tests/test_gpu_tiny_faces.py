"""Faces at the smallest kept area (1e-24 box^2) in boxes far from unit size: the area rule is decided on the
face's FP64 vertices, whatever FP32 says of lines that lie closer together than it resolves.  Needs a GPU."""
import numpy as np
import pytest

from synth import MLP
from tests import parity

pytestmark = pytest.mark.gpu


def triangle_net(a, b, leg, z0, lift):
    """F(x, y, z) = z - z0 as one unit that is active everywhere, and three units without a weight in F whose
    planes cut the face z = z0 into seven: x = a, y = b and x + y = a + b + leg bound a right triangle."""
    r = np.sqrt(0.5)
    W = np.array([[0.0, 0.0, 1.0], [1.0, 0.0, 0.0], [0.0, 1.0, 0.0], [r, r, 0.0]])
    c = np.array([lift, -a, -b, -r * (a + b + leg)])
    return MLP([W], [c], np.array([1.0, 0.0, 0.0, 0.0]), -lift - z0, name="tiny_triangle")


def placed(box, leg, count):
    rng = np.random.default_rng(11)
    for _ in range(count):
        a, b, z0 = rng.uniform(0.05, 0.2, 3) * box
        yield triangle_net(a, b, leg, z0, 8.0 * box), np.array([[a + 0.3 * box, b + 0.4 * box, z0 - 0.1 * box]])


# legs on both sides of the line: an area of half the smallest kept one, and of eight times it
@pytest.mark.parametrize("precision,schedule", [("fp64", "persistent"), ("fp64", "levels"), ("mixed", "persistent"),
                                                ("sliced", "levels")])
@pytest.mark.parametrize("box", [1e3, 1e5])
@pytest.mark.parametrize("times,faces", [(0.5, 6), (8.0, 7)], ids=["below", "above"])
def test_smallest_area(oracle_mod, times, faces, box, precision, schedule):
    import paper_2106_10031_gb300 as am
    leg = np.sqrt(2.0 * times * 1e-24) * box             # area leg^2 / 2
    up = np.array([[0.0, 0.0, 1.0]])
    with am.Mesher(max_cells=1 << 8, max_neurons=64, max_width=8) as m:
        for mlp, o in placed(box, leg, 24):
            net, ref = oracle_mod.mesh_from_rays(mlp, o, up, 0.2 * box, box=box)
            assert len(ref.faces) == faces
            m.reset()
            m.release_nets()
            nid = m.load_mlp(mlp)
            m.seed(nid, o, up, 0.2 * box)
            m.march(box=box, precision=precision, schedule=schedule)
            # coordinates are of the order of the box, the vertices of the triangle 1e-12 of it apart
            parity.compare(ref, m.get_mesh(nid), mlp.N, rtol=1e-9)
