"""Two contexts of different sizes alive in one process: each keeps working whatever sizes of nets the
other was made for (the kernels are shared, their shared memory is sized per context).  Needs a GPU."""
import numpy as np
import pytest

from synth import sphere_net, trigger_points
from tests import parity

pytestmark = pytest.mark.gpu
RAY = (np.zeros((1, 3)), np.array([[1.0, 0.0, 0.0]]))


def everything(m, nid, mlp):
    """Every kernel whose shared memory is sized by the context: composes, triggers and marches."""
    rng = np.random.default_rng(0)
    bits = rng.integers(0, 2, (3, (mlp.N + 63) // 64 * 64), dtype=np.uint8)
    bits[:, mlp.N:] = 0
    keys = np.packbits(bits, axis=1, bitorder="little").view(np.uint64)
    out = [m.compose(nid, keys, p)[0] for p in ("fp64", "mixed", "tensor")]
    pts = trigger_points(64, 3)
    m.reset()
    out.append(np.asarray(m.seed_pairs(nid, pts, 8)[2]))
    m.reset()
    out.append(np.asarray(m.seed_sphere_trace(nid, pts[:4])[1]))
    meshes = []
    for precision, schedule in (("fp64", "persistent"), ("mixed", "persistent"), ("fp64", "levels"), ("mixed", "levels")):
        m.reset()
        m.seed(nid, *RAY)
        m.march(precision=precision, schedule=schedule)
        meshes.append(parity.gpu_faces(m.get_mesh(nid)))
    return out, meshes


@pytest.mark.parametrize("first", [4096, 64], ids=["large-first", "small-first"])
def test_two_sizes_alive(first):
    import paper_2106_10031_gb300 as am
    second = 64 + 4096 - first
    mlp = sphere_net(seed=5, width=16, depth=3)
    with am.Mesher(max_cells=1 << 14, max_neurons=first, max_width=min(first, 512)) as a:
        na = a.load_mlp(mlp)
        alone, meshes = everything(a, na, mlp)
        with am.Mesher(max_cells=1 << 14, max_neurons=second, max_width=min(second, 512)) as b:
            nb = b.load_mlp(mlp)
            for m, nid in ((a, na), (b, nb), (a, na)):
                got, faces = everything(m, nid, mlp)
                for x, y in zip(alone, got):
                    assert np.array_equal(x, y, equal_nan=True)
                for x, y in zip(meshes, faces):
                    assert {k: f[0] for k, f in x.items()} == {k: f[0] for k, f in y.items()}
        again, _ = everything(a, na, mlp)
        assert all(np.array_equal(x, y, equal_nan=True) for x, y in zip(alone, again))
