"""The per-cell path at the edges of its dispatch: layer widths where the compose changes its mapping
(a lane per row and column, two rows per lane, a row per lane; the double-float splits), unit
counts around the 32-bit words and the 32-word chunks of the active list, and faces that the
one-pass polygon and the warp clip meet with few rows and with the box's rows among their edges.  Needs a GPU."""
import numpy as np
import pytest

from synth import geometric_init, tiny_net
from tests import parity

pytestmark = pytest.mark.gpu
X_RAY = np.array([[1.0, 0.0, 0.0]])

WIDTHS = [(1, 2, 3), (7, 8, 9), (15, 16, 17, 5), (31, 32, 33), (63, 64, 65), (127, 128, 129), (130, 255, 256, 257),
          (66, 84, 110), (32, 32, 32), (300, 300, 300, 157)]


def _words(bits):
    n, N = bits.shape
    pad = np.zeros((n, (N + 63) // 64 * 64), dtype=np.uint8)
    pad[:, :N] = bits
    return np.packbits(pad, axis=1, bitorder="little").view(np.uint64)


@pytest.mark.parametrize("widths", WIDTHS, ids=lambda w: "x".join(map(str, w)))
def test_compose_widths(oracle_mod, widths):
    import paper_2106_10031_gb300 as am
    mlp = geometric_init(list(widths), 7, 0.05)
    net = oracle_mod.OracleNet(mlp)
    rng = np.random.default_rng(1)
    S = rng.integers(0, 2, (5, mlp.N)).astype(np.uint8)
    S[0], S[1] = 0, 1                                    # no active unit, every unit
    ref = []
    for s in S:
        A, aF = net.compose(s)
        ref.append(np.vstack([(1.0 - 2.0 * s)[:, None] * A, aF[None, :]]))
    ref = np.asarray(ref)
    with am.Mesher(max_cells=1 << 10, max_neurons=mlp.N, max_width=max(widths)) as m:
        nid = m.load_mlp(mlp)
        r64, _ = m.compose(nid, _words(S), "fp64")
        rdf, edf = m.compose(nid, _words(S), "mixed")
    # FP64 in another order of summation: (n + 4) 2^-53 of the products per layer, far below this
    scale = 1.0 + np.abs(ref).max()
    assert np.abs(r64 - ref).max() <= 1e-12 * scale
    # double-float: within its own bound (and the reference's rounding)
    assert np.all(np.abs(rdf - ref).sum(axis=2) <= edf + 1e-12 * scale)
    assert edf.max() < 1e-3 * scale


@pytest.mark.parametrize("precision,schedule", [("fp64", "persistent"), ("fp64", "levels"), ("mixed", "persistent"),
                                                ("sliced", "levels")])
@pytest.mark.parametrize("make,box", [
    (lambda: tiny_net((4, 4), 4), 1.5),                  # fewer rows than a warp; the box bounds most faces
    (lambda: geometric_init([33, 31], 5, 0.05, recenter=True), 1.5),
    (lambda: geometric_init([17, 9, 40], 6, 0.05, recenter=True), 1.5),
    (lambda: tiny_net((3, 3), 3), 1.5),                  # every face is open
], ids=["4x4", "33x31", "17x9x40", "3x3"])
def test_march_edges(oracle_mod, make, box, precision, schedule):
    import paper_2106_10031_gb300 as am
    mlp = make()
    d = X_RAY
    net, ref = oracle_mod.mesh_from_rays(mlp, np.zeros((1, 3)), d, 2.0, box=box)
    with am.Mesher(max_cells=1 << 16, max_neurons=max(64, mlp.N), max_width=max(mlp.widths)) as m:
        nid = m.load_mlp(mlp)
        m.seed(nid, np.zeros((1, 3)), d, 2.0)
        m.march(box=box, precision=precision, schedule=schedule)
        mesh, st = m.get_mesh(nid), m.stats()
    r = parity.compare(ref, mesh, mlp.N, rtol=1e-5 if precision == "mixed" else 1e-9)
    assert st["faces"] == r["faces"] > 0 and mesh.n_open_faces == ref.open_faces()
    assert mesh.n_open_faces > 0                         # each of these surfaces meets the box


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_one_pass_faces_count_no_cuts(precision):
    # the counter holds cuts applied one by one: several a face without candidates, none for the faces that
    # close in one pass (all but the few that the sequential clip takes)
    import paper_2106_10031_gb300 as am
    mlp = geometric_init([33, 31], 5, 0.05, recenter=True)
    per_cell = {}
    with am.Mesher(max_cells=1 << 16, max_neurons=64, max_width=33) as m:
        nid = m.load_mlp(mlp)
        for candidates in ("none", "nearest"):
            m.reset()
            m.seed(nid, np.zeros((1, 3)), X_RAY, 2.0)
            m.march(precision=precision, candidates=candidates)
            st = m.stats()
            per_cell[candidates] = st["cuts"] / st["cells"]
    assert per_cell["none"] >= 3.0                       # a closed polygon takes three cuts or more
    assert per_cell["nearest"] < 0.5


def _clip(C, aF):
    """The polygon {aF [x; 1] = 0, C [x; 1] <= 0}, cut row by row out of a large square (or None)."""
    n = aF[:3] / np.linalg.norm(aF[:3])
    u = np.cross(n, np.eye(3)[np.argmin(np.abs(n))])
    u /= np.linalg.norm(u)
    w, p0 = np.cross(n, u), -aF[3] / np.linalg.norm(aF[:3]) * n
    P = [p0 + 5.0 * (a * u + b * w) for a, b in ((-1, -1), (1, -1), (1, 1), (-1, 1))]
    for c in C:
        v = [c[:3] @ p + c[3] for p in P]
        P = [q for i in range(len(P)) for q in
             ([P[i - 1] + v[i - 1] / (v[i - 1] - v[i]) * (P[i] - P[i - 1])] if (v[i - 1] <= 0) != (v[i] <= 0) else [])
             + ([P[i]] if v[i] <= 0 else [])]
        if len(P) < 3:
            return None
    return np.array(P)


@pytest.mark.parametrize("precision,schedule", [("fp64", "persistent"), ("mixed", "persistent"), ("sliced", "levels")])
def test_seeds_outside_the_box(oracle_mod, precision, schedule):
    # rays that meet a sphere of radius about 0.6 in a box of half-width 0.45: 16 of 40 seed points lie
    # outside the box, 14 of them on cells without a face in it, two on faces that the box cuts.  The
    # oracle's pivoting starts on the face, so for these two it starts from a point of the cut face.
    import paper_2106_10031_gb300 as am
    mlp, box = geometric_init([32, 32, 32, 32], 21, 0.05), 0.45
    d = np.random.default_rng(3).normal(size=(40, 3))
    d /= np.linalg.norm(d, axis=1)[:, None]
    o = np.zeros((40, 3))
    net, seeds = oracle_mod.OracleNet(mlp), []
    for key, x in oracle_mod.seed_cells(net, o, d, 2.0):
        P = [x] if np.abs(x).max() <= box else _clip(*net.cell_rows(oracle_mod.key_to_state(key, mlp.N), box))
        if P is not None:
            seeds.append((key, np.mean(P, axis=0)))
    assert len(seeds) == 26
    ref = oracle_mod.march(net, seeds, box)
    with am.Mesher(max_cells=1 << 16, max_neurons=mlp.N, max_width=32) as m:
        nid = m.load_mlp(mlp)
        m.seed(nid, o, d, 2.0)
        m.march(box=box, precision=precision, schedule=schedule)
        mesh, st = m.get_mesh(nid), m.stats()
    parity.compare(ref, mesh, mlp.N, rtol=1e-5 if precision == "mixed" else 1e-9)
    assert st["empty_faces"] > 0
