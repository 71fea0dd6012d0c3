"""Performance cases of the analytic-marching library: what its users have it do, by size.

A case is a dict of plain values.  ``prepare`` makes what a program holds before the call (a context
with its nets loaded, trigger points, activation patterns, training samples), ``run`` makes one
pass through the public entry points and returns what they compute, ``work`` the bytes and flops
that pass cannot do without, ``exact`` the same outputs from plain numpy / torch in 64 bits.

Kinds:
  mesh     trigger, march and take the mesh of one net or of several nets of one context
  compose  the affine rows of given activation patterns (device arrays in and out)
  trigger  seed cells alone, from random pairs of samples or by sphere tracing
  train    Adam steps of the learned constraint proposal

The march discovers faces in no fixed order, so a mesh is returned in a reproducible one: small
meshes on the host through ``canonicalize``, large ones on the device by a hash of the face keys.
"""
import copy
import ctypes as C
import functools
import math
import zlib

import numpy as np
import torch

import paper_2106_10031_gb300 as am
from paper_2106_10031_gb300 import mesher
from synth import nets as synth

BOX = 1.5            # the clip box of every march
REACH = 1.4          # every shape below closes inside this radius, where its trigger rays end
PAIRS = 1024         # segments of the random-pair trigger of the large meshes (16 samples for each)


# ------------------------------------------------------------------------------------------
# the cases


def _mesh(name, arch, widths, precision, seeding="ray", candidates="nearest", out="device", latent=0, skip=0):
    named = {"name": name} if name else {}
    return named | {"kind": "mesh", "arch": arch, "widths": widths, "precision": precision, "seeding": seeding,
                    "candidates": candidates, "out": out, "latent": latent, "skip": skip}


def listed():
    return [
        # the smallest call: a hand-built convex polytope (126 faces), default precision, exported
        # from the host in canonical order; launch and host latency
        _mesh("mesh_polytope12", "polytope", "12x6x3x2", "fp64", out="host"),
        # a small shape net (about 10,000 faces) in mixed precision, exported from the host
        _mesh("mesh_32x4_mixed", "plain", "32x4", "mixed", out="host"),
        # the default march of an ordinary net (about 50,000 faces) from one ray
        _mesh("mesh_64x4_fp64", "plain", "64x4", "fp64"),
        # the paper's D6-W60 shape (a width that fills no tile) on the tensor-core path
        _mesh("mesh_60x6_sliced", "plain", "60x6", "sliced", seeding="pairs"),
        # several small nets of one context in one march (an asset batch)
        _mesh("mesh_batch6_mixed", "plain", "32x4,64x4,64x6,32x6,48x4,64x4", "mixed"),
        # residual blocks (Sec. 5.1), which march in FP64
        _mesh("mesh_residual24x6_fp64", "residual", "24x6", "fp64"),
        # a latent-conditioned decoder with a skip-concat, whole mesh (about 850,000 faces)
        _mesh("mesh_decoder128x8_sliced", "decoder", "128x8", "sliced", seeding="pairs", latent=256, skip=4),
        # the largest: the benchmark's step, the whole 3-[256]x8-1 mesh (about 1.6 M faces) with
        # the learned candidates
        _mesh("mesh_256x8_learned", "plain", "256x8", "sliced", seeding="pairs", candidates="learned"),
        # the compose alone of a full-size decoder's cells on the tensor cores
        {"name": "compose_decoder512x8_sliced", "kind": "compose", "widths": "512x8", "precision": "sliced",
         "n": 4000, "latent": 256, "skip": 4},
        # the compose with certified error bounds of a ragged batch
        {"name": "compose_100x6_mixed", "kind": "compose", "widths": "100x6", "precision": "mixed", "n": 1501,
         "latent": 0, "skip": 0},
        # the random-pair trigger of the benchmark's net: 16,384 samples, up to 1024 seed cells
        {"name": "trigger_pairs_256x8", "kind": "trigger", "how": "pairs", "widths": "256x8", "n": 1024, "steps": 0},
        # training the learned proposal of a 3-[256]x8-1 net (batch 1024, as the benchmark trains it)
        {"name": "train_256x8", "kind": "train", "widths": "256x8", "hidden": 256, "batch": 1024, "steps": 8},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["mesh", "mesh", "mesh", "mesh", "mesh", "compose", "compose", "trigger", "train"])
    if kind == "mesh":
        sub = rng.choice(["march", "march", "sliced", "sliced", "batch", "residual", "decoder"])
        if sub == "march":
            prec = rng.choice(["fp64", "mixed"])
            d = rng.randint(3, 6)
            w = _log_int(rng, 24, 440 // d)
            return _mesh(None, "plain", "%dx%d" % (w, d), prec, seeding=rng.choice(["ray", "pairs"]),
                         out="host" if w * d < 160 else "device")
        if sub == "sliced":
            d = rng.randint(4, 8)
            w = _log_int(rng, 48, 1200 // d)
            return _mesh(None, "plain", "%dx%d" % (w, d), "sliced", seeding="pairs")
        if sub == "batch":
            parts = ["%dx%d" % (_log_int(rng, 24, 64), rng.randint(4, 6)) for _ in range(rng.randint(2, 6))]
            return _mesh(None, "plain", ",".join(parts), rng.choice(["fp64", "mixed"]))
        if sub == "residual":
            return _mesh(None, "residual", "%dx%d" % (rng.randint(12, 40), rng.choice([4, 5, 6])), "fp64")
        return _mesh(None, "decoder", "%dx%d" % (_log_int(rng, 48, 136), rng.randint(5, 8)), "sliced", seeding="pairs",
                     latent=rng.randint(5, 256), skip=rng.randint(2, 4))
    if kind == "compose":
        d = rng.randint(4, 8)
        w = _log_int(rng, 32, 512)
        lat = rng.choice([0, rng.randint(5, 256)])
        return {"kind": "compose", "widths": "%dx%d" % (w, d), "precision": rng.choice(["fp64", "mixed", "sliced", "sliced"]),
                "n": _log_int(rng, 16, min(6000, 12_000_000 // (w * d))), "latent": lat,
                "skip": rng.randint(2, 4) if lat else 0}
    if kind == "trigger":
        how = rng.choice(["pairs", "pairs", "trace"])
        return {"kind": "trigger", "how": how, "widths": "%dx%d" % (_log_int(rng, 24, 256), rng.randint(3, 8)),
                "n": _log_int(rng, 16, 1024), "steps": _log_int(rng, 4, 24) if how == "trace" else 0}
    return {"kind": "train", "widths": "%dx%d" % (_log_int(rng, 32, 256), rng.randint(4, 8)), "hidden": 256,
            "batch": _log_int(rng, 100, 1024), "steps": rng.randint(2, 8)}


# ------------------------------------------------------------------------------------------
# the inputs


def _widths(text):
    """'64x4' -> [64] * 4."""
    w, d = (int(v) for v in text.split("x"))
    return [w] * d


def _closed(net):
    """Whether F < 0 at the origin and F > 0 on the sphere of radius REACH around it: a shape that
    closes well inside the box, as a fitted shape does."""
    d = np.random.default_rng(0).normal(size=(600, 3))
    f = _forward(net, np.concatenate([np.zeros((1, 3)), REACH * d / np.linalg.norm(d, axis=1, keepdims=True)]))[0]
    return f[0] < 0.0 and bool(np.all(f[1:] > 0.0))


@functools.lru_cache(maxsize=64)
def _shape(arch, text, latent, skip, index):
    """The net of a case: the first closed shape among those drawn for its sizes."""
    if arch == "polytope":
        return synth.polytope_max_of_planes()
    ws = _widths(text)
    for k in range(500):
        s = zlib.crc32(repr((arch, text, latent, skip, index, k)).encode())
        if arch == "residual":
            net = synth.residual_net(seed=s, width=ws[0], depth=len(ws))
        elif latent:
            net = synth.decoder_net(seed=s, width=ws[0], depth=len(ws), latent_dim=latent, skip_layer=skip)
        else:
            net = synth.geometric_init(ws, s, 0.05, recenter=True)
        if _closed(net):
            return net
    raise RuntimeError("no closed shape among 500 nets")


def _rotation(seed):
    q, r = np.linalg.qr(np.random.default_rng(seed).normal(size=(3, 3)))
    q = q * np.sign(np.diag(r))
    return q * np.linalg.det(q)


def _net(case, text, seed, index=0):
    """The case's shape in a pose of its own, its hidden units in an order of their own: other
    weights for every seed, a mesh of the same size."""
    net = copy.deepcopy(_shape(case.get("arch", "plain"), text, case.get("latent", 0), case.get("skip", 0), index))
    R, rng = _rotation(seed), np.random.default_rng(seed + 1)
    for l in range(1, net.L + 1):
        o = 0 if l == 1 else (net.widths[l - 2] if l == net.skip_layer else None)
        if o is not None:
            net.weights[l - 1][:, o:o + 3] = net.weights[l - 1][:, o:o + 3] @ R.T
        if l in net.shortcuts and net.shortcuts[l][0] == 0:
            net.shortcuts[l] = (0, net.shortcuts[l][1] @ R.T)
    if not net.shortcuts:
        for l in range(1, net.L + 1):
            p = rng.permutation(net.widths[l - 1])
            net.weights[l - 1], net.biases[l - 1] = net.weights[l - 1][p].copy(), net.biases[l - 1][p].copy()
            if l < net.L:
                W = net.weights[l]
                W[:, :len(p)] = W[:, p]
            else:
                net.w_out = net.w_out[p].copy()
    return net


def _units(case):
    if case.get("arch") == "polytope":
        return [23]
    return [sum(_widths(t)) for t in case["widths"].split(",")]


def _faces(case):
    """About how many faces the nets of a mesh case have (measured: 0.4 to 0.9 N^2)."""
    return [126 if case["arch"] == "polytope" else 0.7 * n * n for n in _units(case)]


def _stream():
    return torch.cuda.Stream()


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    s = {"case": case, "stream": _stream()}
    texts = case["widths"].split(",")
    nets = [_net(case, t, seed, i) for i, t in enumerate(texts)]
    s["nets"] = nets
    n_max, w_max = max(n.N for n in nets), max(max(n.widths) for n in nets)
    cells = int(4 * sum(_faces(case))) + 16384 if case["kind"] == "mesh" else 1 << 14
    m = s["m"] = am.Mesher(max_cells=cells, max_neurons=n_max, max_width=w_max, stream=s["stream"].cuda_stream)
    if case["kind"] == "train":
        L, N, H = nets[0].L, nets[0].N, case["hidden"]
        n = case["batch"] * 4
        p = [rng.normal(0.0, math.sqrt(2.0 / i), (o, i)) for i, o in ((7 + L, H), (H, H), (H, N))]
        p = [p[0], np.zeros(H), p[1], np.zeros(H), p[2] / math.sqrt(2.0), np.full(N, math.log(1.0 / 31.0))]
        s["params"] = np.concatenate([v.ravel() for v in p]).astype(np.float32)
        m.proposal_init(7 + L, H, N, max_batch=case["batch"], seed=0)
        m.proposal_set_params(s["params"])
        X, Y = _samples(rng, n, L, N)
        s["X"], s["Y"] = torch.as_tensor(X, device="cuda"), torch.as_tensor(Y, device="cuda")
        return s
    s["ids"] = [m.load_mlp(n) for n in nets]
    if case["kind"] == "compose":
        keys = _patterns(nets[0], rng.uniform(-1.2, 1.2, (case["n"], 3)))
        s["keys"] = torch.as_tensor(keys.view(np.int64), device="cuda")
        return s
    if case["kind"] == "trigger":
        s["points"] = _trigger_points(case, seed)
        return s
    s["points"] = _trigger_points({"how": "pairs", "n": PAIRS}, seed)
    s["ray"] = (np.zeros((1, 3)), _rotation(seed)[None, :, 0])
    if case["candidates"] == "learned":
        # the proposal a program keeps beside its net: trained on faces marched before
        m.seed(0, *s["ray"], R=REACH)
        m.march(box=BOX, precision="sliced", max_cells=20000)
        m.proposal_init(7 + nets[0].L, 256, nets[0].N, max_batch=1024, seed=seed % 1000)
        X, Y = m.proposal_samples(0, max_samples=16384)
        m.proposal_train(X, Y, batch=1024, steps=32, lr=2e-3)
        m.reset()
    return s


def _trigger_points(case, seed):
    """Start points of the tracing walks, or 16 samples for every pair wanted: uniform in a ball
    around the shape, turned with it."""
    rng = np.random.default_rng(5)
    n = 16 * case["n"] if case["how"] == "pairs" else case["n"]
    d = rng.normal(size=(n, 3))
    d *= REACH * rng.uniform(size=(n, 1)) ** (1.0 / 3.0) / np.linalg.norm(d, axis=1, keepdims=True)
    return d @ _rotation(seed).T


def _samples(rng, n, L, N):
    """Training samples as marched faces give them: entry point, unit normal, offset, the active
    fraction of every layer; about six edge neurons of N."""
    x = rng.uniform(-1.0, 1.0, (n, 3))
    nrm = rng.normal(size=(n, 3))
    nrm /= np.linalg.norm(nrm, axis=1, keepdims=True)
    X = np.concatenate([x, nrm, -(x * nrm).sum(1, keepdims=True), rng.normal(0.5, 0.06, (n, L))], 1).astype(np.float32)
    Y = np.zeros((n, N), dtype=np.float32)
    Y[np.arange(n)[:, None], rng.integers(0, N, (n, 6))] = 1.0
    return X, Y


# ------------------------------------------------------------------------------------------
# one pass


def run(s):
    case, m = s["case"], s["m"]
    with torch.cuda.stream(s["stream"]):
        if case["kind"] == "train":
            losses = m.proposal_train(s["X"], s["Y"], batch=case["batch"], steps=case["steps"], lr=1e-3)
            return {"losses": losses, "params": m.proposal_params()}
        if case["kind"] == "compose":
            net, n = s["nets"][0], case["n"]
            rows = torch.empty((n, net.N + 1, 4), dtype=torch.float64, device="cuda")
            err = torch.empty((n, net.N + 1), dtype=torch.float32, device="cuda")
            st = m.lib.am_compose(m.ctx, s["ids"][0], C.c_void_p(s["keys"].data_ptr()), n, mesher.PRECISIONS[case["precision"]],
                                  C.c_void_p(rows.data_ptr()), C.c_void_p(err.data_ptr()))
            if st != 0:
                raise RuntimeError(m.lib.am_last_error(m.ctx).decode())
            return {"rows": rows, "err": err} if case["precision"] == "mixed" else {"rows": rows}
        m.reset()
        if case["kind"] == "trigger":
            if case["how"] == "pairs":
                return list(m.seed_pairs(s["ids"][0], s["points"], case["n"]))
            return list(m.seed_sphere_trace(s["ids"][0], s["points"], eta=1.0, max_steps=case["steps"], eps=1e-12))
        for i in s["ids"]:
            if case["seeding"] == "pairs":
                m.seed_pairs(i, s["points"], PAIRS)
            else:
                m.seed(i, *s["ray"], R=REACH)
        m.march(box=BOX, precision=case["precision"], candidates=case["candidates"])
        out = []
        for i in s["ids"]:
            if case["out"] == "host":
                h = mesher.canonicalize(m.get_mesh(i))
                out.append([h.xyz, h.face_offsets, h.face_vertices, h.edge_planes, h.face_keys.view(np.int64)])
            else:
                d = m.get_mesh_device(i)
                keys = d["face_keys"]
                out.append(_ordered(d["xyz"], d["face_offsets"], d["face_vertices"], d["edge_planes"], keys,
                                    torch.argsort(_mix(keys))))
        return out


def _mix(keys):
    """One 64-bit hash per face key (a multilinear hash with fixed odd multipliers)."""
    c = (torch.arange(1, keys.shape[1] + 1, device=keys.device, dtype=torch.int64) * -7046029254386353131) ^ 0x5DEECE66D2B79F5
    k = keys ^ (keys >> 29)
    return (k * (c | 1)).sum(1)


def _ordered(xyz, off, fv, fe, keys, perm):
    """The mesh with its faces in the order `perm`, every ring started at the corner with the
    smallest pair of planes, and its vertices numbered by first appearance."""
    dev = fv.device
    F, K, V = keys.shape[0], fv.shape[0], xyz.shape[0]
    lens = off[1:] - off[:-1]
    face = torch.repeat_interleave(torch.arange(F, device=dev), lens, output_size=K)
    at = torch.arange(K, device=dev)
    j = at - off[face]
    e = fe.to(torch.int64)
    before = e[torch.where(j == 0, at + lens[face] - 1, at - 1)]
    code = ((torch.minimum(before, e) << 20) | torch.maximum(before, e)) * 64 + j
    first = torch.full((F,), 1 << 62, device=dev, dtype=torch.int64).scatter_reduce_(0, face, code, "amin") & 63
    lens2 = lens[perm]
    off2 = torch.zeros(F + 1, device=dev, dtype=torch.int64)
    off2[1:] = torch.cumsum(lens2, 0)
    new = torch.repeat_interleave(torch.arange(F, device=dev), lens2, output_size=K)
    p = perm[new]
    q = first[p] + at - off2[new]
    src = off[p] + torch.where(q >= lens[p], q - lens[p], q)
    v = fv[src].to(torch.int64)
    seen = torch.full((V,), K, device=dev, dtype=torch.int64).scatter_reduce_(0, v, at, "amin")
    order = torch.argsort(seen)
    rank = torch.empty_like(order)
    rank[order] = torch.arange(V, device=dev)
    return [xyz[order], off2, rank[v].to(torch.int32), fe[src], keys[perm]]


# ------------------------------------------------------------------------------------------
# what a pass cannot do without


def work(case):
    if case["kind"] == "train":
        ws = _widths(case["widths"])
        I, H, O, B, T = 7 + len(ws), case["hidden"], sum(ws), case["batch"], case["steps"]
        P = H * I + H + H * H + H + O * H + O
        # forward, weight gradients, input gradients of the two upper layers; Adam reads and
        # writes the weights and both moments
        flops = T * (2 * B * (H * I + H * H + O * H) * 2 + 2 * B * (H * H + O * H))
        return {"bytes": T * (4 * B * (I + O) + 6 * 4 * P) + 4 * P, "flops": flops}
    if case["kind"] == "compose":
        ws = _widths(case["widths"])
        N, n = sum(ws), case["n"]
        wbytes = 8 * sum(a * b for a, b in zip(ws, ws[1:]))
        flops = n * sum(8 * a * b // 2 for a, b in zip(ws, ws[1:]))      # half the units are active
        return {"bytes": n * (N / 8 + 32 * (N + 1)) + wbytes, "flops": flops}
    if case["kind"] == "trigger":
        # evaluations through the active units: every sample once, about 20 halvings per segment,
        # and the steps of a walk with their gradients
        ws = _widths(case["widths"])
        n = case["n"]
        evals = 16 * n + 20 * n if case["how"] == "pairs" else n * (2 * case["steps"] + 20)
        return {"bytes": n * (16 * 24 if case["how"] == "pairs" else 24) + 24 * n,
                "flops": evals * sum(a * b for a, b in zip([3] + ws, ws))}
    by = fl = 0.0
    for text, f in zip(case["widths"].split(","), _faces(case)):
        ws = [12, 6, 3, 2] if case["arch"] == "polytope" else _widths(text)
        N = sum(ws)
        # a face of about six corners: its rows from a neighbour's (half the later layers change,
        # one column through half the units, then the rows' rank-1 update), the tests of every row
        rows = sum(a * b / 2 for a, b in zip(ws, ws[1:])) + 8 * N / 2
        fl += f * (rows + 8 * 6 * (N + 6))
        by += f * (8 * ((N + 63) // 64) + 6 * 8 + 8 + 24)
    return {"bytes": by, "flops": fl}


# ------------------------------------------------------------------------------------------
# the same outputs from plain 64-bit arithmetic


def _folded(net):
    """Per layer (A, C): pre_l = A h_{l-1} + C [x; 1] (the latent code and the skip folded in)."""
    out = []
    z = np.zeros(0) if net.latent is None else net.latent
    for l in range(1, net.L + 1):
        W, b = net.weights[l - 1], net.biases[l - 1]
        Cl = np.zeros((W.shape[0], 4))
        Cl[:, 3] = b
        A = None
        if l == 1:
            Wx = W
        else:
            A, Wx = W[:, :net.widths[l - 2]], W[:, net.widths[l - 2]:]
        if Wx.shape[1]:
            Cl[:, :3] += Wx[:, :3]
            Cl[:, 3] += Wx[:, 3:] @ z
        if l in net.shortcuts and net.shortcuts[l][0] == 0:
            Cl[:, :3] += net.shortcuts[l][1]
        out.append((A, Cl))
    return out


def _forward(net, x):
    """F (n,) and the active units (n, N) at the points x (n, 3)."""
    x1 = np.concatenate([x, np.ones((len(x), 1))], 1)
    hs, act = [], []
    for l, (A, Cl) in enumerate(_folded(net), start=1):
        a = x1 @ Cl.T
        if A is not None:
            a += hs[-1] @ A.T
        if l in net.shortcuts and net.shortcuts[l][0] > 0:
            src, S = net.shortcuts[l]
            a += hs[src - 1] if S is None else hs[src - 1] @ S.T
        act.append(a > 0.0)
        hs.append(np.maximum(a, 0.0))
    return hs[-1] @ net.w_out + net.b_out, np.concatenate(act, 1)


def _words(bits):
    """(n, N) booleans as (n, ceil(N / 64)) uint64 key words."""
    n, N = bits.shape
    pad = np.zeros((n, (N + 63) // 64 * 64), dtype=bool)
    pad[:, :N] = bits
    return np.ascontiguousarray(np.packbits(pad, axis=1, bitorder="little")).view(np.uint64)


def _patterns(net, x):
    return _words(_forward(net, x)[1])


def _compose(net, bits):
    """(n, N, 4) maps of every unit and (n, 4) of F in the cells with the given active units."""
    n, zs, hs, o = len(bits), [], [], 0
    for l, (A, Cl) in enumerate(_folded(net), start=1):
        z = np.broadcast_to(Cl, (n,) + Cl.shape).copy()
        if A is not None:
            z += np.matmul(A, hs[-1])
        if l in net.shortcuts and net.shortcuts[l][0] > 0:
            src, S = net.shortcuts[l]
            z += hs[src - 1] if S is None else np.matmul(S, hs[src - 1])
        b = bits[:, o:o + len(Cl)]
        o += len(Cl)
        zs.append(z)
        hs.append(np.where(b[:, :, None], z, 0.0))
    F = np.einsum("k,nkc->nc", net.w_out, hs[-1])
    F[:, 3] += net.b_out
    return np.concatenate(zs, 1), F


def _clip(rows, F):
    """The plane F clipped by rows [n | c] x <= 0: ring of (plane of the edge out of the corner)."""
    n = F[:3] / np.linalg.norm(F[:3])
    p0 = -F[3] * F[:3] / (F[:3] @ F[:3])
    u = np.cross(n, np.eye(3)[np.argmin(np.abs(n))])
    u /= np.linalg.norm(u)
    w = np.cross(n, u)
    B = np.stack([np.append(u, 0.0), np.append(w, 0.0), np.append(p0, 1.0)], 1)
    g = rows @ B                                    # (rows, 3): a half-plane each
    nr = np.linalg.norm(g[:, :2], axis=1)
    g = g / np.where(nr > 0.0, nr, 1.0)[:, None]
    P = np.array([[-9.0, -9.0, 1.0], [9.0, -9.0, 1.0], [9.0, 9.0, 1.0], [-9.0, 9.0, 1.0]])
    E = [-1, -2, -3, -4]
    for _ in range(200):
        d = g @ P.T
        k = int(np.argmax(d.max(1)))
        if d[k].max() <= 1e-10:
            return P[:, :2] @ np.stack([u, w]) + p0, E
        out = d[k] > 0.0
        if out.all():
            return None, []
        m = len(P)
        ia = next(i for i in range(m) if out[i] and not out[i - 1])
        ib = next(i for i in range(m) if out[i] and not out[(i + 1) % m])
        keep = [(ib + 1 + i) % m for i in range(m - int(out.sum()))]
        new = []
        for a, b in ((ia - 1, ia), (ib, (ib + 1) % m)):
            da, db = d[k, a], d[k, b]
            new.append(P[a] + da / (da - db) * (P[b] - P[a]))
        P, E = np.concatenate([P[keep], np.stack(new)]), [E[i] for i in keep[:-1]] + [E[ia - 1], k, E[ib]]
    return None, []


def _march(net, x0):
    """The whole mesh reached from the cell of the point x0 on the surface, all faces clipped by all rows."""
    N, kw = net.N, (net.N + 63) // 64
    box = np.zeros((6, 4))
    for i in range(6):
        box[i, i // 2] = -1.0 if i % 2 else 1.0
        box[i, 3] = -BOX
    first = _forward(net, x0[None])[1][0]
    level, seen = [first], {first.tobytes()}
    faces = []
    while level:
        bits = np.stack(level)
        Z, F = _compose(net, bits)
        Z = np.where(bits[:, :, None], -Z, Z)
        level = []
        for b, z, f in zip(bits, Z, F):
            rows = np.concatenate([z, box])
            P, E = _clip(rows, f)
            if P is None or len(E) < 3:
                continue
            pairs = [(E[i - 1], E[i]) for i in range(len(E))]
            M = np.stack([np.stack([rows[p][:3], rows[q][:3], f[:3]]) for p, q in pairs])
            c = np.stack([np.array([rows[p][3], rows[q][3], f[3]]) for p, q in pairs])
            faces.append((b, E, np.linalg.solve(M, -c[:, :, None])[:, :, 0]))
            for e in E:
                if e < N:
                    nb = b.copy()
                    nb[e] = not nb[e]
                    t = nb.tobytes()
                    if t not in seen:
                        seen.add(t)
                        level.append(nb)
    off, fv, fe, xyz, ids = [0], [], [], [], {}
    for b, E, X in faces:
        for i, e in enumerate(E):
            lo, hi = sorted((E[i - 1], e))
            k = b.copy()
            k[[p for p in (lo, hi) if p < N]] = False
            v = ids.setdefault((lo, hi, k.tobytes()), len(ids))
            if v == len(xyz):
                xyz.append(X[i])
            fv.append(v)
            fe.append(e)
        off.append(len(fv))
    keys = _words(np.stack([f[0] for f in faces])).reshape(len(faces), kw)
    return np.stack(xyz), np.array(off), np.array(fv), np.array(fe), keys


def _root(net, o, d, R):
    """The point the dichotomy along o + t d, t in [0, R], ends in."""
    lo, hi = 0.0, R
    (flo, fhi), (blo, bhi) = _forward(net, np.stack([o + lo * d, o + hi * d]))
    for _ in range(200):
        if (blo == bhi).all():
            break
        t = 0.5 * (lo + hi)
        f, b = _forward(net, (o + t * d)[None])
        if (f[0] < 0.0) == (flo < 0.0) and f[0] != 0.0:
            lo, flo, blo = t, f[0], b[0]
        else:
            hi, fhi, bhi = t, f[0], b[0]
    return o + (lo + flo / (flo - fhi) * (hi - lo)) * d


def exact(case, seed):
    if case["kind"] == "mesh":
        if "," in case["widths"] or case["seeding"] != "ray" or sum(_faces(case)) > 15000:
            return None                              # minutes in plain numpy
        net = _net(case, case["widths"], seed)
        x0 = _root(net, np.zeros(3), _rotation(seed)[:, 0], REACH)
        xyz, off, fv, fe, keys = (torch.from_numpy(np.ascontiguousarray(v if v.dtype != np.uint64 else v.view(np.int64)))
                                  for v in _march(net, x0))
        if case["out"] == "host":                   # ascending by key as one unsigned integer
            u = keys.numpy().view(np.uint64)
            perm = torch.from_numpy(np.lexsort([u[:, w] for w in range(u.shape[1])]))
        else:
            perm = torch.argsort(_mix(keys))
        out = _ordered(xyz, off, fv.to(torch.int32), fe.to(torch.int32), keys, perm)
        return [[out[0], None, None, None, None]]
    rng = np.random.default_rng(seed)
    net = _net(case, case["widths"], seed)
    if case["kind"] == "compose":
        n = case["n"]
        if n * sum(8 * a * b for a, b in zip(net.widths, net.widths[1:])) > 1.2e11:
            return None
        act = _forward(net, rng.uniform(-1.2, 1.2, (n, 3)))[1]
        rows = np.empty((n, net.N + 1, 4))
        for i in range(0, n, 256):
            Z, F = _compose(net, act[i:i + 256])
            rows[i:i + 256, :net.N] = np.where(act[i:i + 256, :, None], -Z, Z)
            rows[i:i + 256, net.N] = F
        return {"rows": rows, "err": None} if case["precision"] == "mixed" else {"rows": rows}
    if case["kind"] == "train":
        return _exact_train(case, net, rng)
    return _exact_trigger(case, net, _trigger_points(case, seed))


def _gradient(net, x):
    """F and grad F (the gradient of each point's own affine piece) at the points x."""
    F, act = _forward(net, x)
    o, g, gx = act.shape[1], np.broadcast_to(net.w_out, (len(x), len(net.w_out))), 0.0
    for A, Cl in reversed(_folded(net)):
        o -= len(Cl)
        g = np.where(act[:, o:o + len(Cl)], g, 0.0)
        gx = gx + g @ Cl[:, :3]
        g = None if A is None else g @ A
    return F, gx


def _roots(net, o, d):
    """The points the dichotomies along o + t d, t in [0, 1], end in; NaN where F has one sign."""
    lo, hi = np.zeros(len(o)), np.ones(len(o))
    (flo, blo), (fhi, bhi) = _forward(net, o), _forward(net, o + d)
    ok = flo * fhi < 0.0
    for _ in range(200):
        go = ok & (blo != bhi).any(1)
        if not go.any():
            break
        t = 0.5 * (lo + hi)
        f, b = _forward(net, o + t[:, None] * d)
        left = go & ((f < 0.0) == (flo < 0.0)) & (f != 0.0)
        right = go & ~left
        lo, flo, blo = np.where(left, t, lo), np.where(left, f, flo), np.where(left[:, None], b, blo)
        hi, fhi, bhi = np.where(right, t, hi), np.where(right, f, fhi), np.where(right[:, None], b, bhi)
    t = lo + flo / np.where(flo == fhi, 1.0, flo - fhi) * (hi - lo)
    return np.where(ok[:, None], o + t[:, None] * d, np.nan)


def _exact_trigger(case, net, x):
    if case["how"] == "pairs":
        F = _forward(net, x)[0]
        neg, pos = np.nonzero(F < 0.0)[0], np.nonzero(F > 0.0)[0]
        n = min(len(neg), len(pos), case["n"])
        return [None, None, _roots(net, x[neg[:n]], x[pos[:n]] - x[neg[:n]])]
    x = x.copy()
    live = np.ones(len(x), dtype=bool)
    for _ in range(case["steps"]):
        F, g = _gradient(net, x)
        live &= (np.abs(F) > 1e-12) & (g != 0.0).any(1)
        x[live] -= F[live, None] * g[live]
    F, g = _gradient(net, x)
    nrm = np.linalg.norm(g, axis=1)
    u = g / np.where(nrm > 0.0, nrm, 1.0)[:, None]
    h = 2.0 * np.abs(F) / np.where(nrm > 0.0, nrm, 1.0) + 1e-9
    return [None, _roots(net, x - h[:, None] * u, 2.0 * h[:, None] * u)]


def _exact_train(case, net, rng):
    """Adam on the mean binary cross-entropy, everything in 64 bits (the library's products take
    BF16 operands, so the two agree to their rounding)."""
    L, N, H, B = net.L, net.N, case["hidden"], case["batch"]
    p = [rng.normal(0.0, math.sqrt(2.0 / i), (o, i)) for i, o in ((7 + L, H), (H, H), (H, N))]
    p = [p[0], np.zeros(H), p[1], np.zeros(H), p[2] / math.sqrt(2.0), np.full(N, math.log(1.0 / 31.0))]
    X, Y = _samples(rng, 4 * B, L, N)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    p = [torch.as_tensor(v.astype(np.float32), device=dev).double().requires_grad_() for v in p]
    X, Y = torch.as_tensor(X, device=dev).double(), torch.as_tensor(Y, device=dev).double()
    ms, vs, losses = [torch.zeros_like(v) for v in p], [torch.zeros_like(v) for v in p], []
    for t in range(case["steps"]):
        i = t % 4 * B
        h = torch.relu(X[i:i + B] @ p[0].T + p[1])
        h = torch.relu(h @ p[2].T + p[3])
        z = h @ p[4].T + p[5]
        loss = (torch.nn.functional.softplus(z) - Y[i:i + B] * z).mean()
        losses.append(float(loss.detach()))
        for v, g, a, b in zip(p, torch.autograd.grad(loss, p), ms, vs):
            a.mul_(0.9).add_(0.1 * g)
            b.mul_(0.999).add_(0.001 * g * g)
            with torch.no_grad():
                v -= 1e-3 * (a / (1.0 - 0.9 ** (t + 1))) / (torch.sqrt(b / (1.0 - 0.999 ** (t + 1))) + 1e-8)
    return {"losses": np.array(losses), "params": np.concatenate([v.detach().cpu().numpy().ravel() for v in p])}
