"""Timed cases of the library's public entry points: graph construction from a
point cloud, halo partitioning, and the message-passing model forward and
backward in its three numeric forms (BF16 at H = 128, BF16 at other widths,
FP32).

A case is a dict of plain values; ``kind`` says which entry points a pass
calls:

* ``knn``         ``build_knn`` on ``n`` points with ``k`` neighbours.
* ``multiscale``  ``build_multiscale`` on nested levels ``n0 < n1 < n``.
* ``partition``   ``partition_halo`` of a kNN graph into ``parts`` parts with
                  ``hops`` halo hops; ``given`` says whether the caller brings
                  the parts (regions that need not cover the cloud) or the
                  library bisects the cloud.
* ``train``       ``Model.forward`` with loss and ``Model.backward``; returns
                  loss, predictions and the whole parameter gradient.
* ``infer``       ``Model.forward`` without targets; returns the predictions.

Clouds: ``sphere`` is uniform on the unit sphere in random order; ``body`` is a
car-like closed surface (an ellipsoid and two boxes, uniform by area, points
inside another primitive left out) in Morton order, as surface mesh files keep
neighbours close.  Everything is made on the GPU from the seed alone.
"""
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_2411_17164_gb300 import xmgn

OUT = 4        # predicted channels: pressure and three shear-stress components
IN_NODE = 6    # position and unit normal
LN_EPS = 1e-5


def listed():
    return [
        # the smallest cloud that is used in earnest: launches and host round trips count
        dict(name="knn_sphere_2k", kind="knn", cloud="sphere", n=2000, k=6),
        # the ordinary single-body surface cloud
        dict(name="knn_body_200k", kind="knn", cloud="body", n=200_000, k=6),
        # the three nested levels of the multi-scale graph, the largest graph build
        dict(name="multiscale_1250k", kind="multiscale", cloud="body", n0=50_000, n1=250_000, n=1_250_000, k=6,
             k_cross=3),
        # a 2M-point body cut by the library into 16 parts for a 15-layer model
        dict(name="partition_2m_16", kind="partition", cloud="body", n=2_000_000, parts=16, hops=15, given=False),
        # 64 regions brought by the caller, sizes spread over more than a factor of ten, gaps between them
        dict(name="regions_1m_64", kind="partition", cloud="body", n=1_000_000, parts=64, hops=15, given=True),
        # a training step on the smallest graph, the full 15 layers: latency
        dict(name="train_bf16_sphere_2k", kind="train", cloud="sphere", n=2000, H=128, L=15, dtype="bf16", fourier=0,
             parts=0),
        # the whole training step of one unpartitioned body
        dict(name="train_bf16_body_200k", kind="train", cloud="body", n=200_000, H=128, L=15, dtype="bf16", fourier=0,
             parts=0),
        # a short model over the batch of halo partitions of a larger body, as a batched step runs them
        dict(name="train_bf16_batch_500k", kind="train", cloud="body", n=500_000, H=128, L=2, dtype="bf16", fourier=0,
             parts=16),
        # prediction on a large surface with Fourier features of the coordinates
        dict(name="infer_bf16_body_700k", kind="infer", cloud="body", n=700_000, H=128, L=4, dtype="bf16", fourier=3,
             parts=0),
        # the paper's production width, the layer blocks of a short model
        dict(name="train_h512_body_50k", kind="train", cloud="body", n=50_000, H=512, L=2, dtype="bf16", fourier=0,
             parts=0),
        # prediction at a width between the two, on a ragged medium cloud
        dict(name="infer_h256_body_30k", kind="infer", cloud="body", n=30_011, H=256, L=3, dtype="bf16", fourier=0,
             parts=0),
        # the FP32 form, with which partitions are run one at a time and gradients are checked
        dict(name="train_fp32_body_30k", kind="train", cloud="body", n=30_000, H=128, L=15, dtype="fp32", fourier=0,
             parts=0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["knn", "multiscale", "partition", "bf16", "bf16", "bf16", "wide", "fp32"])
    cloud = rng.choice(["body", "body", "sphere"])
    if what == "knn":
        return dict(kind="knn", cloud=cloud, n=_log(rng, 2000, 1_200_000), k=rng.choice([3, 6, 6, 6, 8, 16]))
    if what == "multiscale":
        n = _log(rng, 8000, 1_250_000)
        n1 = max(400, int(n * rng.uniform(0.1, 0.4)))
        return dict(kind="multiscale", cloud=cloud, n0=max(100, int(n1 * rng.uniform(0.1, 0.4))), n1=n1, n=n, k=6,
                    k_cross=rng.choice([1, 3, 3]))
    if what == "partition":
        n = _log(rng, 5000, 1_500_000)
        given = rng.random() < 0.5  # runs of the point order are compact regions only on a body
        return dict(kind="partition", cloud="body" if given else cloud, n=n,
                    parts=rng.randint(2, max(2, min(24, n // 4000))), hops=rng.choice([2, 4, 8, 15]), given=given)
    kind = rng.choice(["train", "train", "infer"])
    if what == "bf16":
        n = _log(rng, 2000, 300_000)
        L = rng.choice([1, 2, 3, 5, 15]) if n < 200_000 else rng.choice([1, 2, 3])
        return dict(kind=kind, cloud=cloud, n=n, H=128, L=L, dtype="bf16", fourier=rng.choice([0, 0, 3]),
                    parts=rng.choice([0, 0, 4, 8]) if n >= 20_000 else 0)
    if what == "wide":
        H = rng.choice([256, 512, 512])
        return dict(kind=kind, cloud=cloud, n=_log(rng, 2000, 40_000 if H == 512 else 80_000), H=H,
                    L=rng.choice([1, 2]), dtype="bf16", fourier=0, parts=0)
    n = _log(rng, 2000, 60_000)
    return dict(kind=kind, cloud=cloud, n=n, H=rng.choice([64, 128, 128, 256]), L=rng.choice([1, 2, 3]), dtype="fp32",
                fourier=rng.choice([0, 0, 3]), parts=rng.choice([0, 0, 4]) if n >= 20_000 else 0)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _morton(p):
    lo = p.amin(0)
    q = ((p - lo) / (p.amax(0) - lo).clamp_min(1e-30) * 1023.0).long().clamp_(0, 1023)
    code = torch.zeros(len(p), dtype=torch.long, device=p.device)
    for b in range(10):
        for a in range(3):
            code |= ((q[:, a] >> b) & 1) << (3 * b + a)
    return torch.sort(code, stable=True).indices


_ELL = (2.0, 0.9, 0.6)
_BOXES = (((-0.8, -0.65, 0.2), (0.7, 0.65, 0.9)), ((-1.85, -0.8, -0.55), (1.85, 0.8, -0.1)))


def _body(n, g):
    """n random points, uniform by area, of the union's surface, and their unit normals (in random order)."""
    dev = "cuda"
    ax = torch.tensor(_ELL, device=dev, dtype=torch.float64)
    p0 = 1.6075
    a, b, c = _ELL
    area = [4 * math.pi * (((a * b) ** p0 + (a * c) ** p0 + (b * c) ** p0) / 3) ** (1 / p0)]
    for lo, hi in _BOXES:
        d = [h - l for l, h in zip(lo, hi)]
        area.append(2 * (d[0] * d[1] + d[0] * d[2] + d[1] * d[2]))
    gmax = max(a * b, a * c, b * c)
    pts, nrm, have = [], [], 0
    while have < n:
        m = 2 * (n - have) + 1024
        # the ellipsoid is thinned below, so it gets that much more
        u = torch.randn((int(m * 2.2 * area[0] / sum(area)), 3), generator=g, device=dev, dtype=torch.float64)
        u /= u.norm(dim=1, keepdim=True)
        dens = ((b * c * u[:, 0]) ** 2 + (a * c * u[:, 1]) ** 2 + (a * b * u[:, 2]) ** 2).sqrt() / gmax
        u = u[torch.rand(len(u), generator=g, device=dev, dtype=torch.float64) < dens]
        u = u[: int(m * area[0] / sum(area))]
        p, q = [u * ax], [(u / ax) / (u / ax).norm(dim=1, keepdim=True)]
        for (lo, hi), s in zip(_BOXES, area[1:]):
            lo, hi = (torch.tensor(v, device=dev, dtype=torch.float64) for v in (lo, hi))
            d = hi - lo
            k = int(m * s / sum(area))
            fa = torch.stack([d[1] * d[2], d[0] * d[2], d[0] * d[1]])
            w = torch.rand(k, generator=g, device=dev, dtype=torch.float64) * fa.sum()
            axis = (w > fa[0]).long() + (w > fa[0] + fa[1]).long()
            side = (torch.rand(k, generator=g, device=dev) < 0.5).double()
            x = lo + torch.rand((k, 3), generator=g, device=dev, dtype=torch.float64) * d
            x.scatter_(1, axis[:, None], (lo + side[:, None] * d).gather(1, axis[:, None]))
            p.append(x)
            q.append(torch.zeros_like(x).scatter_(1, axis[:, None], (2 * side - 1)[:, None]))
        owner = torch.cat([torch.full((len(x),), i, device=dev) for i, x in enumerate(p)])
        p, q = torch.cat(p), torch.cat(q)
        ok = (((p / ax) ** 2).sum(1) >= 1 - 1e-9) | (owner == 0)
        for i, (lo, hi) in enumerate(_BOXES):
            lo, hi = (torch.tensor(v, device=dev, dtype=torch.float64) for v in (lo, hi))
            ok &= ~((p > lo + 1e-9) & (p < hi - 1e-9)).all(1) | (owner == i + 1)
        p, q = p[ok], q[ok]
        o = torch.randperm(len(p), generator=g, device=dev)
        pts.append(p[o])
        nrm.append(q[o])
        have += len(p)
    return torch.cat(pts)[:n], torch.cat(nrm)[:n]


def _cloud(case, g):
    """(points, normals), float32; nested levels keep the prefix property."""
    n = case["n"]
    if case["cloud"] == "sphere":
        p = torch.randn((n, 3), generator=g, device="cuda", dtype=torch.float64)
        p /= p.norm(dim=1, keepdim=True)
        q = p
    else:
        p, q = _body(n, g)
        cuts = [0] + ([case["n0"], case["n1"]] if case["kind"] == "multiscale" else []) + [n]
        o = torch.cat([lo + _morton(p[lo:hi]) for lo, hi in zip(cuts, cuts[1:])])
        p, q = p[o], q[o]
    return p.float().contiguous(), q.float().contiguous()


def _regions(n, parts, g):
    """Part ids of `parts` compact regions: runs of the point order with log-uniform sizes and gaps (-1) between them."""
    size = torch.exp(torch.rand(parts, generator=g, device="cuda") * math.log(16.0)).cpu().numpy().astype(np.float64)
    size = np.maximum(1, np.floor(size / size.sum() * 0.6 * n)).astype(np.int64)
    gap = (n - int(size.sum())) // parts
    part = np.full(n, -1, dtype=np.int32)
    at = 0
    for p in range(parts):
        part[at:at + size[p]] = p
        at += int(size[p]) + gap
    return torch.from_numpy(part).cuda()


def _blocks(H, L, in_enc):
    """(name, shape, fan in) of the flat parameter vector's blocks, in order."""
    got = []

    def mlp(prefix, fin, fout, ln):
        got.append((prefix + ".W1", (fin, H), fin))
        got.append((prefix + ".b1", (H,), fin))
        got.append((prefix + ".W2", (H, fout), H))
        got.append((prefix + ".b2", (fout,), H))
        if ln:
            got.append((prefix + ".g", (fout,), 0))
            got.append((prefix + ".be", (fout,), 0))

    mlp("ne", in_enc, H, True)
    mlp("ee", 4, H, True)
    for l in range(L):
        mlp("e%d" % l, 3 * H, H, True)
        mlp("n%d" % l, 2 * H, H, True)
    mlp("dec", H, OUT, False)
    return got


def _caps(case):
    """Node and edge capacity of a graph result.  A program that keeps graphs in buffers of one size (for a captured
    step, or a pool of them) fixes these in advance, from the sizes alone."""
    n = case["n"]
    if case["kind"] == "knn":
        return n, int(1.5 * case["k"] * n) + 64
    if case["kind"] == "multiscale":
        return n, int(1.5 * (case["k"] * (case["n0"] + case["n1"] + n) + 2 * case["k_cross"] * (n - case["n0"]))) + 64
    P, hops = case["parts"], case["hops"]
    m = n / P
    nb = int(min(P * n, P * (1.2 * m + 12 * hops * math.sqrt(m) + 24 * hops * hops)))
    return nb, int(7.5 * nb)


def _fixed(parts, pad, size):
    """The arrays one after another in a buffer of `size` elements, -1 behind them."""
    return torch.cat([*parts, pad[: size - sum(len(p) for p in parts)]])


def _params(case, g):
    """Weights of a model some way into training: scaled normal matrices, small biases, scales near one."""
    got = []
    for name, shape, fan in _blocks(case["H"], case["L"], IN_NODE + 6 * case["fourier"]):
        v = torch.randn(math.prod(shape), generator=g, device="cuda")
        if name.endswith(".g"):
            v = 1 + 0.1 * v
        elif name.endswith(".be"):
            v = 0.1 * v
        else:
            v = v * (1 if ".W" in name else 0.1) / math.sqrt(fan)
        got.append(v)
    return torch.cat(got)


def _targets(xyz, g):
    f = torch.randn((OUT, 8, 3), generator=g, device="cuda")
    amp = torch.randn((OUT, 8), generator=g, device="cuda") * math.sqrt(1 / 8)
    phi = torch.rand((OUT, 8), generator=g, device="cuda") * 2 * math.pi
    t = torch.empty((len(xyz), OUT), device="cuda")
    for c in range(OUT):
        t[:, c] = (amp[c] * torch.sin(2 * math.pi * (xyz[:, None, :] * f[c]).sum(-1) + phi[c])).sum(-1)
    return t


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    xyz, nrm = _cloud(case, g)
    st = dict(case=case, xyz=xyz)
    if case["kind"] in ("knn", "multiscale", "partition"):
        nodes, edges = _caps(case)
        st["pad32"] = torch.full((3 * edges,), -1, dtype=torch.int32, device="cuda")
        st["pad64"] = torch.full((nodes + 1,), -1, dtype=torch.int64, device="cuda")
        st["pad8"] = torch.full((nodes,), 255, dtype=torch.uint8, device="cuda")
    if case["kind"] in ("knn", "multiscale"):
        return st
    graph = xmgn.build_knn(xyz, 6)
    if case["kind"] == "partition":
        st["graph"] = graph
        st["given"] = _regions(case["n"], case["parts"], g) if case["given"] else None
        return st
    if case["parts"]:
        graph = xmgn.partition_halo(graph, xyz, case["parts"], case["L"])
    st["graph"] = graph
    st["model"] = xmgn.Model(case["H"], case["L"], graph, dtype=case["dtype"], n_norm=case["n"],
                             fourier=case["fourier"])
    st["params"] = _params(case, g)
    st["node_in"] = torch.cat([xyz, nrm], 1).contiguous()
    st["targets"] = _targets(xyz, g) if case["kind"] == "train" else None
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(state):
    case, xyz = state["case"], state["xyz"]
    if case["kind"] in ("knn", "multiscale"):
        if case["kind"] == "knn":
            g = xmgn.build_knn(xyz, case["k"])
        else:
            g = xmgn.build_multiscale(xyz, [case["n0"], case["n1"], case["n"]], case["k"], case["k_cross"])
        return {"row_ptr": g["row_ptr"],
                "edges": _fixed([g["col"], g["recv"], g["csc_perm"]], state["pad32"], 3 * _caps(case)[1])}
    if case["kind"] == "partition":
        b = xmgn.partition_halo(state["graph"], xyz, case["parts"], case["hops"], part_in=state["given"])
        nodes, edges = _caps(case)
        out = {"row_ptr": _fixed([b["row_ptr"]], state["pad64"], nodes + 1),
               "edges": _fixed([b["col"], b["recv"], b["csc_perm"]], state["pad32"], 3 * edges),
               "gid": _fixed([b["gid"]], state["pad32"], nodes), "hop": _fixed([b["hop"]], state["pad8"], nodes)}
        if state["given"] is None:
            out["part"] = b["part"]
        out.update({k: np.array(b[k], dtype=np.int64) for k in ("node_ptr", "edge_ptr", "inner_cnt")})
        return out
    m, p, nin = state["model"], state["params"], state["node_in"]
    y = torch.zeros((case["n"], OUT), device=xyz.device)
    if case["kind"] == "infer":
        m.forward(p, nin, xyz, y=y)
        return {"y": y}
    loss = torch.zeros((), device=xyz.device)
    grad = torch.zeros_like(p)
    m.forward(p, nin, xyz, targets=state["targets"], y=y, loss=loss)
    m.backward(p, nin, xyz, state["targets"], grad)
    return {"loss": loss, "y": y, "grad": grad}


def _edges(n, k):
    return int(1.18 * k * n)  # directed edges after symmetrisation, of these clouds


def work(case):
    n = case["n"]
    if case["kind"] == "knn":
        return {"bytes": 12 * n + 8 * (n + 1) + 12 * _edges(n, case["k"]), "flops": 0}
    if case["kind"] == "multiscale":
        e = sum(_edges(m, case["k"]) for m in (case["n0"], case["n1"], n)) + 2 * case["k_cross"] * (n - case["n0"])
        return {"bytes": 12 * n + 8 * (n + 1) + 12 * e, "flops": 0}
    if case["kind"] == "partition":
        e = _edges(n, 6)
        # each node and edge read once; the batch (at least the inner nodes and their edges) written once
        cover = 0.6 if case["given"] else 1.0
        read = (4 if case["given"] else 12) * n + 8 * n + 4 * e
        return {"bytes": int(read + cover * (13 * n + 12 * e)), "flops": 0}
    H, L, e = case["H"], case["L"], _edges(n, 6)
    in_enc = IN_NODE + 6 * case["fourier"]
    params = sum(math.prod(s) for _, s, _ in _blocks(H, L, in_enc))
    # products of the method, with the edge MLP's node blocks applied once per node
    mac = n * (in_enc * H + H * H) + e * (4 * H + H * H) + L * (e * 2 * H * H + n * 5 * H * H) + n * (H * H + OUT * H)
    io = 4 * params + n * (4 * IN_NODE + 12 + 4 * OUT) + 8 * n + 8 * e
    if case["kind"] == "infer":
        return {"bytes": io, "flops": 2 * mac}
    return {"bytes": io + 4 * params + 4 * OUT * n + 4 * e, "flops": 6 * mac}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def _ln(x, g, b):
    mu = x.mean(-1, keepdim=True)
    d = x - mu
    return d * torch.rsqrt((d * d).mean(-1, keepdim=True) + LN_EPS) * g + b


def _mlp(w, pre, x1):
    """The MLP after its first product x1 (bias not yet added)."""
    z = torch.nn.functional.silu(x1 + w[pre + ".b1"]) @ w[pre + ".W2"] + w[pre + ".b2"]
    return _ln(z, w[pre + ".g"], w[pre + ".be"]) if pre + ".g" in w else z


def exact(case, seed):
    if case["kind"] not in ("train", "infer"):
        return None
    H, L, n = case["H"], case["L"], case["n"]
    st = prepare(case, seed)
    g = st["graph"]
    xyz, nin = st["xyz"].double(), st["node_in"].double()
    recv, send = g["recv"].long(), g["col"].long()
    gid = g["gid"].long() if "gid" in g else torch.arange(n, device=xyz.device)
    inner = g["hop"] == 0 if "hop" in g else torch.ones(n, dtype=torch.bool, device=xyz.device)
    tgt = st["targets"].double() if st["targets"] is not None else None
    flat = st["params"].double()
    st.clear()
    flat.requires_grad_(case["kind"] == "train")
    w, at = {}, 0
    feats = [nin[gid]]
    for q in range(case["fourier"]):
        ang = (2 << q) * math.pi * xyz[gid]
        feats += [torch.sin(ang), torch.cos(ang)]
    feats = torch.cat(feats, 1)
    for name, shape, _ in _blocks(H, L, feats.shape[1]):
        k = math.prod(shape)
        w[name] = flat[at:at + k].view(shape)
        at += k
    d = xyz[gid[send]] - xyz[gid[recv]]
    ef = torch.cat([d, d.norm(dim=1, keepdim=True)], 1)

    def layer(l, h, e):
        W = w["e%d.W1" % l]
        m = _mlp(w, "e%d" % l, (h @ W[:H])[recv] + (h @ W[H:2 * H])[send] + e @ W[2 * H:])
        a = torch.zeros_like(h).index_add_(0, recv, m)
        W = w["n%d.W1" % l]
        return h + _mlp(w, "n%d" % l, h @ W[:H] + a @ W[H:]), e + m

    with torch.set_grad_enabled(case["kind"] == "train"):
        h = _mlp(w, "ne", feats @ w["ne.W1"])
        e = _mlp(w, "ee", ef @ w["ee.W1"])
        for l in range(L):
            h, e = checkpoint(layer, l, h, e, use_reentrant=False) if case["kind"] == "train" else layer(l, h, e)
        yb = _mlp(w, "dec", h @ w["dec.W1"])[inner]
        y = torch.zeros((n, OUT), device=xyz.device, dtype=torch.float64)
        y[gid[inner]] = yb.detach()
        if case["kind"] == "infer":
            return {"y": y}
        loss = ((yb - tgt[gid[inner]]) ** 2).sum() / (OUT * n)
        grad, = torch.autograd.grad(loss, flat)
    return {"loss": loss.detach(), "y": y, "grad": grad}
