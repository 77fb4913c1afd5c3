"""The work that this library's speed is judged by: calls of the public entry points as a
user's program makes them, over the range of sizes that the package's own workloads span
(synth.single_pair, torus_sequence, ellipsoid_pair, batched_job): 1k to 200k points per frame,
162 to 100k template vertices, 3 to 5 grid levels of 4 to 256 vertices per axis, both payloads.

Kinds of case:
  step          the next `iters` iterations of an open frame (pdg_step), then the template at the
                updated grids (pdg_deform): the body of every fit
  batch         the same for several sequences advanced together (pdg_batch_step): serving
  frame         one whole frame of a sequence (pdg_fit_frame and pdg_get_vertices): set-up,
                iterations, advance to the next frame
  eval          loss and gradients of all grid levels at given grids (autograd.grid_loss and its
                backward): the differentiable use, an external optimiser's step
  precondition  the grid preconditioner of one level on a given gradient (pdg_precondition)
  static        the same without a context and without allocation (pdg_precondition_static)
  deform        a frame's deformation applied to arbitrary points (pdg_deform): dense
                attributes, other meshes
  fit_mesh      iterations of the template fit to a keyframe cloud (pdg_fit_mesh)

Which outputs: the isometry term's gradient is the sign of each edge's stretch, and Adam divides
every gradient by its own size, so where a value is zero in exact arithmetic (a grid vertex far
from every point, an edge moved rigidly in the first iterations of a zero-initialised frame) the
sign of a rounding error decides.  Steps therefore start from given grids and return moved points,
which only the well-determined vertices near the points reach, and the frames run without the
isometry term (the paper's ablation); gradients come whole from the eval and the preconditioner
cases, which have no such step between input and output.
"""
import functools
import math

import numpy as np
import torch

from paper_2509_18097_gb300 import binding as B
from paper_2509_18097_gb300 import synth
from paper_2509_18097_gb300.autograd import grid_loss

AXES = {"ellipsoid": (1.0, 0.7, 0.5), "sphere": (1.0, 1.0, 1.0)}
SIGMA = 0.01  # grid values of a fit in progress, N(0, SIGMA^2)
LR0 = 2.5e-4  # a late, small learning rate (a twentieth of the default): one flipped sign moves a point by little
ALPHA, W_ISO = 5.56, 250.0
MAX_POW2 = 128  # largest level of the Cayley payload


def _res(text):
    return tuple(int(n) for n in text.split("/"))


def listed():
    return [
        # the small single-pair fit: latency and launches are all there is
        dict(name="step_2k", kind="step", shape="sphere", mesh=8, n_src=2048, n_tgt=2048, res="8/16/32",
             payload="displacement", iters=4),
        # one sequence of the paper's frame size (20k points, some dropped) with its 6-D payload
        dict(name="step_cayley_20k", kind="step", shape="torus", mesh=100, n_src=20000, n_tgt=18013,
             res="16/32/64/128", payload="cayley", iters=4),
        # the benchmark's frame pair: 50 412 vertices, 100k + 100k points
        dict(name="step_100k", kind="step", shape="ellipsoid", mesh=71, n_src=100000, n_tgt=100000,
             res="16/32/64/128", payload="displacement", iters=4),
        # the largest served job: 200k points, finest level 256^3
        dict(name="step_200k_256", kind="step", shape="ellipsoid", mesh=100, n_src=200000, n_tgt=199999,
             res="16/32/64/128/256", payload="displacement", iters=4),
        # serving: eight sequences of different sizes in one step, most levels not a power of two
        dict(name="batch_8", kind="batch", jobs=8, n_pts=12000, finest=108, iters=3),
        # a frame of the noisy torus sequence, forth and back between two clouds
        dict(name="frame_20k", kind="frame", shape="torus", mesh=100, n_src=18013, n_tgt=18013, res="16/32/64/128",
             payload="displacement", iters=8),
        # loss and gradients for an outer optimiser at the benchmark's size
        dict(name="eval_100k", kind="eval", shape="ellipsoid", mesh=71, n_src=100000, n_tgt=100000,
             res="16/32/64/128", w_iso=W_ISO),
        # the preconditioner alone at the largest level, and at a size with a factor 3
        dict(name="precondition_256", kind="precondition", n=256, lam=1.265625),
        dict(name="precondition_108", kind="precondition", n=108, lam=0.84375),
        # the allocation-free form on a small grid: a handful of launches
        dict(name="static_32", kind="static", n=32, lam=0.375),
        # a dense cloud carried along with a fitted frame
        dict(name="deform_1m", kind="deform", n=1000003, res="16/32/64/128", payload="displacement"),
        # the keyframe's template fit at the benchmark's mesh, the paper's lambda
        dict(name="fit_mesh_50k", kind="fit_mesh", mesh=71, n=100000, lam=16.0, iters=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _levels(rng, most, pow2):
    finest = math.exp(rng.uniform(math.log(32), math.log(min(most, MAX_POW2) if pow2 else most)))
    L = rng.randint(3, 5)
    r = [finest / 2 ** (L - 1 - l) for l in range(L)]
    r = [2 ** int(round(math.log2(max(n, 4.0)))) if pow2 else max(4, synth.smooth23(n)) for n in r]
    return "/".join(str(n) for n in r)


def draw(rng):
    kind = rng.choice(["step", "step", "batch", "frame", "eval", "precondition", "static", "deform", "fit_mesh"])
    if kind in ("step", "frame", "eval"):
        n = _log(rng, 1000, {"step": 150000, "frame": 50000, "eval": 100000}[kind])
        shape = rng.choice(["sphere", "ellipsoid", "torus"])
        mesh = max(4, int(round(math.sqrt(n / (4 if shape == "torus" else 20)))))
        c = dict(kind=kind, shape=shape, mesh=mesh, n_src=n, n_tgt=max(500, int(n * rng.uniform(0.7, 1.1))))
        if kind == "eval":
            return dict(c, res=_levels(rng, 192, False), w_iso=rng.choice([0.0, W_ISO]))
        payload = rng.choice(["displacement"] * 3 + ["cayley"])
        c.update(res=_levels(rng, MAX_POW2 if payload == "cayley" else 192, payload == "cayley" or rng.random() < 0.4),
                 payload=payload, iters=rng.randint(1, 4) if kind == "step" else rng.randint(2, 8))
        return c
    if kind == "batch":
        return dict(kind=kind, jobs=rng.randint(2, 8), n_pts=_log(rng, 1000, 12000), finest=_log(rng, 32, 108),
                    iters=rng.randint(1, 3))
    if kind == "precondition":
        return dict(kind=kind, n=rng.choice(synth.SMOOTH_SIZES), lam=round(rng.uniform(0.25, 4.0), 4))
    if kind == "static":
        return dict(kind=kind, n=2 ** rng.randint(1, 6), lam=round(rng.uniform(0.25, 4.0), 4))
    if kind == "deform":
        payload = rng.choice(["displacement", "cayley"])
        return dict(kind=kind, n=_log(rng, 100, 1000000), payload=payload,
                    res=_levels(rng, MAX_POW2 if payload == "cayley" else 192, payload == "cayley"))
    return dict(kind=kind, mesh=_log(rng, 4, 71), n=_log(rng, 1000, 100000), lam=round(rng.uniform(1.0, 32.0), 3),
                iters=rng.randint(1, 4))


# ------------------------------------------------------------------------------------ inputs


@functools.lru_cache(maxsize=32)
def _mesh(shape, k):
    """Template (vertices, edges): a geodesic sphere or ellipsoid of frequency k, a 2k x k torus."""
    v, _, e = synth.torus_mesh(2 * k, k) if shape == "torus" else synth.geodesic_sphere(k, AXES[shape])
    return v, e


def _cloud(rng, shape, n, s):
    """n points of the frame at deformation s in [0, 1] (0: the template's own surface)."""
    if shape == "torus":  # noisy scan, as torus_sequence_frame
        p = synth.twist_bend(synth.torus_points(rng, n), 0.1 * s)
        p = p + 0.002 * rng.standard_normal(p.shape)
    else:
        p = synth.sinusoid(synth.ellipsoid_points(rng, n, AXES[shape]), (0.05 if shape == "ellipsoid" else 0.1) * s)
    return p.astype(np.float32)


def _rng(seed):
    return np.random.Generator(np.random.PCG64(seed))


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _thetas(seed, res, channels, sigma=SIGMA):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return [torch.randn((n**3, channels), generator=g, device="cuda") * sigma for n in res]


class _Handle:
    """Owns a context or a batch for as long as a state lives."""

    def __init__(self, h, destroy):
        self.h, self.destroy = h, destroy

    def __del__(self):
        self.destroy(self.h)


def _context(v, e, src, max_pts, **cfg):
    return _Handle(B.pdg_create(B.pdg_config_default(**cfg), v, e, src, max_pts=max_pts), B.pdg_destroy)


def _open_frame(case, seed):
    """A context in an open frame, started from given grids."""
    res, payload = _res(case["res"]), case.get("payload", "displacement")
    r = _rng(seed)
    v, e = _mesh(case["shape"], case["mesh"])
    src, tgt = _cloud(r, case["shape"], case["n_src"], 0.0), _cloud(r, case["shape"], case["n_tgt"], 1.0)
    ctx = _context(v, e, src, max(len(src), len(tgt)), res=res, payload=payload, lr0=LR0,
                   w_iso=case.get("w_iso", W_ISO))
    B.pdg_begin_frame(ctx.h, _dev(tgt))
    th = _thetas(seed, res, 6 if payload == "cayley" else 3)
    for l, t in enumerate(th):
        B.pdg_write_theta(ctx.h, l, t)
    return ctx, _dev(v), th


def _batch_cases(case, seed):
    """The members of a batch: sizes spread a factor of four around the case's, like batched_job."""
    r = _rng(1000 + case["jobs"])  # the mix is the case's own; the clouds are the seed's
    out = []
    for i in range(case["jobs"]):
        n = int(case["n_pts"] * math.exp(r.uniform(-0.7, 0.7)))
        shape = ("sphere", "torus", "ellipsoid")[i % 3]
        L = 3 + i % 3
        finest = max(16, case["finest"] * math.exp(r.uniform(-0.7, 0.0))) if i else case["finest"]
        res = [max(4, synth.smooth23(finest / 2 ** (L - 1 - l))) for l in range(L)]
        out.append(dict(shape=shape, mesh=max(4, int(math.sqrt(n / (4 if shape == "torus" else 20)))), n_src=n,
                        n_tgt=max(500, int(n * r.uniform(0.8, 1.1))), res="/".join(map(str, res))))
    return [(c, seed * 64 + i) for i, c in enumerate(out)]


def _dense(seed, n):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn((n**3, 3), generator=g, device="cuda")


def prepare(case, seed):
    kind = case["kind"]
    s = dict(kind=kind, iters=case.get("iters"))
    if kind == "step":
        s["ctx"], s["verts"], _ = _open_frame(case, seed)
    elif kind == "eval":
        s["ctx"], _, th = _open_frame(case, seed)
        s["thetas"] = [t.reshape(n, n, n, 3).requires_grad_() for t, n in zip(th, _res(case["res"]))]
    elif kind == "batch":
        members = [_open_frame(c, sd) for c, sd in _batch_cases(case, seed)]
        s["ctxs"], s["verts"] = [m[0] for m in members], [m[1] for m in members]
        s["batch"] = _Handle(B.pdg_batch_create(len(members)), B.pdg_batch_destroy)
        B.pdg_batch_set(s["batch"].h, [c.h for c in s["ctxs"]])
    elif kind == "frame":
        r = _rng(seed)
        v, e = _mesh(case["shape"], case["mesh"])
        src = _cloud(r, case["shape"], case["n_src"], 0.0)
        s["frames"] = [_dev(_cloud(r, case["shape"], case["n_tgt"], 1.0)), _dev(src)]
        s["ctx"] = _context(v, e, src, max(case["n_src"], case["n_tgt"]), res=_res(case["res"]),
                            payload=case["payload"], lr0=LR0, w_iso=0.0)
        s["n"], s["at"] = len(v), 0
    elif kind in ("precondition", "static"):
        s.update(n=case["n"], lam=case["lam"], g=_dense(seed, case["n"]))
        if kind == "precondition":
            v, e = _mesh("sphere", 4)
            s["ctx"] = _context(v, e, v, len(v), res=(case["n"],), lambda0=case["lam"])
    elif kind == "deform":
        v, e = _mesh("ellipsoid", 8)
        res = _res(case["res"])
        s["ctx"] = _context(v, e, v, len(v), res=res, payload=case["payload"])
        for l, t in enumerate(_thetas(seed, res, 6 if case["payload"] == "cayley" else 3)):
            B.pdg_write_theta(s["ctx"].h, l, t)
        s["pts"] = _deform_points(case, seed)
    else:
        s.update(lam=case["lam"], **_mesh_inputs(case, seed))
        s["ctx"] = _context(s["v"], s["e"], s["p0"], len(s["p0"]), res=(8, 16))
        s["p0"] = _dev(s["p0"])
    torch.cuda.synchronize()
    return s


def _deform_points(case, seed):
    return _dev(_cloud(_rng(seed), "ellipsoid", case["n"], 0.5))


def _mesh_inputs(case, seed):
    v, e = _mesh("ellipsoid", case["mesh"])
    p0 = synth.sinusoid(synth.ellipsoid_points(_rng(seed), case["n"]), 0.02).astype(np.float32)
    return dict(v=v, e=e, p0=p0)


# ------------------------------------------------------------------------------------ a pass


def _moved(ctx, verts):
    return B.pdg_deform(ctx.h, verts, torch.empty_like(verts))


def run(s):
    kind = s["kind"]
    if kind == "step":
        B.pdg_step(s["ctx"].h, s["iters"])
        return _moved(s["ctx"], s["verts"])
    if kind == "batch":
        B.pdg_batch_step(s["batch"].h, s["iters"])
        return [_moved(c, v) for c, v in zip(s["ctxs"], s["verts"])]
    if kind == "frame":
        st = B.pdg_fit_frame(s["ctx"].h, s["frames"][s["at"]], s["iters"])
        s["at"] ^= 1
        out = torch.empty((s["n"], 3), device="cuda")
        return [B.pdg_get_vertices(s["ctx"].h, out), st.loss_total, st.cd_mesh, st.cd_pts]
    if kind == "eval":
        loss = grid_loss(s["ctx"].h, s["thetas"])
        # the loss has single precision: its terms are summed in 32 bits
        return [loss.detach().float(), *torch.autograd.grad(loss, s["thetas"])]
    if kind == "precondition":
        return B.pdg_precondition(s["ctx"].h, 0, s["g"], torch.empty_like(s["g"]))
    if kind == "static":
        out = torch.empty_like(s["g"])
        if B.pdg_precondition_static(s["n"], s["lam"], s["g"], out) != B.OK:
            raise RuntimeError("pdg_precondition_static failed")
        return out
    if kind == "deform":
        return _moved(s["ctx"], s["pts"])
    st = B.pdg_fit_mesh(s["ctx"].h, s["p0"], s["iters"], s["lam"])
    x, pg = torch.empty((len(s["v"]), 3), device="cuda"), torch.empty((len(s["v"]), 3), device="cuda")
    return [B.pdg_get_vertices(s["ctx"].h, x), B.pdg_read(s["ctx"].h, B.BUF_MESH_PGRAD, 0, pg), st.loss_total]


# ------------------------------------------------------------------------------------ work


def _mesh_size(shape, k):
    return (2 * k * k, 6 * k * k) if shape == "torus" else (10 * k * k + 2, 30 * k * k)


def _step_work(c, update):
    """One iteration: points, targets and edges in, the touched grid values; with the update the
    grids and both Adam moments in and out, else the gradients out."""
    C = 6 if c.get("payload") == "cayley" else 3
    V, E = _mesh_size(c["shape"], c["mesh"])
    Q, M, res = V + c["n_src"], c["n_tgt"], _res(c["res"])
    G, G_near = sum(n**3 for n in res), sum(min(n**3, 8 * Q) for n in res)
    flops = Q * len(res) * 8 * C * 4 + 30 * 8 * (Q + 2 * M) + 30 * E
    moved = 24 * Q + 12 * M + 12 * E
    if not update:
        return dict(bytes=moved + 4 * C * (G_near + G), flops=flops)
    fft = sum(6 * 2.5 * n**3 * max(1.0, math.log2(n)) for n in res if n > 1) * C
    return dict(bytes=moved + 4 * C * 6 * G, flops=flops + fft + 12 * C * G)


def _times(w, k):
    return {x: k * y for x, y in w.items()}


def _sum(ws):
    return {x: sum(w[x] for w in ws) for x in ("bytes", "flops")}


def work(case):
    kind = case["kind"]
    if kind == "step":
        return _times(_step_work(case, True), case["iters"])
    if kind == "batch":
        return _sum([_times(_step_work(c, True), case["iters"]) for c, _ in _batch_cases(case, 0)])
    if kind == "frame":
        return _sum([_times(_step_work(case, True), case["iters"]), dict(bytes=24 * case["n_tgt"], flops=0)])
    if kind == "eval":
        return _step_work(case, False)
    if kind in ("precondition", "static"):
        n = case["n"]
        return dict(bytes=24 * n**3, flops=6 * 2.5 * 3 * n**3 * max(1.0, math.log2(n)))
    C = 6 if case.get("payload") == "cayley" else 3
    if kind == "deform":
        res = _res(case["res"])
        near = sum(min(n**3, 8 * case["n"]) for n in res)
        return dict(bytes=24 * case["n"] + 4 * C * near, flops=case["n"] * len(res) * 8 * C * 2)
    V, E = _mesh_size("ellipsoid", case["mesh"])
    # points in, matches and gradient; two solves that read and write the vertices and the edges
    return dict(bytes=case["iters"] * (12 * case["n"] + 24 * V + 2 * (24 * V + 8 * E) + 72 * V),
                flops=case["iters"] * (30 * 8 * (case["n"] + V) + 2 * 100 * (12 * E + 12 * V)))


# ------------------------------------------------------------------------------------ in 64 bits


def _corners(x, n, lo=-1.5, hi=1.5):
    """Vertex indices and trilinear weights [N, 8] of points x in a level of n vertices per axis."""
    u = ((x - lo) / (hi - lo) * (n - 1)).clamp(0, n - 1)
    i = u.floor().clamp(max=n - 2)
    f, i = u - i, i.long()
    idx, w = [], []
    for d in range(8):
        b = [d & 1, d >> 1 & 1, d >> 2]
        idx.append(((i[:, 2] + b[2]) * n + i[:, 1] + b[1]) * n + i[:, 0] + b[0])
        w.append(math.prod(f[:, a] if b[a] else 1 - f[:, a] for a in range(3)))
    return torch.stack(idx, 1), torch.stack(w, 1)


def _deformed(x, thetas, res):
    """The points x [N, 3] moved by the level average of the grids, payload by channel count."""
    T = torch.zeros((len(x), thetas[0].shape[1]), dtype=torch.float64, device=x.device)
    for t, n in zip(thetas, res):
        idx, w = _corners(x, n)
        for c in range(8):
            T += w[:, c : c + 1] * t[idx[:, c]].double()
    T /= len(res)
    if T.shape[1] == 3:
        return x + T
    z, t = T[:, :3], T[:, 3:]
    Z = torch.zeros((len(x), 3, 3), dtype=torch.float64, device=x.device)
    Z[:, 0, 1], Z[:, 0, 2], Z[:, 1, 2] = -z[:, 2], z[:, 1], -z[:, 0]
    Z = Z - Z.transpose(1, 2)
    eye = torch.eye(3, dtype=torch.float64, device=x.device)
    return ((eye + Z) @ torch.linalg.solve(eye - Z, x.unsqueeze(2))).squeeze(2) + t


def _nearest(a, b):
    """Index of the nearest point of b for every point of a, by exhaustive search."""
    chunk = max(1, (1 << 26) // len(b))
    out = []
    for s in range(0, len(a), chunk):
        q = a[s : s + chunk]
        d = sum((q[:, k : k + 1] - b[None, :, k]) ** 2 for k in range(3))
        out.append(d.argmin(1))
    return torch.cat(out)


def _chamfer(a, b):
    """Robust Chamfer distance of a (differentiable) and b."""
    with torch.no_grad():
        ab, ba = _nearest(a, b), _nearest(b, a)
    phi = lambda s: (s * torch.exp(-ALPHA * s)).mean()  # noqa: E731
    return phi(((a - b[ab]) ** 2).sum(1)) + phi(((a[ba] - b) ** 2).sum(1))


def _exact_eval(case, seed):
    res = _res(case["res"])
    r = _rng(seed)
    v, e = _mesh(case["shape"], case["mesh"])
    src, tgt = _cloud(r, case["shape"], case["n_src"], 0.0), _cloud(r, case["shape"], case["n_tgt"], 1.0)
    x, tgt, e = _dev(np.concatenate([v, src])).double(), _dev(tgt).double(), _dev(e).long()
    th = [t.double().requires_grad_() for t in _thetas(seed, res, 3)]
    y, V = _deformed(x, th, res), len(v)
    length = lambda p: ((p[e[:, 0]] - p[e[:, 1]]) ** 2).sum(1).sqrt()  # noqa: E731
    iso = (length(y) - length(x)).abs().mean()
    loss = _chamfer(y[:V], tgt) + _chamfer(y[V:], tgt) + case["w_iso"] * iso
    grads = torch.autograd.grad(loss, th)
    return [loss.detach(), *(g.reshape(n, n, n, 3) for g, n in zip(grads, res))]


def _exact_precondition(g, n, lam):
    """(I + lam L)^-2 in the cosine basis that diagonalises the free-boundary grid Laplacian."""
    k = torch.arange(n, dtype=torch.float64, device=g.device)
    Cm = torch.cos(math.pi * k[:, None] * (k[None, :] + 0.5) / n) * math.sqrt(2.0 / n)
    Cm[0] /= math.sqrt(2.0)
    mu = 4 * torch.sin(math.pi * k / (2 * n)) ** 2
    scale = (1 + lam * (mu[:, None, None] + mu[None, :, None] + mu[None, None, :])) ** -2.0
    out = torch.empty((n**3, 3), dtype=torch.float64, device=g.device)
    for c in range(3):
        a = g[:, c].double().reshape(n, n, n)
        for m in (Cm, None, Cm.T):
            if m is None:
                a = a * scale
            else:
                for _ in range(3):  # transform the last axis, bring the next one to its place
                    a = (a.reshape(-1, n) @ m.T).reshape(n, n, n).permute(2, 0, 1).contiguous()
        out[:, c] = a.reshape(-1)
    return out


def _exact_fit_mesh(case, seed):
    m = _mesh_inputs(case, seed)
    x, p0, e = _dev(m["v"]).double(), _dev(m["p0"]).double(), _dev(m["e"]).long()

    def apply(h):
        d = case["lam"] * (h[e[:, 0]] - h[e[:, 1]])
        return h.index_add(0, e[:, 0], d).index_add(0, e[:, 1], d, alpha=-1)

    def solve(b):  # conjugate gradients on I + lam L, per channel
        h, r, p = torch.zeros_like(b), b, b
        rr = (r * r).sum(0)
        for _ in range(400):
            q = apply(p)
            a = rr / (p * q).sum(0).clamp(min=1e-300)
            h, r = h + a * p, r - a * q
            new = (r * r).sum(0)
            if bool((new <= 1e-28 * (b * b).sum(0)).all()):
                break
            p, rr = r + new / rr.clamp(min=1e-300) * p, new
        return h

    m1, m2 = torch.zeros_like(x), torch.zeros_like(x)
    lr = float(np.float32(B.MESH_LR))
    for k in range(1, case["iters"] + 1):
        x = x.detach().requires_grad_()
        loss = _chamfer(x, p0)
        pg = solve(solve(torch.autograd.grad(loss, x)[0]))
        m1, m2 = 0.9 * m1 + 0.1 * pg, 0.999 * m2 + 0.001 * pg * pg
        x = x.detach() - lr * (m1 / (1 - 0.9**k)) / ((m2 / (1 - 0.999**k)).sqrt() + 1e-8)
    return [x, pg, float(loss.detach())]


def exact(case, seed):
    kind = case["kind"]
    if kind == "eval":
        return _exact_eval(case, seed)
    if kind in ("precondition", "static"):
        return _exact_precondition(_dense(seed, case["n"]), case["n"], float(np.float32(case["lam"])))
    if kind == "deform":
        res = _res(case["res"])
        th = _thetas(seed, res, 6 if case["payload"] == "cayley" else 3)
        return torch.cat([_deformed(x.double(), th, res) for x in _deform_points(case, seed).split(1 << 18)])
    if kind == "fit_mesh":
        return _exact_fit_mesh(case, seed)
    return None  # iterations of the fit: signs decided by rounding (see above) set trajectories apart
