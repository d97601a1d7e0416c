"""The measured cases: what a program that uses this solver has it do, through the Python binding.

A case is a dict of plain values; `listed()` holds the ones that are always timed and `draw()`
gives more of the same ranges.  The kinds are the calls of the public interface:

  operator     one product with the boundary operator (eq. discrete_sys of the paper)
  targets      the double layer at points in the domain (a plot, a probe, a coupled code)
  gmres        one boundary solve from a zero start
  matrix_free  the same solve with the operator in its matrix-free form
  volume       the volume potential at every tree node
  step         one heat step of a running trajectory
  batch        one step of several problems by a graph launch
  net          loss and gradient of the learned start's network on a minibatch

Domains are the unit disk minus a circle ("annulus") or minus five-armed starfish holes
("starfish").  Data are smooth: densities and right-hand sides are trigonometric on each curve,
and the trajectories of the step cases are manufactured from u = V + W with V a sum of Gaussians
that vanish at the boundary (so that B, extended by zero, stays smooth) and W homogeneous,
W - alpha^2 Lap W = 0, from sources outside the domain.  Mixed precision has binary32 accuracy,
and its fields and products are kept in binary32, as a program that asks for it records them.
"""
import functools
import json
import math

import numpy as np
import torch

import paper_1007_5335_gb300 as mh

DEV = "cuda"
TAU = 2.0 * math.pi
CYCLE = 32          # time levels after which a trajectory's data repeat


def listed():
    star = {"domain": "starfish", "holes": 5, "npc": 1024, "geometry": 2, "alpha2": 1e-3}
    ring = {"domain": "annulus", "holes": 1, "npc": 128, "geometry": 0, "alpha2": 1e-2}
    tree = {"q": 8, "min_level": 4, "max_level": 8, "tol": 2e-9, "p": 20}
    return [
        # the smallest call: a product with the operator of the two-circle domain (latency)
        {"name": "operator_small_f64", "kind": "operator", "prec": 0, **ring},
        # a product with the stored operator of the starfish domain, 302 MB of binary64
        {"name": "operator_large_f64", "kind": "operator", "prec": 0, **star},
        # a field probed at scattered points of the domain, accurately
        {"name": "targets_f64", "kind": "targets", "prec": 0, "targets": 2000, **star},
        # a stationary problem: one solve to the tolerance the paper uses
        {"name": "gmres_mixed", "kind": "gmres", "prec": 1, **star},
        # a long boundary, where the matrix-free form is taken for its memory
        {"name": "matrix_free_f64", "kind": "matrix_free", "prec": 0, **dict(star, npc=2048),
         "q": 8, "min_level": 4, "max_level": 8, "tol": 1e-6, "p": 20},
        # the volume potential alone, on the adaptive tree of the benchmark's size
        {"name": "volume_mixed", "kind": "volume", "prec": 1, "geometry": 2, "alpha2": 1e-3, **dict(tree, tol=5e-10)},
        # ... and in binary64 with an odd number of nodes per box side and a lower order
        {"name": "volume_f64", "kind": "volume", "prec": 0, "geometry": 3, "alpha2": 2.7e-3,
         "q": 5, "min_level": 4, "max_level": 7, "tol": 2e-7, "p": 15},
        # a step of the small problem with caller-supplied extension: launches and host round trips
        {"name": "step_small_f64", "kind": "step", "prec": 0, "ext": "array", **ring,
         "q": 4, "min_level": 4, "max_level": 4, "tol": 0.0, "p": 20},
        # the benchmark's size in the two precisions, step by step
        {"name": "step_mixed", "kind": "step", "prec": 1, "ext": "const", **star, **tree},
        {"name": "step_f64", "kind": "step", "prec": 0, "ext": "const", **star, **tree},
        # independent problems of uneven size advanced together
        {"name": "batch_mixed", "kind": "batch", "prec": 1, "problems": 4, "holes": 3, "npc": 480, "geometry": 11,
         "domain": "starfish", "alpha2": 1.5e-3, "q": 8, "min_level": 4, "max_level": 6, "tol": 1e-6, "p": 16},
        # a minibatch of the learned start's training on the starfish boundary
        {"name": "net_grad", "kind": "net", "samples": 64, "modes": 256, "width": 256, **star},
    ]


def draw(rng):
    def log(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    def even(lo, hi):
        # half of the curves have a power of two nodes, the others any even count
        n = log(lo, hi)
        return 2 ** int(round(math.log2(n))) if rng.random() < 0.5 else 2 * int(round(n / 2))

    kind = rng.choice(("operator", "targets", "gmres", "matrix_free", "volume", "step", "step", "batch", "net"))
    case = {"kind": kind, "prec": rng.randrange(2), "geometry": rng.randrange(2, 1000)}
    if kind != "volume":
        ring = kind in ("operator", "gmres", "step") and rng.random() < 0.25
        case["domain"] = "annulus" if ring else "starfish"
        case["holes"] = 1 if ring else rng.randint(1, 6)
        npc = even(96, 512) if ring else even(256, 1024)
        case["npc"] = max(96, min(npc, 1024))
        # a screening length the boundary grid resolves, up to the paper's largest
        case["alpha2"] = round(log(max(1e-4, (TAU / case["npc"]) ** 2), 1e-2), 7)
    else:
        case["alpha2"] = round(log(1e-4, 1e-2), 7)
    if kind in ("volume", "step", "batch", "matrix_free"):
        case["q"] = rng.choice((4, 5, 6, 7, 8, 8))
        case["min_level"] = rng.choice((4, 4, 5)) if case["q"] < 8 else 4
        case["max_level"] = rng.randint(6, 8)
        case["tol"] = float("%.2g" % log({4: 1e-4, 5: 1e-5, 6: 1e-6, 7: 1e-7, 8: 1e-8}[case["q"]], 1e-2))
        case["p"] = rng.randint(10, 24)
    if kind == "targets":
        case["targets"] = int(log(50, 1900))
    if kind == "matrix_free":
        case["prec"], case["p"] = 0, max(18, case["p"])
    if kind == "step":
        case["ext"] = rng.choice(("const", "const", "array"))
    if kind == "batch":
        case.update(problems=rng.randint(2, 4), holes=rng.randint(1, 3), npc=min(case["npc"], 512), prec=1)
        case["alpha2"] = max(case["alpha2"], round((TAU / case["npc"]) ** 2, 7))
        case["max_level"] = 6
    if kind == "net":
        case["prec"], case["samples"] = 1, int(log(1, 500))
        case["modes"] = 4 * rng.randint(4, case["npc"] // 8)
        case["width"] = 8 * rng.randint(2, 48)
    return case


# ------------------------------------------------------------------ domains

def _curves(case):
    """(cx, cy, r0, eps, s, N) per curve: r(t) = r0 (1 + eps cos 5t), y = cy + s r sin t."""
    n = case["npc"]
    out = [(0.0, 0.0, 1.0, 0.0, 1.0, n)]
    if case["domain"] == "annulus":
        return out + [(0.2, 0.0, 0.3, 0.0, -1.0, n)]
    r0 = min(0.12, 0.27 / math.sqrt(case["holes"]))
    reach, gap = 1.3 * r0, 0.05
    rng = np.random.default_rng([case["geometry"], 17])
    lim = 1.0 - reach - gap
    while len(out) <= case["holes"]:
        c = rng.uniform(-lim, lim, 2)
        if math.hypot(*c) <= lim and all(math.hypot(c[0] - k[0], c[1] - k[1]) >= 2 * reach + gap for k in out[1:]):
            out.append((float(c[0]), float(c[1]), r0, 0.3, -1.0, n))
    return out


def _on_curve(c, t):
    """Position, first and second parameter derivative of curve c at t, each (n, 2)."""
    cx, cy, r0, eps, s, _ = c
    r, r1, r2 = r0 * (1 + eps * np.cos(5 * t)), -5 * r0 * eps * np.sin(5 * t), -25 * r0 * eps * np.cos(5 * t)
    co, si = np.cos(t), np.sin(t)
    p = np.stack([cx + r * co, cy + s * r * si], 1)
    d = np.stack([r1 * co - r * si, s * (r1 * si + r * co)], 1)
    dd = np.stack([r2 * co - 2 * r1 * si - r * co, s * (r2 * si + 2 * r1 * co - r * si)], 1)
    return p, d, dd


def _nodes_of(case, times=1):
    return [_on_curve(c, TAU * np.arange(times * c[5]) / (times * c[5]))[0] for c in _curves(case)]


def _gap(c, xy):
    """Radial distance of points from curve c, positive on the side of the domain."""
    t = np.arctan2(c[4] * (xy[:, 1] - c[1]), xy[:, 0] - c[0])
    return c[4] * (c[2] * (1 + c[3] * np.cos(5 * t)) - np.hypot(xy[:, 0] - c[0], xy[:, 1] - c[1]))


def _inside(case, xy):
    ok = np.ones(len(xy), bool)
    for c in _curves(case):
        ok &= _gap(c, xy) > 0
    return ok


# ------------------------------------------------------------------ meshes

_KEYS = ("kind", "domain", "holes", "npc", "geometry", "q", "min_level", "max_level", "tol")


def _key(case):
    return json.dumps({k: case[k] for k in _KEYS if k in case}, sort_keys=True)


@functools.lru_cache(maxsize=32)
def _gaussians(key):
    """Centres and widths of the Gaussians of V: far enough from every curve to vanish there."""
    case = json.loads(key)
    rng = np.random.default_rng([case["geometry"], 29])
    if "domain" not in case:
        ang, rad = rng.uniform(0, TAU, 20), 0.6 * np.sqrt(rng.uniform(0, 1, 20))
        return np.stack([rad * np.cos(ang), rad * np.sin(ang), rng.uniform(0.025, 0.06, 20)], 1)
    dense = np.concatenate([_on_curve(c, TAU * np.arange(400) / 400)[0] for c in _curves(case)])
    out = []
    while len(out) < 20:
        xy = rng.uniform(-0.9, 0.9, 2)
        if not _inside(case, xy[None])[0]:
            continue
        s = np.min(np.hypot(dense[:, 0] - xy[0], dense[:, 1] - xy[1])) / 6.8
        if s >= 0.018:
            out.append((xy[0], xy[1], min(s, rng.uniform(0.018, 0.06))))
    return np.array(out)


def _refine_field(key):
    g = _gaussians(key)

    def field(xy):
        out = np.zeros(len(xy))
        for i, (cx, cy, s) in enumerate(g):
            out += (1.0 if i % 2 else -1.0) * np.exp(-((xy[:, 0] - cx) ** 2 + (xy[:, 1] - cy) ** 2) / (2 * s * s))
        return out
    return field


def _grid(l, ix, iy, xi):
    w = 2.0 / (1 << l)
    x = -1.0 + (ix[:, None, None] + 0.5) * w + 0.5 * w * xi[None, None, :]
    y = -1.0 + (iy[:, None, None] + 0.5) * w + 0.5 * w * xi[None, :, None]
    return np.stack(np.broadcast_arrays(x, y), -1).reshape(-1, 2)


@functools.lru_cache(maxsize=8)
def _mesh(key):
    """The volume nodes in tree order (Morton order of the leaves, then iy q + ix), in plain numpy."""
    case = json.loads(key)
    q, lmin, lmax = case["q"], case["min_level"], case["max_level"]
    xi = np.polynomial.legendre.leggauss(q)[0]
    half = np.concatenate([0.5 * xi - 0.5, 0.5 * xi + 0.5])         # the children's nodes on the parent's axis
    L = np.ones((2 * q, q))
    for a in range(q):
        for m in range(q):
            if m != a:
                L[:, a] *= (half - xi[m]) / (xi[a] - xi[m])
    field = _refine_field(key) if case["tol"] > 0 and lmax > lmin else None
    split = [np.zeros((1 << l, 1 << l), bool) for l in range(lmax + 1)]
    have = [np.zeros((1 << l, 1 << l), bool) for l in range(lmax + 1)]
    have[0][0, 0] = True
    for l in range(lmax):
        ix, iy = np.nonzero(have[l])
        if l < lmin:
            go = np.ones(len(ix), bool)
        elif field is None:
            break
        else:
            own = field(_grid(l, ix, iy, xi)).reshape(-1, q, q)
            both = np.einsum("va,nab,ub->nvu", L, own, L)
            w = 2.0 / (1 << l)
            x = -1.0 + (ix[:, None] + 0.5) * w + 0.5 * w * half[None]
            y = -1.0 + (iy[:, None] + 0.5) * w + 0.5 * w * half[None]
            pts = np.stack(np.broadcast_arrays(x[:, None, :], y[:, :, None]), -1).reshape(-1, 2)
            go = np.abs(field(pts).reshape(both.shape) - both).max((1, 2)) > case["tol"]
        split[l][ix[go], iy[go]] = True
        have[l + 1] = np.repeat(np.repeat(split[l], 2, 0), 2, 1)
    for l in range(lmax - 1, 0, -1):                                 # 2:1 balance, edges and corners
        pad = np.pad(split[l], 1)
        near = np.zeros_like(split[l])
        for dx in range(3):
            for dy in range(3):
                near |= pad[dx:dx + near.shape[0], dy:dy + near.shape[1]]
        split[l - 1] |= near.reshape(near.shape[0] // 2, 2, -1, 2).any((1, 3))
    keys, blocks = [], []
    for l in range(lmax + 1):
        have_l = np.ones((1, 1), bool) if l == 0 else np.repeat(np.repeat(split[l - 1], 2, 0), 2, 1)
        ix, iy = np.nonzero(have_l & ~split[l])
        z = np.zeros(len(ix), np.int64)
        for b in range(lmax + 1):
            z |= (((ix << (lmax - l)) >> b) & 1) << (2 * b) | (((iy << (lmax - l)) >> b) & 1) << (2 * b + 1)
        keys.append(z)
        blocks.append(_grid(l, ix, iy, xi).reshape(len(ix), q * q, 2))
    return np.concatenate(blocks)[np.argsort(np.concatenate(keys))].reshape(-1, 2)


def _tree(ctx, case):
    fn = _refine_field(_key(case)) if case["tol"] > 0 and case["max_level"] > case["min_level"] else None
    return mh.Tree(ctx, (-1.0, -1.0, 2.0), case["q"], case["min_level"], case["max_level"], fn,
                   case["tol"] if fn else float("inf"))


# ------------------------------------------------------------------ inputs

def _k0(z):
    return torch.special.modified_bessel_k0(torch.as_tensor(z)).numpy()


class _Field:
    """u(x, k) = V + W at time level k, from the seed; `smooth` takes low trigonometric modes for V
    (problems whose B is extended by the caller), else the Gaussians of the mesh."""

    def __init__(self, case, seed):
        self.a2 = case["alpha2"]
        rng = np.random.default_rng([seed, 5])
        self.smooth = case.get("ext") == "array"
        self.g = rng.integers(-1, 2, (8, 2)).astype(float) if self.smooth else _gaussians(_key(case))
        n = len(self.g)
        self.phase = rng.uniform(0, TAU, n)
        self.src = []
        for c in _curves(case) if "domain" in case else []:
            if c[4] > 0:
                b = rng.uniform(0, TAU)
                self.src.append((1.2 * math.cos(b), 1.2 * math.sin(b), 0.2))
            else:
                self.src.append((c[0], c[1], c[2] * (1 - c[3])))
        self.amp = rng.uniform(0.3, 1.0, n + len(self.src)) * rng.choice((-1.0, 1.0), n + len(self.src))
        self.turn = rng.uniform(0, TAU, n + len(self.src))

    def basis(self, xy, inside=None):
        """V's functions, (1 - alpha^2 Lap) of them, and W's (zero at points outside the domain)."""
        x = torch.as_tensor(xy, device=DEV)
        V, B = [], []
        for i, g in enumerate(self.g):
            if self.smooth:
                v = torch.sin(math.pi * (g[0] * x[:, 0] + g[1] * x[:, 1]) + self.phase[i])
                V.append(v)
                B.append(v * (1 + self.a2 * math.pi ** 2 * (g[0] ** 2 + g[1] ** 2)))
            else:
                d2, s2 = (x[:, 0] - g[0]) ** 2 + (x[:, 1] - g[1]) ** 2, g[2] ** 2
                v = torch.exp(-d2 / (2 * s2))
                V.append(v)
                B.append(v * (1 - self.a2 * (d2 / s2 - 2) / s2))
        at = np.ones(len(xy), bool) if inside is None else inside
        W = np.zeros((len(self.src), len(xy)))
        al = math.sqrt(self.a2)
        for j, (sx, sy, d) in enumerate(self.src):
            W[j, at] = _k0(np.hypot(xy[at, 0] - sx, xy[at, 1] - sy) / al) / _k0(np.array([d / al]))
        return torch.stack(V), torch.stack(B), torch.as_tensor(W, device=DEV)

    def coef(self, k):
        return torch.as_tensor(self.amp * np.cos(TAU * k / CYCLE + self.turn), device=DEV)


def _modes(case, seed, times=1):
    """A smooth periodic function on the curves' nodes (times-fold grids), from the seed."""
    rng, out = np.random.default_rng([seed, 7]), []
    for c in _curves(case):
        t = TAU * np.arange(times * c[5]) / (times * c[5])
        a, f = rng.uniform(-1, 1, 9), rng.uniform(0, TAU, 9)
        out.append(sum(a[m] / (1 + m) * np.cos(m * t + f[m]) for m in range(9)))
    return np.concatenate(out)


def _points(case, seed):
    """Points of the domain, none closer than 0.02 node spacings to a curve."""
    rng, got = np.random.default_rng([seed, 9]), np.zeros((0, 2))
    while len(got) < case["targets"]:
        xy = rng.uniform(-1, 1, (4 * case["targets"], 2))
        ok = np.ones(len(xy), bool)
        for c in _curves(case):
            ok &= _gap(c, xy) > 0.03 * TAU * c[2] * 1.6 / c[5]
        got = np.concatenate([got, xy[ok]])
    return got[:case["targets"]]


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device=DEV)


def _parts(case):
    """The problems of a batch: other holes, other node counts."""
    return [dict(case, kind="step", geometry=case["geometry"] + j, npc=2 * round(case["npc"] * f / 2),
                 holes=1 + (case["holes"] + j) % 3) for j, f in zip(range(case["problems"]), (1.0, 0.8, 0.6, 1.0))]


def _trajectory(ctx, case, seed):
    tree, bnd = _tree(ctx, case), mh.Boundary(ctx, _nodes_of(case), 8)
    array = case.get("ext") == "array"
    prob = mh.Problem(ctx, tree, bnd, case["alpha2"], case["p"], mh.MH_EXT_ARRAY if array else mh.MH_EXT_CONST)
    nodes = tree.nodes().cpu().numpy()
    inside = _inside(case, nodes)
    field, on = _Field(case, seed), _dev(inside).double()
    V, B, W = field.basis(nodes, inside)
    fV, _, fW = field.basis(np.concatenate(_nodes_of(case)))
    s = {"prob": prob, "F": [], "f": [], "b": [], "i": 0, "prec": case["prec"],
         "sigma": torch.zeros(bnd.n, dtype=torch.float64, device=DEV)}
    n = len(V)
    for k in range(CYCLE):
        c, d = field.coef(k), field.coef(k + 1)
        u, b = c[:n] @ V + c[n:] @ W, d[:n] @ B
        s["F"].append((b - u) / case["alpha2"] * on)
        s["f"].append(d[:n] @ fV + d[n:] @ fW)
        s["b"].append(b if array else None)
        if k == 0:
            s["u"] = u * on
    s["un"] = torch.empty_like(s["u"])
    return s


def prepare(case, seed):
    torch.zeros(1, device=DEV)
    ctx, kind = mh.Context(torch.cuda.current_device()), case["kind"]
    s = {"kind": kind, "ctx": ctx, "prec": case.get("prec", 0), "alpha": math.sqrt(case["alpha2"])}
    if kind == "volume":
        s["tree"], s["p"] = _tree(ctx, case), case["p"]
        field = _Field(case, seed)
        _, B, _ = field.basis(s["tree"].nodes().cpu().numpy())
        s["b"] = field.coef(0)[:len(B)] @ B
        s["out"] = torch.empty_like(s["b"])
        mh.mh_volume_potential(ctx, s["tree"], s["alpha"], s["p"], s["b"], s["out"], s["prec"])   # the tables
    elif kind == "step":
        s.update(_trajectory(ctx, case, seed))
    elif kind == "batch":
        s["parts"] = [_trajectory(ctx, c, seed + 1000 * j) for j, c in enumerate(_parts(case))]
        s["batch"] = mh.Batch(ctx, [t["prob"] for t in s["parts"]])
        s["F"], s["f"] = ([t[k][0].clone() for t in s["parts"]] for k in ("F", "f"))
        s["u"], s["sigma"], s["i"] = [t["u"] for t in s["parts"]], [t["sigma"] for t in s["parts"]], 0
    elif kind == "net":
        s["bnd"] = mh.Boundary(ctx, _nodes_of(case), 8)
        s["net"] = mh.Net(ctx, s["bnd"], case["modes"], case["width"])
        par, X, T = _network(case, seed)
        s["net"].set_params(np.concatenate([a.reshape(-1) for a in par]))
        s["X"], s["T"] = _dev(X), _dev(T)
        s["grad"] = torch.empty(s["net"].n_params, dtype=torch.float32, device=DEV)
    else:
        s["bnd"] = mh.Boundary(ctx, _nodes_of(case), 8)
        s["x"] = _dev(_modes(case, seed))
        s["out"] = torch.zeros_like(s["x"])
        if kind == "matrix_free":
            s["tree"] = _tree(ctx, case)
            s["prob"] = mh.Problem(ctx, s["tree"], s["bnd"], case["alpha2"], case["p"])
            s["prob"].matrix_free(True)
        elif kind == "targets":
            s["xy"] = _dev(_points(case, seed))
            s["out"] = torch.empty(case["targets"], dtype=torch.float64, device=DEV)
        if kind != "matrix_free":   # the operator is assembled by the first call that needs it
            mh.mh_double_layer_apply(ctx, s["bnd"], s["alpha"], s["x"], torch.empty_like(s["x"]), prec=s["prec"])
    return s


def _kept(s, *out):
    return [t.float() if s["prec"] else t for t in out]


def run(s):
    kind, ctx = s["kind"], s["ctx"]
    if kind == "operator":
        return _kept(s, mh.mh_double_layer_apply(ctx, s["bnd"], s["alpha"], s["x"], s["out"], prec=s["prec"]))
    if kind == "targets":
        return _kept(s, mh.mh_double_layer_apply(ctx, s["bnd"], s["alpha"], s["x"], s["out"], s["xy"], s["prec"]))
    if kind in ("gmres", "matrix_free"):
        s["out"].zero_()
        mh.mh_gmres_solve(ctx, s["bnd"], s["alpha"], s["x"], s["out"], 1e-10, 100, s["prec"])
        return [s["out"]]           # refined to a binary64 residual in either precision
    if kind == "volume":
        return _kept(s, mh.mh_volume_potential(ctx, s["tree"], s["alpha"], s["p"], s["b"], s["out"], s["prec"]))
    if kind == "step":
        k = s["i"] % CYCLE
        mh.heat_step(ctx, s["prob"], s["u"], s["F"][k], s["f"][k], s["un"], s["sigma"], s["b"][k], 1e-10, s["prec"])
        s["u"], s["un"], s["i"] = s["un"], s["u"], s["i"] + 1
        return _kept(s, s["u"], s["sigma"])
    if kind == "batch":
        k = s["i"] % CYCLE
        torch._foreach_copy_(s["F"] + s["f"], [t["F"][k] for t in s["parts"]] + [t["f"][k] for t in s["parts"]])
        s["batch"].step(s["u"], s["F"], s["f"], s["sigma"], 1e-10, s["prec"])
        s["i"] += 1
        return _kept(s, *s["u"], *s["sigma"])
    return [s["net"].loss_grad(s["X"], s["T"], s["grad"]), s["grad"]]


# ------------------------------------------------------------------ work

def work(case):
    kind, size = case["kind"], 4.0 if case.get("prec") else 8.0
    n = float(sum(c[5] for c in _curves(case))) if "domain" in case else 0.0
    if kind == "net":
        d, w = (case["holes"] + 1) * 2 * case["modes"], case["width"]
        par = 2 * d * w + 2 * w * w + 3 * w + d
        return {"bytes": 4.0 * (2 * par + 2 * d * case["samples"]), "flops": 6.0 * par * case["samples"]}
    if kind == "operator":
        return {"bytes": size * n * n + 16 * n, "flops": 2 * n * n}
    if kind == "gmres":
        return {"bytes": size * n * n + 16 * n, "flops": 20 * n * n}
    if kind == "targets":      # 68 operations for a kernel value of the pair sums
        return {"bytes": 24.0 * case["targets"] + 8 * n, "flops": 68.0 * case["targets"] * n}
    P, qq = 2 * case["p"] + 1, case["q"] ** 2
    if kind == "matrix_free":  # expansions of the boxes along the curves, neighbours, Alpert nodes; 10 products
        return {"bytes": 16 * n, "flops": 10 * n * (27 * 2 * P * P / 16 + 2 * 48 + 4 * P + 64)}
    if kind == "batch":
        every = [work(c) for c in _parts(case)]
        return {k: sum(w[k] for w in every) for k in ("bytes", "flops")}
    nodes = float(len(_mesh(_key(case))))
    leaves = nodes / qq
    flops = leaves * (9 * 2 * qq * qq + 4 * P * qq + 36 * 2 * P * P)
    if kind == "volume":
        return {"bytes": 16 * nodes, "flops": flops}
    flops += 20 * n * n + 68 * 16 * n * 9 * qq + leaves * (2 * P * qq)
    return {"bytes": 24 * nodes + size * n * n + 24 * n, "flops": flops}


# ------------------------------------------------------------------ 64-bit values

def _network(case, seed):
    rng = np.random.default_rng([seed, 3])
    d, w, n = (case["holes"] + 1) * 2 * case["modes"], case["width"], case["samples"]
    par = []
    for o, i in ((w, d), (w, w), (w, w), (d, w)):
        par += [(rng.standard_normal((o, i)) / math.sqrt(i)).astype(np.float32),
                (0.1 * rng.standard_normal(o)).astype(np.float32)]
    return par, rng.standard_normal((n, d)).astype(np.float32), rng.standard_normal((n, d)).astype(np.float32)


def _k1(z):
    return torch.special.modified_bessel_k1(z)


def _matrix(case, times, rows):
    """The continuous operator sigma + (1/pi) int K sigma ds on a times-fold grid, rows of every
    rows-th node: periodic trapezoid rule with Kress's logarithmic weights for the part
    I1(r/alpha) log(4 sin^2) of K1, windowed to a few alpha so that nothing cancels."""
    al, cs = math.sqrt(case["alpha2"]), _curves(case)
    ts = [TAU * np.arange(times * c[5]) / (times * c[5]) for c in cs]
    geo = [[torch.as_tensor(a) for a in _on_curve(c, t)] for c, t in zip(cs, ts)]
    out = []
    for j, (x, dx, ddx) in enumerate(geo):
        line = []
        for k, (y, dy, ddy) in enumerate(geo):
            N = len(y)
            h, sp = TAU / N, dy.norm(dim=1)
            nx, ny = dy[:, 1] / sp, -dy[:, 0] / sp
            ax, ay = y[None, :, 0] - x[::rows, None, 0], y[None, :, 1] - x[::rows, None, 1]
            r = torch.hypot(ax, ay)
            r = torch.where(r == 0, torch.ones_like(r), r)
            dn = (ax * nx + ay * ny) / r * (sp / al)
            K = _k1(r / al) * dn
            if j != k:
                line.append(K * (h / math.pi))
                continue
            at = torch.arange(0, N, rows)
            lag = (torch.arange(N)[None] - at[:, None]) % N
            near = r < 8 * al
            z = torch.where(near, r / al, torch.zeros_like(r))
            k1 = torch.where(near, 0.5 * torch.special.i1(z) * dn * torch.exp(-(z / 3.0) ** 8), torch.zeros_like(r))
            m = torch.arange(1, N // 2, dtype=torch.float64)
            i = torch.arange(N, dtype=torch.float64)
            R = torch.zeros(N, dtype=torch.complex128)
            R[1:N // 2] = 1.0 / m
            R = -(2 * TAU / N) * torch.fft.ifft(R).real * N - 2 * TAU / N ** 2 * torch.cos(math.pi * i)
            s2 = 4 * torch.sin(lag * (math.pi / N)) ** 2
            K2 = K - k1 * torch.log(torch.where(lag == 0, torch.ones_like(s2), s2))
            diag = -(ddy[:, 0] * nx + ddy[:, 1] * ny) / (2 * sp ** 2) * sp
            K2[torch.arange(len(at)), at] = diag[at]
            A = (K2 * h + k1 * R[lag]) / math.pi
            A[torch.arange(len(at)), at] += 1.0
            line.append(A)
        out.append(torch.cat(line, 1))
    return torch.cat(out)


def _layer(case, seed):
    """U^h at the target points from the density itself: trapezoid sums on grids fine enough for
    the distance (32-fold, 1024-fold for points within 0.4 node spacings of the curve)."""
    al, xy = math.sqrt(case["alpha2"]), _points(case, seed)
    rng, dens = np.random.default_rng([seed, 7]), []
    for c in _curves(case):
        a, f = rng.uniform(-1, 1, 9), rng.uniform(0, TAU, 9)
        dens.append((a, f))
    total = torch.zeros(len(xy), dtype=torch.float64, device=DEV)
    for c, (a, f) in zip(_curves(case), dens):
        close = _gap(c, xy) < 1.6 * 0.4 * TAU * c[2] * 1.6 / c[5]
        for which, times in ((~close, 32), (close, 1024)):
            at = np.nonzero(which)[0]
            if not len(at):
                continue
            t = TAU * np.arange(times * c[5]) / (times * c[5])
            y, d, _ = _on_curve(c, t)
            sig = sum(a[m] / (1 + m) * np.cos(m * t + f[m]) for m in range(9))
            g = torch.as_tensor(np.stack([y[:, 0], y[:, 1], d[:, 1] * sig, -d[:, 0] * sig]), device=DEV) # n |y'| sigma
            x = torch.as_tensor(xy[at], device=DEV)
            step = max(1, int(3e7) // g.shape[1])
            for i in range(0, len(at), step):
                ax, ay = g[0] - x[i:i + step, :1], g[1] - x[i:i + step, 1:]
                r = torch.hypot(ax, ay)
                v = (_k1(r / al) * (ax * g[2] + ay * g[3]) / r).sum(1) * (TAU / len(t)) / al
                total[torch.as_tensor(at[i:i + step], device=DEV)] += v
    return -total / (TAU * case["alpha2"])


def exact(case, seed):
    kind = case["kind"]
    if kind == "operator":
        times = 4 if case["npc"] * (case["holes"] + 1) <= 7000 else 2
        return [_matrix(case, times, times) @ torch.as_tensor(_modes(case, seed, times))]
    if kind == "targets":
        return [_layer(case, seed)]
    if kind in ("gmres", "matrix_free"):
        times = 2 if case["npc"] * (case["holes"] + 1) <= 6200 else 1
        A = _matrix(case, times, 1).to(DEV)
        return [torch.linalg.solve(A, torch.as_tensor(_modes(case, seed, times), device=DEV))[::times].contiguous()]
    if kind == "volume":
        field = _Field(case, seed)
        V, _, _ = field.basis(_mesh(_key(case)))
        return [field.coef(0)[:len(V)] @ V]
    if kind == "step" and case["ext"] == "const":
        return [_solution(case, seed), None]
    if kind == "batch":
        parts = _parts(case)
        return [_solution(c, seed + 1000 * j) for j, c in enumerate(parts)] + [None] * len(parts)
    if kind == "net":
        par, X, T = _network(case, seed)
        par = [torch.as_tensor(a, device=DEV).double().requires_grad_() for a in par]
        h = torch.as_tensor(X, device=DEV).double()
        for i in range(4):
            h = h @ par[2 * i].T + par[2 * i + 1]
            h = torch.tanh(h) if i < 3 else h
        loss = (h - torch.as_tensor(T, device=DEV).double()).square().mean() / 2
        loss.backward()
        return [float(loss), torch.cat([a.grad.reshape(-1) for a in par])]
    return None


def _solution(case, seed):
    nodes = _mesh(_key(case))
    inside, field = _inside(case, nodes), _Field(case, seed)
    V, _, W = field.basis(nodes, inside)
    c = field.coef(1)
    return (c[:len(V)] @ V + c[len(V):] @ W) * _dev(inside)
