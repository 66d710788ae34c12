"""Performance cases of the library: what its users have it do, through the Python binding.

``listed()`` names the workloads, ``draw(rng)`` gives further sizes and options of the same
kinds, ``prepare`` makes a workload's inputs on the GPU together with the context that a
program keeps, ``run`` is one call (or one training step), ``work`` the bytes and operations
that the call cannot do without, and ``exact`` the result in 64 bits by direct sums.

Kinds:
  eval      one evaluation of v and s (a diagnostic, or one stage of a caller's own integrator)
  step      one RK4 step in place as a captured graph (a simulation's time loop)
  batch     one RK4 step of many independent systems at once (parameter studies)
  scalar    potential and gradient of monopoles (the scalar reference case)
  filament  velocity at the nodes of vortex filaments
  train     one training step of the selector network: loss, gradient and Adam
"""
import math

import torch

from paper_1201_5430_gb300 import LHV, _lib, api

# Gaussian core of the ring workloads (2 pi R / 1000) and of the cube and blob workloads.
RING_A = 2.0 * math.pi / 1000.0
CLOUD_A = 0.01
EPS = 1e-6
LEAF = 64


def listed():
    return [
        # The smallest configuration: 4096 elements of a cube, launches and host reads count.
        {"name": "eval_cube_4096", "kind": "eval", "dist": "cube", "n": 4096, "p": 8, "core": True,
         "precision": "fp32"},
        # An ordinary singular cloud of odd size in the default arithmetic.
        {"name": "eval_cube_100003", "kind": "eval", "dist": "cube", "n": 100003, "p": 12, "core": False,
         "precision": "fp32"},
        # The single vortex ring in the default arithmetic.
        {"name": "eval_ring_262144", "kind": "eval", "dist": "ring", "n": 262144, "p": 12, "core": True,
         "precision": "fp32"},
        # A short step of a simulation: a small ring, where latency and launches count.
        {"name": "step_ring_32768", "kind": "step", "dist": "ring", "n": 32768, "p": 12, "core": True,
         "precision": "tf32x3"},
        # The sphere surface of the timing tables: two-dimensional density, odd leaf counts.
        {"name": "eval_sphere_1048576", "kind": "eval", "dist": "sphere", "n": 1 << 20, "p": 12, "core": False,
         "precision": "tf32x3"},
        # Two offset rings of 2^20 elements: sparse tree, far field and near field alike.
        {"name": "eval_offset_2097152", "kind": "eval", "dist": "offset", "n": 1 << 21, "p": 16, "core": True,
         "precision": "tf32x3"},
        # The largest: one RK4 step of the leapfrogging pair of rings.
        {"name": "step_leapfrog_4194304", "kind": "step", "dist": "leapfrog", "n": 1 << 22, "p": 16, "core": True,
         "precision": "tf32x3"},
        # Independent blob clouds of uneven size, one RK4 step of all of them.
        {"name": "batch_blobs_16", "kind": "batch", "nsys": 16, "n_lo": 5000, "n_hi": 50000, "p": 12,
         "precision": "tf32x3"},
        # The scalar reference case of the timing tables.
        {"name": "scalar_cube_1048576", "kind": "scalar", "dist": "cube", "n": 1 << 20, "p": 12,
         "precision": "tf32x3"},
        # Double precision, as for reference solutions.
        {"name": "eval_ring_f64_32768", "kind": "eval", "dist": "ring", "n": 32768, "p": 12, "core": True,
         "precision": "fp64"},
        # A closed vortex filament ring.
        {"name": "filament_ring_262144", "kind": "filament", "nfil": 1, "n": 262144, "p": 16, "closed": True,
         "precision": "tf32x3"},
        # One training step of the selector network on its training set's size.
        {"name": "train_selector_800", "kind": "train", "rows": 800},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case.  Sizes are log-uniform; their upper ends keep every draw below the cost of
    the largest listed case."""
    kind = rng.choice(["eval", "eval", "eval", "step", "step", "batch", "scalar", "filament", "f64", "train"])
    if kind == "train":
        return {"kind": "train", "rows": _log_int(rng, 1, 4096)}
    precision = rng.choice(["fp32", "tf32x3"])
    p = rng.choice([8, 10, 12, 14, 16] if precision == "fp32" else [8, 12, 16])
    if kind == "f64":
        return {"kind": "eval", "dist": rng.choice(["ring", "cube"]), "n": _log_int(rng, 1000, 50000),
                "p": rng.choice([8, 12]), "core": True, "precision": "fp64"}
    if kind == "batch":
        lo = _log_int(rng, 500, 20000)
        return {"kind": "batch", "nsys": _log_int(rng, 2, 64), "n_lo": lo, "n_hi": int(lo * rng.uniform(1, 4)), "p": p,
                "precision": precision}
    if kind == "scalar":
        return {"kind": "scalar", "dist": rng.choice(["cube", "sphere"]), "n": _log_int(rng, 2000, 600000), "p": p,
                "precision": precision}
    if kind == "filament":
        return {"kind": "filament", "nfil": rng.choice([1, 2, 5]), "n": _log_int(rng, 5000, 400000), "p": p,
                "closed": rng.random() < 0.7, "precision": precision}
    if kind == "step":
        return {"kind": "step", "dist": rng.choice(["ring", "leapfrog", "offset"]), "n": _log_int(rng, 4000, 600000),
                "p": p, "core": True, "precision": precision}
    dist = rng.choice(["cube", "cube", "sphere", "ring", "leapfrog", "offset"])
    core = dist != "sphere" and (dist != "cube" or rng.random() < 0.5)
    return {"kind": "eval", "dist": dist, "n": _log_int(rng, 1500, 400000 if precision == "fp32" else 1200000), "p": p,
            "core": core, "precision": precision}


# ---- inputs --------------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _f4(a, dtype):
    """[n, 3] in 64 bits -> the binding's [n, 4] layout: rounded to FP32 once, fourth lane zero."""
    out = torch.zeros((a.shape[0], 4), dtype=dtype, device="cuda")
    out[:, :3] = a.float().to(dtype)
    return out


def _ring(n, g, gamma=1.0, centre=(0.0, 0.0, 0.0), tilt=0.0, sigma=0.03):
    f64 = dict(dtype=torch.float64, device="cuda")
    th = 2.0 * math.pi * torch.arange(n, **f64) / n
    j = sigma * torch.randn((2, n), generator=g, **f64)
    zero = torch.zeros_like(th)
    x = torch.stack([(1.0 + j[0]) * th.cos(), (1.0 + j[0]) * th.sin(), j[1]], 1)
    w = gamma * (2.0 * math.pi / n) / (4.0 * math.pi) * torch.stack([-th.sin(), th.cos(), zero], 1)
    c, s = math.cos(math.radians(tilt)), math.sin(math.radians(tilt))
    q = torch.tensor([[1.0, 0.0, 0.0], [0.0, c, -s], [0.0, s, c]], **f64)
    return x @ q.T + torch.tensor(centre, **f64), w @ q.T


def _elements(dist, n, seed):
    """Positions and strengths ([n, 3], 64 bits) of one system."""
    g = _gen(seed)
    f64 = dict(dtype=torch.float64, device="cuda")
    if dist == "cube":
        return torch.rand((n, 3), generator=g, **f64), torch.randn((n, 3), generator=g, **f64)
    if dist == "sphere":
        x = torch.randn((n, 3), generator=g, **f64)
        return x / x.norm(dim=1, keepdim=True), torch.randn((n, 3), generator=g, **f64)
    if dist == "ring":
        return _ring(n, g)
    xa, wa = _ring((n + 1) // 2, g)
    if dist == "leapfrog":
        xb, wb = _ring(n // 2, g, centre=(0.0, 0.0, 0.1))
    else:
        xb, wb = _ring(n // 2, g, gamma=-1.0, centre=(0.0, 0.0, 1.5), tilt=30.0)
    return torch.cat([xa, xb]), torch.cat([wa, wb])


def _blob_sizes(case):
    """Sizes of a batch's systems: spread evenly over the logarithm between n_lo and n_hi."""
    k = max(case["nsys"] - 1, 1)
    return [int(round(case["n_lo"] * (case["n_hi"] / case["n_lo"]) ** (((i * 7) % case["nsys"]) / k)))
            for i in range(case["nsys"])]


def _blobs(case, seed):
    """Gaussian blob clouds, eight blobs a system, strengths with quadrature weight 1/N_s."""
    g = _gen(seed)
    f64 = dict(dtype=torch.float64, device="cuda")
    xs, ws, off = [], [], [0]
    for n in _blob_sizes(case):
        centre = 0.2 + 0.6 * torch.rand((8, 3), generator=g, **f64)
        xs.append(centre[torch.arange(n, device="cuda") % 8] + 0.05 * torch.randn((n, 3), generator=g, **f64))
        ws.append(torch.randn((n, 3), generator=g, **f64) / (4.0 * math.pi * n))
        off.append(off[-1] + n)
    return off, torch.cat(xs), torch.cat(ws)


def _filaments(case, seed):
    """Coaxial rings (or arcs of 350 degrees), nodes jittered by a fifth of the segment length."""
    g = _gen(seed)
    f64 = dict(dtype=torch.float64, device="cuda")
    m = case["nfil"]
    off = [case["n"] * k // m for k in range(m + 1)]
    xs = []
    for k in range(m):
        n = off[k + 1] - off[k]
        turn = 2.0 * math.pi if case["closed"] else 2.0 * math.pi * 350.0 / 360.0
        th = turn * torch.arange(n, **f64) / n
        j = 0.2 * turn / n * torch.randn((2, n), generator=g, **f64)
        r = 1.0 - 0.1 * (k % 3) + j[0]
        xs.append(torch.stack([r * th.cos(), r * th.sin(), 0.25 * k + j[1]], 1))
    gamma = 0.5 + torch.rand((m,), generator=g, **f64)
    per_node = torch.cat([gamma[k].expand(off[k + 1] - off[k]) for k in range(m)])
    return off, [bool(case["closed"])] * m, torch.cat(xs), per_node.float()


def _network(rows, seed):
    """Feature rows in [-1, 1], labels (one leaf label in five rows), weights of a He-uniform
    start and the moments of a training run under way."""
    g = _gen(seed)
    f32 = dict(dtype=torch.float32, device="cuda")
    sizes = [(64, 12), (64, 64), (64, 64), (21, 64)]
    w = torch.cat([((2.0 * torch.rand((o * i,), generator=g, **f32) - 1.0) * math.sqrt(6.0 / i)) for o, i in sizes])
    st = {"X": 2.0 * torch.rand((rows, _lib.MLP_IN), generator=g, **f32) - 1.0,
          "yp": torch.randint(0, 17, (rows,), generator=g, device="cuda", dtype=torch.int32),
          "yl": torch.randint(0, 4, (rows,), generator=g, device="cuda", dtype=torch.int32),
          "W32": w, "W": w.bfloat16(), "b": 0.1 * torch.randn((_lib.MLP_NB,), generator=g, **f32)}
    st["yl"][torch.arange(rows, device="cuda") % 5 != 0] = -1
    for k, n in (("W", _lib.MLP_NW), ("b", _lib.MLP_NB)):
        st["m" + k] = 0.01 * torch.randn((n,), generator=g, **f32)
        st["v" + k] = 1e-4 * (0.5 + torch.rand((n,), generator=g, **f32))
    st["t"] = 50
    return st


# ---- a program's state, its call, and what the call needs -----------------------------------

def _core(case):
    if case["kind"] in ("scalar", "filament"):
        return 0.0
    if case["kind"] == "batch":
        return CLOUD_A
    return (CLOUD_A if case["dist"] == "cube" else RING_A) if case["core"] else 0.0


def prepare(case, seed):
    if case["kind"] == "train":
        return dict(_network(case["rows"], seed), kind="train")
    dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
    # a time loop runs on a stream of its own, which a captured step needs; other calls on the current one
    loop = case["kind"] in ("step", "batch")
    stream = torch.cuda.Stream() if loop else None
    ctx = LHV(p=case["p"], leaf_max=LEAF, core_a=_core(case), eps=EPS, precision=case["precision"], stream=stream)
    st = {"kind": case["kind"], "ctx": ctx, "dt": 5e-4}
    if case["kind"] == "batch":
        st["off"], x, w = _blobs(case, seed)
        st["x4"], st["w4"] = _f4(x, dtype), _f4(w, dtype)
    elif case["kind"] == "filament":
        st["off"], st["closed"], x, gamma = _filaments(case, seed)
        st["x4"], st["gamma"] = _f4(x, dtype), gamma.to(dtype)
    else:
        x, w = _elements(case["dist"], case["n"], seed)
        st["x4"] = _f4(x, dtype)
        if case["kind"] == "scalar":
            st["q"] = w[:, 0].float().to(dtype).contiguous()
        else:
            st["w4"] = _f4(w, dtype)
    if loop:
        st["x0"], st["w0"] = st["x4"].clone(), st["w4"].clone()
        stream.wait_stream(torch.cuda.current_stream())
        ctx.set_graph(True)
    return st


def run(st):
    kind = st["kind"]
    if kind == "eval":
        v4, s4 = st["ctx"].evaluate_velocity_stretching(st["x4"], st["w4"])
        return {"v": v4, "s": s4}
    if kind in ("step", "batch"):
        with torch.cuda.stream(st["ctx"].stream):  # the step's state comes in, and is advanced in place
            st["x4"].copy_(st["x0"])
            st["w4"].copy_(st["w0"])
        if kind == "step":
            st["ctx"].step(st["x4"], st["w4"], st["dt"])
        else:
            st["ctx"].step_batched(st["off"], st["x4"], st["w4"], st["dt"])
        return {"x": st["x4"], "w": st["w4"]}
    if kind == "scalar":
        return {"pg": st["ctx"].evaluate_potential_gradient(st["x4"], st["q"])}
    if kind == "filament":
        return {"v": st["ctx"].evaluate_filaments(st["off"], st["closed"], st["x4"], st["gamma"])}
    loss, gW, gb = api.mlp_loss_grad(st["X"], st["yp"], st["yl"], st["W"], st["b"])
    st["t"] += 1
    api.mlp_adam(st["W32"], st["W"], gW, st["mW"], st["vW"], st["b"], gb, st["mb"], st["vb"], st["t"], 1e-3)
    return {"loss": loss, "gW": gW, "gb": gb, "W32": st["W32"], "W": st["W"], "b": st["b"],
            "mW": st["mW"], "vW": st["vW"], "mb": st["mb"], "vb": st["vb"]}


def _neighbours(case, n):
    """About how many sources the near field of one element holds: the 27 boxes around it, with
    leaves of the core radius (5.95 a at eps = 1e-6) or of about half the leaf bound."""
    few = 27.0 * LEAF / 2
    if case["kind"] == "batch":
        return max(few, 0.12 * n)
    if case["kind"] == "filament":
        return 3.0 * LEAF
    if not _core(case):
        return min(n, few if case.get("dist") == "cube" else few / 2)
    box = 3.0 * 5.95 * _core(case)
    if case["dist"] == "cube":
        return min(n, max(few, n * box ** 3))
    return min(n, max(few / 4, 0.75 * n * box / (2.0 * math.pi) / (1 if case["dist"] in ("ring", "leapfrog") else 2)))


def work(case):
    """Elements read and results written once; the near-field pairs (46 operations for v and s,
    18 for a potential and its gradient, about 45 for a segment), and per element forming and
    evaluating an expansion of p^2 terms, with translations of the same order."""
    if case["kind"] == "train":
        nw = _lib.MLP_NW
        return {"bytes": case["rows"] * (_lib.MLP_IN + 2) * 4 + nw * 30, "flops": 6 * case["rows"] * nw}
    size = 8 if case["precision"] == "fp64" else 4
    sizes = _blob_sizes(case) if case["kind"] == "batch" else [case["n"]]
    evals = 4 if case["kind"] in ("step", "batch") else 1
    pair, term = {"scalar": (18, 10), "filament": (45, 25)}.get(case["kind"], (46, 60))
    n = sum(sizes)
    flops = sum(k * (pair * _neighbours(case, k) + term * case["p"] ** 2) for k in sizes)
    lanes = {"scalar": 4 + 1 + 4, "filament": 4 + 1 + 4}.get(case["kind"], 16)
    return {"bytes": n * lanes * size, "flops": evals * flops}


# ---- the same results in 64 bits -------------------------------------------------------------

def _direct(x, w, a):
    """v and s of every element by direct sums in 64 bits (x, w: [n, 3])."""
    n = x.shape[0]
    src = torch.cat([w, torch.linalg.cross(w, x)], 1)  # w_j x (x_i - x_j) = w_j x x_i - w_j x x_j
    v, s = torch.empty_like(x), torch.empty_like(x)
    rows = max(1, (1 << 25) // n)
    for b in range(0, n, rows):
        e = min(n, b + rows)
        xi, wi = x[b:e], w[b:e]
        r = torch.cdist(xi, x, compute_mode="donot_use_mm_for_euclid_dist")
        own = (torch.arange(e - b, device=x.device), torch.arange(b, e, device=x.device))
        r[own] = 1.0
        i2 = 1.0 / (r * r)
        f = i2 / r
        if a > 0.0:
            u = r / a
            d = math.sqrt(2.0 / math.pi) * torch.exp(-0.5 * u * u)
            f *= torch.erf(u / math.sqrt(2.0)) - u * d
            g = (d / a ** 3 - 3.0 * f) * i2
        else:
            g = -3.0 * f * i2
        f[own] = 0.0
        g[own] = 0.0
        g *= (wi * xi).sum(1, keepdim=True) - wi @ x.T
        F, G = f @ src, g @ src
        v[b:e] = torch.linalg.cross(F[:, :3], xi) - F[:, 3:]
        s[b:e] = torch.linalg.cross(F[:, :3], wi) + torch.linalg.cross(G[:, :3], xi) - G[:, 3:]
    return v, s


def _direct_scalar(x, q):
    n = x.shape[0]
    src = torch.cat([torch.ones((n, 1), dtype=x.dtype, device=x.device), x], 1) * q[:, None]
    out = torch.empty((n, 4), dtype=x.dtype, device=x.device)
    rows = max(1, (1 << 25) // n)
    for b in range(0, n, rows):
        e = min(n, b + rows)
        r = torch.cdist(x[b:e], x, compute_mode="donot_use_mm_for_euclid_dist")
        i1 = torch.where(r > 0.0, 1.0 / r, 0.0)
        F = i1 ** 3 @ src
        out[b:e, :3] = F[:, 1:] - F[:, :1] * x[b:e]
        out[b:e, 3] = i1 @ q
    return out


def _direct_filaments(off, closed, x, gamma):
    """Each segment's closed form at every node that it neither starts nor ends at."""
    n = x.shape[0]
    nxt = torch.arange(1, n + 1, device=x.device)
    live = torch.ones(n, dtype=torch.bool, device=x.device)
    for k in range(len(off) - 1):
        nxt[off[k + 1] - 1] = off[k]
        live[off[k + 1] - 1] = closed[k]
    y, gam = x[nxt], torch.where(live, gamma, 0.0) / (4.0 * math.pi)
    v = torch.empty_like(x)
    rows = max(1, (1 << 23) // n)
    for b in range(0, n, rows):
        e = min(n, b + rows)
        r1, r2 = x[b:e, None] - x[None], x[b:e, None] - y[None]
        c = torch.linalg.cross(r1, r2)
        l1, l2 = r1.norm(dim=2), r2.norm(dim=2)
        k = (1.0 / l1 + 1.0 / l2) / (l1 * l2 + (r1 * r2).sum(2)) * gam
        i = torch.arange(b, e, device=x.device)[:, None]
        k = torch.where((i == torch.arange(n, device=x.device)) | (i == nxt), 0.0, k)
        v[b:e] = (k[..., None] * c).sum(1)
    return v


def _rk4(x, w, a, dt):
    kx, kw = _direct(x, w, a)
    sx, sw = kx.clone(), kw.clone()
    for c, weight in ((0.5, 2.0), (0.5, 2.0), (1.0, 1.0)):
        kx, kw = _direct(x + c * dt * kx, w + c * dt * kw, a)
        sx += weight * kx
        sw += weight * kw
    return x + dt / 6.0 * sx, w + dt / 6.0 * sw


def _pad(a):
    return torch.cat([a, torch.zeros_like(a[:, :1])], 1)


def _train_exact(rows, seed):
    st = {k: v.double() if torch.is_tensor(v) and v.is_floating_point() else v for k, v in _network(rows, seed).items()}
    ws, bs, i, j = [], [], 0, 0
    for o, n in ((64, 12), (64, 64), (64, 64), (21, 64)):
        ws.append(st["W"][i:i + o * n].reshape(o, n).requires_grad_())
        bs.append(st["b"][j:j + o].clone().requires_grad_())
        i, j = i + o * n, j + o
    h = st["X"]
    for k in range(3):
        h = torch.relu(h @ ws[k].T + bs[k])
    z = h @ ws[3].T + bs[3]
    has = st["yl"] >= 0
    loss = torch.nn.functional.cross_entropy(z[:, :17], st["yp"].long())
    loss = loss + torch.nn.functional.cross_entropy(z[has, 17:], st["yl"][has].long())
    grads = torch.autograd.grad(loss, ws + bs)
    gW, gb = torch.cat([g.reshape(-1) for g in grads[:4]]), torch.cat(grads[4:])
    out, t = {"loss": loss.detach().reshape(1), "gW": gW, "gb": gb, "W": None}, st["t"] + 1
    for k, theta, g in (("W", "W32", gW), ("b", "b", gb)):
        m, v = 0.9 * st["m" + k] + 0.1 * g, 0.999 * st["v" + k] + 0.001 * g * g
        out["m" + k], out["v" + k] = m, v
        out[theta] = st[theta] - 1e-3 * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
    return out


def exact(case, seed):
    if case["kind"] == "train":
        return _train_exact(case["rows"], seed)
    if case["kind"] == "batch":
        if 4 * sum(n * n for n in _blob_sizes(case)) > 2.5e10:
            return None
        off, x, w = _blobs(case, seed)
        x, w = x.float().double(), w.float().double()
        parts = [_rk4(x[b:e], w[b:e], CLOUD_A, 5e-4) for b, e in zip(off, off[1:])]
        return {"x": _pad(torch.cat([q[0] for q in parts])), "w": _pad(torch.cat([q[1] for q in parts]))}
    if case["kind"] == "filament":
        if case["n"] ** 2 > 4e9:
            return None
        off, closed, x, gamma = _filaments(case, seed)
        return {"v": _pad(_direct_filaments(off, closed, x.float().double(), gamma.double()))}
    if case["n"] ** 2 * (4 if case["kind"] == "step" else 1) > 2.5e10:
        return None
    x, w = (t.float().double() for t in _elements(case["dist"], case["n"], seed))
    if case["kind"] == "scalar":
        return {"pg": _direct_scalar(x, w[:, 0])}
    if case["kind"] == "step":
        x, w = _rk4(x, w, _core(case), 5e-4)
        return {"x": _pad(x), "w": _pad(w)}
    v, s = _direct(x, w, _core(case))
    return {"v": _pad(v), "s": _pad(s)}
