"""The work that users of this library have it do, as cases that can be timed.

A case is one call of a public entry point of paper_1507_05925_gb300.bie on one
geometry (or one batch of geometries): elastance and mobility solves in every
precision, with direct and with FMM pair sums, batches of small problems, and
single operator applications.  Sizes are those of this repository's benchmark
and tests (four discs, 100 stars, 400 and 10,000 ellipses, ragged bodies,
batches of requests); draw() gives more of the same ranges.

Geometries are bodies on a lattice, jittered as far as a gap of five node
spacings between neighbours allows (the resolution the trapezoidal rule needs),
with shapes and loads from the seed; node counts a body belong to the case, so
that two seeds are the same discretisation of two arrangements of bodies.  A
program keeps one context and one CUDA stream of its own for all its calls, as
bench.py does; "host" cases pass numpy arrays on the default stream.

The FP32 operator (precision "mixed" of apply_operator) is the operator of the
mixed solves' inner iterations and is measured there.
"""
import math
import zlib

import numpy as np
import torch

from paper_1507_05925_gb300 import bie

_PREC = {"fp64": bie.FP64, "mixed": bie.MIXED, "mixed_ff": bie.MIXED_FF}
_DEV = "cuda"
_kept = {}


def _context():
    """The program's library context."""
    if "ctx" not in _kept:
        _kept["ctx"] = bie.Context(torch.cuda.current_device())
    return _kept["ctx"]


def _stream():
    """The program's own stream (its iterations can be replayed as CUDA graphs there)."""
    if "stream" not in _kept:
        _kept["stream"] = torch.cuda.Stream()
    return _kept["stream"]


def listed():
    return [
        # the smallest call: four conductors of 128 nodes, the latency of a whole solve
        _case("elastance_4_discs", "elastance", 4, "discs", 128, 128, "mixed_ff"),
        # a first program: four ragged bodies, host arrays, the options' defaults (FP64 GMRES)
        _case("mobility_4_ragged_default", "mobility", 4, "mixed", 91, 300, "fp64", host=True),
        # a medium elastance problem at the default precision
        _case("elastance_36_stars_fp64", "elastance", 36, "stars", 128, 301, "fp64"),
        # the benchmark's headline: 100 stars of 256 nodes, direct sums, float-float refinement
        _case("elastance_100_stars", "elastance", 100, "stars", 256, 256, "mixed_ff"),
        # the same with FMM pair sums, the order the benchmark takes
        _case("elastance_100_stars_fmm", "elastance", 100, "stars", 256, 256, "mixed_ff", fmm=30),
        # a suspension with FP64 residuals
        _case("mobility_64_ellipses_mixed", "mobility", 64, "ellipses", 128, 128, "mixed"),
        # the benchmark's suspension of 400 ellipses with direct sums
        _case("mobility_400_ellipses", "mobility", 400, "ellipses", 128, 128, "mixed_ff"),
        # the largest: 10,000 ellipses (640,000 nodes) with FMM pair sums
        _case("mobility_10000_ellipses_fmm", "mobility", 10000, "ellipses", 64, 64, "mixed_ff", fmm=36),
        # throughput: a batch of 128 four-disc problems
        _case("elastance_batch_128", "elastance_batch", 4, "discs", 128, 128, "mixed_ff", problems=128),
        # served requests of up to 64 bodies, solved together
        _case("mobility_batch_8_requests", "mobility_batch", 64, "mixed", 64, 256, "mixed_ff", problems=8),
        # one matvec for a caller's own Krylov method, FP64, a ragged suspension
        _case("operator_stokes_fp64", "operator", 101, "ellipses", 90, 165, "fp64", kind=1),
        # the same for a large conductor problem, through the FMM
        _case("operator_fmm_laplace_fp64", "operator_fmm", 2500, "ellipses", 64, 64, "fp64", fmm=36, kind=0),
    ]


def _case(name, call, bodies, shape, lo, hi, precision, fmm=0, host=False, problems=1, kind=-1, formulation=0,
          precond=0):
    if kind < 0:
        kind = 0 if call.startswith("elastance") else 1
    c = dict(call=call, kind=kind, bodies=bodies, shape=shape, nodes_lo=lo, nodes_hi=hi, precision=precision, fmm=fmm,
             host=host, problems=problems, formulation=formulation, precond=precond)
    return dict(c, name=name) if name else c


def draw(rng):
    """One more case: a family by how it is used, its node count over the logarithm of its range."""
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def shape_and_nodes(stars=True):
        shape = rng.choice(["discs", "ellipses", "mixed", "stars"] if stars else ["ellipses", "mixed"])
        n = log_int(*{"discs": (32, 200), "ellipses": (48, 256), "mixed": (96, 256), "stars": (128, 320)}[shape])
        if rng.random() < 0.5:
            return shape, n, n
        return shape, max(24, int(0.7 * n)), int(1.3 * n)

    u = rng.random()
    kind = rng.randrange(2)
    if u < 0.5:  # a solve with direct sums
        prec = rng.choice(["fp64", "mixed", "mixed_ff", "mixed_ff"])
        cap = {"fp64": (9000, 4500), "mixed": (25600, 12800), "mixed_ff": (51200, 40000)}[prec][kind]
        shape, lo, hi = shape_and_nodes()
        M = log_int(256, cap)
        return _case("", "mobility" if kind else "elastance", max(2, 2 * M // (lo + hi)), shape, lo, hi, prec,
                     host=rng.random() < 0.25, formulation=int(rng.random() < 0.15), precond=int(rng.random() < 0.1))
    if u < 0.7:  # a solve with FMM sums
        n = rng.choice([64, 96, 128])
        M = log_int(12000, 400000)
        return _case("", "mobility" if kind else "elastance", M // n, "ellipses", n if rng.random() < 0.5 else n - 13, n,
                     "mixed_ff", fmm=rng.randrange(30, 39))
    if u < 0.8:  # a batch of small problems
        return _case("", "mobility_batch" if kind else "elastance_batch", rng.randrange(2, 7), "discs", 48, log_int(64, 144),
                     "mixed_ff", problems=log_int(4, 200))
    if u < 0.87:  # a batch of requests
        return _case("", "mobility_batch" if kind else "elastance_batch", rng.randrange(8, 49), "mixed", 64, 256,
                     "mixed_ff", problems=rng.randrange(2, 9))
    shape, lo, hi = shape_and_nodes(stars=False)
    if u < 0.95:  # one direct operator application
        prec = rng.choice(["fp64", "mixed_ff"])
        M = log_int(512, {"fp64": 30000, "mixed_ff": 51200}[prec])
        return _case("", "operator", max(2, 2 * M // (lo + hi)), shape, lo, hi, prec, kind=kind)
    M = log_int(20000, 300000)
    return _case("", "operator_fmm", 2 * M // (lo + hi), shape, lo, hi, rng.choice(["fp64", "mixed_ff"]),
                 fmm=rng.randrange(30, 39), kind=kind)


# ------------------------------------------------------------------ inputs ----
def _node_counts(case, problem):
    """Nodes of each body: the case's own (the discretisation does not depend on the seed)."""
    key = "{bodies} {shape} {nodes_lo} {nodes_hi} {kind}".format(**case) + " %d" % problem
    r = np.random.default_rng(zlib.crc32(key.encode()))
    nb = case["bodies"]
    if case["call"].endswith("_batch") and nb > 6:  # requests differ in their number of bodies
        nb = int(r.integers(1, nb + 1))
    return r.integers(case["nodes_lo"], case["nodes_hi"] + 1, nb)


def _geometry(case, counts, rng):
    """Bodies on a lattice, evaluated on the GPU: dict of the arrays of bie_geometry (device tensors)."""
    nb = counts.size
    stars = {"stars": np.ones(nb, bool), "mixed": rng.random(nb) < 0.5}.get(case["shape"], np.zeros(nb, bool))
    a = np.where(stars, rng.uniform(0.5, 1.0, nb), 1.0)  # a star's mean radius; a disc's radius; a major semi-axis
    if case["shape"] == "discs":
        a = rng.uniform(0.5, 1.0, nb)
    b = a.copy() if case["shape"] == "discs" else rng.uniform(0.34, 1.0, nb)
    eps = rng.uniform(0.0, 0.3, nb)
    arms = rng.integers(3, 7, nb)
    phi = rng.uniform(0.0, 2.0 * math.pi, nb)
    # lattice: room for the largest body and five of the coarsest node spacings
    big, speed = {"discs": (1.0, 1.0), "ellipses": (1.0, 1.0)}.get(case["shape"], (1.3, 2.23))
    need = 2.0 * big + 5.0 * speed * 2.0 * math.pi / counts.min()
    pitch = max(3.2 if case["bodies"] <= 1000 else 0.0, need)
    side = int(math.ceil(math.sqrt(nb)))
    slot = rng.permutation(side * side)[:nb]
    jit = 0.5 * (pitch - need)
    cx = (slot // side) * pitch + rng.uniform(-jit, jit, nb)
    cy = (slot % side) * pitch + rng.uniform(-jit, jit, nb)
    start = np.zeros(nb + 1, np.int32)
    start[1:] = np.cumsum(counts)
    cnt = torch.from_numpy(counts.astype(np.int64)).to(_DEV)
    par = torch.from_numpy(np.stack([cx, cy, a, b, eps, arms.astype(np.float64), phi, stars.astype(np.float64),
                                     start[:-1].astype(np.float64), counts.astype(np.float64)])).to(_DEV)
    q = torch.repeat_interleave(par, cnt, dim=1)
    cx, cy, a, b, eps, arms, phi, star, first, n = q
    t = 2.0 * math.pi * (torch.arange(q.shape[1], device=_DEV, dtype=torch.float64) - first) / n
    c, s = torch.cos(t), torch.sin(t)
    # ellipse: (a cos t, b sin t) turned by phi
    cp, sp = torch.cos(phi), torch.sin(phi)
    e = [(cp * u - sp * v, sp * u + cp * v) for u, v in ((a * c, b * s), (-a * s, b * c), (-a * c, -b * s))]
    # star: r = a (1 + eps cos(arms (t - phi)))
    ph = arms * (t - phi)
    r, r1, r2 = a * (1 + eps * torch.cos(ph)), -a * eps * arms * torch.sin(ph), -a * eps * arms * arms * torch.cos(ph)
    p = [(r * c, r * s), (r1 * c - r * s, r1 * s + r * c), (r2 * c - 2 * r1 * s - r * c, r2 * s + 2 * r1 * c - r * s)]
    is_star = star > 0.5
    x, y, dx, dy, ddx, ddy = (torch.where(is_star, v, u).contiguous() for m in range(3) for u, v in zip(e[m], p[m]))
    return dict(x=x + cx, y=y + cy, dx=dx, dy=dy, ddx=ddx, ddy=ddy, body_start=torch.from_numpy(start).to(_DEV))


def _load(case, nb, rng):
    """Charges, or (Fx, Fy, T) a body: N(0, 1), the net charge or force removed."""
    if case["kind"] == 0:
        q = rng.standard_normal(nb)
        return q - q.mean()
    ft = rng.standard_normal((nb, 3))
    ft[:, :2] -= ft[:, :2].mean(axis=0, keepdims=True)
    return ft.reshape(-1)


def _inputs(case, seed):
    """One (geometry, load) a problem, on the GPU."""
    out = []
    for p in range(case["problems"]):
        rng = np.random.default_rng([seed, p])
        g = _geometry(case, _node_counts(case, p), rng)
        nb = g["body_start"].numel() - 1
        out.append((g, torch.from_numpy(_load(case, nb, rng)).to(_DEV)))
    return out


def _density(case, n, seed):
    gen = torch.Generator(device=_DEV)
    gen.manual_seed(seed)
    return torch.randn(n, dtype=torch.float64, device=_DEV, generator=gen)


def prepare(case, seed):
    ins = _inputs(case, seed)
    st = dict(case=case, ctx=_context(), stream=None if case["host"] else _stream())
    if case["call"].startswith("operator"):
        g = ins[0][0]
        v = _density(case, g["x"].numel() * (case["kind"] + 1), seed)
        return dict(st, geom=g, inp=v, out=torch.empty_like(v))
    st["opts"] = bie.make_opts(precision=_PREC[case["precision"]], fmm_order=case["fmm"],
                               formulation=case["formulation"], precond=case["precond"])
    if case["call"].endswith("_batch"):
        sizes = [ld.numel() for _, ld in ins]
        out = torch.empty(sum(sizes), dtype=torch.float64, device=_DEV)
        return dict(st, geoms=[g for g, _ in ins], loads=[ld for _, ld in ins], out=out, outs=list(out.split(sizes)))
    g, ld = ins[0]
    out = torch.empty_like(ld)
    dens = torch.empty(g["x"].numel() * (case["kind"] + 1), dtype=torch.float64, device=_DEV)
    if case["host"]:
        g = {k: v.cpu().numpy() for k, v in g.items()}
        ld, out, dens = ld.cpu().numpy(), out.cpu().numpy(), dens.cpu().numpy()
    return dict(st, geom=g, load=ld, out=out, density=dens)


def run(state):
    case, ctx, stream = state["case"], state["ctx"], state["stream"]
    call, kind = case["call"], case["kind"]
    if call == "operator":
        rc = bie.apply_operator(ctx, state["geom"], kind, _PREC[case["precision"]], state["inp"], state["out"],
                                stream=stream)
        res = state["out"]
    elif call == "operator_fmm":
        rc = bie.apply_operator_fmm_prec(ctx, state["geom"], kind, case["fmm"], _PREC[case["precision"]], state["inp"],
                                         state["out"], stream=stream)
        res = state["out"]
    elif call.endswith("_batch"):
        solve = bie.mobility_solve_batch if kind else bie.elastance_solve_batch
        rc, _, _ = solve(ctx, state["geoms"], state["loads"], state["outs"], opts=state["opts"], stream=stream)
        res = state["out"]
    else:
        solve = bie.mobility_solve if kind else bie.elastance_solve
        rc, _ = solve(ctx, state["geom"], state["load"], state["out"], state["density"], opts=state["opts"],
                      stream=stream)
        res = {"out": state["out"], "density": state["density"]}
    if rc < 0:
        raise RuntimeError("%s: status %d: %s" % (call, rc, ctx.last_error()))
    return res


# -------------------------------------------------------------------- work ----
# Floating-point operations of one ordered pair of nodes (Laplace: r, |r|^2,
# q/|r|^2 and its sum; Stokes: two dot products and a product more), and the
# operator applications a solve to 1e-12 takes on such bodies (block-Jacobi
# preconditioned GMRES: measured 12 to 16 and 30 to 40).
_PAIR, _APPLY = (10.0, 18.0), (16.0, 35.0)


def work(case):
    M = [int(_node_counts(case, p).sum()) for p in range(case["problems"])]
    nb = [_node_counts(case, p).size for p in range(case["problems"])]
    c = case["kind"] + 1
    op = case["call"].startswith("operator")
    nbytes = 48.0 * sum(M) + 4.0 * sum(nb) + (16.0 * c * sum(M) if op else 16.0 * sum(nb) * (1 if c == 1 else 3))
    if not op and not case["call"].endswith("_batch"):
        nbytes += 8.0 * c * sum(M)  # the density
    if case["fmm"]:  # near field: 3 x 3 leaves of about 30 nodes; translations: 27 boxes a leaf, c^2 sums of order p
        one = sum(M) * (270.0 * _PAIR[case["kind"]] + 2.0 * 27.0 / 30.0 * case["fmm"] ** 2 * (1, 3)[case["kind"]])
    else:
        one = sum(float(m) * (m - 1) for m in M) * _PAIR[case["kind"]]
    return {"bytes": nbytes, "flops": one * (1.0 if op else _APPLY[case["kind"]])}


# ------------------------------------------------- the same in 64-bit torch ----
def _nodes(g):
    """Quadrature data of the trapezoidal rule."""
    start = g["body_start"].long()
    cnt = start[1:] - start[:-1]
    N = cnt.numel()
    body = torch.repeat_interleave(torch.arange(N, device=_DEV), cnt)
    speed = torch.hypot(g["dx"], g["dy"])
    w = speed * 2.0 * math.pi / cnt[body]

    def per_body(v):
        return torch.zeros(N, dtype=torch.float64, device=_DEV).index_add_(0, body, v)

    length = per_body(w)
    xc, yc = per_body(w * g["x"]) / length, per_body(w * g["y"]) / length
    kappa = (g["dx"] * g["ddy"] - g["dy"] * g["ddx"]) / speed ** 3
    return dict(x=g["x"], y=g["y"], w=w, nx=g["dy"] / speed, ny=-g["dx"] / speed, kappa=kappa, body=body, N=N,
                xc=xc, yc=yc, px=-(g["y"] - yc[body]), py=g["x"] - xc[body])


def _rows(d, kind, lo, hi):
    """Rows lo..hi (nodes) of 1/2 I + K + L."""
    r = slice(lo, hi)
    rx, ry = d["x"][r, None] - d["x"][None], d["y"][r, None] - d["y"][None]
    i = torch.arange(hi - lo, device=_DEV)
    r2 = rx * rx + ry * ry
    r2[i, lo + i] = 1.0
    k = (rx * d["nx"][r, None] + ry * d["ny"][r, None]) / r2
    w = d["w"][None]
    same = (d["body"][r, None] == d["body"][None]).double()
    if kind == 0:
        k = -k / (2.0 * math.pi)
        k[i, lo + i] = -d["kappa"][r] / (4.0 * math.pi)
        A = (k + same) * w
        A[i, lo + i] += 0.5
        return A
    k = -k / r2 / math.pi
    tx, ty, kap = -d["ny"][r], d["nx"][r], -d["kappa"][r] / (2.0 * math.pi)
    A = torch.empty((hi - lo, 2, d["x"].numel(), 2), dtype=torch.float64, device=_DEV)
    for a, (ra, ta, pa) in enumerate(((rx, tx, d["px"]), (ry, ty, d["py"]))):
        for b, (rb, tb, pb) in enumerate(((rx, tx, d["px"]), (ry, ty, d["py"]))):
            e = k * ra * rb
            e[i, lo + i] = kap * ta * tb
            A[:, a, :, b] = (e + same * ((1.0 if a == b else 0.0) + pa[r, None] * pb[None])) * w
    i2 = torch.arange(2 * (hi - lo), device=_DEV)
    A = A.view(2 * (hi - lo), -1)
    A[i2, 2 * lo + i2] += 0.5
    return A


def _apply_rows(d, kind, v):
    M = d["x"].numel()
    step = max(1, min(M, (1 << 26) // M))
    return torch.cat([_rows(d, kind, s, min(M, s + step)) @ v for s in range(0, M, step)])


def _solve(d, kind, f):
    """A nu = f: dense, Krylov (Arnoldi, twice orthogonalised), corrected until the residual is rounding."""
    M = d["x"].numel()
    n = f.numel()
    A = torch.empty((n, n), dtype=torch.float64, device=_DEV)
    step = max(1, min(M, (1 << 25) // M))
    for s in range(0, M, step):
        e = min(M, s + step)
        A[s * (kind + 1):e * (kind + 1)] = _rows(d, kind, s, e)
    if n <= 4096:
        x = torch.linalg.solve(A, f)
        return x + torch.linalg.solve(A, f - A @ x)
    x, fn = torch.zeros_like(f), float(f.norm())
    for _ in range(4):
        r = f - A @ x
        beta = float(r.norm())
        if not beta > 2e-16 * fn:
            break
        m = 160
        V = torch.zeros((m + 1, n), dtype=torch.float64, device=_DEV)
        H = torch.zeros((m + 1, m), dtype=torch.float64, device=_DEV)
        V[0] = r / beta
        used = m
        for j in range(m):
            q = A @ V[j]
            for _twice in range(2):
                h = V[:j + 1] @ q
                q = q - h @ V[:j + 1]
                H[:j + 1, j] += h
            H[j + 1, j] = q.norm()
            V[j + 1] = q / H[j + 1, j]
            if j % 8 == 7:
                e1 = torch.zeros(j + 2, 1, dtype=torch.float64)
                e1[0] = beta
                Hh = H[:j + 2, :j + 1].cpu()
                y = torch.linalg.lstsq(Hh, e1).solution
                if float((Hh @ y - e1).norm()) < 1e-15 * fn:
                    used = j + 1
                    break
        e1 = torch.zeros(used + 1, 1, dtype=torch.float64)
        e1[0] = beta
        y = torch.linalg.lstsq(H[:used + 1, :used].cpu(), e1).solution[:, 0].to(_DEV)
        x = x + y @ V[:used]
        del V
    return x


def _at(d, kind, nu, px, py):
    """The single layer of nu at points inside the bodies."""
    rx, ry = px[:, None] - d["x"][None], py[:, None] - d["y"][None]
    r2 = rx * rx + ry * ry
    lg = -0.5 * torch.log(r2)
    if kind == 0:
        return (lg @ (d["w"] * nu)) / (2.0 * math.pi)
    f1, f2 = d["w"] * nu[0::2], d["w"] * nu[1::2]
    xy = rx * ry / r2
    return torch.stack([(lg + rx * rx / r2) @ f1 + xy @ f2, xy @ f1 + (lg + ry * ry / r2) @ f2], 1) / (4.0 * math.pi)


def _solution(g, kind, load):
    d = _nodes(g)
    b = d["body"]
    if kind == 0:
        nu = _solve(d, 0, load[b])
        return _at(d, 0, nu, d["xc"], d["yc"]), nu
    ft = load.view(-1, 3)
    f = torch.stack([ft[b, 0] + ft[b, 2] * d["px"], ft[b, 1] + ft[b, 2] * d["py"]], 1).reshape(-1)
    nu = _solve(d, 1, f)
    dist = torch.hypot(d["px"], d["py"])
    near = torch.full((d["N"],), math.inf, dtype=torch.float64, device=_DEV).scatter_reduce_(0, b, dist, "amin")
    h = 0.25 * near
    u0, u1, u2 = (_at(d, 1, nu, d["xc"] + ex * h, d["yc"] + ey * h) for ex, ey in ((0, 0), (1, 0), (0, 1)))
    om = ((u1[:, 1] - u0[:, 1]) - (u2[:, 0] - u0[:, 0])) / (2.0 * h)
    return torch.stack([u0[:, 0], u0[:, 1], om], 1).reshape(-1), nu


def exact(case, seed):
    M = max(int(_node_counts(case, p).sum()) for p in range(case["problems"]))
    kind = case["kind"]
    if case["call"].startswith("operator"):
        if float(M) * M * (1 + 3 * kind) > 4e10:
            return None
        g = _inputs(case, seed)[0][0]
        return _apply_rows(_nodes(g), kind, _density(case, M * (kind + 1), seed))
    if M * (kind + 1) > 26000:
        return None
    res = [_solution(g, kind, ld) for g, ld in _inputs(case, seed)]
    if case["call"].endswith("_batch"):
        return torch.cat([r[0] for r in res])
    return {"out": res[0][0], "density": res[0][1]}
