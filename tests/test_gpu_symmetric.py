"""Symmetric pair sums (one CTA per unordered pair of tiles) at the edges of
their tiles, against the oracle and the directed kernels, and the smaller
workspace that a cap forces."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import synth  # noqa: E402
from oracle import geometry, laplace, stokes  # noqa: E402
from paper_1507_05925_gb300 import bie  # noqa: E402
from test_gpu_parity import TOL32, TOL64, TOL_SOLVE, rel2, rel_max, to_dev  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_05925_gb300 import build
    build.build()
    c = bie.Context(0)
    yield c
    bie.tune_clear()
    c.close()


def bodies_of(counts):
    """Ellipses and discs with the given node counts on a grid of pitch 3.2."""
    side = int(np.ceil(np.sqrt(len(counts))))
    curves = []
    for i, n in enumerate(counts):
        x, y = 3.2 * (i % side), 3.2 * (i // side)
        curves.append(synth.ellipse(x, y, 1.0, 0.4 + 0.05 * (i % 9), 0.3 * i, n) if i % 2 else synth.disc(x, y, 0.8, n))
    return synth.assemble(curves)


# one tile, exact and ragged tiles of 32, sizes at which the larger tiles are chosen
COUNTS = {"8": [8], "31": [13, 18], "32": [16, 16], "33": [8, 25], "1057": [151] * 7, "4097": [241] * 17,
          "12001": [267] * 43 + [520]}


@pytest.mark.parametrize("kind", [bie.LAPLACE, bie.STOKES])
@pytest.mark.parametrize("name", list(COUNTS))
def test_symmetric_fp64_operator(ctx, kind, name):
    g = bodies_of(COUNTS[name])
    geo = geometry.nodes(g)
    M = geo["M"]
    assert M == int(name)
    gd = to_dev(g)
    v = np.random.default_rng(M).standard_normal(M * (kind + 1))
    vin = torch.from_numpy(v).cuda()
    out = torch.empty_like(vin)
    bie.tune_clear()
    assert bie.apply_operator(ctx, gd, kind, bie.FP64, vin, out) == bie.OK
    sym = out.cpu().numpy()
    out.fill_(float("nan"))
    assert bie.apply_operator(ctx, gd, kind, bie.FP64, vin, out) == bie.OK
    assert np.array_equal(sym, out.cpu().numpy())  # fixed order
    # the directed kernel (a uniform plan, installed untimed)
    assert bie.tune(ctx, gd, kind, bie.FP64, splits=3)[0] == bie.OK
    assert bie.apply_operator(ctx, gd, kind, bie.FP64, vin, out) == bie.OK
    bie.tune_clear()
    directed = out.cpu().numpy()
    assert rel_max(sym, directed) <= 2 * TOL64
    if M <= 5000:
        ref = (laplace if kind == 0 else stokes).apply(geo, v)
        print(f"kind={kind} M={M}: symmetric {rel_max(sym, ref):.2e}, directed {rel_max(directed, ref):.2e}")
        assert rel_max(sym, ref) <= TOL64
        assert rel_max(directed, ref) <= TOL64


def test_workspace_cap_takes_the_smaller_plans(ctx):
    """A cap below the symmetric plans' workspace but above the directed ones'
    solves as before, through a context and through the server."""
    g = bodies_of([256] * 16)
    N, M = 16, 4096
    q = synth.charges(N, np.random.default_rng(3))
    ref = laplace.solve(g, q)["phi"]
    cap = int(0.85 * bie.workspace_bytes(bie.LAPLACE, N, M))
    small = bie.Context(0, workspace_cap_bytes=cap)
    phi = np.empty(N)
    rc, info = bie.elastance_solve(small, g, q, phi)
    assert rc == bie.OK, small.last_error()
    assert rel2(phi, ref) <= TOL_SOLVE
    small.close()
    srv = bie.Server(0, workers=1, hbm_cap_bytes=cap)
    phi[:] = np.nan
    t = srv.submit(bie.LAPLACE, g, q, phi)
    assert t > 0
    rc, info, _ = srv.wait(t)
    st = srv.stats()
    srv.close()
    assert rc == bie.OK and rel2(phi, ref) <= TOL_SOLVE
    assert st["peak_inflight_bytes"] <= cap


def ragged(total, seed):
    """Ragged bodies (8 to 300 nodes) in random order on a grid of pitch 2.6, some
    close to each other, `total` nodes in all."""
    rng = np.random.default_rng(seed)
    counts = []
    while sum(counts) < total - 400:
        counts.append(int(rng.choice([8, 31, 32, 33, 64, 97, 128, 200, 256, 300])))
    counts.append(total - sum(counts))
    side = int(np.ceil(np.sqrt(len(counts))))
    slots = rng.permutation(side * side)[:len(counts)]
    curves = []
    for n, s in zip(counts, slots):
        x, y = 2.6 * (s // side), 2.6 * (s % side)
        curves.append(synth.ellipse(x, y, 1.2, rng.uniform(0.4, 1.2), rng.uniform(0, 3), n))
    return synth.assemble(curves)


# tiles of 128 (the last with 1, 127 and 128 nodes), of 192 and 256
@pytest.mark.parametrize("kind", [bie.LAPLACE, bie.STOKES])
@pytest.mark.parametrize("M", [5505, 5631, 5632, 21505, 25857])
def test_symmetric_fp32_operator(ctx, kind, M):
    g = ragged(M, M)
    assert g["x"].size == M
    gd = to_dev(g)
    v = np.random.default_rng(M + 1).standard_normal(M * (kind + 1))
    vin = torch.from_numpy(v).cuda()
    out = torch.empty_like(vin)
    bie.tune_clear()
    assert bie.apply_operator(ctx, gd, kind, bie.FP64, vin, out) == bie.OK
    ref = out.cpu().numpy()
    res = []
    for _ in range(2):
        out.fill_(float("nan"))
        assert bie.apply_operator(ctx, gd, kind, bie.MIXED, vin, out) == bie.OK
        res.append(out.cpu().numpy())
    assert np.array_equal(res[0], res[1])  # fixed order
    assert bie.tune(ctx, gd, kind, bie.MIXED, splits=7)[0] == bie.OK  # the directed kernel
    assert bie.apply_operator(ctx, gd, kind, bie.MIXED, vin, out) == bie.OK
    bie.tune_clear()
    e_sym, e_dir = rel_max(res[0], ref), rel_max(out.cpu().numpy(), ref)
    print(f"kind={kind} M={M}: symmetric {e_sym:.2e}, directed {e_dir:.2e}")
    assert e_sym <= TOL32[kind]
    assert e_dir <= TOL32[kind]
