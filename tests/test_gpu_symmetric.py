"""Symmetric pair sums (one CTA per unordered pair of tiles) at the edges of
their tiles, against the oracle and the directed kernels, and the smaller
workspace that a cap forces."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import synth  # noqa: E402
from oracle import geometry, laplace, stokes  # noqa: E402
from paper_1507_05925_gb300 import bie  # noqa: E402
from test_gpu_parity import TOL64, TOL_SOLVE, rel2, rel_max, to_dev  # noqa: E402

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
