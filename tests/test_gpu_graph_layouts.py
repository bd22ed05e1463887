"""Captured GMRES iterations of one context and stream while the bodies change:
geometries of equal numbers of bodies and nodes whose bodies' sizes, interior
points or FMM orders differ lay the workspace out differently and launch other
grids, and a graph captured for one must not serve another.  Every solve is
bitwise the one of the same context on the default stream, which captures
nothing."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import synth  # noqa: E402
from oracle import laplace, stokes  # noqa: E402
from paper_1507_05925_gb300 import bie  # noqa: E402
from test_gpu_parity import TOL_SOLVE, rel2, to_dev  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_05925_gb300 import build
    build.build()
    c = bie.Context(0)
    yield c
    c.close()


def bodies_of(counts, interior=False):
    g = synth.assemble([synth.ellipse(3.0 * i, 0.3 * (i % 2), 1.0, 0.7, 0.4 * i, n) for i, n in enumerate(counts)])
    if interior:
        g["interior_pt"] = np.array([[3.0 * i + 0.05, 0.3 * (i % 2)] for i in range(len(counts))]).reshape(-1)
    return g


def solve(ctx, g, kind, stream, **opts):
    N = g["body_start"].size - 1
    rng = np.random.default_rng(N)
    load = synth.charges(N, rng) if kind == bie.LAPLACE else synth.forces_torques(N, rng).reshape(-1)
    gd = to_dev(g)
    if "interior_pt" in g:
        gd["interior_pt"] = torch.from_numpy(g["interior_pt"]).cuda()
    ld = torch.from_numpy(load).cuda()
    out = torch.full((load.size,), float("nan"), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    fn = bie.elastance_solve if kind == bie.LAPLACE else bie.mobility_solve
    rc, info = fn(ctx, gd, ld, out, opts=bie.make_opts(**opts), stream=stream)
    torch.cuda.synchronize()
    assert rc == bie.OK, (rc, ctx.last_error(), info)
    assert info["graph_replay"] == (0 if stream is None else 1)
    return out.cpu().numpy()


# the largest body (its rows of the FP64 preconditioner's grid), the sum of the blocks
# (96^2 + 96^2 and 95^2 + 97^2 round to one slot), the order of the bodies
LAYOUTS = {"largest body": [(96, 96, 40), (95, 97, 40)], "sum of blocks": [(150, 150), (100, 200), (60, 240)],
           "order": [(60, 90, 150), (150, 60, 90)], "first without blocks": [(344, 344), (8, 680)]}


@pytest.mark.parametrize("prec", [bie.FP64, bie.MIXED, bie.MIXED_FF])
@pytest.mark.parametrize("kind", [bie.LAPLACE, bie.STOKES])
@pytest.mark.parametrize("name", list(LAYOUTS))
def test_graphs_follow_the_bodies(ctx, name, kind, prec):
    stream = torch.cuda.Stream()
    solve(ctx, bodies_of((400, 400, 400)), kind, None, precision=prec)  # a workspace that fits all the others
    for counts in LAYOUTS[name] + LAYOUTS[name][:1]:
        for interior in (False, True):
            g = bodies_of(counts, interior)
            out = solve(ctx, g, kind, stream, precision=prec)
            assert np.array_equal(out, solve(ctx, g, kind, None, precision=prec)), (counts, interior)
            if not interior:
                N = len(counts)
                rng = np.random.default_rng(N)
                ref = (laplace.solve(g, synth.charges(N, rng))["phi"] if kind == bie.LAPLACE else
                       stokes.solve(g, synth.forces_torques(N, rng))["UW"].reshape(-1))
                assert rel2(out, ref) <= TOL_SOLVE


@pytest.mark.parametrize("kind", [bie.LAPLACE, bie.STOKES])
def test_graphs_follow_the_fmm_order(ctx, kind):
    """Outer orders 35 and 36 have one inner order, 18, but lay the tree's arrays out
    differently in a buffer that order 38 made: the iteration captured at 35 must not be
    replayed at 36."""
    g = synth.assemble([synth.ellipse(3.2 * (i % 12), 3.2 * (i // 12), 1.0, 0.6, 0.3 * i, 64) for i in range(144)])
    stream = torch.cuda.Stream()
    opts = dict(precision=bie.MIXED_FF)
    outs = [solve(ctx, g, kind, stream, fmm_order=p, **opts) for p in (38, 35, 36, 36)]
    for p, out in zip((38, 35, 36, 36), outs):
        assert np.array_equal(out, solve(ctx, g, kind, None, fmm_order=p, **opts)), p
