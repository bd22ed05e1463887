"""FMM with few large bodies: trees that are mostly empty, whose blocks go over several
boxes, against the direct FP64 sums and, solved, against the direct solution."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import synth  # noqa: E402
from paper_1507_05925_gb300 import bie  # noqa: E402
from test_gpu_fmm import TOL_FMM  # noqa: E402
from test_gpu_parity import TOL_SOLVE, rel2, rel_max, to_dev  # noqa: E402

pytestmark = pytest.mark.gpu


# bodies, nodes a body, distance; the leaf level and its boxes a block: 6 and 1 (the line is a
# tree 1/32 full), 7 and 4, 8 and 10, 9 and 32
CASES = [(2, 3000, 3.0), (1, 20000, 3.0), (2, 12000, 3.0), (3, 1500, 40.0)]


@pytest.mark.parametrize("kind", [bie.LAPLACE, bie.STOKES])
@pytest.mark.parametrize("bodies,n,pitch", CASES)
def test_fmm_of_few_large_bodies(kind, bodies, n, pitch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_05925_gb300 import build
    build.build()
    ctx = bie.Context(0)
    g = synth.assemble([synth.ellipse(pitch * (i % 3), pitch * (i // 3), 1.0, 0.8, 0.5 * i, n) for i in range(bodies)])
    gd = to_dev(g)
    rng = np.random.default_rng(bodies)
    v = torch.from_numpy(rng.standard_normal(bodies * n * (kind + 1))).cuda()
    out = torch.empty_like(v)
    assert bie.apply_operator(ctx, gd, kind, bie.FP64, v, out) == bie.OK
    ref = out.cpu().numpy()
    for prec, order, tol in ((bie.FP64, 36, TOL_FMM[36]), (bie.MIXED_FF, 36, TOL_FMM[36]), (bie.MIXED, 18, 2e-5)):
        got = []
        for _ in range(2):
            out.fill_(float("nan"))
            assert bie.apply_operator_fmm_prec(ctx, gd, kind, order, prec, v, out) == bie.OK, ctx.last_error()
            got.append(out.cpu().numpy())
        print(f"kind={kind} {bodies} x {n} prec={prec}: {rel_max(got[0], ref):.2e}")
        assert rel_max(got[0], ref) <= tol
        assert np.array_equal(got[0], got[1])  # fixed order
    if bodies > 1:
        load = synth.charges(bodies, rng) if kind == bie.LAPLACE else synth.forces_torques(bodies, rng).reshape(-1)
        sol = {}
        fn = bie.elastance_solve if kind == bie.LAPLACE else bie.mobility_solve
        for order in (0, 36):
            sol[order] = np.empty(load.size)
            rc, info = fn(ctx, g, load, sol[order], opts=bie.make_opts(precision=bie.MIXED_FF, fmm_order=order))
            assert rc == bie.OK, (ctx.last_error(), info)
        assert rel2(sol[36], sol[0]) <= TOL_SOLVE
    ctx.close()
