"""FP64 GMRES with the block-Jacobi preconditioner in FP64 arithmetic: bodies at
the edges of the row tiles (32 rows a CTA) and of the largest block (640
unknowns; larger bodies keep the identity), against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import synth  # noqa: E402
from oracle import laplace, stokes  # noqa: E402
from paper_1507_05925_gb300 import bie  # noqa: E402
from test_gpu_parity import TOL_SOLVE, rel2, to_dev  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,counts", [(0, (8, 31, 32, 33, 65)), (0, (639, 40)), (0, (640, 641, 64)),
                                         (1, (8, 15, 16, 17, 33)), (1, (319, 320)), (1, (321, 48))])
def test_fp64_gmres_block_jacobi(kind, counts):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_05925_gb300 import build
    build.build()
    ctx = bie.Context(0)
    g = synth.assemble([synth.ellipse(3.0 * i, 0.4 * (i % 2), 1.0, 0.5 + 0.08 * i, 0.4 * i, n)
                        for i, n in enumerate(counts)])
    N = len(counts)
    rng = np.random.default_rng(5)
    if kind == 0:
        load = synth.charges(N, rng)
        ref, fn = laplace.solve(g, load)["phi"], bie.elastance_solve
    else:
        FT = synth.forces_torques(N, rng)
        load = FT.reshape(-1)
        ref, fn = stokes.solve(g, FT)["UW"].reshape(-1), bie.mobility_solve
    gd, ld = to_dev(g), torch.from_numpy(load).cuda()
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    for st in (None, stream):  # kernel by kernel, and replayed from a graph
        out = torch.empty(ref.size, dtype=torch.float64, device="cuda")
        rc, info = fn(ctx, gd, ld, out, opts=bie.make_opts(precision=bie.FP64, restart=6), stream=st)
        torch.cuda.synchronize()
        assert rc == bie.OK, (rc, ctx.last_error(), info)
        assert info["rel_residual"] <= 1e-12
        e = rel2(out.cpu().numpy(), ref)
        print(f"kind={kind} {counts}: {e:.2e} {info['iters']} iterations")
        assert e <= TOL_SOLVE
    ctx.close()
