"""FP64 GMRES where one body is far larger than the preconditioner's blocks: its rows keep
the identity and are copied by as many CTAs as the grid has for a body, in strides."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import synth  # noqa: E402
from oracle import laplace, stokes  # noqa: E402
from paper_1507_05925_gb300 import bie  # noqa: E402
from test_gpu_parity import TOL_SOLVE, rel2, to_dev  # noqa: E402

pytestmark = pytest.mark.gpu


# with 61 bodies a body has 20 CTAs, which copy 5,120 rows a stride; with two, one for every
# 256 rows of the large one
@pytest.mark.parametrize("kind,large,small,count", [(0, 5121, 8, 60), (0, 6000, 16, 60), (0, 4000, 64, 1),
                                                    (1, 2561, 8, 60), (1, 321, 16, 20)])
def test_fp64_gmres_with_one_large_body(kind, large, small, count):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_05925_gb300 import build
    build.build()
    ctx = bie.Context(0)
    curves = [synth.disc(0.0, 0.0, 2.0, large)]
    curves += [synth.ellipse(5.0 + 3.0 * (i % 8), 3.0 * (i // 8), 1.0, 0.8, 0.4 * i, small) for i in range(count)]
    g = synth.assemble(curves)
    rng = np.random.default_rng(5)
    if kind == 0:
        load = synth.charges(count + 1, rng)
        ref, fn = laplace.solve(g, load)["phi"], bie.elastance_solve
    else:
        FT = synth.forces_torques(count + 1, rng)
        load = FT.reshape(-1)
        ref, fn = stokes.solve(g, FT)["UW"].reshape(-1), bie.mobility_solve
    gd, ld = to_dev(g), torch.from_numpy(load).cuda()
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    out = torch.empty(ref.size, dtype=torch.float64, device="cuda")
    rc, info = fn(ctx, gd, ld, out, opts=bie.make_opts(precision=bie.FP64, restart=6), stream=stream)
    torch.cuda.synchronize()
    assert rc == bie.OK, (rc, ctx.last_error(), info)
    assert rel2(out.cpu().numpy(), ref) <= TOL_SOLVE
    ctx.close()
