"""The FP32 Arnoldi step of the refinement's inner solves in its three forms: blocks
fetched into shared memory (fewer bodies than SMs), one body a CTA without the
fetch, and more bodies than CTAs (with the clusters of the block inversion for
few and for many bodies); block sizes that the fetch takes and leaves
(bytes no multiple of 16, above 313 rows, above the largest block), against the
oracle or, with hundreds of bodies, the FP64 solve."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import synth  # noqa: E402
from oracle import laplace, stokes  # noqa: E402
from paper_1507_05925_gb300 import bie  # noqa: E402
from test_gpu_parity import TOL_SOLVE, rel2, to_dev  # noqa: E402

pytestmark = pytest.mark.gpu


def run(kind, gd, load, size, precision, stream=None):
    ctx = bie.Context(0)
    out = torch.empty(size, dtype=torch.float64, device="cuda")
    fn = bie.elastance_solve if kind == 0 else bie.mobility_solve
    rc, info = fn(ctx, gd, torch.from_numpy(load).cuda(), out, opts=bie.make_opts(precision=precision), stream=stream)
    torch.cuda.synchronize()
    assert rc == bie.OK, (rc, ctx.last_error(), info)
    ctx.close()
    return out.cpu().numpy(), info


@pytest.mark.parametrize("kind,counts", [(0, (12, 33, 40, 313)), (0, (314, 320, 64)), (0, (640, 641, 48)), (0, (72,)),
                                         (1, (20, 33, 156)), (1, (157, 160)), (1, (321, 40))])
def test_blocks(kind, counts):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_05925_gb300 import build
    build.build()
    g = synth.assemble([synth.ellipse(3.0 * i, 0.4 * (i % 2), 1.0, 0.6 + 0.08 * i, 0.4 * i, n)
                        for i, n in enumerate(counts)])
    rng = np.random.default_rng(6)
    if kind == 0:
        load = synth.charges(len(counts), rng)
        ref = laplace.solve(g, load)["phi"]
    else:
        FT = synth.forces_torques(len(counts), rng)
        load, ref = FT.reshape(-1), stokes.solve(g, FT)["UW"].reshape(-1)
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    for st in (None, stream):  # kernel by kernel, and replayed from a graph
        got, info = run(kind, to_dev(g), load, ref.size, bie.MIXED, st)
        e = rel2(got, ref) if ref.any() else np.abs(got).max()  # one body: its potential is 0
        print(f"kind={kind} {counts}: {e:.2e} {info['iters']} iterations")
        assert e <= TOL_SOLVE


@pytest.mark.parametrize("kind,rows,cols,n", [(0, 10, 15, 32), (0, 8, 19, 32), (0, 20, 20, 32), (1, 25, 25, 16), (0, 4, 6, 160), (1, 4, 6, 130),
                                              (1, 10, 15, 40)])
def test_many_bodies(kind, rows, cols, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_05925_gb300 import build
    build.build()
    N = rows * cols
    g = synth.assemble([synth.ellipse(3.0 * (i % cols), 3.0 * (i // cols), 1.0, 0.6 + 0.3 * ((i * 7) % 10) / 10, 0.4 * i, n)
                        for i in range(N)])
    rng = np.random.default_rng(8)
    load = synth.charges(N, rng) if kind == 0 else synth.forces_torques(N, rng).reshape(-1)
    size = N if kind == 0 else 3 * N
    ref, _ = run(kind, to_dev(g), load, size, bie.FP64)
    got, info = run(kind, to_dev(g), load, size, bie.MIXED)
    e = rel2(got, ref)
    print(f"kind={kind} {N} bodies: {e:.2e} {info['iters']} iterations")
    assert e <= TOL_SOLVE
