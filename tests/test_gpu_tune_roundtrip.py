"""bie_tune's answer, installed in a table without it, brings the timed plan back."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import synth  # noqa: E402
from paper_1507_05925_gb300 import bie  # noqa: E402
from test_gpu_parity import to_dev  # noqa: E402

pytestmark = pytest.mark.gpu


# sizes at which the symmetric kernels are well ahead; the tiles that they may have (FP32
# Laplace: the rule's, of 128 nodes here, or the tuner's other candidate of 256)
@pytest.mark.parametrize("kind,prec,bodies,tiles", [
    (bie.LAPLACE, bie.FP64, 40, (32, 64, 128, 256)), (bie.STOKES, bie.FP64, 40, (32, 64, 128, 256)),
    (bie.LAPLACE, bie.MIXED, 64, (128, 256)), (bie.LAPLACE, bie.MIXED, 260, (256,)),
    (bie.STOKES, bie.MIXED, 100, (128,)), (bie.STOKES, bie.MIXED, 260, (192,)),
    (bie.LAPLACE, bie.MIXED_FF, 200, (256,))])
def test_installing_the_count_brings_the_plan_back(kind, prec, bodies, tiles):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_05925_gb300 import build
    build.build()
    side = 17
    g = to_dev(synth.assemble([synth.ellipse(3.2 * (i % side), 3.2 * (i // side), 1.0, 0.6, 0.3 * i, 127 + i % 3)
                               for i in range(bodies)]))
    M = g["x"].numel()
    v = torch.randn(M * (kind + 1), dtype=torch.float64, device="cuda")
    ctx = bie.Context(0)
    bie.tune_clear()

    def apply():
        out = torch.full_like(v, float("nan"))
        assert bie.apply_operator(ctx, g, kind, prec, v, out) == bie.OK
        torch.cuda.synchronize()
        return out.cpu().numpy()

    try:
        rc, S, ms = bie.tune(ctx, g, kind, prec)
        assert rc == bie.OK and ms > 0
        assert -S in [(M + t - 1) // t for t in tiles], S
        tuned = apply()
        bie.tune_clear()
        assert bie.tune(ctx, g, kind, prec, splits=7)[:2] == (bie.OK, 7)
        assert not np.array_equal(apply(), tuned)  # another order of the sums
        assert bie.tune(ctx, g, kind, prec, splits=S)[:2] == (bie.OK, S)
        assert np.array_equal(apply(), tuned)
        if prec == bie.FP64 or kind == bie.STOKES:
            for bad in (-1, S - 1, -(2 ** 31)):  # counts that no symmetric plan has
                assert bie.tune(ctx, g, kind, prec, splits=bad)[0] == bie.ERR_INVALID
            assert np.array_equal(apply(), tuned)  # a refused count changes nothing
    finally:
        bie.tune_clear()
        ctx.close()


def test_count_names_the_tiles():
    """FP32 Laplace sums of 8,128 nodes: 64 tiles are of 128 nodes (the rule's plan), 32 of
    256, which any other negative count also installs."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_05925_gb300 import build
    build.build()
    g = to_dev(synth.assemble([synth.ellipse(3.2 * (i % 8), 3.2 * (i // 8), 1.0, 0.6, 0.3 * i, 127) for i in range(64)]))
    v = torch.randn(8128, dtype=torch.float64, device="cuda")
    ctx = bie.Context(0)
    outs = {}
    try:
        for S in (None, -64, -32, -1):
            bie.tune_clear()
            if S is not None:
                assert bie.tune(ctx, g, bie.LAPLACE, bie.MIXED, splits=S)[:2] == (bie.OK, -64 if S == -64 else -32)
            out = torch.empty_like(v)
            assert bie.apply_operator(ctx, g, bie.LAPLACE, bie.MIXED, v, out) == bie.OK
            torch.cuda.synchronize()
            outs[S] = out.cpu().numpy()
    finally:
        bie.tune_clear()
        ctx.close()
    assert np.array_equal(outs[None], outs[-64]) and np.array_equal(outs[-32], outs[-1])
    assert not np.array_equal(outs[-64], outs[-32])
