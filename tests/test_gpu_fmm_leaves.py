"""FMM operator with leaves of very different populations (empty ones, a few
nodes, more nodes than an evaluation block holds targets and stages sources),
in every precision, against the direct FP64 sums."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import synth  # noqa: E402
from paper_1507_05925_gb300 import bie  # noqa: E402
from test_gpu_fmm import TOL_FMM  # noqa: E402
from test_gpu_parity import rel_max, to_dev  # noqa: E402

pytestmark = pytest.mark.gpu


def uneven(n_dense):
    rng = np.random.default_rng(n_dense)
    curves = [synth.disc(0.1, 0.2, 0.05, n_dense)]
    for k in range(10):
        curves.append(synth.ellipse(3.0 + 3.0 * (k % 4), 3.0 * (k // 4), 1.0, rng.uniform(0.4, 1.0),
                                    rng.uniform(0, 3), int(rng.integers(8, 90))))
    return synth.assemble(curves)


@pytest.mark.parametrize("kind", [bie.LAPLACE, bie.STOKES])
@pytest.mark.parametrize("n_dense", [40, 127, 300, 1500])
def test_fmm_operator_uneven_leaves(kind, n_dense):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_05925_gb300 import build
    build.build()
    ctx = bie.Context(0)
    g = to_dev(uneven(n_dense))
    M = g["x"].numel()
    v = torch.from_numpy(np.random.default_rng(7).standard_normal(M * (kind + 1))).cuda()
    out = torch.empty_like(v)
    assert bie.apply_operator(ctx, g, kind, bie.FP64, v, out) == bie.OK
    ref = out.cpu().numpy()
    for prec, order, tol in ((bie.FP64, 36, TOL_FMM[36]), (bie.MIXED_FF, 36, TOL_FMM[36]), (bie.MIXED, 18, 2e-5)):
        out.fill_(float("nan"))
        assert bie.apply_operator_fmm_prec(ctx, g, kind, order, prec, v, out) == bie.OK, ctx.last_error()
        got = out.cpu().numpy()
        err = rel_max(got, ref)
        print(f"kind={kind} dense={n_dense} prec={prec}: {err:.2e}")
        assert err <= tol
        assert bie.apply_operator_fmm_prec(ctx, g, kind, order, prec, v, out) == bie.OK
        assert np.array_equal(got, out.cpu().numpy())  # fixed order
    ctx.close()


# Orders on both sides of the FP32 translation kernel's instances (12, 16, 20, 24,
# 32, 48, 64) and of the numbers of splits.  The same expansions in FP64 are the
# reference, so that only rounding differs: FP32 sums as above 2e-5; float-float
# products (2^-46) summed in FP64, with the expansions' own FP64 rounding, 1e-11.
@pytest.mark.parametrize("kind", [bie.LAPLACE, bie.STOKES])
@pytest.mark.parametrize("order", [2, 7, 12, 13, 16, 17, 20, 21, 24, 25, 32, 33, 48, 49, 64])
def test_fmm_operator_orders(kind, order):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_05925_gb300 import build
    build.build()
    ctx = bie.Context(0)
    g = to_dev(uneven(300))
    v = torch.from_numpy(np.random.default_rng(8).standard_normal(g["x"].numel() * (kind + 1))).cuda()
    out = torch.empty_like(v)
    got = {}
    for prec in (bie.FP64, bie.MIXED_FF, bie.MIXED):
        out.fill_(float("nan"))
        assert bie.apply_operator_fmm_prec(ctx, g, kind, order, prec, v, out) == bie.OK, ctx.last_error()
        got[prec] = out.cpu().numpy()
    for prec, tol in ((bie.MIXED_FF, 1e-11), (bie.MIXED, 2e-5)):
        err = rel_max(got[prec], got[bie.FP64])
        print(f"kind={kind} order={order} prec={prec}: {err:.2e}")
        assert err <= tol
    ctx.close()
