"""The FP64 FMM operator against the direct FP64 sums at orders on both sides of the
instances of the translation kernels (16, 20, 36 and 64), on a tree of three levels of
shifts: an absolute check of their coefficients, which the sweep of precisions against
the FP64 expansions does not give."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import synth  # noqa: E402
from paper_1507_05925_gb300 import bie  # noqa: E402
from test_gpu_fmm import TOL_FMM  # noqa: E402
from test_gpu_parity import rel_max, to_dev  # noqa: E402

pytestmark = pytest.mark.gpu

# A source lies within sqrt(1/2) box sides of its box's centre and a target's box centre two
# sides off at least: the terms decay like RHO^p.  50 stands for 1/(1 - RHO) = 2.2 and the
# ratio of the far sum of |q|/r to the sums themselves; Stokes takes the expansions' derivative
# (p).  Below that, the rounding that TOL_FMM has at order 36.
RHO = 0.5 ** 0.5 / (2.0 - 0.5 ** 0.5)


@pytest.mark.parametrize("kind", [bie.LAPLACE, bie.STOKES])
def test_fmm_operator_orders_against_direct_sums(kind):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_05925_gb300 import build
    build.build()
    ctx = bie.Context(0)
    g = to_dev(synth.assemble([synth.ellipse(3.2 * (i % 12), 3.2 * (i // 12), 1.0, 0.5 + 0.003 * i, 0.3 * i, 64)
                               for i in range(144)]))
    v = torch.from_numpy(np.random.default_rng(6).standard_normal(g["x"].numel() * (kind + 1))).cuda()
    out = torch.empty_like(v)
    assert bie.apply_operator(ctx, g, kind, bie.FP64, v, out) == bie.OK
    ref = out.cpu().numpy()
    for p in (12, 16, 17, 20, 21, 36, 37, 38, 48, 63, 64):
        out.fill_(float("nan"))
        assert bie.apply_operator_fmm(ctx, g, kind, p, v, out) == bie.OK, ctx.last_error()
        err = rel_max(out.cpu().numpy(), ref)
        tol = 50.0 * (p if kind == bie.STOKES else 1) * RHO ** p + TOL_FMM[36]
        print(f"kind={kind} order={p}: {err:.2e} (bound {tol:.2e})")
        assert err <= tol
    ctx.close()
