"""The kernels' reciprocals (csrc/pair_math.cuh) against 1/x in extended precision, over
mantissas and exponents, and at the ends of the range."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import synth  # noqa: E402
from paper_1507_05925_gb300 import bie  # noqa: E402
from test_gpu_parity import to_dev  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_05925_gb300 import build
    build.build()


def reciprocal(x):
    xd = torch.from_numpy(np.ascontiguousarray(x)).cuda()
    out = torch.full((2 * x.size,), float("nan"), dtype=torch.float64, device="cuda")
    assert bie.test_rcp(xd, out) == bie.OK
    torch.cuda.synchronize()
    out = out.cpu().numpy()
    return out[:x.size], out[x.size:]


def test_reciprocal_over_mantissas_and_exponents():
    rng = np.random.default_rng(2)
    n = 1 << 20
    m = np.concatenate([1.0 + np.arange(4096) / 4096.0, np.nextafter(1.0 + np.arange(1, 4097) / 4096.0, 0.0),
                        rng.uniform(1.0, 2.0, n)])
    x = np.ldexp(m, rng.integers(-1021, 1021, m.size)) * rng.choice([-1.0, 1.0], m.size)
    exact = np.longdouble(1.0) / x.astype(np.longdouble)
    err = np.abs(reciprocal(x)[0].astype(np.longdouble) - exact) / np.spacing(np.abs(exact).astype(np.float64))
    print(f"largest error {float(err.max()):.4f} ulp")
    # the last rounding, |e|^3 < 2^-57 (1/16 ulp at most), and the roundings of e, e + e^2
    assert float(err.max()) <= 0.5 + 2.0 ** -4 + 2.0 ** -15


def test_reciprocal_at_the_ends():
    x = np.array([np.inf, -np.inf, np.finfo(np.float64).max, 2.0 ** 1023, 0.0, -0.0, 2.0 ** -1074, np.nan])
    r, _ = reciprocal(x)
    assert np.array_equal(r[:4], [0.0, -0.0, 0.0, 0.0])  # (1/x of the middle two is below 2^-1022)
    assert r[4] == np.inf and r[5] == -np.inf and r[6] == np.inf and np.isnan(r[7])


def test_fp32_reciprocal():
    rng = np.random.default_rng(3)
    n = 1 << 20
    x = np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(-125, 125, n)).astype(np.float32)
    _, r = reciprocal(x.astype(np.float64))
    exact = 1.0 / x.astype(np.float64)
    err = np.abs(r - exact) / np.spacing(exact.astype(np.float32))
    print(f"largest error {err.max():.6f} ulp")
    assert err.max() <= 0.5 + 2.0 ** -20  # the last rounding and e^2 <= 2^-44
    _, r = reciprocal(np.array([np.inf, -np.inf, 2.0 ** -140, 0.0, np.nan]))
    assert r[0] == 0.0 and r[1] == 0.0 and r[2] == np.inf and r[3] == np.inf and np.isnan(r[4])


@pytest.mark.parametrize("n", [40, 300])
def test_bodies_whose_squared_distance_overflows(n):
    """Bodies of radius 1e150 at a distance of 1e157: their |r|^2 is infinite and the pair
    adds nothing; the operator acts body by body.  (Laplace: the torques of Stokes bodies
    of this size overflow.)"""
    ctx = bie.Context(0)
    bodies = [synth.disc(0.0, 0.0, 1e150, n), synth.ellipse(1e157, 0.0, 1e150, 0.6e150, 0.0, n)]
    v = np.random.default_rng(n).standard_normal(2 * n)

    def apply(curves, density):
        out = torch.empty(density.size, dtype=torch.float64, device="cuda")
        assert bie.apply_operator(ctx, to_dev(synth.assemble(curves)), bie.LAPLACE, bie.FP64,
                                  torch.from_numpy(density).cuda(), out) == bie.OK
        torch.cuda.synchronize()
        return out.cpu().numpy()

    both = apply(bodies, v)
    half = v.size // 2
    alone = np.concatenate([apply(bodies[:1], v[:half].copy()), apply(bodies[1:], v[half:].copy())])
    ctx.close()
    assert np.all(np.isfinite(alone))
    assert np.max(np.abs(both - alone)) <= 1e-13 * np.max(np.abs(alone))
