"""Device memory that a solve reserves for its pair sums' partial slots."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import synth  # noqa: E402
from paper_1507_05925_gb300 import bie  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_05925_gb300 import build
    build.build()


def _reserved(kind, g, load, **opts):
    """Bytes that the server reserves for a request of these options, run alone."""
    srv = bie.Server(0, workers=1)
    out = np.empty(load.size)
    t = srv.submit(kind, g, load, out, opts=bie.make_opts(**opts))
    assert t > 0
    rc, info, _ = srv.wait(t)
    peak = srv.stats()["peak_inflight_bytes"]
    srv.close()
    assert rc == bie.OK, info
    return peak, out


@pytest.mark.parametrize("kind", [bie.LAPLACE, bie.STOKES])
def test_only_the_sums_of_the_call_reserve_slots(kind):
    """160 bodies of 128 nodes: at 20,480 nodes the FP32 sums keep 107 to 160 slots, the
    float-float and FP64 ones 5 to 160; FMM solves keep one."""
    N, n = 160, 128
    M = N * n
    side = 13
    g = synth.assemble([synth.ellipse(3.2 * (i % side), 3.2 * (i // side), 1.0, 0.7, 0.3 * i, n) for i in range(N)])
    rng = np.random.default_rng(8)
    load = synth.charges(N, rng) if kind == bie.LAPLACE else synth.forces_torques(N, rng).reshape(-1)
    slot = 8 * M * (kind + 1)
    direct, ref = _reserved(kind, g, load, precision=bie.MIXED_FF)
    half, out_half = _reserved(kind, g, load, precision=bie.MIXED_FF, fmm_order=-36)
    fmm, out = _reserved(kind, g, load, precision=bie.MIXED_FF, fmm_order=36)
    assert direct - fmm >= 100 * slot
    assert half <= direct and half - fmm >= 100 * slot  # FP32 direct sums inside
    fmm_paper, _ = _reserved(kind, g, load, precision=bie.MIXED_FF, fmm_order=36, formulation=1)
    assert fmm_paper > fmm  # the FP64 sum of its right-hand side
    for o in (out_half, out):
        assert np.linalg.norm(o - ref) <= 1e-9 * np.linalg.norm(ref)
    whole = bie.workspace_bytes(kind, N, M)  # of whichever options need most
    assert whole >= direct


def test_batches_of_changing_size_and_stream():
    """The copy tables that a context keeps between batches: larger and smaller batches, on
    two streams, from device and host arrays, each bitwise as in a context of its own."""
    from test_gpu_parity import to_dev
    ctx = bie.Context(0)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for k, P in enumerate((3, 200, 5, 700, 1, 40)):
        geoms = [synth.four_discs(seed=300 + 10 * k + p % 7, n=24 + 8 * (p % 3)) for p in range(P)]
        loads = [synth.charges(4, np.random.default_rng(p)) for p in range(P)]
        res = []
        for c, stream in ((ctx, streams[k % 2]), (bie.Context(0), None)):
            gs = [to_dev(g) if p % 3 else g for p, g in enumerate(geoms)]
            ls = [torch.from_numpy(q).cuda() if p % 2 else q for p, q in enumerate(loads)]
            outs = [torch.empty(4, dtype=torch.float64, device="cuda") if p % 2 else np.empty(4) for p in range(P)]
            torch.cuda.synchronize()
            rc, _, _ = bie.elastance_solve_batch(c, gs, ls, outs, opts=bie.make_opts(precision=bie.MIXED_FF), stream=stream)
            torch.cuda.synchronize()
            assert rc == bie.OK, c.last_error()
            res.append([o.cpu().numpy() if p % 2 else o for p, o in enumerate(outs)])
            if c is not ctx:
                c.close()
        assert all(np.array_equal(a, b) for a, b in zip(*res)), P
    ctx.close()


def test_full_device_takes_the_smaller_plans():
    """With little device memory left, a call whose symmetric plan's slots do not fit runs
    with the directed one's, as it does under a workspace cap."""
    from test_gpu_parity import TOL64, rel_max, to_dev
    N, n = 1000, 120
    M = N * n
    side = 32
    g = to_dev(synth.assemble([synth.ellipse(3.2 * (i % side), 3.2 * (i // side), 1.0, 0.7, 0.3 * i, n)
                               for i in range(N)]))
    v = torch.randn(M, dtype=torch.float64, device="cuda")
    out = torch.empty_like(v)
    ctx = bie.Context(0)
    assert bie.apply_operator(ctx, g, bie.LAPLACE, bie.FP64, v, out) == bie.OK
    torch.cuda.synchronize()
    ref = out.cpu().numpy()
    assert bie.tune(ctx, g, bie.LAPLACE, bie.FP64, splits=1)[0] == bie.OK  # the directed kernel, now loaded too
    assert bie.apply_operator(ctx, g, bie.LAPLACE, bie.FP64, v, out) == bie.OK
    torch.cuda.synchronize()
    ctx.close()
    bie.tune_clear()
    slots = 8 * M * 400  # the symmetric plan has more
    torch.cuda.empty_cache()
    try:
        held = torch.empty(torch.cuda.mem_get_info()[0] - (256 << 20), dtype=torch.uint8, device="cuda")
    except torch.OutOfMemoryError:
        pytest.skip("the device's free memory is not one piece")
    ctx = bie.Context(0)
    try:
        assert torch.cuda.mem_get_info()[0] < slots
        out.fill_(float("nan"))
        rc = bie.apply_operator(ctx, g, bie.LAPLACE, bie.FP64, v, out)
        torch.cuda.synchronize()
        err = ctx.last_error()
    finally:
        ctx.close()
        del held
        torch.cuda.empty_cache()
    assert rc == bie.OK, err
    assert rel_max(out.cpu().numpy(), ref) <= 2 * TOL64
