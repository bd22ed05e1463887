"""Several threads, each with its own context and stream, solving problems whose
kernels need different amounts of shared memory (block-Jacobi blocks of 16 to 600
unknowns, FMM of two orders) at the same time: every solve is as it is alone."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import synth  # noqa: E402
from paper_1507_05925_gb300 import bie  # noqa: E402
from test_gpu_parity import to_dev  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", [bie.LAPLACE, bie.STOKES])
def test_concurrent_solves(kind):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_05925_gb300 import build
    build.build()
    counts = [(16, 20), (70, 90), (130, 64), (230, 60), (300, 40), (65, 66, 67), (150, 290), (16, 16)]
    jobs = []
    for k, c in enumerate(counts):
        g = synth.assemble([synth.ellipse(3.0 * i, 0.3 * i, 1.0, 0.7, 0.4 * i, n) for i, n in enumerate(c)])
        rng = np.random.default_rng(k)
        load = synth.charges(len(c), rng) if kind == bie.LAPLACE else synth.forces_torques(len(c), rng).reshape(-1)
        jobs.append((to_dev(g), torch.from_numpy(np.ascontiguousarray(load)).cuda(), (0, 24, 36)[k % 3]))
    torch.cuda.synchronize()

    def run(job, repeats, results):
        geom, load, order = job
        ctx, stream = bie.Context(0), torch.cuda.Stream()
        fn = bie.elastance_solve if kind == bie.LAPLACE else bie.mobility_solve
        with torch.cuda.stream(stream):
            for _ in range(repeats):
                out = torch.empty_like(load)
                rc, _ = fn(ctx, geom, load, out, opts=bie.make_opts(precision=bie.MIXED_FF, fmm_order=order),
                           stream=stream)
                stream.synchronize()
                results.append((rc, out.cpu().numpy(), ctx.last_error()))
        ctx.close()

    alone = []
    for job in jobs:
        r = []
        run(job, 1, r)
        assert r[0][0] >= 0, r[0]
        alone.append(r[0][1])
    together = [[] for _ in jobs]
    threads = [threading.Thread(target=run, args=(job, 25, r)) for job, r in zip(jobs, together)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for k, results in enumerate(together):
        assert len(results) == 25
        for rc, out, err in results:
            assert rc >= 0, (k, rc, err)
            assert np.array_equal(out, alone[k])  # fixed order: bitwise
