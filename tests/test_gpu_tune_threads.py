"""Tuned plans that change while another thread solves: a call chooses its plans
once, so that it lays out the workspace it has sized.  Every solve, in a context
of its own whose workspace is exactly what it asked for, is right."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import synth  # noqa: E402
from oracle import laplace  # noqa: E402
from paper_1507_05925_gb300 import bie  # noqa: E402
from test_gpu_parity import TOL_SOLVE, rel2  # noqa: E402

pytestmark = pytest.mark.gpu


def test_plans_change_while_solving():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_05925_gb300 import build
    build.build()
    g = synth.assemble([synth.ellipse(3.0 * i, 0.2 * i, 1.0, 0.7, 0.4 * i, 128) for i in range(8)])
    q = synth.charges(8, np.random.default_rng(4))
    ref = laplace.solve(g, q)["phi"]
    stop = threading.Event()
    errors = []

    def retune():
        ctx = bie.Context(0)
        while not stop.is_set():
            for prec in (bie.FP64, bie.MIXED, bie.MIXED_FF):
                rc, _, _ = bie.tune(ctx, g, bie.LAPLACE, prec, splits=16)  # the most that the size allows
                if rc != bie.OK:
                    errors.append((rc, ctx.last_error()))
            bie.tune_clear()
        ctx.close()

    t = threading.Thread(target=retune)
    t.start()
    try:
        for k in range(60):
            ctx = bie.Context(0)
            phi = np.full(8, np.nan)
            rc, info = bie.elastance_solve(ctx, g, q, phi, opts=bie.make_opts(precision=k % 3))
            assert rc == bie.OK, (k, rc, ctx.last_error(), info)
            assert rel2(phi, ref) <= TOL_SOLVE
            ctx.close()
    finally:
        stop.set()
        t.join()
        bie.tune_clear()
    assert not errors
