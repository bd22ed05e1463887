"""Batches whose problems are large enough for the symmetric FP32 pair sums (tiles
of each problem by itself): problems of very different sizes, none a multiple of
the tile, against their solo solves."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import synth  # noqa: E402
from paper_1507_05925_gb300 import bie  # noqa: E402
from test_gpu_parity import TOL_SOLVE, rel2, to_dev  # noqa: E402

pytestmark = pytest.mark.gpu


def grid(count, n, seed):
    rng = np.random.default_rng(seed)
    return synth.assemble([synth.ellipse(3.0 * (i % 7), 3.0 * (i // 7), 1.0, rng.uniform(0.5, 1.0), rng.uniform(0, 3),
                                         n + int(rng.integers(0, 9))) for i in range(count)])


# sizes in nodes: about 1,000 (8 tiles of 128) to 5,000, and one of 80
@pytest.mark.parametrize("kind,sizes", [(0, [(30, 70)] * 7 + [(2, 40), (15, 67), (31, 129)]),
                                        (1, [(24, 66)] * 6 + [(2, 40), (15, 69), (30, 101)]),
                                        (1, [(36, 131)] * 8 + [(20, 150)]), (0, [(40, 160)] * 14)])
def test_batch_against_solo(kind, sizes):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_05925_gb300 import build
    build.build()
    rng = np.random.default_rng(3)
    geoms = [grid(count, n, k) for k, (count, n) in enumerate(sizes)]
    loads = []
    for count, _ in sizes:
        loads.append(synth.charges(count, rng) if kind == 0 else synth.forces_torques(count, rng).reshape(-1))
    dev = [to_dev(g) for g in geoms]
    ql = [torch.from_numpy(np.ascontiguousarray(q)).cuda() for q in loads]
    outs = [torch.full((q.numel(),), float("nan"), dtype=torch.float64, device="cuda") for q in ql]
    solo = bie.elastance_solve if kind == 0 else bie.mobility_solve
    batch = bie.elastance_solve_batch if kind == 0 else bie.mobility_solve_batch
    opts = bie.make_opts(precision=bie.MIXED)
    ctx = bie.Context(0)
    for _ in range(2):
        rc, infos, status = batch(ctx, dev, ql, outs, opts=opts)
        torch.cuda.synchronize()
        assert rc == bie.OK and not any(status), (rc, status, ctx.last_error())
    got = [o.cpu().numpy() for o in outs]
    for k in range(0, len(sizes), 3):
        ref = torch.empty_like(outs[k])
        rc, _ = solo(ctx, dev[k], ql[k], ref, opts=opts)
        torch.cuda.synchronize()
        assert rc == bie.OK
        e = rel2(got[k], ref.cpu().numpy())
        print(f"kind={kind} problem {k} {sizes[k]}: {e:.2e} {infos[k]['iters']} iterations")
        assert e <= TOL_SOLVE
    ctx.close()
