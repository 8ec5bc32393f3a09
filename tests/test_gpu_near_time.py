"""Solves on the coarse mesh itself in calls of few samples, which wait for their slowest one: the mixed path agrees with the
FP64 path and is not slower than it, for inputs among which some shift nearly meets an eigenvalue.

Tolerance 1e-10 relative, that of every per-sample value.  Times: best of seven calls each; the mixed path takes 0.5 to
0.95 of the FP64 path's, and took 1.4 to 1.6 of it where one sample ran into a second solve in FP64."""
import time

import numpy as np
import pytest

from oracle import lattice
from synthetic_inputs import Level, shifts

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def B():
    from paper_2103_03407_gb300 import binding, build

    build.build()
    if not torch.cuda.is_available():
        pytest.fail("a GPU test ran without a CUDA device")
    return binding


@pytest.mark.parametrize("n,seed", [(8, 0), (16, 0), (16, 2), (32, 1), (64, 1), (128, 0), (128, 1)])
def test_few_samples(B, n, seed):
    lv = Level(n, n, 32, 6, 64, 8)
    z, delta, got, ms = lattice.cbc(lv.N, lv.s), shifts(seed, [lv])[0], [], []
    for prec in (B.MQ_PREC_MIXED, B.MQ_PREC_FP64):
        with B.Context(0) as ctx:
            ctx.mq_set_coefficient(1.0, lv.s, 0, 2.0)
            ctx.mq_set_levels([lv])
            ctx.mq_set_lattice(0, z)
            ctx.mq_set_shifts(0, delta)
            ctx.mq_set_precision(prec)
            out = torch.empty((lv.R, 16, 4), dtype=torch.float64, device="cuda")
            best = 1e9
            for _ in range(7):
                torch.cuda.synchronize()
                t = time.perf_counter()
                ctx.mq_eval_level_device(0, 0, 16, out)
                torch.cuda.synchronize()
                best = min(best, time.perf_counter() - t)
            ms.append(best)
            got.append(out.cpu().numpy()[..., 1])
    assert np.abs(got[0] - got[1]).max() <= 1e-10 * got[1].max()
    assert ms[0] <= ms[1], ms
