"""Streamed solves under a caller's cap on the refinement steps: three steps suffice on every mesh (two up to 1/512) at the
default target, with the values of an uncapped call.

Tolerance 1e-10 relative, that of every per-sample value."""
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


@pytest.mark.parametrize("n,cap,tol", [(64, 2, 0.0), (512, 2, 0.0), (512, 3, 1e-8), (1024, 3, 0.0), (1024, 3, 1e-8)])
def test_capped_refinement_converges(B, n, cap, tol):
    lv = Level(n, 32, 64, 8, 64, 4)
    z, delta, got = lattice.cbc(lv.N, lv.s), shifts(1, [lv])[0], []
    for steps in (0, cap):
        with B.Context(0) as ctx:
            ctx.mq_set_coefficient(1.0, lv.s, 0, 2.0)
            ctx.mq_set_levels([lv])
            ctx.mq_set_lattice(0, z)
            ctx.mq_set_shifts(0, delta)
            ctx.mq_set_precision(B.MQ_PREC_MIXED, tol)
            ctx.mq_set_solver_options(0.0, 0, steps)
            got.append(ctx.mq_eval_level(0, 3, 11)[0][..., 1])
            assert ctx.mq_get_stats()["noconv"] == 0
    assert np.abs(got[0] - got[1]).max() <= 1e-10 * got[0].max()
