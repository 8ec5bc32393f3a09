"""FP64 solves of the streaming tier with coefficients far from one: the refinement stops where it stops for a coefficient of
one, and the eigenvalue is exactly that multiple (squares of the solution beyond FP32's range included).

No tolerance: products with powers of two are exact."""
import numpy as np
import pytest

from synthetic_inputs import Level

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def B():
    from paper_2103_03407_gb300 import binding, build

    build.build()
    if not torch.cuda.is_available():
        pytest.fail("a GPU test ran without a CUDA device")
    return binding


@pytest.mark.parametrize("n,nc,tol", [(128, 32, 0.0), (128, 32, 1e-14), (256, 16, 1e-12), (32, 8, 1e-10)])
def test_any_scale(B, n, nc, tol):
    got = []
    for e in (0, -96, -64, 64, 96):
        with B.Context(0) as ctx:
            ctx.mq_set_coefficient(2.0 ** e, 8, 0, 2.0)
            ctx.mq_set_levels([Level(n, nc, 8, 3, 64, 2)])
            ctx.mq_set_precision(B.MQ_PREC_FP64, tol)
            ctx.mq_set_level_config(0, 1, 0, 0)
            lam = ctx.mq_eval_point(0, np.zeros(8))
            st = ctx.mq_get_stats()
        got.append([v * 2.0 ** -e for v in lam[:2]] + [st[k] for k in ("fine_iters_mean", "outer_iters_mean", "noconv")])
    assert all(g == got[0] for g in got) and got[0][-1] == 0
