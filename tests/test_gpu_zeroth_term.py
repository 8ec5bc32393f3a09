"""A zeroth term far below the terms: with all parameters zero the tensor-core coefficients are exactly that term, in the
resident, streamed and separable forms (no tolerance: nothing is rounded), and an eigenvalue is found for it."""
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


@pytest.mark.parametrize("n,s,family", [(8, 16, 1), (16, 64, 0), (16, 100, 0), (128, 65, 0)])
@pytest.mark.parametrize("a0", [1.0 / 3.0, 2.0 / 3.0 * 2.0 ** -8, 1e-5 / 3.0, 1e-20])
def test_zero_parameters_give_the_zeroth_term(B, n, s, family, a0):
    with B.Context(0) as ctx:
        ctx.mq_set_coefficient(a0, s, family, 2.0)
        ctx.mq_set_levels([Level(n, n, s, s, 8, 2)])
        ctx.mq_set_precision(B.MQ_PREC_MIXED)
        d = torch.empty((3, 2 * n * n), dtype=torch.float64, device="cuda")
        ctx.mq_coefficients_device(n, s, torch.zeros((3, s), dtype=torch.float64, device="cuda"), 3, s, d)
        assert bool((d == a0).all())
        lam = ctx.mq_eval_point(0, np.zeros(s))[0]
    h = 1.0 / n  # the first sine mode of a constant coefficient
    c = np.cos(np.pi * h)
    ref = a0 * (4.0 - 4.0 * c) / (h * h * (6.0 + 4.0 * c + 2.0 * c * c) / 12.0)
    assert abs(lam / ref - 1.0) < 0.05  # (the mass matrix couples the sine modes: the mode is not exactly the eigenvector)
