"""Tensor-core coefficients at the ends of their domain |y| <= 1, in the resident, streamed and separable forms, against the
long-double reference; one row with the signs of the terms at a centroid, where it makes the sums largest.

Tolerance: four units of FP64 rounding of the largest |a|, as inside the parameters' own range."""
import numpy as np
import pytest

from synthetic_inputs import Level, random_points

from test_gpu_coefficients import B, reference  # noqa: F401

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,s,family", [(8, 16, 1), (16, 32, 0), (16, 48, 0), (16, 64, 1), (16, 80, 0), (16, 96, 0), (16, 300, 0),
                                        (8, 80, 2), (128, 65, 0), (128, 257, 0)])
def test_ends_of_the_domain(B, n, s, family):  # noqa: F811
    Y = 2.0 * random_points(n + s, 4, s)
    Y[0], Y[1] = 1.0, -1.0
    if n <= 16:
        c, zero = n * n // 2 + 1, reference(n, np.zeros(s), 1.0, family)
        unit = [np.float64(reference(n, np.eye(1, s, j)[0], 1.0, family)[c] - zero[c]) for j in range(s)]
        Y[2] = np.where(np.array(unit) < 0, -1.0, 1.0)
    with B.Context(0) as ctx:
        if family == 2:
            ctx.mq_set_islands(s, 4.0 / 3.0, 2.0, 4.0 / 3.0, 2.0)
        else:
            ctx.mq_set_coefficient(1.0, s, family, 2.0)
        ctx.mq_set_levels([Level(n, n, s, s, 8, 2)])
        ctx.mq_set_precision(B.MQ_PREC_MIXED)
        d = torch.empty((4, 2 * n * n), dtype=torch.float64, device="cuda")
        ctx.mq_coefficients_device(n, s, torch.from_numpy(Y).cuda(), 4, s, d)
    for y, got in zip(Y, d.cpu().numpy()):
        ref = reference(n, y, 1.0, family)
        assert float(np.abs(got - ref).max()) <= 4 * 2.0 ** -52 * float(np.abs(ref).max())
