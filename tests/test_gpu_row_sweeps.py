"""The sweeps by windows of rows (launches of at least 2^24 nodes) against the four-node sweeps (few samples) and
the oracle: the smallest and larger meshes, whose last group of rows is short on every level, one and several
tiles per sample, one and several levels of the cycle by rows (sample counts on both sides of the limits), and the
reaction term.

The sweeps form the same values by the same expressions, so the iterates of both forms agree but for the
grouping of the sums <v, z>.  Tolerance 1e-12 relative against both, as for the other streamed values at the
residual target 1e-10: the solve error enters the Rayleigh quotient squared, the rest is rounding of the sums."""
import numpy as np
import pytest

from oracle import lattice, mlqmc
from synthetic_inputs import Level, shifts

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

DECAYS = (4.0 / 3.0, 2.0, 4.0 / 3.0, 2.0)


@pytest.fixture(scope="module")
def B():
    from paper_2103_03407_gb300 import binding, build

    build.build()
    if not torch.cuda.is_available():
        pytest.fail("a GPU test ran without a CUDA device")
    return binding


@pytest.mark.parametrize("n,nc,family,pts", [(64, 16, 0, 1366), (64, 16, 2, 1366), (128, 16, 0, 342), (128, 16, 0, 1366),
                                            (256, 32, 0, 86), (256, 32, 2, 86)])
def test_sweeps_by_rows(B, n, nc, family, pts):
    lv = Level(n, nc, 16, 4, 2048, 3)
    z = lattice.cbc(lv.N, lv.s)
    delta = shifts(n + pts, [lv])[0]
    some = sorted({0, pts // 2, pts - 1})
    with B.Context(0) as ctx:
        if family == 2:
            ctx.mq_set_islands(lv.s, *DECAYS)
        else:
            ctx.mq_set_coefficient(1.0, lv.s, 0, 2.0)
        ctx.mq_set_levels([lv])
        ctx.mq_set_lattice(0, z)
        ctx.mq_set_shifts(0, delta)
        ctx.mq_set_precision(B.MQ_PREC_MIXED, 1e-10)
        ctx.mq_set_eig_options(1e-10)
        many, _ = ctx.mq_eval_level(0, 5, 5 + pts)
        few = np.stack([ctx.mq_eval_level(0, 5 + k, 6 + k)[0][:, 0] for k in some], 1)
    top = np.abs(many[..., 1]).max()
    assert np.abs(many[:, some, 1] - few[..., 1]).max() <= 1e-12 * top
    ref = mlqmc.level_samples(lv, None, z, delta, [5 + k for k in some[::2]], 1.0, DECAYS if family == 2 else 2.0, family)
    assert np.abs(many[:, some[::2], 1] - ref[..., 1]).max() <= 1e-12 * top
