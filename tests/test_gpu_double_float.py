"""The streaming tier's mixed path with its residual and Rayleigh quotient in double-float
arithmetic, against the oracle at the edges of its tiles: rows shorter than one four-node group's
neighbourhood (mesh 1/4), tiles with partial rows, one and several tiles per sample, odd sample
counts, both smoothers and the reaction term.

Tolerance 1e-12 relative: the residual target 1e-10 leaves ~3e-17 of solve error in the Rayleigh
quotient and the eigen target 1e-10 ~1e-19; the double-float sums are good to a few 2^-48 (4e-15) of
the distance between the coarse and the fine eigenvalue; the oracle's own sparse solves and sums
are in FP64 on systems of condition up to ~1e6.  The islands' coarse mesh does not resolve them, and
the eigenvector error enters their two-grid values ~1e4 times more strongly: still below 1e-12.
"""
import numpy as np
import pytest

from oracle import lattice, mlqmc
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


@pytest.mark.parametrize("n,nc,R,pts,nu,family", [(4, 2, 3, 1, 1, 0), (8, 4, 2, 5, 1, 0), (16, 8, 3, 3, 2, 0),
                                                  (32, 8, 3, 3, 1, 0), (64, 8, 1, 3, 1, 0), (64, 16, 3, 1, 2, 0),
                                                  (256, 32, 1, 1, 1, 0), (16, 8, 3, 3, 1, 2), (64, 16, 3, 1, 1, 2)])
def test_streamed_values_match_the_oracle(B, n, nc, R, pts, nu, family):
    lv = Level(n, nc, 16, 4, 64, max(R, 2))
    z = lattice.cbc(lv.N, lv.s)
    delta = shifts(n + nc, [lv])[0]
    decays = (4.0 / 3.0, 2.0, 4.0 / 3.0, 2.0)
    with B.Context(0) as ctx:
        if family == 2:
            ctx.mq_set_islands(lv.s, *decays)
        else:
            ctx.mq_set_coefficient(1.0, lv.s, 0, 2.0)
        ctx.mq_set_levels([lv])
        ctx.mq_set_lattice(0, z)
        ctx.mq_set_shifts(0, delta)
        ctx.mq_set_precision(B.MQ_PREC_MIXED, 1e-10)
        ctx.mq_set_eig_options(1e-10)
        ctx.mq_set_level_config(0, 1, 0, nu)
        ps, _ = ctx.mq_eval_level(0, 5, 5 + pts)
    ref = mlqmc.level_samples(lv, None, z, delta, list(range(5, 5 + pts)), 1.0, decays if family == 2 else 2.0, family)
    assert np.abs(ps[..., 1] - ref[..., 1]).max() <= 1e-12 * np.abs(ref[..., 1]).max()
