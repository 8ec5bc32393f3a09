"""FP64 fine solves by the default tier on both sides of its limits (mesh 1/128 for any number of samples, meshes 1/32
and 1/64 from 2^21 nodes in a call), with a previous level on a finer mesh and on the coarse mesh itself,
against the per-sample kernel, as single points and as a range.

Tolerance 1e-10 relative, that of every per-sample value (both tiers stop at a relative residual of 1e-6, which
moves a value by at most ~3e-13)."""
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


@pytest.mark.parametrize("n,nc,np_,R,pts", [(128, 16, 64, 3, 1), (64, 16, 32, 7, 73), (64, 16, 32, 8, 64), (64, 32, 32, 8, 65),
                                           (32, 8, 16, 23, 89), (32, 16, 16, 16, 129)])
def test_default_tier(B, n, nc, np_, R, pts):
    levels = [Level(np_, min(nc, np_), 8, 3, 256, R), Level(n, nc, 16, 4, 256, R)]
    ds = shifts(n + pts, levels)
    z = [lattice.cbc(lv.N, lv.s) for lv in levels]
    got = []
    for tier in (0, 1 << 20):
        with B.Context(0) as ctx:
            ctx.mq_set_coefficient(1.0, 16, 0, 2.0)
            ctx.mq_set_levels(levels)
            for l in range(2):
                ctx.mq_set_lattice(l, z[l])
                ctx.mq_set_shifts(l, ds[l])
            ctx.mq_set_precision(B.MQ_PREC_FP64)
            ctx.mq_set_tier(tier)
            ps, _ = ctx.mq_eval_level(1, 3, 3 + pts)
            got.append(ps)
    assert np.abs(got[0] - got[1])[..., :3].max() <= 1e-10 * np.abs(got[1][..., :3]).max()
