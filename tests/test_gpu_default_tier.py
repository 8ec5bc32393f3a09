"""Which tier the default takes, told by the number of kernels of a call (the streaming tier launches one per sweep): on both
sides of the FP64 limits (mesh 1/128 for any number of samples, 1/32 and 1/64 from 2^21 nodes in the call), for
points and ranges, under an explicit limit, with islands, and in the mixed path."""
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


@pytest.mark.parametrize("n,R,pts,prec,tier,family,streamed", [
    (128, 2, 1, 0, 0, 0, True), (128, 2, 1, 0, 1 << 20, 0, False), (64, 8, 64, 0, 0, 0, True), (64, 7, 73, 0, 0, 0, False),
    (64, 8, 64, 0, 1 << 20, 0, False), (64, 7, 73, 0, 64, 0, True), (32, 16, 128, 0, 0, 0, True), (32, 23, 89, 0, 0, 0, False),
    (16, 16, 512, 0, 0, 0, False), (128, 2, 1, 0, 0, 2, False), (32, 2, 1, 1, 0, 0, True), (16, 2, 1, 1, 0, 0, False)])
def test_default_tier_by_launches(B, n, R, pts, prec, tier, family, streamed):
    lv = Level(n, 8, 8, 3, 512, R)
    with B.Context(0) as ctx:
        if family == 2:
            ctx.mq_set_islands(8, 4.0 / 3.0, 2.0, 4.0 / 3.0, 2.0)
        else:
            ctx.mq_set_coefficient(1.0, 8, 0, 2.0)
        ctx.mq_set_levels([lv])
        ctx.mq_set_lattice(0, lattice.cbc(64, 8))
        ctx.mq_set_shifts(0, shifts(n + pts, [lv])[0])
        ctx.mq_set_precision(prec)
        ctx.mq_set_tier(tier)
        ctx.mq_eval_level(0, 0, pts)
        assert (ctx.mq_get_launch_count() > 40) == streamed
        if pts == 1:  # one parameter vector counts as one sample
            ctx.mq_reset_sums()
            ctx.mq_eval_point(0, np.zeros(8))
            assert (ctx.mq_get_launch_count() > 40) == streamed
