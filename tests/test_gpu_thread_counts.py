"""The threads per CTA of the per-sample kernel change the order of its sums and nothing else: with a loose eigen target,
where the start vector of every point shows in its eigenvalue, all counts give the same values.

Tolerance: the sums of a step (FP32 in the mixed path) round differently, 1e-6 relative of a correction; at the target 1e-3
the last correction is 1e-3 of the vector and the eigenvalue second order in what is left, below 1e-9.  Chains of
another length move it by 3e-7."""
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


@pytest.mark.parametrize("n,nc", [(8, 8), (16, 8), (32, 32)])
@pytest.mark.parametrize("prec", [0, 1])
def test_threads_do_not_change_the_chains(B, n, nc, prec):
    s, got = 16, []
    lv = Level(n, nc, s, s if n == nc else 4, 1024, 8)
    z, delta = lattice.cbc(64, s), shifts(n, [lv])[0]
    for threads in (0, 32, 64, 128, 256, 512):
        with B.Context(0) as ctx:
            ctx.mq_set_coefficient(1.0, s, 0, 2.0)
            ctx.mq_set_levels([lv])
            ctx.mq_set_lattice(0, z)
            ctx.mq_set_shifts(0, delta)
            ctx.mq_set_precision(prec)
            ctx.mq_set_eig_options(1e-3)
            ctx.mq_set_cta_threads(0, threads)
            got.append(ctx.mq_eval_level(0, 0, 1024)[0][..., :2])
    for v in got[1:]:
        assert np.abs(v - got[0]).max() <= 1e-9 * np.abs(got[0]).max()
