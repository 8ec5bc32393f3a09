"""Solves on the coarse mesh itself (the previous level's mesh is the coarse mesh, with a longer truncation),
which the FP32 kernel solves for the change of the eigenvector, with an FP64 solve behind it, and (from
coarse mesh 1/8 on, where the default residual target allows it) the fine solves beside them: against the oracle at the workload tolerance 1e-10
relative, over the smallest meshes, chain lengths, the reaction term, and a truncation so close to the coarse one
that the shift almost meets the eigenvalue (s' = S + 1: the last term changes the eigenvalue by ~1e-4 and less)."""
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


@pytest.mark.parametrize("nf,nc,sp,S,family,pts", [(4, 2, 8, 3, 0, 3), (16, 8, 24, 5, 0, 400), (16, 8, 6, 5, 0, 40),
                                                  (16, 8, 24, 5, 2, 40), (64, 32, 24, 5, 0, 3), (64, 32, 9, 8, 0, 5),
                                                  (512, 256, 9, 4, 0, 1)])
def test_previous_level_on_the_coarse_mesh(B, nf, nc, sp, S, family, pts):
    levels = [Level(nc, nc, sp, sp, 512, 3), Level(nf, nc, 2 * sp, S, 512, 3)]
    ds = shifts(nf + sp, levels)
    z = [lattice.cbc(lv.N, lv.s) for lv in levels]
    with B.Context(0) as ctx:
        if family == 2:
            ctx.mq_set_islands(2 * sp, *DECAYS)
        else:
            ctx.mq_set_coefficient(1.0, 2 * sp, 0, 2.0)
        ctx.mq_set_levels(levels)
        for l in range(2):
            ctx.mq_set_lattice(l, z[l])
            ctx.mq_set_shifts(l, ds[l])
        ctx.mq_set_precision(B.MQ_PREC_MIXED)
        ps, _ = ctx.mq_eval_level(1, 7, 7 + pts)
    ks = sorted({0, pts // 2, pts - 1})
    ref = mlqmc.level_samples(levels[1], levels[0], z[1], ds[1], [7 + k for k in ks], 1.0, DECAYS if family == 2 else 2.0,
                              family)
    for i, k in enumerate(ks):
        c = slice(1 if nc >= 8 else 2, 3)
        assert np.all(np.abs(ps[:, k, c] - ref[:, i, c]) <= 1e-10 * np.abs(ref[:, i, c])), k
