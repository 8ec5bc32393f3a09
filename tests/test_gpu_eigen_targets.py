"""Eigen-residual targets around and below what an iterate of 48 bits reaches: every sample converges, in few iterations,
whatever the mesh, the target and the contrast of the coefficients.

Tolerances: the eigenvalues of both precisions are exact to the square of the target; their sums are good to about
2e-12 on mesh 1/128 (mixed: 48 bits; FP64: eps lambda_max / lambda_1), the two-grid values to 1e-10 as everywhere."""
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


@pytest.mark.parametrize("n,tol", [(4, 3.3e-14), (16, 3e-14), (16, 5.2e-13), (32, 1e-13), (32, 2.1e-12), (64, 3e-13),
                                   (64, 8.3e-12), (128, 1e-12), (128, 3.3e-11)])
@pytest.mark.parametrize("family", [0, 2])
def test_targets_are_reached(B, n, tol, family):
    lv = Level(n, n, 16, 16, 64, 4)
    z, delta = lattice.cbc(lv.N, lv.s), shifts(n, [lv])[0]
    got = []
    for prec in (B.MQ_PREC_MIXED, B.MQ_PREC_FP64):
        with B.Context(0) as ctx:
            if family == 2:
                ctx.mq_set_islands(lv.s, 4.0 / 3.0, 2.0, 4.0 / 3.0, 2.0)
            else:
                ctx.mq_set_coefficient(1.0, lv.s, 0, 2.0)
            ctx.mq_set_levels([lv])
            ctx.mq_set_lattice(0, z)
            ctx.mq_set_shifts(0, delta)
            ctx.mq_set_precision(prec)
            ctx.mq_set_eig_options(tol)
            got.append(ctx.mq_eval_level(0, 3, 19)[0][..., 0])
            st = ctx.mq_get_stats()
            assert st["noconv"] == 0 and st["coarse_iters_max"] <= 40
    assert np.abs(got[0] - got[1]).max() <= 2e-12 * got[1].max()


@pytest.mark.parametrize("nc,contrast", [(8, 1e3), (16, 1e2), (32, 1e1), (64, 1e1), (128, 1.0)])
def test_contrast_of_coefficient_arrays(B, nc, contrast):
    nf, nb, got = 2 * nc, 16, []
    for prec in (0, 1):
        a = []
        for n in (nf, nc):
            x = (np.arange(n) + 0.5) / n
            inside = np.maximum(abs(x[:, None] - 0.5), abs(x[None, :] - 0.5)) < 0.25
            cell = np.where(inside, contrast, 1.0)[None] * (1.0 + np.arange(nb) / (16.0 * nb))[:, None, None]
            a.append(torch.from_numpy(np.ascontiguousarray(np.stack([cell, cell], 1).reshape(nb, -1))).cuda())
        out = torch.empty((nb, 4), dtype=torch.float64, device="cuda")
        stat = torch.empty((nb, 4), dtype=torch.int32, device="cuda")
        outer = torch.zeros((nb, 2), dtype=torch.int32, device="cuda")
        B.mq_twogrid_samples_noalloc(nf, nc, 0, prec, nb, a[0], a[1], None, out, stat, outer)
        torch.cuda.synchronize()
        s = stat.cpu().numpy()
        assert not s[:, 3].any() and s[:, 0].max() <= 60
        got.append(out.cpu().numpy()[:, :2])
    assert np.abs(got[0] - got[1]).max() <= 1e-10 * got[0].max()
