"""The streaming tier's FP32 MINRES keeps 12 Lanczos vectors and combines them into the solution: solves that end
one iteration before, at and after a combination and after the second one (iteration caps below a
reduction that no solve reaches earlier), on meshes with one and with several tiles, both smoothers
and the reaction term, level by level and as one graph (whose iterations run in pairs), against the oracle.

Tolerance 1e-12 relative, as for the other streamed values at the residual target 1e-10 (the solve error enters
the Rayleigh quotient squared, below 1e-16; what is left is rounding of the sums on both sides); the refinement
reaches the target whatever an inner solve leaves, so an error in the combination would show as flagged samples
(MQNoConvergence) as well."""
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


@pytest.mark.parametrize("n,nc,nu,family,cap", [(16, 8, 1, 0, 12), (32, 8, 1, 0, 13), (64, 16, 1, 0, 11), (64, 16, 1, 0, 12),
                                               (64, 16, 1, 0, 13), (64, 16, 1, 0, 25), (64, 16, 2, 0, 13), (64, 16, 1, 2, 13),
                                               (128, 16, 1, 0, 24)])
def test_solves_around_a_combination(B, n, nc, nu, family, cap):
    lv = Level(n, nc, 16, 4, 64, 3)
    z = lattice.cbc(lv.N, lv.s)
    delta = shifts(n + cap, [lv])[0]
    got = []
    for graph in (False, True):
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
            ctx.mq_set_solver_options(1e-30, cap, 0)
            ctx.mq_set_level_config(0, 1, 0, nu)
            out = torch.empty((lv.R, 3, 4), dtype=torch.float64, device="cuda")
            if graph:
                ctx.mq_graph_capture([(0, 5, 8)], [out])
                ctx.mq_graph_launch()
            else:
                ctx.mq_eval_level_device(0, 5, 8, out)
                st = ctx.mq_get_stats()
                assert st["fine_iters_max"] % cap == 0  # every solve ran into the cap
            torch.cuda.synchronize()
            got.append(out.cpu().numpy())
    assert np.array_equal(got[0], got[1])
    ref = mlqmc.level_samples(lv, None, z, delta, [5, 6, 7], 1.0, DECAYS if family == 2 else 2.0, family)
    assert np.abs(got[0][..., 1] - ref[..., 1]).max() <= 1e-12 * np.abs(ref[..., 1]).max()
