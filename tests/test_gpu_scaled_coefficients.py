"""Coefficients times a power of two: every eigenvalue is exactly that multiple, functionals and all counters stay what
they are, whatever the precision and the kernel (FP32 sums of squares would leave FP32's range at 2^-64 and 2^64
long before the values themselves do).

No tolerance: products with powers of two are exact, and nothing here may round differently (the exponents are
multiples of the library's own step of scale, 2^32)."""
import numpy as np
import pytest

from synthetic_inputs import Level, random_points

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def B():
    from paper_2103_03407_gb300 import binding, build

    build.build()
    if not torch.cuda.is_available():
        pytest.fail("a GPU test ran without a CUDA device")
    return binding


@pytest.mark.parametrize("nf,nc,np_", [(16, 8, 8), (32, 16, 0), (64, 32, 32), (16, 16, 0)])
@pytest.mark.parametrize("prec", [0, 1])
def test_coefficient_arrays(B, nf, nc, np_, prec):
    s, nb = 16, 24
    dY = torch.from_numpy(random_points(5, nb, s)).cuda()
    with B.Context(0) as ctx:
        ctx.mq_set_coefficient(1.0, s, 0, 2.0)
        ctx.mq_set_levels([Level(nf, nc, s, 4, 64, 2)])
        a = []
        for n, k in ((nf, s), (nc, 4), (np_, 8)):
            a.append(torch.empty((nb, 2 * n * n), dtype=torch.float64, device="cuda") if n else None)
            if n:
                ctx.mq_coefficients_device(n, k, dY, nb, s, a[-1])
    ref = None
    for e in (0, -64, -32, 32, 64):
        out = torch.empty((nb, 4), dtype=torch.float64, device="cuda")
        stat = torch.empty((nb, 4), dtype=torch.int32, device="cuda")
        outer = torch.zeros((nb, 2), dtype=torch.int32, device="cuda")
        af, ac, ap = (None if v is None else v * 2.0 ** e for v in a)
        B.mq_twogrid_samples_noalloc(nf, nc, np_, prec, nb, af, ac, ap, out, stat, outer)
        torch.cuda.synchronize()
        got = [(out * 2.0 ** -e).cpu().numpy(), stat.cpu().numpy(), outer.cpu().numpy()]
        assert not got[1][:, 3].any()
        ref = ref or got
        assert all(np.array_equal(x, y) for x, y in zip(got, ref)), e


@pytest.mark.parametrize("n,nc,prec,tier,nu,qoi", [(16, 16, 1, -1, 0, 0), (64, 64, 1, -1, 0, 1), (16, 8, 1, 0, 0, 0),
                                                  (32, 8, 1, 1, 0, 0), (64, 8, 1, 1, 0, 1), (64, 16, 1, 1, 2, 0),
                                                  (256, 32, 1, 1, 0, 0), (32, 8, 0, 0, 0, 0)])
def test_zeroth_term(B, n, nc, prec, tier, nu, qoi):
    s, got = 8, []
    for e in (0, 32, 64):
        with B.Context(0) as ctx:
            ctx.mq_set_coefficient(2.0 ** e, s, 0, 2.0)
            ctx.mq_set_levels([Level(n, nc, s, s if n == nc else 3, 64, 2)])
            ctx.mq_set_precision(prec)
            ctx.mq_set_qoi(qoi)
            ctx.mq_set_level_config(0, tier, 0, nu)
            lam = ctx.mq_eval_point(0, np.zeros(s))
            st = ctx.mq_get_stats()
        scale = [2.0 ** -e, 1.0 if qoi else 2.0 ** -e]
        got.append([v * f for v, f in zip(lam[:2], scale)] + [st[k] for k in ("coarse_iters_mean", "fine_iters_mean", "noconv")])
    assert got[0] == got[1] == got[2] and got[0][-1] == 0
