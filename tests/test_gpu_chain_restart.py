"""A sample without an eigenvalue (a coefficient that is not a number) leaves the other points of its warm-start
chain alone: only it is flagged, and every other value is the one it has in a call without such samples.

Tolerance 1e-10 relative, that of every per-sample value (the neighbours start from another vector)."""
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


@pytest.mark.parametrize("nf,nc", [(8, 8), (16, 8), (32, 32)])
@pytest.mark.parametrize("prec", [0, 1])
def test_one_bad_sample_in_a_chain(B, nf, nc, prec):
    s, nb = 8, 20000  # chains of tens of samples
    dY = torch.from_numpy(random_points(5, nb, s)).cuda()
    with B.Context(0) as ctx:
        ctx.mq_set_coefficient(1.0, s, 0, 2.0)
        ctx.mq_set_levels([Level(nf, nc, s, 4, 64, 2)])
        a_f, a_c = (torch.empty((nb, 2 * n * n), dtype=torch.float64, device="cuda") for n in (nf, nc))
        ctx.mq_coefficients_device(nf, s, dY, nb, s, a_f)
        ctx.mq_coefficients_device(nc, 4, dY, nb, s, a_c)
    bad = np.arange(1000, nb, 997)
    got = []
    for rows in ([], bad):
        a_c[rows, 0] = float("nan")
        out = torch.empty((nb, 4), dtype=torch.float64, device="cuda")
        stat = torch.empty((nb, 4), dtype=torch.int32, device="cuda")
        outer = torch.zeros((nb, 2), dtype=torch.int32, device="cuda")
        B.mq_twogrid_samples_noalloc(nf, nc, 0, prec, nb, None if nf == nc else a_f, a_c, None, out, stat, outer)
        torch.cuda.synchronize()
        assert np.array_equal(np.nonzero(stat.cpu().numpy()[:, 3])[0], rows)
        got.append(np.delete(out.cpu().numpy()[:, :2], bad, 0))
    assert np.abs(got[1] - got[0]).max() <= 1e-10 * np.abs(got[0]).max()
