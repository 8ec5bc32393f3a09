"""The tensor-core coefficient kernels at the edges of their dispatch, against a long-double evaluation of
eq. coeff_s: contractions of one to five K steps (sample slices resident) and six (streamed), ragged
sample and triangle tiles, more tiles than one wave of CTAs, an output that is only 8-byte aligned, a
zeroth term far above the terms (the FP64 form of the fold), the separable form with odd and prefix
truncations on both triangle planes, and the piecewise zeroth term.

Tolerance: four units of FP64 rounding of the largest |a| (half of one rounds the result; the tables'
FP64 sines and products and the slices' remainders stay below one more for these sums of terms; the
fixed-point sums add less than a hundredth).  The reference is in long double, because FP64 sines of
arguments up to 72 pi would by themselves be off by more than that for the islands' terms.
"""
import numpy as np
import pytest

from oracle import fem
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


LD = np.longdouble
PI = LD("3.14159265358979323846264338327950288")


def reference(n, y, a0, family, which=0):
    """a (or, which = 1, b) at the centroids of mesh 1/n in long double: lower plane, then upper plane."""
    s = y.size
    j = np.arange(1, s + 1).astype(LD)
    out = []
    for plane in range(2):
        i = np.arange(n).astype(LD)
        x1, x2 = (3 * i + (2 - plane)) / LD(3 * n), (3 * i + (1 + plane)) / LD(3 * n)
        if family < 2:
            k1, k2 = np.array(fem.psi_pairs(s, family)).T
            t = (y.astype(LD) * j ** -2)[:, None] * np.sin(PI * k2.astype(LD)[:, None] * x2)  # [s, rows]
            T = np.zeros((n, k1.max()), dtype=LD)
            np.add.at(T.T, k1 - 1, t)
            S = np.sin(PI * np.arange(1, k1.max() + 1).astype(LD)[:, None] * x1)
            out.append(LD(a0) + T.dot(S))
            continue
        p = (LD(4) / 3, LD(2))
        sig = (2.0, 0.3) if which else (0.01, 0.011)
        band = lambda t: ((t > 0.125) & (t < 0.375)) | ((t > 0.625) & (t < 0.875))  # noqa: E731
        inside = band(x2)[:, None] & band(x1)[None, :]
        # (the library multiplies the FP64 constants)
        v = np.where(inside, LD(sig[0] * (np.pi / np.sqrt(2.0))), LD(sig[1]))
        for m in range(1, s + 1):
            k, r = (m + 1) // 2, 0 if m % 2 else 1
            w = LD(sig[r]) * LD(k) ** -p[r] * np.sin(PI * 8 * (k + 1) * x2)[:, None] * np.sin(PI * 8 * k * x1)[None, :]
            v = v + LD(y[m - 1]) * np.where(inside if r == 0 else ~inside, w, LD(0))
        out.append(v)
    return np.stack(out).reshape(-1)


@pytest.mark.parametrize("n,s,nb,family,a0,offset", [
    (2, 16, 1, 1, 2.5, 0), (4, 32, 129, 1, 2.5, 1), (8, 48, 130, 0, 1.0, 0), (16, 49, 5, 0, 1.0, 0), (64, 64, 600, 0, 1.0, 0),
    (32, 80, 257, 1, 2.5, 0), (32, 81, 257, 1, 2.5, 0), (16, 40, 3, 0, 1e9, 0), (16, 300, 3, 0, 1e9, 1),
    (128, 65, 3, 0, 1.0, 0), (128, 257, 1, 0, 1.0, 0), (256, 700, 2, 0, 1.0, 0), (128, 257, 2, 0, 1e9, 0),
    (8, 17, 131, 2, 1.0, 0), (16, 96, 3, 2, 1.0, 1)])
def test_coefficients_at_the_edges_of_the_dispatch(B, n, s, nb, family, a0, offset):
    Y = random_points(7 * n + s, nb, s)
    Y[0] = np.where(np.arange(s) % 2, -0.5, 0.5 - 2.0 ** -53)  # the ends of the range
    dY = torch.from_numpy(Y).cuda()
    buf = torch.empty(nb * 2 * n * n + offset, dtype=torch.float64, device="cuda")
    with B.Context(0) as ctx:
        if family == 2:
            ctx.mq_set_islands(s, 4.0 / 3.0, 2.0, 4.0 / 3.0, 2.0)
        else:
            ctx.mq_set_coefficient(a0, s, family, 2.0)
        ctx.mq_set_levels([Level(n, n, s, s, 8, 2)])
        ctx.mq_set_precision(B.MQ_PREC_MIXED)
        for which, k in ((0, s), (0, max(1, s - 3))) + (((1, s),) if family == 2 else ()):
            d = buf[offset:].view(nb, 2 * n * n)
            (ctx.mq_reaction_coefficients_device if which else ctx.mq_coefficients_device)(n, k, dY, nb, s, d)
            got = d.cpu().numpy()
            for b in np.unique(np.linspace(0, nb - 1, 12).astype(int)):
                ref = reference(n, Y[b][:k], a0, family, which)
                top = max(float(np.abs(ref).max()), 1.0 if family < 2 else 0.0)
                assert float(np.abs(got[b].astype(LD) - ref).max()) <= 4 * 2.0 ** -52 * top, (which, k, b)
