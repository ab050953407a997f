"""The FP64 stencil and field on values of any size: the seven values of a point are aligned as 59-bit integers.

Error bound of tpcg_apply_laplacian: per point 2^-52 of the sum of the magnitudes it adds (one FP64 rounding of the
result and 2^-58 of the largest value per term), against the same sum in extended precision.  Scaling the field by a
power of two scales every step exactly, so those results are compared bit for bit; next to the ends of the FP64 range
the plain FP64 form runs instead.
"""
import numpy as np
import pytest

from inputs import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_03377_gb300 import build

    build.build()


def neighbours(x, bcs):
    """(start, end) neighbours of every point per axis (x, y, z) under the ghost rules of the boundary conditions."""
    out = []
    for m in range(3 if x.shape[0] > 1 else 2):
        d = 2 - m
        first, last = np.take(x, [0], d), np.take(x, [-1], d)
        lo = last if bcs[m] == "P" else first if bcs[m] in ("N", "ND") else np.zeros_like(first)
        hi = first if bcs[m] == "P" else last if bcs[m] in ("N", "DN") else np.zeros_like(first)
        e = np.concatenate([lo, x, hi], d)
        out.append((np.take(e, range(x.shape[d]), d), np.take(e, range(2, x.shape[d] + 2), d)))
    return out


def apply_gpu(pl, x):
    xd = torch.from_numpy(np.ascontiguousarray(x)).cuda()
    wd = torch.full_like(xd, float("nan"))
    pl.laplacian(xd, wd)
    return wd.cpu().numpy()


@pytest.mark.parametrize("shape", [(33, 9, 5), (64, 17, 3), (3, 3, 3), (40, 24, 1)])
@pytest.mark.parametrize("bcs", [("P", "D", "N"), ("DN", "P", "ND")])
@pytest.mark.parametrize("h", [(1.0, 1.0, 1.0), (0.5, 0.5, 0.5), (1.0, 0.5, 2.0)])
def test_laplacian_any_magnitude(shape, bcs, h):
    from paper_2501_03377_gb300 import Plan

    nx, ny, nz = shape
    pl = Plan(nx, ny, nz, bcs, h)
    base = synth.random_field(nx, ny, nz, seed=41)
    wide = base * np.exp(12.0 * synth.random_field(nx, ny, nz, seed=42))  # neighbours many orders apart
    sparse = np.where(np.abs(base) > 1.5, base, 0.0)
    for x in (base, wide, sparse, np.zeros_like(base)):
        w = apply_gpu(pl, x)
        X = x.astype(np.longdouble)
        ref, mag = np.zeros_like(X), np.zeros_like(X)
        for m, (lo, hi) in enumerate(neighbours(X, bcs)):
            ref += (2 * X - lo - hi) / np.longdouble(h[m]) ** 2
            mag += (2 * np.abs(X) + np.abs(lo) + np.abs(hi)) / np.longdouble(h[m]) ** 2
        rounds = 1 if len(set(h)) == 1 else 4  # one rounding; unequal spacings: a conversion, product and sums per axis
        assert np.all(np.abs(w - ref) <= rounds * 2.0**-52 * mag)
        if x is not wide:  # (its smallest values would leave the normal range)
            for k in (900, -900):
                assert np.array_equal(apply_gpu(pl, x * 2.0**k) * 2.0**-k, w)
    for k in (1015, -1010):  # the plain FP64 form: a handful of roundings
        w = apply_gpu(pl, base * 2.0**k) * 2.0**-k
        assert np.abs(w - apply_gpu(pl, base)).max() <= 1e-13 * np.abs(w).max()


@pytest.mark.parametrize("h", [(1.0, 0.25, 2.0), (0.3, 1.0, 0.7)])
def test_field_scaling(h):
    """(lo - hi) / (2 h): exact differences and one rounding where 1 / (2 h) is a power of two, two otherwise."""
    from paper_2501_03377_gb300 import Plan

    nx, ny, nz, bcs = 35, 18, 6, ("N", "P", "D")
    pl = Plan(nx, ny, nz, bcs, h)
    for scale in (1.0, 2.0**1000, 2.0**-1015):
        u = synth.random_field(nx, ny, nz, seed=43) * scale
        ud = torch.from_numpy(u).cuda()
        out = [torch.empty_like(ud) for _ in range(3)]
        pl.efield(ud, *out)
        for m, (lo, hi) in enumerate(neighbours(u, bcs)):
            assert np.array_equal(out[m].cpu().numpy(), (lo - hi) * (0.5 / h[m]))
