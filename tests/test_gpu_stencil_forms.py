"""The FP64 stencil where its two forms (aligned integers; plain FP64 next to the ends of the range) could differ from the
plain sum of the terms."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_03377_gb300 import build

    build.build()


def apply_gpu(pl, x):
    xd = torch.from_numpy(np.ascontiguousarray(x)).cuda()
    wd = torch.full_like(xd, float("nan"))
    pl.laplacian(xd, wd)
    return wd.cpu().numpy()


@pytest.mark.parametrize("bad", [np.inf, -np.inf])
@pytest.mark.parametrize("shape", [(8, 6, 1), (35, 9, 1), (8, 6, 5)])
@pytest.mark.parametrize("h", [(1.0, 1.0, 1.0), (1.0, 0.5, 2.0)])
def test_infinity_stays_an_infinity(shape, h, bad):
    """A lone infinity: itself at its point, its negative at its neighbours, nothing elsewhere."""
    from paper_2501_03377_gb300 import Plan

    nx, ny, nz = shape
    pl = Plan(nx, ny, nz, ("D", "D", "D"), h)
    x = np.zeros((nz, ny, nx))
    k = nz // 2
    x[k, 3, 4] = bad
    ref = np.zeros_like(x)
    ref[k, 3, 4] = bad
    for d in (-1, 1):
        ref[k, 3 + d, 4] = ref[k, 3, 4 + d] = -bad
        if nz > 1:
            ref[k + d, 3, 4] = -bad
    assert np.array_equal(apply_gpu(pl, x), ref)
    pl.close()


def neighbours(x, axis):
    """Start and end neighbours of every point along an array axis, Dirichlet ghosts."""
    z = np.zeros_like(np.take(x, [0], axis))
    e = np.concatenate([z, x, z], axis)
    return np.take(e, range(x.shape[axis]), axis), np.take(e, range(2, x.shape[axis] + 2), axis)


@pytest.mark.parametrize("shape", [(33, 9, 7), (20, 34, 3), (40, 24, 1)])
@pytest.mark.parametrize("h", [(1.0, 1.0, 2.0), (1.0, 0.49, 1.0), (2.0**-8, 1.0, 16.0), (1.0, 0.01, 3.0), (0.1, 1.0, 10.0),
                               (50.0, 1.0, 0.02)])
def test_unequal_spacings_large_values_on_a_weak_axis(shape, h):
    """Every second plane, row or column 2^12 to 2^40 times larger than the others: where the axis across them has the
    small weight, the other axes' differences must keep their own accuracy.

    Bound as for any sum of the seven terms in FP64: 4 x 2^-52 of the sum of their magnitudes (a conversion, a product and
    the sums of the axes), per point, against extended precision.
    """
    from paper_2501_03377_gb300 import Plan

    nx, ny, nz = shape
    pl = Plan(nx, ny, nz, ("D", "D", "D"), h)
    rng = np.random.default_rng(51)
    base = rng.standard_normal((nz, ny, nx))
    for axis in range(3):
        if base.shape[axis] == 1:
            continue
        odd = np.indices(base.shape)[axis] % 2 == 1
        for k in (12, 26, 40):
            x = np.where(odd, np.ldexp(base, k), base)
            w = apply_gpu(pl, x)
            X = x.astype(np.longdouble)
            ref, mag = np.zeros_like(X), np.zeros_like(X)
            for m in range(3):
                if X.shape[2 - m] == 1:
                    continue
                lo, hi = neighbours(X, 2 - m)
                ref += (2 * X - lo - hi) / np.longdouble(h[m]) ** 2
                mag += (2 * np.abs(X) + np.abs(lo) + np.abs(hi)) / np.longdouble(h[m]) ** 2
            worst = (np.abs(w - ref) / mag).max()
            assert worst <= 4 * 2.0**-52, (axis, k, float(worst * 2.0**52))
    pl.close()


@pytest.mark.parametrize("shape", [(3, 700, 5), (8, 33, 4), (16, 16, 3), (5, 51, 1), (257, 3, 6), (255, 4, 3), (3, 3, 900)])
def test_field_on_narrow_planes(shape):
    """Planes below, at and above the 256 columns of a block: the exact differences, one rounding each (1 / (2 h) a power of
    two) or two."""
    from paper_2501_03377_gb300 import Plan

    nx, ny, nz = shape
    h = (1.0, 0.3, 0.25)
    pl = Plan(nx, ny, nz, ("D", "D", "D"), h)
    u = np.random.default_rng(52).standard_normal((nz, ny, nx))
    ud = torch.from_numpy(u).cuda()
    out = [torch.full_like(ud, float("nan")) for _ in range(3)]
    pl.efield(ud, *out)
    for m in range(3 if nz > 1 else 2):
        lo, hi = neighbours(u, 2 - m)
        assert np.array_equal(out[m].cpu().numpy(), (lo - hi) * (0.5 / h[m]))
    pl.close()


@pytest.mark.parametrize("narrow", [(8, 512, 512), (3, 700, 998)])
def test_field_of_a_narrow_grid_costs_what_a_wide_one_does(narrow):
    """The same number of points, twice the time at most (tiles 32 columns wide: 3.4 and 7 times)."""
    from paper_2501_03377_gb300 import Plan

    def best(shape):
        nx, ny, nz = shape
        pl = Plan(nx, ny, nz, ("D", "D", "D"))
        u = torch.zeros((nz, ny, nx), dtype=torch.float64, device="cuda")
        out = [torch.empty_like(u) for _ in range(3)]
        times = []
        for _ in range(8):
            t = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            t[0].record()
            for _ in range(10):
                pl.efield(u, *out)
            t[1].record()
            torch.cuda.synchronize()
            times.append(t[0].elapsed_time(t[1]))
        pl.close()
        return min(times)

    assert best(narrow) <= 2.0 * best((512, 512, 8))
