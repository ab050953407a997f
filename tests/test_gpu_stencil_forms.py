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
