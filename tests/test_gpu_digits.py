"""The FP64 form's mode products on the tensor cores (digit slices): sizes at the edges of their tiles.

The 64-wide K tiles, 128-column blocks, 16-wide K steps, 32-row data tiles and the bound of 256 points each have a
size below, at and above them; axes past 256 points mix the digit products with the FP64 ones.  Tolerance of the
preconditioner: 1e-12, the bar of the FP64 form (six products of length <= 256, each O(l 2^-53) of its operands).
The reference applies the three products with the plan's own eigenpairs (checked against eq. lap1d elsewhere): a
dense eigensolver's smallest eigenvalues are off by eps ||L|| / lambda, more than the tolerance at these lengths.
Scaling the input by a power of two scales every step exactly, so the outputs are compared bit for bit.
"""
import numpy as np
import pytest

from inputs import synth
from tests._util import rel_err

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_03377_gb300 import build

    build.build()


def reference(pl, r):
    axes = [pl.eigenpairs(m) for m in range(3)]
    lam = [np.array(a[0]) for a in axes]
    V = [np.array(a[1]).reshape(len(a[0]), len(a[0])) for a in axes]
    modes = lambda t, m: np.einsum("kc,kji->cji", m[2], np.einsum("jc,kji->kci", m[1], t @ m[0], optimize=True),  # noqa: E731
                                   optimize=True)
    s = lam[2][:, None, None] + lam[1][None, :, None] + lam[0][None, None, :]
    g = np.divide(1.0, s, out=np.zeros_like(s), where=s > 0)
    return modes(modes(r, V) * g, [v.T for v in V])


SHAPES = [(3, 3, 3), (16, 15, 17), (63, 8, 5), (64, 33, 4), (65, 9, 3), (127, 7, 3), (128, 32, 6), (129, 8, 4),
          (255, 5, 3), (256, 8, 3), (4, 256, 5), (5, 3, 255), (192, 66, 1), (300, 6, 4), (7, 257, 1), (257, 300, 1)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("bcs", [("P", "D", "N"), ("DN", "ND", "D"), ("N", "P", "P")])
def test_precond_edges(shape, bcs):
    from paper_2501_03377_gb300 import Plan

    nx, ny, nz = shape
    pl = Plan(nx, ny, nz, bcs)
    r = synth.random_field(nx, ny, nz, seed=31)
    ref = reference(pl, r)
    # one double of slack in front: rows that are only 8-byte aligned
    buf = torch.zeros(r.size + 1, dtype=torch.float64, device="cuda")
    outs = []
    for off, scale in ((0, 1.0), (1, 1.0), (0, 2.0**900), (0, 2.0**-900)):
        rd = buf[off : off + r.size].view(nz, ny, nx)
        rd.copy_(torch.from_numpy(r * scale))
        zd = torch.full((nz, ny, nx), np.nan, dtype=torch.float64, device="cuda")
        pl.precond(rd, zd)
        outs.append(zd.cpu().numpy() / scale)
    assert rel_err(outs[0], ref) <= 1e-12
    for z in outs[1:]:
        assert np.array_equal(z, outs[0])


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_non_finite_input_spreads(bad):
    from paper_2501_03377_gb300 import Plan

    pl = Plan(40, 24, 12, ("P", "D", "N"))
    r = synth.random_field(40, 24, 12, seed=32)
    r[3, 5, 7] = bad
    zd = torch.zeros((12, 24, 40), dtype=torch.float64, device="cuda")
    pl.precond(torch.from_numpy(r).cuda(), zd)
    assert not bool(torch.isfinite(zd).any())


def test_zero_rows_and_zero_input():
    from paper_2501_03377_gb300 import Plan

    pl = Plan(40, 24, 12, ("P", "D", "N"))
    r = np.zeros((12, 24, 40))
    zd = torch.ones((12, 24, 40), dtype=torch.float64, device="cuda")
    pl.precond(torch.from_numpy(r).cuda(), zd)
    assert bool((zd == 0).all())
    r[5, 7] = synth.random_field(40, 1, 1, seed=33)[0, 0]  # one row of the field
    ref = reference(pl, r)
    pl.precond(torch.from_numpy(r).cuda(), zd)
    assert rel_err(zd.cpu().numpy(), ref) <= 1e-12


@pytest.mark.parametrize("shape", [(130, 200, 200), (40, 208, 200), (200, 256, 40)])
def test_precond_many_tiles_a_block(shape):
    """Passes of 5 to 10 data tiles per block, with one and two column blocks and with an eigenbasis that stays resident:
    the rings, the accumulators and the eight row-exponent buffers go round."""
    from paper_2501_03377_gb300 import Plan

    nx, ny, nz = shape
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert max(ny * nz, nx * nz, nx * ny) > 4 * 32 * sms
    pl = Plan(nx, ny, nz, ("P", "D", "N"))
    r = synth.random_field(nx, ny, nz, seed=34)
    # rows and planes of their own magnitude: a row's exponent read from another tile's buffer shows
    r *= np.exp2(np.random.default_rng(35).integers(-40, 40, (nz, ny, 1)))
    rd = torch.from_numpy(r).cuda()
    zd = torch.full_like(rd, float("nan"))
    pl.precond(rd, zd)
    assert rel_err(zd.cpu().numpy(), reference(pl, r)) <= 1e-12
    pl.close()
