"""The default sweep grain, set again, is the default: small grids get back the launch grids of a plan left alone."""
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


@pytest.mark.parametrize("prec", ["fp64", "fp16", "bf16x3"])
@pytest.mark.parametrize("shape", [(40, 24, 12), (64, 64, 1), (33, 40, 7)])
def test_default_grain_set_again_is_the_default(shape, prec):
    from paper_2501_03377_gb300 import Plan, binding

    nx, ny, nz = shape
    pl = Plan(nx, ny, nz, ("P", "D", "N"), prec=prec)
    eta = torch.from_numpy(synth.random_field(nx, ny, nz, seed=81)).cuda()

    def solve():
        u = torch.zeros_like(eta)
        st, info = pl.solve(eta, u, tol=1e-8, maxit=60, zero_guess=True)
        assert st == 0
        return u, info

    u0, i0 = solve()
    coarse = []
    for grain in (64, 4):
        pl.set_option(binding.TPCG_OPT_SWEEP_GRAIN, grain)
        u, info = solve()
        coarse.append(torch.equal(u, u0) and info["rel_res_true"] == i0["rel_res_true"])
    assert coarse[1]
    # (the grain matters here: other blocks, other order of the sums)
    assert not coarse[0]
    pl.close()
