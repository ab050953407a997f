"""FP64 plans on streams of their own, many solves in flight: the digit passes of one plan start while the sweeps and passes
of others hold SMs, and every solve ends with the bits it has alone."""
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


def test_concurrent_solves_equal_solo_solves():
    from paper_2501_03377_gb300 import Plan
    from paper_2501_03377_gb300.binding import TPCG_ZERO_GUESS, tpcg_solve_batched

    shapes = [(64, 64, 32), (32, 48, 64), (96, 64, 40), (130, 60, 20), (64, 256, 16), (48, 48, 48), (200, 40, 30), (64, 64, 1)]
    nrhs, bcs = 24, ("P", "D", "N")
    streams = [torch.cuda.Stream() for _ in shapes]
    plans = [Plan(*sh, bcs, prec="fp64", stream=st.cuda_stream) for sh, st in zip(shapes, streams)]
    etas, solo = [], []
    for i, (nx, ny, nz) in enumerate(shapes):
        etas.append(torch.stack([torch.from_numpy(synth.random_field(nx, ny, nz, seed=100 + i)) for _ in range(nrhs)]).cuda())
    torch.cuda.synchronize()
    for pl, e in zip(plans, etas):
        u = torch.zeros_like(e[0])
        torch.cuda.synchronize()
        st, info = pl.solve(e[0], u, tol=1e-10, maxit=40, zero_guess=True)
        assert st == 0
        torch.cuda.synchronize()
        solo.append(u)
    ups = [torch.zeros_like(e) for e in etas]
    torch.cuda.synchronize()
    for _ in range(4):
        st, infos = tpcg_solve_batched([pl.handle for pl in plans], [nrhs] * len(plans), [e.data_ptr() for e in etas],
                                       [u.data_ptr() for u in ups], [1e-10] * len(plans), 40, TPCG_ZERO_GUESS)
        torch.cuda.synchronize()
        assert st == 0
        for u, ref in zip(ups, solo):
            for r in range(nrhs):
                assert torch.equal(u[r], ref)
    for pl in plans:
        pl.close()
