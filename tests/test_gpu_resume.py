"""A chunk of iterations whose recurrence met the tolerance while the true residual did not: the rest of the chunk pauses,
the check at its end fails, and the next chunk goes on from the device's iteration count.  The outcome must not depend on
how the host cut the solve into chunks."""
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


KEYS = ("iters", "checks", "precond_applies", "rel_res_true", "rel_res_recur")


@pytest.mark.parametrize("shape,bcs", [((64, 64, 32), ("P", "D", "N")), ((96, 80, 1), ("P", "P", "P"))])
@pytest.mark.parametrize("prec", ["fp64", "fp16", "bf16x3"])
def test_outcome_after_failed_checks_does_not_depend_on_the_chunks(shape, bcs, prec):
    """Tolerances at the attainable residual and below it.  A fresh plan's chunks are 4, 2, 2, .. (FP64: 2, 1, 1, ..); a plan
    that has solved before begins with as many iterations as that solve took, up to 12."""
    from paper_2501_03377_gb300 import Plan, binding

    nx, ny, nz = shape
    eta = torch.from_numpy(synth.random_field(nx, ny, nz, seed=91)).cuda()
    most = 0
    for tol in (2e-15, 1e-15, 5e-16, 2e-16, 1e-16):
        out = []
        for primed, graphs in ((None, 0), (1e-2, 0), (1e-14, 0), (None, 1), (1e-14, 1)):
            stream = torch.cuda.Stream()
            pl = Plan(nx, ny, nz, bcs, prec=prec, stream=stream.cuda_stream)
            pl.set_option(binding.TPCG_OPT_GRAPHS, graphs)
            torch.cuda.synchronize()
            u = torch.zeros_like(eta)
            if primed:
                pl.solve(eta, u, tol=primed, maxit=40, zero_guess=True)
            st, info = pl.solve(eta, u, tol=tol, maxit=14, zero_guess=True)
            torch.cuda.synchronize()
            out.append((st, u, info))
            pl.close()
        st0, u0, i0 = out[0]
        most = max(most, i0["checks"])
        for st, u, info in out[1:]:
            assert st == st0 and torch.equal(u, u0)
            assert [info[k] for k in KEYS] == [i0[k] for k in KEYS]
    assert most >= 2  # a check failed and the solve went on


@pytest.mark.parametrize("prec", ["fp16", "bf16x3"])
def test_deferred_updates_after_failed_checks(prec):
    """The ring of recorded directions follows the device's count too: same outcome from every cut into chunks."""
    from paper_2501_03377_gb300 import Plan, binding

    nx, ny, nz, bcs = 64, 64, 32, ("P", "D", "N")
    eta = torch.from_numpy(synth.random_field(nx, ny, nz, seed=92)).cuda()
    most = 0
    for tol in (1e-15, 5e-16, 2e-16):
        out = []
        for primed in (None, 1e-2, 1e-14):
            pl = Plan(nx, ny, nz, bcs, prec=prec)
            pl.set_option(binding.TPCG_OPT_DEFER_U, 1)
            u = torch.zeros_like(eta)
            if primed:
                pl.solve(eta, u, tol=primed, maxit=40, zero_guess=True)
            st, info = pl.solve(eta, u, tol=tol, maxit=20, zero_guess=True)
            torch.cuda.synchronize()
            out.append((st, u, info))
            pl.close()
        most = max(most, out[0][2]["checks"])
        for st, u, info in out[1:]:
            assert st == out[0][0] and torch.equal(u, out[0][1])
            assert [info[k] for k in KEYS] == [out[0][2][k] for k in KEYS]
    assert most >= 2
