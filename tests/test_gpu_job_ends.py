"""Ends that only a held-up GPU reaches, presented to the host code by hooks (no wait runs out here)."""
import ctypes
import subprocess

import pytest

from inputs import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def hooks(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import os

    from paper_2501_03377_gb300 import build

    lib = build.build()
    out = str(tmp_path_factory.mktemp("hooks") / "hooks.so")
    src = os.path.join(os.path.dirname(__file__), "_job_hooks.cu")
    subprocess.run([build._nvcc(), *build.ARCH, *build.COMMON, "-shared", src,
                    "-o", out, lib, "-Xlinker", "-rpath=" + os.path.dirname(lib)], check=True)
    return ctypes.CDLL(out)


def plan_and_fields(prec):
    from paper_2501_03377_gb300 import Plan

    bcs = ("P", "D", "N")
    pl = Plan(40, 24, 12, bcs, prec=prec)
    eta = torch.from_numpy(synth.random_field(40, 24, 12, seed=71)).cuda()
    return pl, eta, torch.zeros_like(eta)


@pytest.mark.parametrize("prec", ["fp64", "bf16x3"])
def test_application_that_gave_up_is_reported_once(hooks, prec):
    from paper_2501_03377_gb300 import binding

    pl, r, z = plan_and_fields(prec)
    apply = lambda: binding.tpcg_precond_apply(pl.handle, r.data_ptr(), z.data_ptr())  # noqa: E731
    assert apply() == 0
    torch.cuda.synchronize()
    ref = z.clone()
    hooks.hook_give_up(pl.handle)
    z.zero_()
    assert apply() == binding.TPCG_ERR_TIMEOUT
    torch.cuda.synchronize()
    assert not bool(z.any())  # nothing was enqueued
    st, info = pl.solve(r, z.clone(), tol=1e-10, maxit=50, zero_guess=True)
    assert st == 0
    assert apply() == 0
    torch.cuda.synchronize()
    assert torch.equal(z, ref)
    pl.close()


@pytest.mark.parametrize("prec", ["fp64", "fp16", "bf16x3"])
@pytest.mark.parametrize("timeout", [0, 1])
def test_chunk_without_progress_ends_the_solve(hooks, prec, timeout):
    """A read-back in which no iteration completed, or a wait gave up, ends the solve in two steps (its end and the report
    of it) with an error; the plan solves again afterwards."""
    from paper_2501_03377_gb300 import binding

    pl, eta, u = plan_and_fields(prec)
    steps = ctypes.c_int(0)
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    st = hooks.hook_stalled_chunk(pl.handle, ptr(eta), ptr(u), timeout, ctypes.byref(steps))
    assert st == (binding.TPCG_ERR_TIMEOUT if timeout else binding.TPCG_ERR_NOT_CONVERGED)
    assert steps.value == 2
    st, info = pl.solve(eta, u, tol=1e-10, maxit=50, zero_guess=True)
    assert st == 0 and info["rel_res_true"] <= 1e-10
    pl.close()
