"""No two CTAs that allocate TMEM fit one SM.

tcgen05.alloc waits without a limit, and a pass launched early holds its columns while it waits for the pass before it,
so the exclusion must not rest on register counts: every tensor-core launch asks for more than half of an SM's shared
memory.  The sizes are read from a captured application (grid, block and dynamic shared memory of each kernel).
"""
import re

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SM_SHARED = 228 * 1024
RESERVED = 1024  # the system's share of every CTA


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_03377_gb300 import build

    build.build()


@pytest.mark.filterwarnings("ignore:DEBUG")
@pytest.mark.parametrize("prec", ["fp64", "bf16", "fp16", "tf32", "bf16x3"])
@pytest.mark.parametrize("shape", [(16, 3, 3), (64, 64, 32), (64, 48, 1), (37, 21, 9), (128, 64, 130), (256, 256, 5)])
def test_tensor_core_launches_fill_half_an_sm(shape, prec, tmp_path):
    from paper_2501_03377_gb300 import Plan, binding

    nx, ny, nz = shape
    stream = torch.cuda.Stream()
    pl = Plan(nx, ny, nz, ("P", "D", "N"), prec=prec, stream=stream.cuda_stream)
    r = torch.ones((nz, ny, nx), dtype=torch.float64, device="cuda")
    z = torch.empty_like(r)
    torch.cuda.synchronize()
    for slices, fuse in ((1, 1), (1, 0), (0, 1), (0, 0)):
        pl.set_option(binding.TPCG_OPT_SLICES, slices)
        pl.set_option(binding.TPCG_OPT_FUSE_G, fuse)
        graph = torch.cuda.CUDAGraph(keep_graph=True)
        graph.enable_debug_mode()
        with torch.cuda.graph(graph, stream=stream):
            pl.precond(r, z)
        dot = tmp_path / f"{slices}{fuse}.dot"
        graph.debug_dump(str(dot))
        kernels = re.findall(r"\| (\w+)\\<\\<\\<(\d+),(\d+),(\d+)\\>\\>\\>", dot.read_text())
        tensor = [(name, int(smem)) for name, _, _, smem in kernels
                  if re.search(r"k_(modeprod_tc|modeprod_pair|modeprod_oz|frontal_pair|tube_pair)", name)]
        assert len(tensor) >= 3, kernels
        for name, smem in tensor:
            assert 2 * (smem + RESERVED) > SM_SHARED, (name, smem)
    pl.close()
