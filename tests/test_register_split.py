"""setmaxnreg: the warps of a warpgroup have to meet between two of them, or what each holds is undefined.

Read from the sources: in a role's code a barrier stands between one setmaxnreg and the next, and what the warpgroups give
away and take goes back to the launch's split.
"""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2501_03377_gb300", "csrc")


def _kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        code = re.sub(r"//[^\n]*", "", open(path).read())
        for body in re.split(r"__global__", code)[1:]:
            if "setmaxnreg" in body:
                yield os.path.basename(path), body


def test_a_barrier_between_two_register_splits_of_a_warpgroup():
    seen = 0
    for name, body in _kernels():
        parts = re.split(r"setmaxnreg\.", body)
        seen += len(parts) - 1
        for between in parts[1:-1]:  # from one setmaxnreg to the next
            assert re.search(r"__syncthreads\(\)|bar\.sync|else if \(warp", between), (name, between[:200])
    assert seen >= 4


def test_register_split_is_the_launch_again_at_the_end():
    for name, body in _kernels():
        moves = re.findall(r"setmaxnreg\.(inc|dec)\.sync\.aligned\.u32 (\d+)", body)
        assert sorted(m for m, _ in moves) == ["dec", "dec", "inc", "inc"], name
        low, high = min(int(v) for _, v in moves), max(int(v) for _, v in moves)
        ends = {int(v) for _, v in moves} - {low, high}
        assert len(ends) == 1 and low < min(ends) < high, name
