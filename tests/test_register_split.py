"""setmaxnreg: the warps of a warpgroup have to meet between two of them, or what each holds is undefined.

Read from the sources: between two block barriers a kernel gives registers away in one place and takes them in one, so
that no warpgroup passes two setmaxnreg without a barrier in between; and what its warpgroups hold is never more than the
launch's registers.
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


def test_a_barrier_between_two_register_splits():
    seen = 0
    for name, body in _kernels():
        for segment in body.split("__syncthreads();"):
            moves = re.findall(r"setmaxnreg\.(inc|dec)", segment)
            assert len(moves) == len(set(moves)), (name, moves)
            seen += len(moves)
    assert seen >= 4


def test_register_split_is_the_launch_again_at_the_end():
    for name, body in _kernels():
        moves = re.findall(r"setmaxnreg\.(inc|dec)\.sync\.aligned\.u32 (\d+)", body)
        (give, low), (take, high), (back1, end1), (back2, end2) = moves
        assert (give, take, back1, back2) == ("dec", "inc", "inc", "dec"), name
        assert end1 == end2 and int(low) < int(end1) < int(high), name
