"""Orders within kernels on which progress depends and which a run does not show: read from the sources."""
import glob
import os
import re

import pytest

from paper_2506_18145_b200 import build as rbuild


def kernels(path):
    """Bodies of a file's kernels, without comments."""
    with open(path) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    starts = [m.start() for m in re.finditer(r"__global__", text)] + [len(text)]
    return [text[a:b] for a, b in zip(starts, starts[1:])]


# A kernel's successor may allocate tensor memory before it waits.  Let in ahead of the kernel's own allocation it could take the columns of
# an SM and wait for blocks that wait for them.  (The single-token step's In Proj lets in first: what follows it holds no tensor memory.)
@pytest.mark.parametrize("path", [p for p in sorted(glob.glob(os.path.join(rbuild.CSRC, "*.cu"))) if os.path.basename(p) != "rom_step.cu"],
                         ids=os.path.basename)
def test_tensor_memory_is_allocated_before_the_successor_comes_in(path):
    for body in kernels(path):
        alloc = body.find("tcgen05.alloc")
        let_in = re.search(r"pdl_trigger\(\)|pdl_sync\(\)", body)
        if alloc >= 0 and let_in:
            assert alloc < let_in.start()


# bar.sync, bar.arrive and the tensor-memory instructions (all of the .aligned kind) take a whole warp, converged: after a branch by lane the
# warp is brought together by name.
@pytest.mark.parametrize("before,after", [
    (r"cur_z\.load", r"bar_sync\(warp\)"),                    # gate rows and the next tile's operands, up to the hand-over
    (r"fetch_rows\(t0\)", r"tm_store16\("),                   # rows' indices, up to the first sweep
    (r"V16<bf16>::store", r"tcgen05\.dealloc"),               # outputs of the last step, up to the end
])
def test_lanes_of_the_one_launch_scan_meet_before_aligned_instructions(before, after):
    body, = kernels(os.path.join(rbuild.CSRC, "rom_scan_ring.cu"))
    for m in re.finditer(before, body):
        end = re.search(after, body[m.end():])
        if end:
            assert "__syncwarp();" in body[m.end():m.end() + end.start()]
