"""Properties of the CUDA sources that no run can show (CPU)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2207_08393_b200", "csrc")


def test_no_read_only_loads_in_kernels_that_start_early():
    """Every kernel may be scheduled while the launch before it still writes what it will read (griddepcontrol.wait is its
    first statement), and a read-only load promises that the data stay as they are for the kernel's lifetime."""
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cu", ".cuh")):
            continue
        for number, line in enumerate(open(os.path.join(CSRC, name)), 1):
            code = line.split("//")[0]
            assert not re.search(r"__ldg\b|__restrict__|ld\.global\.nc", code), "%s:%d" % (name, number)


def test_a_warp_barrier_stands_before_copies_into_slots_of_other_lanes():
    """Bricks: a lane copies 16 bytes, its own slot and its neighbour's, so the neighbour has to have read its slot before.  A
    shuffle in between orders no memory accesses; only __syncwarp() does."""
    code = [line.split("//")[0] for line in open(os.path.join(CSRC, "dc_brick.cuh"))]
    reads = [i for i, line in enumerate(code) if "u[m] = e[m * W];" in line]
    copies = [i for i, line in enumerate(code) if "cp_async16(e - odd" in line]
    assert len(reads) == len(copies) == 1 and reads[0] < copies[0]
    assert any("__syncwarp();" in line for line in code[reads[0]:copies[0]])
