"""Kernels that start before the one ahead of them ends promise the compiler nothing about its output."""

import glob
import os
import re

import paper_0807_2387_gb300 as pkg

CSRC = os.path.join(os.path.dirname(os.path.abspath(pkg.__file__)), "csrc")
#: what a plan holds from its creation on, which no kernel of an evaluation writes
CONSTANTS = {"mul", "tw"}


def test_chained_kernels_take_plain_pointers():
    """A kernel that calls wait_previous_kernel is resident while its producer still writes.  A __restrict__
    parameter says that nobody else writes the data during the kernel, so the compiler may read it through
    the non-coherent path or ahead of the wait."""
    seen = []
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        for kernel in re.split(r"\n(?=template|__global__)", open(path).read()):
            head, _, body = kernel.partition("{")
            body = body.split("\n}\n")[0]
            if "__global__" not in head or "wait_previous_kernel();" not in body:
                continue
            seen.append(re.search(r"(\w+)\(", head[head.index("void"):].split("__launch_bounds__(256)")[-1]).group(1))
            assert set(re.findall(r"__restrict__\s+(\w+)", head)) <= CONSTANTS, seen[-1]
            assert not re.search(r"__ldg\((?!mul|tw)", body), seen[-1]
    assert sorted(seen) == ["k_fft_cols", "k_fft_rows_fwd", "k_fft_rows_inv"]
