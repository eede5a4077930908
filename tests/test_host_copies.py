"""Copies from host variables: CUDA may read the source after the call has returned, so a
value set by the host goes to the device as a kernel argument, and a copy's source is an
array that lives until the next wait."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2303_05688_gb300", "csrc")


def test_no_copy_to_the_device_from_a_scalar_on_the_stack():
    copies = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"cudaMemcpyAsync\(([^;]*?),\s*(cudaMemcpy\w+)\s*,", text, re.S):
            copies += 1
            dst, src = m.group(1).split(",")[:2]
            if m.group(2) == "cudaMemcpyHostToDevice":
                assert not src.strip().startswith("&"), (os.path.basename(path), m.group(0))
    assert copies > 20
