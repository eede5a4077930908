"""The scan's and the radix sort's ways out of an unanswered look back (-m gpu): the library
linked with a sort.cu that allows no polls, so that a tile which finds a predecessor's word
unknown forms its prefix itself.  Scans in place (a matrix's row pointers) and out of place,
sums of 32 and 64 bits, sorts of keys alone and with values."""
import glob
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
LIMIT = "constexpr uint32_t kLookLimit = 1u << 18;"

_RUN = """
import sys
import paper_2303_05688_gb300 as asci
asci._LIB_PATH = sys.argv[1]
import torch
from tests import test_gpu_scan as scan, test_gpu_sort as sort
for n in (4097, 131_073, 300_001):
    for repeat in (1, 2, 5000):
        scan.test_run_positions(torch, n, repeat)
for nd in (4096, 8193, 20_000):
    scan.test_row_pointers(torch, nd)
for n in (4097, 8193, 100_003, 300_001):
    for kind in ("wide", "one digit", "two values", "sorted", "reversed"):
        sort.test_sort_over_tiles(n, kind)
maps = open("/proc/self/maps").read()
assert sys.argv[1] in maps and "lib/libasci.so" not in maps
print("AGREE")
"""


def test_tiles_that_get_no_answer(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_05688_gb300 import build
    build.build()
    text = open(os.path.join(build.CSRC, "sort.cu")).read()
    assert text.count(LIMIT) == 1
    (tmp_path / "sort.cu").write_text(text.replace(LIMIT, "constexpr uint32_t kLookLimit = 0u;"))
    obj, lib = str(tmp_path / "sort.o"), str(tmp_path / "libasci_lost.so")
    subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-c",
                    str(tmp_path / "sort.cu"), "-o", obj], check=True, capture_output=True)
    objs = [o for o in glob.glob(os.path.join(build.OBJ, "*.o")) if not o.endswith("/sort.o")]
    subprocess.run([build._nvcc(), *build.ARCH, "-shared", "-o", lib, obj, *objs, "-lpthread"],
                   check=True, capture_output=True)
    r = subprocess.run([sys.executable, "-c", _RUN, lib], cwd=ROOT, capture_output=True, text=True,
                       env=dict(os.environ, PYTHONPATH=ROOT), timeout=600)
    assert r.returncode == 0 and "AGREE" in r.stdout, r.stderr[-2000:]
