"""Building a handle where the host has no more threads or memory, or for a
matrix with an empty row: a status, not the end of the process.  Each in a
process of its own, the first under an address-space limit in which no thread's
stack fits; without a GPU the build ends at its first CUDA call, behind the
host's work."""
import subprocess
import sys

import pytest

from conftest import ROOT

PROGRAM = """
import resource, sys
import numpy as np
from paper_2605_14170_gb300 import mbbp
from paper_2605_14170_gb300.inputs import named_code
code, R, room = sys.argv[1], int(sys.argv[2]), int(sys.argv[3])
H = np.ascontiguousarray(named_code(code).HZ, np.uint8)

def build(H=H, R=R):
    try:
        mbbp.mbbp_build_bases(H, R, 1)
        return 0
    except mbbp.MBBPError as e:
        return e.status

first = build(named_code("bb72").HZ, 1)
size = int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()
resource.setrlimit(resource.RLIMIT_AS, (size + room, resource.RLIM_INFINITY))
second = build()
resource.setrlimit(resource.RLIMIT_AS, (resource.RLIM_INFINITY, resource.RLIM_INFINITY))
print(first, second, build())
"""


def _run(code, R, room):
    r = subprocess.run([sys.executable, "-c", PROGRAM, code, str(R), str(room)], cwd=ROOT, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    return [int(x) for x in r.stdout.split()]


def test_build_without_further_threads():
    """No thread can start (1 MB more for the heap): the calling one does the
    work, with the result of an unlimited build."""
    first, second, third = _run("bb72", 8, 1 << 20)
    assert first == second == third


@pytest.mark.parametrize("code,R", [("gb882", 64)])
def test_build_without_memory(code, R):
    """No memory for the tables: MBBP_E_NOMEM, and the next build succeeds as
    far as the first did."""
    first, second, third = _run(code, R, 0)
    assert second == 5 and third == first


def test_build_with_an_empty_row():
    """A row of H without entries (a small code: its layout search swaps the
    edges of a row)."""
    program = PROGRAM.split("first =")[0] + "H[5] = 0\nprint(build(), build(named_code('bb72').HZ, 4))"
    r = subprocess.run([sys.executable, "-c", program, "bb72", "4", "0"], cwd=ROOT, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, (r.returncode, r.stderr[-2000:])
    with_empty, without = (int(x) for x in r.stdout.split())
    assert with_empty == without
