"""Building a handle where the host has no more threads or memory: a status,
not the end of the process.  Run in a process of its own under an address-space
limit, in which no thread's stack fits; without a GPU the build ends at its
first CUDA call, behind the host's work."""
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
