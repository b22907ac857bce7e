"""A host without memory is an error code, not an exception that leaves the C interface.  No GPU work."""
import subprocess
import sys

from tests.conftest import ROOT

PROGRAM = """
import ctypes, resource, sys
sys.path.insert(0, sys.argv[1])
import numpy as np
from paper_2503_09357_b200 import binding as pe
desc, keep = pe.make_desc(num_ops=40_000_000, edge_src=np.zeros(0, np.int32), edge_dst=np.zeros(0, np.int32),
                          dur=np.ones(40_000_000, np.int32), num_devices=2)
with open("/proc/self/statm") as f:
    used = int(f.read().split()[0]) * resource.getpagesize()
resource.setrlimit(resource.RLIMIT_AS, (used + (64 << 20), resource.RLIM_INFINITY))   # the scratch arrays take 160 MB each
handle = ctypes.c_void_p(1)
print(pe._lib.pe_graph_validate(ctypes.byref(desc)), pe._lib.pe_graph_create(ctypes.byref(desc), 0, ctypes.byref(handle)), handle.value)
"""


def test_no_memory_is_an_error_code():
    from paper_2503_09357_b200.build import build_libpe
    build_libpe()
    run = subprocess.run([sys.executable, "-c", PROGRAM, ROOT], capture_output=True, text=True, timeout=120)
    assert run.returncode == 0, run.stderr[-500:]
    assert run.stdout.split() == ["-5", "-5", "None"]
