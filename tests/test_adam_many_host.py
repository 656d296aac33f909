"""vlb_adam_step_many checks its tensors before it sets aside anything of the size of the list, and lets no C++ exception
through the C entry: with the address space limited, a list that claims 2^31 - 33 tensors, the first of them
invalid, is refused like any other."""
import subprocess
import sys

CODE = """
import ctypes, os, resource, sys
sys.path.insert(0, os.getcwd())
from paper_1904_10070_gb300 import vlb
L = vlb.lib()
resource.setrlimit(resource.RLIMIT_AS, (8 << 30, 8 << 30))
one = (ctypes.c_void_p * 1)(1)
n = (ctypes.c_int64 * 1)(0)
f = ctypes.c_float
st = L.vlb_adam_step_many(2**31 - 33, n, one, one, one, one, 1, f(1e-3), f(0.9), f(0.999), f(1e-8), None, None)
assert st == vlb.VLB_ERR_ARG, st
"""


def test_a_long_list_is_refused_without_an_exception():
    res = subprocess.run([sys.executable, "-c", CODE], capture_output=True, text=True, timeout=300)
    assert res.returncode == 0, (res.returncode, res.stderr[-500:])
