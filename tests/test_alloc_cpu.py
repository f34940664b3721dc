"""A host allocation that fails inside a C entry is reported as LHE_ERR_OOM; the exception does not cross the C boundary (which would
end the process, so the call runs in one of its own)."""
import subprocess
import sys

from paper_2410_13165_gb300 import _abi, build


def test_a_map_too_large_for_the_host_is_an_error():
    build.build()
    # 2^40 velocities of D4Q33, one Fourier variable each: 300 TB of weights, more than the address space holds
    code = """
import ctypes
from paper_2410_13165_gb300 import _abi
lib = _abi.load()
p = _abi.lhe_lbm_default_params()
p.d = 4
x = (ctypes.c_double * 4)()
a = ctypes.addressof(x)
print(lib.lhe_lbm_stability_map(ctypes.byref(p), a, 1 << 40, 1, a, a))
"""
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.returncode, r.stderr[-500:])
    assert int(r.stdout.split()[-1]) == _abi.ERR_OOM
