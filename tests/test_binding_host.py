"""CPU: the ctypes binding itself."""
import os
import subprocess
import sys

from paper_2406_12580_gb300 import _lib
from paper_2406_12580_gb300 import build as blr_build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_raw_addresses_need_no_torch():
    """A program that passes addresses and a stream as ints runs where torch is not installed."""
    if blr_build.stale():
        blr_build.build()
    code = f"""
import sys
sys.modules["torch"] = None
import paper_2406_12580_gb300 as P
try:  # validated, and refused for its alignment, before anything reaches a GPU
    P.blr_step(4, 8, P.BLR_F32, 1.0, 8, 16, 16, 16, 16, stream=0)
except P.BLRError as e:
    assert e.status == {_lib.BLR_ERR_INVALID_ARG}
else:
    raise AssertionError
"""
    subprocess.run([sys.executable, "-c", code], check=True, cwd=ROOT)
