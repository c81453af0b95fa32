"""Errors for the status bits that kernels set, as pm_check and pm_decompress_noalloc
return them: each bit alone is an error, the first cause wins, no bit is none."""
import ctypes
import subprocess

from paper_1611_01545_gb300 import _lib
from paper_1611_01545_gb300 import build as b

CORRUPT, OVERFLOW, RANGE, TIMEOUT = 1, 2, 4, 8


def test_status_codes(tmp_path):
    src, so = tmp_path / "status.cpp", tmp_path / "status.so"
    src.write_text('#include "status.h"\nextern "C" int status_error(int bits) { return pm::status_error(bits); }\n')
    subprocess.run(["g++", "-shared", "-fPIC", "-I", b.INCLUDE, "-I", b.CSRC, "-o", str(so), str(src)], check=True)
    error = ctypes.CDLL(str(so)).status_error
    assert error(0) == _lib.PM_OK
    assert error(TIMEOUT) == _lib.PM_ERR_TIMEOUT
    assert error(CORRUPT) == _lib.PM_ERR_CORRUPT
    assert error(OVERFLOW) == _lib.PM_ERR_OVERFLOW
    assert error(RANGE) == _lib.PM_ERR_RANGE
    assert error(CORRUPT | TIMEOUT) == _lib.PM_ERR_CORRUPT
    assert error(RANGE | CORRUPT) == _lib.PM_ERR_RANGE
    assert error(OVERFLOW | CORRUPT) == _lib.PM_ERR_OVERFLOW
