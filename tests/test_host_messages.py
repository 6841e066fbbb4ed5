"""Every bounded wait on the device that runs out has a message of its own: the solves of the
inverse form do not report the tensor-memory-accelerator stage of the block Cholesky's solve
kernel 4, which did not run (the kernels' codes are checked in their source)."""
import ctypes as C
import os
import re

import pytest

from tests.host import hostcheck


def test_stage_error_messages():
    try:
        lib = hostcheck.lib()
    except RuntimeError as err:
        pytest.skip(str(err))
    lib.hc_stage_error_text.restype = C.c_char_p
    text = {e: lib.hc_stage_error_text(e).decode() for e in (1, 2, 3)}
    assert "tensor-memory-accelerator" in text[1] and "persistent" in text[2] and "inverse Schur" in text[3]
    src = open(os.path.join(hostcheck.CSRC, "k_inv.cu")).read()
    assert set(re.findall(r"atomicExch\(a\.err, (\w+)\)", src)) == {"KERR_SOLVE_COPY"}
