"""The X-pass probe takes fewer rows than a box has only where the pass itself takes
a row count: the register X pass of the other sizes always runs N*N rows, past the
end of buffers sized for fewer.  Checked on the host, before anything is launched."""
import ctypes as ct
import os

import pytest

from paper_2012_04838_gb300 import binding as B
from paper_2012_04838_gb300 import build


@pytest.fixture(scope="module")
def lib():
    if not os.path.exists(B.lib_path()):
        build.build()
    return B.load()


@pytest.mark.parametrize("prec", [B.FP32_MIXED, B.FP64])
@pytest.mark.parametrize("N", [8, 16, 24, 32, 48, 64, 96, 128, 192, 256, 512, 1024])
def test_rows_the_probe_takes(lib, N, prec):
    n = ct.c_size_t(0)

    def nbytes(rows):
        return lib.psc_xpass_probe_bytes(N, prec, rows, ct.byref(n))

    assert nbytes(N * N) == B.PSC_OK
    # nine input and four output streams of N*N rows fit the buffer
    assert n.value >= 13 * N * N * ((N - 1) // 3 + 1) * (16 if prec == B.FP64 else 8)
    counts = N >= 512 or (N == 256 and prec == B.FP32_MIXED)
    for rows in {64, N * N // 128 * 64, N * N - 64}:
        if 0 < rows < N * N:
            assert nbytes(rows) == (B.PSC_OK if counts else B.PSC_EINVAL), rows
            if not counts:  # the launch itself refuses too (the buffer is never looked at)
                assert lib.psc_xpass_probe(N, prec, rows, ct.c_void_p(256), 1 << 40, None, 1) == B.PSC_EINVAL
