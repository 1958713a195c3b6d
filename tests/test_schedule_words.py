"""The schedule fixes the order of every row's entries, and with it the bits of
every product: its words for a set of patterns are pinned by a digest."""
import ctypes
import hashlib

import numpy as np
import pytest

import synth

# SHA-256 over lane counts 1 to 32 (at most 16 rows per lane) of {entry, word} per slot
# (its first 16 digits)
DIGEST = {(9, 14): "77f1dc4638b747e7", (40, 90): "bd82d144a74ac3fc", (80, 200): "0aa0a985206fe6a8",
          (81, 640): "6037fb1b47739eb7", (150, 400): "16714d8ed4c9c0d6"}


@pytest.mark.parametrize("n,R", list(DIGEST))
def test_schedule_words_are_pinned(n, R):
    from paper_2405_17363_gb300 import build
    f = ctypes.CDLL(build.build()).camp_schedule_build
    f.restype = ctypes.c_int
    f.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int,
                  ctypes.c_void_p, ctypes.c_int, ctypes.POINTER(ctypes.c_int)]
    m = synth.make_mechanism(n, R, 900 + n)
    rp, ci = (np.ascontiguousarray(v, np.int32) for v in (m.row_ptr, m.col_idx))
    h = hashlib.sha256()
    for lc in (1, 2, 4, 8, 16, 32):
        if (n + lc - 1) // lc > 16:
            continue
        L = ctypes.c_int()
        words = np.zeros(2 * 65536, "<u4")
        assert f(n, m.nnz, rp.ctypes.data, ci.ctypes.data, lc, words.ctypes.data, 65536,
                 ctypes.byref(L)) == 0
        h.update(words[:2 * L.value * lc].tobytes())
    assert h.hexdigest()[:16] == DIGEST[n, R]
