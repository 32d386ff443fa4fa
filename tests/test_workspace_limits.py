"""Contractions of a few large rows off 16-byte boundaries stay within the
fixed scratch of tvc_noalloc."""
import ctypes as C

import pytest

import paper_2501_03121_gb300 as tg


@pytest.mark.parametrize("dims, mode", [((2680, 212, 1690), 1), ((1, 395, 2313733, 2), 1), ((147, 1, 97, 1, 1005, 47), 0)])
def test_ragged_columns_fit_the_fixed_scratch(dims, mode):
    lib = tg.load_library()
    lib.tvc_workspace_size.restype = C.c_size_t
    for dtype in range(6):
        need = lib.tvc_workspace_size(len(dims), (C.c_int64 * len(dims))(*dims), mode, dtype)
        assert need <= 32 << 20
