"""The lines that the library finds on the device are those of the host rule
(`paper_1810_08572_gb300/csrc/lines_host.h`), cell by cell: columns, columns cut
at 512 cells, rings, chains and rings longer than the pointer doubling's usual
rounds reach, and couplings without a direction."""
import ctypes as C
import os

import numpy as np
import pytest

from tests.test_line_layout import check_layout, grid_operator, layout, lines_of, shim  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fvs():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1810_08572_gb300 import LIB_PATH, build
    if not os.path.exists(LIB_PATH):
        build()
    from paper_1810_08572_gb300 import fvs as f
    return f


def device_layout(fvs, col, val, n, w):
    sizes = np.zeros(4, np.int64)
    ptr = lambda a: a.ctypes.data_as(C.c_void_p)
    fvs.check(fvs.fvs_line_layout(ptr(col), ptr(val), n, w, ptr(sizes), 0, 0, None, None, None, None, None), "sizes")
    nlines, ngroups, padded, max_len = (int(v) for v in sizes)
    out = dict(nlines=nlines, ngroups=ngroups, padded=padded, max_len=max_len, goff=np.zeros(ngroups + 1, np.int64),
               llen=np.zeros(ngroups * 32, np.int32), cell=np.zeros(padded, np.int32),
               sprev=np.zeros(padded, np.int8), snext=np.zeros(padded, np.int8))
    fvs.check(fvs.fvs_line_layout(ptr(col), ptr(val), n, w, ptr(sizes), ngroups, padded, ptr(out["goff"]),
                                  ptr(out["llen"]), ptr(out["cell"]), ptr(out["sprev"]), ptr(out["snext"])), "layout")
    return out


def sequences(L):
    out = {}
    for _, idx in lines_of(L):
        if len(idx):
            out[int(L["cell"][idx[0]])] = (L["cell"][idx].tolist(), L["sprev"][idx].tolist(), L["snext"][idx].tolist())
    return out


@pytest.mark.parametrize("shape,cz,periodic", [
    ((1, 1, 1), 20.0, False), ((1, 1, 2), 20.0, False), ((5, 7, 12), 20.0, False), ((3, 3, 1030), 20.0, False),
    ((6, 6, 6), 1.15, False), ((17, 19, 33), 1.0, False),
    ((3, 4, 9), 20.0, True), ((2, 3, 600), 20.0, True),
    ((2, 1, 4096), 20.0, False), ((2, 1, 4097), 20.0, False), ((1, 1, 9001), 20.0, False),
    ((1, 2, 4096), 20.0, True), ((1, 1, 5000), 20.0, True)])
def test_lines_found_on_the_device_are_those_of_the_host_rule(fvs, shim, shape, cz, periodic):  # noqa: F811
    col, val, _, _ = grid_operator(*shape, cz=cz, seed=3, periodic_z=periodic)
    n = int(np.prod(shape))
    D = device_layout(fvs, col, val, n, 7)
    H = layout(shim, col, val, n, 7, 512)
    check_layout(D, col, n, 7)
    assert (D["nlines"], D["ngroups"], D["padded"], D["max_len"]) == (H["nlines"], H["ngroups"], H["padded"], H["max_len"])
    assert (D["llen"] == H["llen"]).all() and (D["goff"] == H["goff"]).all()
    assert sequences(D) == sequences(H)


def test_layout_call_refuses_columns_outside_the_rows(fvs):
    sizes = np.zeros(4, np.int64)
    col = np.array([0, 1, 1, 2], np.int32)
    val = np.ones(4)
    ptr = lambda a: a.ctypes.data_as(C.c_void_p)
    for args in ((ptr(col), ptr(val), 2, 2), (None, ptr(val), 2, 2), (ptr(col), ptr(val), 0, 2), (ptr(col), ptr(val), 2, 128)):
        assert fvs.fvs_line_layout(*args, ptr(sizes), 0, 0, None, None, None, None, None) == fvs.FVS_ERR_ARG
        assert fvs.fvs_last_error().startswith("fvs_line_layout")
