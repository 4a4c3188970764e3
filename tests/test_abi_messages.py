"""Messages of refused graphs name the refused values."""
import ctypes

import numpy as np
import pytest
import scipy.sparse as sp

from paper_2510_08695_gb300 import _bpdc


def _message(priors, columns=3):
    lib = _bpdc.load()
    H = sp.csr_matrix(np.array([[1, 1, 0], [0, 1, 1]], np.uint8))
    keep = [_bpdc._csr(m) for m in (H, sp.csr_matrix((1, columns), dtype=np.uint8), sp.csr_matrix((0, 3), dtype=np.uint8))]
    pr = np.ascontiguousarray(priors, dtype=np.float64)
    out = ctypes.c_void_p()
    rc = lib.bpdc_graph_create(*[ctypes.byref(k[0]) for k in keep], pr.ctypes.data_as(ctypes.POINTER(ctypes.c_double)),
                               None, 0, ctypes.byref(out))
    return rc, lib.bpdc_last_error().decode()


@pytest.mark.parametrize("at", [0, 1, 2])
def test_refused_prior(at):
    p = [0.1, 0.1, 0.1]
    p[at] = 0.625
    assert _message(p) == (_bpdc.ERR_INVALID_ARG, f"prior {at} = 0.625 outside (0, 1/2]")


def test_refused_columns():
    rc, text = _message([0.1] * 3, columns=4)
    assert rc == _bpdc.ERR_DIM_MISMATCH and text.endswith("(3, 4, 3)")
