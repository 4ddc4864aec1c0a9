"""The admission limit of mb_apply_H_noalloc: requests whose scratch fits the
array run, whatever launch shape was selected, and one run boundary of rows
counts on row-space grids as documented."""
import ctypes

import numpy as np
import pytest

from paper_1406_4960_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# bands of the 1417-G graphene cell: 80 FP32 ones count 9.2 MB of boundary rows
# and 1.8 MB of overlaps, in FP64 twice that
@pytest.mark.parametrize("prec,nbands,n_int,rc", [
    ("fp32", 80, 77, 0), ("fp32", 1, 77, 0), ("fp64", 80, 77, 1), ("fp64", 56, 77, 0),
    ("fp64", 80, 17, 0),         # too few intervals for three runs: the overlaps alone, 3.7 MB
])
@pytest.mark.parametrize("waves", [0, 1, 8])
def test_admission(prec, nbands, n_int, rc, waves):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1406_4960_gb300 import mb
    lib = mb.load(build_if_missing=True)
    w = W.scaled(W.graphene(), n_int=n_int)
    h = mb.Handle.from_workload(w)
    ng, nb, ldg = h.sizes(0)
    h.plane_kernel_select(1, nbands, prec, -1, waves)
    dt = torch.complex128 if prec == "fp64" else torch.complex64
    g = torch.Generator(device="cuda").manual_seed(2)
    X = torch.randn(nbands, nb, ldg, dtype=dt, device="cuda", generator=g)
    X[:, :, ng:] = 0
    Y = torch.full_like(X, complex(np.nan, np.nan))
    assert lib.mb_apply_H_noalloc(h._h, 0, ctypes.c_void_p(X.data_ptr()), ctypes.c_void_p(Y.data_ptr()), nbands,
                                  mb.PREC[prec], None) == rc
    if rc == 0:
        ref = torch.empty_like(X)
        h.apply_H(0, X, ref, prec)
        torch.cuda.synchronize()
        assert torch.equal(Y, ref)           # the same launches, fixed summation orders
    h.close()
