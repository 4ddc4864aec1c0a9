"""The eigensolver's tiled vector kernels at the edges of their tiles: the FP32
and float-float rotations (one, two and three tiles of 48 columns), the
S-Gram inverse and the small Rayleigh-Ritz problem (FP32 sweeps, and FP64 ones
from a refined FP32 result) at odd and large numbers of roots, and the float-float kernel's element and column remainders.

Tolerances: eigenvalues 1e-6 Ha of the dense FP64 ones as in
test_gpu_eigsolve.py (residual 1e-6 and an error of its square over the gap);
a float-float rotation sums 4 ma products of 48 bits, so its error stays below
4 ma 2^-48 of sum |a||y| (1.6e-12 for ma = 112)."""
import ctypes
import dataclasses

import numpy as np
import pytest

from oracle import eigen as E
from oracle import hamiltonian as Hm
from paper_1406_4960_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mbmod():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1406_4960_gb300 import mb
    mb.load(build_if_missing=True)
    return mb


@pytest.fixture(scope="module")
def dense():
    w = W.tiny()
    mod = Hm.model_from_workload(w, 0)
    return E.generalized_lowest(mod.dense_H(), mod.dense_S(), 95)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("nroots", [9, 43, 85, 86, 95])
def test_roots_at_the_tile_edges(mbmod, dense, nroots, prec):
    w = dataclasses.replace(W.tiny(), nbands=nroots, name=f"tiny-{nroots}")
    h = mbmod.Handle.from_workload(w)
    ev, info = h.eigsolve(nroots, 1e-6, prec)
    assert info.max_residual < 1e-6
    assert np.abs(ev[0] - dense[:nroots]).max() < 1e-6
    h.close()


@pytest.mark.parametrize("ma,mc,n", [(8, 48, 64), (9, 49, 65), (112, 97, 127), (17, 112, 63), (7, 1, 1)])
def test_float_float_rotation_edges(mbmod, ma, mc, n):
    lib = mbmod.load()
    lib.mb_debug_combine_ff.argtypes = [ctypes.c_void_p, ctypes.POINTER(ctypes.c_double), ctypes.c_longlong, ctypes.c_int,
                                        ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p]
    rng = np.random.default_rng(ma + 131 * mc)
    A = rng.standard_normal((ma, n)) + 1j * rng.standard_normal((ma, n))
    Y = rng.standard_normal((ma, mc)) + 1j * rng.standard_normal((ma, mc))
    Ad = torch.from_numpy(A).cuda()
    Cd = torch.full((mc, n), complex(np.nan, np.nan), dtype=torch.complex128, device="cuda")
    rc = lib.mb_debug_combine_ff(Ad.data_ptr(), np.ascontiguousarray(Y).view(np.float64).ctypes.data_as(
        ctypes.POINTER(ctypes.c_double)), n, ma, mc, Cd.data_ptr(), None)
    assert rc == 0
    bound = 4 * ma * 2.0**-48 * (np.abs(Y).T @ np.abs(A))
    assert np.all(np.abs(Cd.cpu().numpy() - Y.T @ A) <= bound)
