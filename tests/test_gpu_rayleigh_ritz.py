"""The eigensolver's FP64 Rayleigh-Ritz problems: orthonormality and values to
FP64, whatever precision the sweeps start in.

Tolerances (u = 2^-53, m columns), first-order bounds of the rounding alone: the
vectors are m-term sums (m u), orthonormalized through m-term products (m u),
then turned by at most six sweeps of m - 1 rotations (8 u each, 48 m u): 50 m u
of orthonormality.  Values and residuals: the sweeps stop at 1e-13 of the
matrix's Frobenius norm, and its projection is two m-term products with vectors
orthonormal to the above: (1e-13 + 100 m u) of the norm.  The returned bands:
sums of nb ng products through S of condition below 1e3 (2e-11 in FP64, and
1e-10 with the float-float rotations, as in test_gpu_eigsolve.py)."""
import ctypes

import numpy as np
import pytest

from paper_1406_4960_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U = 2.0**-53


@pytest.fixture(scope="module")
def handle():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1406_4960_gb300 import mb
    mb.load(build_if_missing=True)
    h = mb.Handle.from_workload(W.tiny())
    yield h
    h.close()


def _unitary(rng, m):
    return np.linalg.qr(rng.standard_normal((m, m)) + 1j * rng.standard_normal((m, m)))[0]


def matrix(kind, m):
    rng = np.random.default_rng(m)
    if kind == "couplings":
        # nothing for FP32 sweeps to do (off-diagonal norm 9e-7 of the matrix's),
        # and a cluster whose couplings are all 1e-4 of their gaps: the largest
        # first corrections that the refinement makes, added up in phase
        r = np.arange(m - 1.0)
        gap = np.abs(r[:, None] - r[None])
        w = 9e-7 / (1e-4 * np.linalg.norm(gap))
        A = np.zeros((m, m), dtype=complex)
        A[0, 0] = 1.0
        A[1:, 1:] = w * (np.diag(r) + 0.99e-4 * gap)
        ph = np.exp(2j * np.pi * rng.random(m))
        return ph[:, None] * A * ph.conj()[None]
    if kind == "multiple":            # roots of multiplicity 1 to 4, and pairs 1e-9 apart
        e = np.repeat(np.arange(m) * 0.1, 1 + np.arange(m) % 4)[:m] + 1e-9 * (np.arange(m) % 2)
    elif kind == "wide":              # 1e-3 to 1e3
        e = np.geomspace(1e-3, 1e3, m)
    else:
        e = rng.standard_normal(m)
    Q = _unitary(rng, m)
    A = (Q * e) @ Q.conj().T
    return 0.5 * (A + A.conj().T)


def rayleigh_ritz(h, A, refined=1):
    n, m = A.shape[:2]
    A = np.ascontiguousarray(A, dtype=np.complex128)
    ev, Y = np.zeros((n, m)), np.zeros((n, m, m), dtype=np.complex128)
    dp = ctypes.POINTER(ctypes.c_double)
    f = h._lib.mb_debug_rayleigh_ritz
    f.argtypes = [ctypes.c_void_p, dp, ctypes.c_int, ctypes.c_int, ctypes.c_int, dp, dp]
    rc = f(h._h, A.view(np.float64).ctypes.data_as(dp), m, n, refined, ev.ctypes.data_as(dp),
           Y.view(np.float64).ctypes.data_as(dp))
    assert rc == 0
    return ev, Y


@pytest.mark.parametrize("m", [2, 6, 15, 16, 17, 41, 64, 65, 95, 112])
@pytest.mark.parametrize("kind", ["couplings", "multiple", "wide", "normal"])
def test_eigenpairs_to_fp64(handle, kind, m):
    if kind == "couplings" and m < 3:
        pytest.skip("a cluster has at least two roots")
    A = np.stack([matrix(kind, m), 2.0 * matrix(kind, m).conj()])
    ev, Y = rayleigh_ritz(handle, A)
    for a, e, y in zip(A, ev, Y):
        assert np.abs(y.conj().T @ y - np.eye(m)).max() < 50 * m * U
        tol = (1e-13 + 100 * m * U) * np.linalg.norm(a)
        assert np.abs(e - np.linalg.eigvalsh(a)).max() < tol
        assert np.abs(a @ y - y * e).max() < tol


@pytest.mark.parametrize("prec,tol", [("fp64", 2e-11), ("fp32", 1e-10)])
@pytest.mark.parametrize("nroots", [8, 52, 85])
def test_bands_are_s_orthonormal(handle, nroots, prec, tol):
    """Subspaces of 10 and 15, 59 and 64, 96 and 101 vectors; the square cell's
    Gamma point has double roots."""
    ng, nb, ldg = handle.sizes(0)
    V = torch.zeros(nroots, nb, ldg, dtype=torch.complex128, device="cuda")
    handle.eigsolve(nroots, 1e-6, prec, evecs=V)
    SV = torch.empty_like(V)
    handle.apply_S(0, V, SV, "fp64")
    G = V.reshape(nroots, -1).conj() @ SV.reshape(nroots, -1).T
    assert (G - torch.eye(nroots, dtype=G.dtype, device="cuda")).abs().max().item() < tol


@pytest.mark.parametrize("n,m", [(76, 112), (77, 112), (305, 56), (305, 57)])
def test_many_problems(handle, n, m):
    """The most that the refinement's workspace holds (max(304, n) 112^2 numbers
    for four matrices a problem), and one more, which takes FP64 sweeps."""
    A = np.stack([(1 + 0.01 * p) * matrix("normal", m) for p in range(n)])
    ev, Y = rayleigh_ritz(handle, A)
    G = Y.conj().transpose(0, 2, 1) @ Y
    assert np.abs(G - np.eye(m)).max() < 50 * m * U
    tol = (1e-13 + 100 * m * U) * np.linalg.norm(A[-1])
    assert np.abs(A @ Y - Y * ev[:, None, :]).max() < tol
