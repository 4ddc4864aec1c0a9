"""The row-space kernel of the H apply on every grid shape it is compiled for,
at its edges: discs that fill more than 3/4 of a side (the unpruned planes),
sides of 64 points whose disc folds onto itself, runs of one row up to the
whole basis, steps that end inside and past the basis, and k-points with
different discs in one batch, against the FP64 oracle.

Tolerances as in test_gpu_apply.py: 1e-10 (FP64) and 2e-5 (FP32) of max |Y|,
and for the row-space density that of test_gpu_scf.py, 1e-11 of its maximum."""
import dataclasses

import numpy as np
import pytest

from oracle import hamiltonian as Hm
from oracle import scf as F
from paper_1406_4960_gb300 import workloads as W

from gpu_util import gmap, lib_block, oracle_block, rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-10, "fp32": 2e-5}

# grid, cell sides (bohr), cutoff (Ha)
GRIDS = {
    "16x16-full": ((16, 16), (4.7, 4.7), 42.0),
    "16x32": ((16, 32), (4.7, 9.4), 12.0),
    "16x32-full": ((16, 32), (4.7, 9.4), 42.0),
    "32x16-full": ((32, 16), (9.4, 4.7), 42.0),
    "32x32-full": ((32, 32), (9.4, 9.4), 36.0),
    "64x16-fold": ((64, 16), (26.0, 4.7), 12.0),
    "16x64-fold": ((16, 64), (4.7, 26.0), 12.0),
    "64x32-fold": ((64, 32), (26.0, 9.4), 8.0),
    "32x64-fold": ((32, 64), (9.4, 26.0), 8.0),
    "64x64-fold": ((64, 64), (26.0, 26.0), 9.0),
}


@pytest.fixture(scope="module")
def mbmod():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1406_4960_gb300 import mb
    mb.load(build_if_missing=True)
    return mb


def _workload(grid, sides, ecut, n_int, nbands):
    w = W.tiny()
    atoms = [W.Atom((0.3 * sides[0], 0.6 * sides[1], 0.8), -2.0, 1.0),
             W.Atom((0.7 * sides[0], 0.1 * sides[1], -1.1), -1.5, 0.9, 4, W.KB_E, W.KB_RC)]
    k = np.array([[0.0, 0.0], [0.11, -0.07]])
    return dataclasses.replace(w, a1=(sides[0], 0.0), a2=(0.0, sides[1]), ecut=ecut, grid=grid, atoms=atoms, kpts=k,
                               breaks=W.uniform_breaks(-4.0, 4.0, n_int), nbands=nbands, name="rowspace")


def _check(mbmod, w, prec, waves=(0,), kernel="rowspace_"):
    h = mbmod.Handle.from_workload(w)
    cdt = np.complex128 if prec == "fp64" else np.complex64
    Xs, perms, refs = [], [], []
    for ik in range(w.nk):
        ng, nb, ldg = h.sizes(ik)
        m = Hm.model_from_workload(w, ik)
        perms.append(gmap(h, m, ik))
        X = W.random_block(w.nbands, nb, ng, seed=70 + ik)
        refs.append(m.apply_H(X))
        Xs.append(torch.from_numpy(lib_block(X, perms[ik], ldg, cdt)).cuda())
    for wv in waves:
        h.plane_kernel_select(w.nk, w.nbands, prec, -1, wv)
        assert h.plane_kernel_name(w.nk, w.nbands, prec).startswith(kernel)
        Ys = [torch.full_like(x, complex(np.nan, np.nan)) for x in Xs]
        h.apply_H_batch(list(range(w.nk)), Xs, Ys, prec)
        torch.cuda.synchronize()
        for ik in range(w.nk):
            Yh = Ys[ik].cpu().numpy()
            assert np.all(Yh[:, :, len(perms[ik]):] == 0)
            err = rel_err(oracle_block(Yh, perms[ik]), refs[ik])
            assert err < TOL[prec], (wv, ik, err)
    h.close()


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("case", list(GRIDS))
def test_every_grid_shape(mbmod, case, prec):
    # 12 splines: runs of a few rows (waves 0) and of a single row (waves 8)
    _check(mbmod, _workload(*GRIDS[case], n_int=9, nbands=3), prec, waves=(0, 8))


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("n_int", [6, 8, 13, 14, 24, 29, 30])
def test_run_lengths_around_a_step(mbmod, n_int, prec):
    # enough bands that a run is the whole basis: 9 to 33 rows, which with the
    # five drain rows end below, at and above multiples of the step (8, 16)
    _check(mbmod, _workload((16, 16), (4.7, 4.7), 5.0, n_int, 100), prec)


@pytest.mark.parametrize("case", ["16x16", "16x16-full"])
@pytest.mark.parametrize("n_int,nbands", [(6, 2), (7, 1), (13, 9), (38, 9), (60, 9), (61, 9), (62, 9), (38, 10)])
def test_small_fp64_clusters(mbmod, case, n_int, nbands):
    """One cluster of CTAs per band: one or two rows a CTA (9 splines) up to eight (64),
    and the sizes just outside (65 splines, 20 bands of two k-points)."""
    grid = {"16x16": ((16, 16), (4.7, 4.7), 12.0), "16x16-full": GRIDS["16x16-full"]}[case]
    small = n_int + 3 <= 64 and 2 * nbands * 8 <= 152
    _check(mbmod, _workload(*grid, n_int=n_int, nbands=nbands), "fp64",
           kernel="rowspace_small_kernel" if small else "rowspace_kernel")


@pytest.mark.parametrize("prec,case,nk,nbands", [
    ("fp32", "16x16-full", 8, 100), ("fp32", "16x32", 4, 100), ("fp32", "32x32-full", 2, 100), ("fp32", "64x16-fold", 2, 100),
    ("fp32", "64x64-fold", 2, 24), ("fp64", "16x16-full", 2, 100), ("fp64", "32x16-full", 2, 100), ("fp64", "64x32-fold", 2, 50)])
def test_runs_across_bands(mbmod, prec, case, nk, nbands):
    """A third more bands than the device holds at once: equal runs that begin
    and end inside a band, of k-points with different discs.  A row's
    operations do not depend on the run it is in, so the result is bitwise that
    of whole bands per run (an explicit target of one run a slot)."""
    w = _workload(*GRIDS[case], n_int=40, nbands=nbands)
    w = dataclasses.replace(w, kpts=np.array([[0.03 * i, -0.02 * i * i / nk] for i in range(nk)]))
    h = mbmod.Handle.from_workload(w)
    g = torch.Generator(device="cuda").manual_seed(5)
    Xs = []
    for ik in range(w.nk):
        ng, nb, ldg = h.sizes(ik)
        x = torch.randn(nbands, nb, ldg, dtype=torch.complex128 if prec == "fp64" else torch.complex64, device="cuda", generator=g)
        x[:, :, ng:] = 0
        Xs.append(x)
    out = []
    for waves in (0, 1):
        h.plane_kernel_select(w.nk, nbands, prec, -1, waves)
        Ys = [torch.full_like(x, complex(np.nan, np.nan)) for x in Xs]
        h.apply_H_batch(list(range(w.nk)), Xs, Ys, prec)
        out.append(Ys)
    torch.cuda.synchronize()
    for a, b in zip(*out):
        assert torch.equal(a, b)
    h.close()


@pytest.mark.parametrize("case,n_int,nbands", [(c, 9, 3) for c in GRIDS] + [("16x32", 24, 40), ("64x16-fold", 14, 20)])
def test_density(mbmod, case, n_int, nbands):
    """The density of random bands on every grid shape, with some bands empty
    (and a whole k-point) and, in the cells of 3 bands, one of negative weight."""
    w = _workload(*GRIDS[case], n_int=n_int, nbands=nbands)
    w = dataclasses.replace(w, kpts=np.array([[0.0, 0.0], [0.11, -0.07], [-0.2, 0.05]]))
    h = mbmod.Handle.from_workload(w)
    models, coefs, blocks = [], [], []
    occ = np.random.default_rng(4).random((w.nk, nbands))
    occ[1] = 0.0
    occ[2, 1] = 0.0
    if nbands == 3:
        occ[0, 2] = -0.3
    for ik in range(w.nk):
        ng, nb, ldg = h.sizes(ik)
        m = Hm.model_from_workload(w, ik)
        X = W.random_block(nbands, nb, ng, seed=40 + ik)
        models.append(m)
        coefs.append(X)
        blocks.append(lib_block(X, gmap(h, m, ik), ldg, np.complex128).ravel())
    evecs = torch.from_numpy(np.concatenate(blocks)).cuda()
    zq, _ = h.zplanes()
    rho = torch.full((len(zq),) + w.grid, float("nan"), dtype=torch.float64, device="cuda")
    h.density(evecs, nbands, occ, rho)
    ref = F.density(models, coefs, occ)
    assert np.abs(rho.cpu().numpy() - ref).max() < 1e-11 * np.abs(ref).max()
    if nbands > 3:
        assert float(rho.min()) >= 0.0
    h.close()
