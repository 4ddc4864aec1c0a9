"""Both forms of the row-space density: sums of squares (few bands) and products
of rows (many) on every grid shape, at the ends of their runs, with Gauss points
per interval below and above a batch of six; the accuracy of few bands where
they vanish; and non-finite coefficients of many.

Tolerances: 1e-11 of the maximum, as in test_gpu_rowspace.py.  At a plane where
the bands vanish for every r, the amplitude sum_j B_j x_j is rounding alone:
with x from a 2D transform (nine stages of at most 4 u on the sum of the
coefficients' moduli) and six products, below 64 u A, A = sum_j B_j sum_G |c_jG|,
so the density is below f / A_c (64 u A)^2."""
import dataclasses

import numpy as np
import pytest

from oracle import hamiltonian as Hm
from oracle import scf as F
from paper_1406_4960_gb300 import workloads as W

from gpu_util import gmap, lib_block
from test_gpu_rowspace import GRIDS, _workload

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

KPTS = np.array([[0.0, 0.0], [0.11, -0.07], [-0.2, 0.05]])


@pytest.fixture(scope="module")
def mbmod():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1406_4960_gb300 import mb
    mb.load(build_if_missing=True)
    return mb


def _density(h, w, blocks, occ):
    rho = torch.full((len(h.zplanes()[0]),) + w.grid, float("nan"), dtype=torch.float64, device="cuda")
    h.density(torch.cat([torch.as_tensor(b, device="cuda").reshape(-1) for b in blocks]), w.nbands, occ, rho)
    return rho


@pytest.mark.parametrize("case,n_int,nbands,nquad", [(c, 9, nb, 6) for c in GRIDS for nb in (1, 12)] + [
    ("16x16-full", n, 1, 6) for n in (6, 12, 13, 60, 61)] + [("64x64-fold", n, 1, 6) for n in (7, 14, 29)] + [
    ("16x32", 20, nb, q) for nb in (1, 12) for q in (5, 7, 16)])
def test_against_the_oracle(mbmod, case, n_int, nbands, nquad):
    w = dataclasses.replace(_workload(*GRIDS[case], n_int=n_int, nbands=nbands), kpts=KPTS, nquad=nquad)
    h = mbmod.Handle.from_workload(w)
    models, coefs, blocks = [], [], []
    occ = 0.2 + 0.1 * np.random.default_rng(6).random((w.nk, nbands))     # (sum f)^2 / sum f^2: close to the number of bands
    for ik in range(w.nk):
        ng, nb, ldg = h.sizes(ik)
        models.append(Hm.model_from_workload(w, ik))
        coefs.append(W.random_block(nbands, nb, ng, seed=10 + ik))
        blocks.append(lib_block(coefs[-1], gmap(h, models[-1], ik), ldg, np.complex128))
    ref = F.density(models, coefs, occ)
    assert np.abs(_density(h, w, blocks, occ).cpu().numpy() - ref).max() < 1e-11 * np.abs(ref).max()
    h.close()


@pytest.mark.parametrize("case", ["16x16-full", "32x16-full", "64x32-fold"])
@pytest.mark.parametrize("nbands", [1, 2])
def test_few_bands_where_they_vanish(mbmod, case, nbands):
    w = dataclasses.replace(_workload(*GRIDS[case], n_int=14, nbands=nbands), kpts=KPTS[1:2])
    h = mbmod.Handle.from_workload(w)
    ng, nb, ldg = h.sizes(0)
    m = Hm.model_from_workload(w, 0)
    t = 6
    q = t * w.nquad + 2
    vals = m.zb.B[q]                                    # of the retained splines at the plane
    rng = np.random.default_rng(8)
    c = np.zeros((nbands, nb, ldg), dtype=np.complex128)
    A = 0.0
    for n in range(nbands):
        b = rng.standard_normal(nb)
        b[t] -= (vals @ b) / vals[t]
        g = rng.standard_normal(ng) + 1j * rng.standard_normal(ng)
        c[n, :, :ng] = b[:, None] * g[None]
        A = max(A, (np.abs(vals) @ np.abs(c[n]).sum(1)))
    occ = np.full((1, nbands), 2.0)
    rho = _density(h, w, [c], occ).cpu().numpy()
    area = w.a1[0] * w.a2[1]
    assert rho[q].max() <= nbands * 2.0 / area * (64 * 2.0**-53 * A) ** 2
    assert rho.max() > 0.1 / area                       # not where the bands are
    h.close()


@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("case", ["16x16-full", "16x32", "64x16-fold"])
def test_nonfinite_coefficient_of_many_bands(mbmod, case, value):
    """As test_gpu_density_nonfinite.py, which has few."""
    nbands, j = 12, 7
    w = dataclasses.replace(_workload(*GRIDS[case], n_int=14, nbands=nbands), kpts=KPTS[1:2])
    h = mbmod.Handle.from_workload(w)
    ng, nb, ldg = h.sizes(0)
    x = torch.randn(nbands, nb, ldg, dtype=torch.complex128, device="cuda", generator=torch.Generator(device="cuda").manual_seed(9))
    x[:, :, ng:] = 0
    occ = np.ones((1, nbands))
    clean = _density(h, w, [x], occ)
    x[2, j, 2] = value
    rho = _density(h, w, [x], occ)
    interval = torch.arange(len(rho), device="cuda") // w.nquad
    reach = (interval >= j + 2 - w.order) & (interval <= j + 1)
    assert reach.any() and not reach.all()
    assert not torch.isfinite(rho[reach]).any()
    assert torch.equal(rho[~reach], clean[~reach])
    h.close()
