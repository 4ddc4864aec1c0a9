"""The row-space density keeps NaN and infinite coefficients visible: the planes
that the coefficient's B-spline reaches are non-finite at every grid point, the
others are those of the finite bands bit for bit (they do not read it), and a
band without electrons does not count."""
import numpy as np
import pytest

from test_gpu_rowspace import GRIDS, _workload

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mbmod():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1406_4960_gb300 import mb
    mb.load(build_if_missing=True)
    return mb


@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("case", ["16x16-full", "16x32", "64x16-fold"])
def test_nonfinite_coefficient_stays_visible(mbmod, case, value):
    n_int, nbands, j = 14, 3, 7
    w = _workload(*GRIDS[case], n_int=n_int, nbands=nbands)
    h = mbmod.Handle.from_workload(w)
    g = torch.Generator(device="cuda").manual_seed(9)
    blocks = []
    for ik in range(w.nk):
        ng, nb, ldg = h.sizes(ik)
        x = torch.randn(nbands, nb, ldg, dtype=torch.complex128, device="cuda", generator=g)
        x[:, :, ng:] = 0
        blocks.append(x)
    occ = np.array([[2.0, 1.0, 0.5], [1.0, 0.0, 0.25]])
    nq = len(h.zplanes()[0])

    def density():
        rho = torch.zeros((nq,) + w.grid, dtype=torch.float64, device="cuda")
        h.density(torch.cat([x.reshape(-1) for x in blocks]), nbands, occ, rho)
        return rho

    clean = density()
    blocks[1][1, j, 2] = value                 # an empty band
    assert torch.equal(density(), clean)
    blocks[0][2, j, 2] = value
    rho = density()
    interval = torch.arange(nq, device="cuda") // w.nquad
    reach = (interval >= j + 2 - w.order) & (interval <= j + 1)      # retained spline j: knot intervals j - order + 2 .. j + 1
    assert reach.any() and not reach.all()
    assert not torch.isfinite(rho[reach]).any()
    assert torch.equal(rho[~reach], clean[~reach])
    h.close()
