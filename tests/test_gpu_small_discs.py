"""Discs of one G or one row of G on every kind of row-space plane (pruned,
full, folded), in runs of a few rows and of whole bands, against the FP64 oracle
at the tolerances of test_gpu_rowspace.py."""
import pytest

from test_gpu_rowspace import _check, _workload

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mbmod():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1406_4960_gb300 import mb
    mb.load(build_if_missing=True)
    return mb


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("n_int,nbands", [(6, 3), (37, 3), (9, 100)])
@pytest.mark.parametrize("grid,sides,ecut", [((16, 16), (4.7, 4.7), 0.4), ((64, 64), (3.0, 3.0), 1.0),
                                             ((16, 64), (4.7, 3.0), 0.3), ((32, 32), (9.4, 3.0), 0.6)])
def test_one_row_of_g(mbmod, grid, sides, ecut, n_int, nbands, prec):
    _check(mbmod, _workload(grid, sides, ecut, n_int, nbands), prec, waves=(0, 8))
