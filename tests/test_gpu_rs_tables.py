"""The row-space potential's table: Gauss points per interval whose planes do
not fill the kernel's batches of loads, and tables of few rows (64 points a CTA)
and of many (256).  Tolerances as in test_gpu_rowspace.py."""
import dataclasses

import pytest

from test_gpu_rowspace import GRIDS, _check, _workload

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mbmod():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1406_4960_gb300 import mb
    mb.load(build_if_missing=True)
    return mb


@pytest.mark.parametrize("nquad", [4, 7, 16])
@pytest.mark.parametrize("case,n_int", [("16x16-full", 7), ("64x32-fold", 40)])
def test_points_per_interval(mbmod, case, n_int, nquad):
    _check(mbmod, dataclasses.replace(_workload(*GRIDS[case], n_int=n_int, nbands=2), nquad=nquad), "fp64")
