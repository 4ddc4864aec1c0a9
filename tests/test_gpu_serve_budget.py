"""Device memory that the solve server reserves for a request of many small
subspace problems: 64 k-points x (16 + 2 guard) blocks of 6 columns, each with
0.26 MB matrices (3 in FP64, 6 in mixed precision) and 0.2 MB of partial
products: 1.2 and 2.1 GB, with 0.6 GB of vectors 1.84 and 2.86 GB."""
import dataclasses

import pytest

from paper_1406_4960_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,budget", [("fp64", 1.85e9), ("fp32", 2.87e9)])
def test_many_small_problems_fit(prec, budget):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1406_4960_gb300 import mb
    mb.load(build_if_missing=True)
    w = W.scaled(W.tiny(), ecut=4.0, n_int=15, nbands=16)
    w = dataclasses.replace(w, kpts=W.random_kpoints(w.a1, w.a2, 64, 3))
    srv = mb.Server(slots=1, hbm_budget_bytes=budget)
    rc, ev, info, lat = srv.wait(srv.submit(w, 16, 1e-6, prec))
    assert rc == 0 and info.max_residual < 1e-6
    assert srv.stats()["peak_bytes"] <= budget
    srv.close()
