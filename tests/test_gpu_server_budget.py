"""The server's account of a request covers what the request allocates: with 14400 boxes of 8 cells
the tables of the boxes (their PML in FP64 and FP32, 13 MB) count as well as factors and vectors."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as W

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1508_02897_gb300.build import build  # noqa: E402

build()
from paper_1508_02897_gb300 import _binding as B  # noqa: E402
from paper_1508_02897_gb300.solver import HelmholtzDDM, Server  # noqa: E402


def test_request_bytes_cover_the_box_tables():
    N, npml, nb, restart = 480, 2, 120, 2
    n = N + 2 * npml
    c = np.ones((n, n))
    om = 2 * np.pi * N / 10.0
    s = HelmholtzDDM(N, npml, om, c, nb, nb, 0, factor=False)
    factor, krylov, scratch = B.hd_query_workspace(s.ctx, 1, restart)
    s.close()
    box = (16 + 8) * (2 * 8 + 2 * 8 + 2)   # a1, 1/a1, a2, 1/a2 of a box of 8 x 8, FP64 and FP32
    held = factor + krylov + scratch + 2 * 8 * n * n + box * nb * nb + 8 * n * n + 2 * 16 * n * n
    srv = Server(hbm_budget_bytes=4 << 30, max_slots=1)
    t = srv.submit(c, W.gaussian_source(N, npml, 0.4, 0.5, 2.0 / N), N, npml, om, nb, nb, 0, restart, 0.99)
    _, _, info = srv.poll(t)
    srv.close()
    assert info["device_bytes"] >= held
