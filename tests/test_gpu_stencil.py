"""Operator at the edges of its tiles: grids with no tile, one tile, ragged strips of every
kind, no PML, and several vectors (grids of 4, 8 and 16 rows per tile), against the oracle's
sparse matrix.  The operator is five products and four sums per component in FP64: 1e-13
relative L2, the bound of the parity tests."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as W
from oracle import Grid, global_operator

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1508_02897_gb300.build import build  # noqa: E402

build()
from paper_1508_02897_gb300.solver import HelmholtzDDM  # noqa: E402


@pytest.mark.parametrize("N,npml,nrhs", [(5, 2, 1), (31, 1, 2), (33, 0, 1), (62, 4, 3), (63, 16, 1), (97, 0, 2),
                                         (900, 16, 2), (1021, 9, 9)])
def test_operator_tiles(N, npml, nrhs):
    c = W.velocity_random_field(N, npml, seed=3) if N > 40 else W.velocity_three_layer(N, npml)
    om = 2 * np.pi * float(c.min()) * N / 10.0
    g = Grid(N, npml, om)
    A = global_operator(g, c)
    s = HelmholtzDDM(N, npml, om, c, -(-N // 200), -(-N // 200), 0, factor=False)
    x = W.random_complex((nrhs, g.n, g.n), seed=5)
    y = s.matvec(torch.from_numpy(x)).cpu().numpy()
    for k in (0, nrhs - 1):
        ref = A @ x[k].ravel()
        assert np.linalg.norm(y[k].ravel() - ref) / np.linalg.norm(ref) < 1e-13
