"""Split-TF32 substitution with 32 right-hand sides per CTA (M = 128) on small uneven boxes: 100 boxes
and 49 to 64 sources take two waves of such CTAs where 16 per CTA (M = 64) would take three.  Every source
gives bitwise the vector it gives alone (M = 64), and matches the FP64 oracle to the FP32 grade
of the products, 2e-4 as elsewhere."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as W
from oracle import DDMPreconditioner, Grid

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1508_02897_gb300 import _binding as B  # noqa: E402
from paper_1508_02897_gb300.build import build  # noqa: E402

build()
from paper_1508_02897_gb300.solver import HelmholtzDDM  # noqa: E402

# owned cells of the ten box columns and rows: widths 16 to 41, or one box column 176 wide (the widest)
CUTS = {"uneven": [7, 33, 8, 11, 9, 25, 7, 10, 13, 8], "widest": [168, 7, 9, 7, 11, 8, 7, 7, 9, 7]}


@pytest.mark.parametrize("name,nrhs", [("uneven", 64), ("uneven", 61), ("widest", 49), ("uneven", 17)])
def test_x3_groups(name, nrhs):
    npml, overlap = 3, 2
    w = CUTS[name]
    cx = [npml + sum(w[:i]) for i in range(len(w) + 1)]
    N = sum(w)
    cy = [npml + (N * i) // 10 for i in range(11)]
    c = W.velocity_random_field(N, npml, seed=2)
    om = 2 * np.pi * float(c.min()) * N / 10.0
    g = Grid(N, npml, om)
    P = DDMPreconditioner(g, c, cx, cy, overlap)
    s = HelmholtzDDM(N, npml, om, c, 10, 10, overlap, cut_x=cx, cut_y=cy, tcore="x3", symmetric=False)
    r = W.random_complex((nrhs, g.n, g.n), seed=8)
    rt = torch.from_numpy(r)
    alone = [s.apply_precond(rt[k]).cpu().numpy() for k in range(nrhs)]
    _, _, need = B.hd_query_workspace(s.ctx, nrhs, 1)
    s.scratch = torch.empty(need, dtype=torch.uint8, device="cuda")
    s.scratch_bytes = need
    z = s.apply_precond(rt).cpu().numpy()
    for k in range(nrhs):
        assert np.array_equal(z[k], alone[k])
    for k in {0, 15, 16, min(31, nrhs - 1), min(32, nrhs - 1), nrhs - 1}:
        ref = P.apply(r[k])
        assert np.linalg.norm(z[k] - ref) / np.linalg.norm(ref) < 2e-4
    s.close()
