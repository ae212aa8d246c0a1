"""Substitution over the symmetric tile storage at the edges of its launch shapes: widths
from less than one tile to the widest box, boxes of unequal widths in one launch (their
segments fall into unequal rounds), few to many boxes (four, two or one CTA per box) and
one to five right-hand sides (groups of four, with a ragged last one).

The tolerances are those of the preconditioner against the FP64 oracle (1e-10 complex FP64,
2e-4 complex FP32: FP32 rounding times the condition number of the local problems); every
right-hand side of a group gives bitwise the vector it gives alone."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as W
from oracle import DDMPreconditioner, Grid

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1508_02897_gb300.build import build  # noqa: E402

build()
from paper_1508_02897_gb300.solver import HelmholtzDDM  # noqa: E402

# name -> N, npml, overlap, cuts along x, cuts along y (interior cells)
SHAPES = {
    "one tile": (10, 2, 0, [0, 10], [0, 10]),                                  # 14 wide
    "uneven widths": (261, 4, 1, [0, 5, 92, 261], [0, 130, 261]),              # 14, 97, 178 wide, four CTAs per box
    "widest": (432, 8, 8, [0, 200, 432], [0, 40, 120, 432]),                   # 224 and 256 wide, two sets
    "two CTAs": (350, 4, 2, [50 * i for i in range(8)], [50 * i for i in range(8)]),      # 49 boxes
    "one CTA": (360, 4, 2, [36 * i for i in range(11)], [36 * i for i in range(11)]),     # 100 boxes
}


@pytest.mark.parametrize("name", list(SHAPES))
@pytest.mark.parametrize("precision,tol", [("c128", 1e-10), ("c64", 2e-4)])
def test_subst_sym_shapes(name, precision, tol):
    N, npml, overlap, cx, cy = SHAPES[name]
    cx, cy = [npml + v for v in cx], [npml + v for v in cy]
    c = W.velocity_random_field(N, npml, seed=11)
    om = 2 * np.pi * float(c.min()) * N / 10.0
    g = Grid(N, npml, om)
    P = DDMPreconditioner(g, c, cx, cy, overlap)
    s = HelmholtzDDM(N, npml, om, c, len(cx) - 1, len(cy) - 1, overlap, precision=precision, cut_x=cx, cut_y=cy)
    r = W.random_complex((5, g.n, g.n), seed=23)
    alone = [s.apply_precond(torch.from_numpy(r[k])).cpu().numpy() for k in range(5)]
    for k in (0, 4):
        ref = P.apply(r[k])
        assert np.linalg.norm(alone[k] - ref) / np.linalg.norm(ref) < tol
    for nrhs in (2, 3, 5):
        z = s.apply_ddm(torch.from_numpy(r[:nrhs]), 1).cpu().numpy()
        for k in range(nrhs):
            assert np.array_equal(z[k], alone[k])
