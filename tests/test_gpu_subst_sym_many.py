"""Substitution over the symmetric tile storage with more boxes than SMs: the small CTAs of narrow
boxes (three or four to an SM), two CTAs to an SM in complex FP64, FP16 and BF16 tiles with one
CTA per box and four sources, ragged groups of sources in each, and boxes of unequal widths in
one launch.

Tolerances as for the other shapes: 1e-10 complex FP64, 2e-4 complex FP32, and for 16-bit tiles those of
their storage rounding (3e-2 FP16 as elsewhere, eight times that BF16, which has three bits less); every source of a group gives bitwise the vector it gives alone."""
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

TOL = {"c128": 1e-10, "c64": 2e-4, "c64h": 3e-2, "c64b": 2.4e-1}


def _cuts(npml, first, rest, count):
    """One box column of `first` owned cells, then `count` of `rest`."""
    return [npml] + [npml + first + rest * i for i in range(count + 1)]


# owned cells of the first box column (8 more with its PML and overlap), boxes per side
SHAPES = {
    "narrow": (14, 13),      # 169 boxes, 19 to 22 wide
    "three tiles": (40, 13),    # 48 wide beside 19: in complex FP64 small CTAs from one source on
    "four tiles": (56, 13),     # 64 wide: in complex FP64 two CTAs to an SM, small ones from two sources on
    "six tiles": (88, 13),      # 96 wide: the widest small CTA; in complex FP64 clusters of two
    "mid": (88, 10),            # 100 boxes: 400 CTAs of four sources, three to an SM in complex FP64
    "seven tiles": (103, 10),   # 111 wide: one large CTA per box, four sources each
}


@pytest.mark.parametrize("name", list(SHAPES))
@pytest.mark.parametrize("precision", ["c128", "c64", "c64h", "c64b"])
def test_subst_sym_many_boxes(name, precision):
    first, nb = SHAPES[name]
    npml, overlap, rest = 3, 2, 9
    N = first + rest * (nb - 1)
    cx = _cuts(npml, first, rest, nb - 1)
    cy = [npml + (N * i) // nb for i in range(nb + 1)]
    c = W.velocity_random_field(N, npml, seed=11)
    om = 2 * np.pi * float(c.min()) * N / 10.0
    g = Grid(N, npml, om)
    P = DDMPreconditioner(g, c, cx, cy, overlap)
    s = HelmholtzDDM(N, npml, om, c, nb, nb, overlap, precision=precision, cut_x=cx, cut_y=cy)
    r = W.random_complex((9, g.n, g.n), seed=23)
    rt = torch.from_numpy(r)
    alone = [s.apply_precond(rt[k]).cpu().numpy() for k in range(9)]
    for k in (0, 8):
        ref = P.apply(r[k])
        assert np.linalg.norm(alone[k] - ref) / np.linalg.norm(ref) < TOL[precision]
    _, _, need = B.hd_query_workspace(s.ctx, 9, 1)
    s.scratch = torch.empty(need, dtype=torch.uint8, device="cuda")
    s.scratch_bytes = need
    for nrhs in (2, 3, 4, 5, 9):
        z = s.apply_precond(rt[:nrhs]).cpu().numpy()
        for k in range(nrhs):
            assert np.array_equal(z[k], alone[k])
    s.close()
