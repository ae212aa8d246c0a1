"""The autotuner on symmetric storage: it reports a ring that the launch has, and changes no result.

With a box 176 wide among 49 the ring of either precision holds two stages and no more (complex FP32:
two sets, two clusters' halves of the tiles, 42 KB a set and stage at least; complex FP64: 90 KB a stage), so
two is the only depth to report; 169 narrow boxes leave several to choose from, 16 at most."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as W

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1508_02897_gb300.build import build  # noqa: E402

build()
from paper_1508_02897_gb300.solver import HelmholtzDDM  # noqa: E402


@pytest.mark.parametrize("precision", ["c64", "c128"])
@pytest.mark.parametrize("first,nb,threads,stages", [(168, 7, {"c64": 448, "c128": 256}, {2}),
                                                     (14, 13, {"c64": 96, "c128": 96}, set(range(1, 17)))])
def test_autotune_reports_what_runs(precision, first, nb, threads, stages):
    npml, overlap, rest = 3, 2, 9
    N = first + rest * (nb - 1)
    cx = [npml] + [npml + first + rest * i for i in range(nb)]
    cy = [npml + (N * i) // nb for i in range(nb + 1)]
    c = W.velocity_random_field(N, npml, seed=11)
    om = 2 * np.pi * float(c.min()) * N / 10.0
    s = HelmholtzDDM(N, npml, om, c, nb, nb, overlap, precision=precision, cut_x=cx, cut_y=cy)
    r = torch.from_numpy(W.random_complex((s.n, s.n), seed=4))
    z = s.apply_precond(r).cpu().numpy()
    t, n, ms = s.autotune()
    assert t == threads[precision] and n in stages and ms > 0
    assert np.array_equal(z, s.apply_precond(r).cpu().numpy())
    assert s.autotune()[:2] == (t, n)   # from the cache
    s.close()
