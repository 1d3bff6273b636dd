"""The midpoint iteration's stop test is taken by the block that finishes last: the evaluations a
step makes are the cap's when no change is small enough and one when every change is, for one
block and for many, on both sides of the gather's widths, with and without Anderson mixing."""
import numpy as np
import pytest

from paper_2606_14073_gb300 import nep_params, spinlat as S, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,n,depth", [(S.SL_PREC_FP64, 5, 0), (S.SL_PREC_FP64, 16385, 0), (S.SL_PREC_MIXED, 33, 2),
                                          (S.SL_PREC_MIXED, 4095, 0), (S.SL_PREC_MIXED, 16385, 0),
                                          (S.SL_PREC_MIXED, 65537, 0)])
def test_evaluations_per_step(prec, n, depth):
    rng = np.random.default_rng(n)
    cells = max(3, int(np.ceil((n / 8.0) ** (1.0 / 3.0))))
    pos, species, box = W.b20_lattice(cells, cells, cells)
    keep = np.sort(rng.permutation(len(pos))[:n])
    per = np.ones(3, np.int32)
    pos = W.wrap(pos + rng.normal(0.0, 0.02, pos.shape), box, per)[keep]
    for tol, want in ((0.0, 4), (1e30, 1)):
        s = S.System(pos, W.random_unit_vectors(rng, n), box, per, species[keep], nep_params.load(), precision=prec,
                     midpoint_iters=4, midpoint_tol=tol, anderson_depth=depth)
        e0 = s.midpoint_evaluations()
        s.step(3, 0.1, 100.0)
        assert s.midpoint_evaluations() - e0 == 3 * want
        st = s.get_state()
        assert np.abs(np.linalg.norm(st["spins"], axis=1) - 1.0).max() < 1e-14
        s.destroy()
