"""List capacities that are too small, over every form of the radial kernel: the call reports the overflow, and
what else lives on the GPU, or is made there afterwards, is as if the call had not been."""
import numpy as np
import pytest

from paper_2606_14073_gb300 import nep_params, spinlat as S, workloads as W

pytestmark = pytest.mark.gpu

KEYS = ("positions", "velocities", "spins", "forces", "fields")


def _make(cells, prec, **kw):
    return S.system_from_workload(W.fege_cube(cells, T=300.0, seed=cells), nep_params.load(), precision=prec, **kw)


def _run(s, steps):
    s.step(steps, 1.0, 300.0)
    return s.get_state()


def _overflow_leaves_no_trace(cells, prec, caps):
    fresh = _make(cells, prec)
    live = _make(cells, prec)
    first = _run(fresh, 3)
    fresh.destroy()
    for c in caps:
        with pytest.raises(S.SpinlatError) as e:
            _make(cells, prec, **c)
        assert e.value.code == S.SL_ENBR_OVERFLOW
    again = _make(cells, prec)
    for s in (live, again):
        state = _run(s, 3)
        for k in KEYS:
            assert np.array_equal(state[k], first[k]), k
        s.destroy()


# rows and sums in two kernels, in one, and one thread per atom (mixed precision beyond 16,384 atoms)
@pytest.mark.parametrize("cells,prec", [(4, S.SL_PREC_FP64), (6, S.SL_PREC_FP64), (4, S.SL_PREC_MIXED),
                                        (9, S.SL_PREC_MIXED), (13, S.SL_PREC_MIXED)])
def test_too_few_angular_rows(cells, prec):
    """An atom has some 21 angular pairs: every capacity here refuses some of them in the radial kernel, too."""
    _overflow_leaves_no_trace(cells, prec, [dict(cap_ang=c) for c in (1, 2, 4, 8, 12, 16)])


@pytest.mark.parametrize("cells,prec", [(4, S.SL_PREC_FP64), (13, S.SL_PREC_MIXED)])
def test_cut_lists(cells, prec):
    """Lists cut at their capacity (an atom has some 110 candidates) hold pairs on one side only."""
    _overflow_leaves_no_trace(cells, prec, [dict(cap_rad=c, cap_ang=min(c, 64)) for c in (1, 7, 32, 64, 100)])
