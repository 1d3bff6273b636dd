"""A batch's two kernels of a launch group (a width each) run side by side over their own slots, and
its rebuild group returns at once unless a slot's rebuild is due: replicas on both sides of the
widths, some rebuilding often and some never, step bit for bit as alone."""
import numpy as np
import pytest

from paper_2606_14073_gb300 import nep_params, spinlat as S, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,cells,skins", [(S.SL_PREC_MIXED, (4, 7, 13), (1.0, 0.02, 1.0)),
                                              (S.SL_PREC_MIXED, (13, 5), (0.02, 1.0)),
                                              (S.SL_PREC_FP64, (4, 8, 13), (0.05, 1.0, 0.02))])
def test_widths_side_by_side(prec, cells, skins):
    make = lambda: [S.system_from_workload(W.fege_cube(c, T=300.0, seed=c), nep_params.load(), precision=prec,  # noqa: E731
                                           skin=k, seed=c, steps_per_graph=3) for c, k in zip(cells, skins)]
    alone, together = make(), make()
    steps = [8 - i for i in range(len(cells))]
    for s, n in zip(alone, steps):
        s.step(n, 1.0, 300.0)
    b = S.Batch(together)
    k = len(cells)
    b.step(steps, [1.0] * k, [300.0] * k, [(0.0, 0.0, 0.0)] * k)
    assert max(s.info()["n_builds"] for s in together) > 1
    for x, y in zip(alone, together):
        p, q = x.get_state(), y.get_state()
        for k in ("positions", "velocities", "spins", "forces", "fields"):
            assert np.array_equal(p[k], q[k]), k


@pytest.mark.parametrize("prec,first,joins", [(S.SL_PREC_MIXED, 4, 13), (S.SL_PREC_FP64, 9, 4)])
def test_a_kernel_that_cannot_be_switched_on(prec, first, joins):
    """A replica that takes other forms of the kernels joins a batch whose graphs have those switched off; the
    switching fails, and the batch captures its graphs again: both replicas step bit for bit as alone."""
    make = lambda: [S.system_from_workload(W.fege_cube(c, T=300.0, seed=c), nep_params.load(), precision=prec,  # noqa: E731
                                           seed=c, steps_per_graph=3) for c in (first, joins)]
    alone, together = make(), make()
    b = S.Batch([together[0], None])
    zero = [(0.0, 0.0, 0.0)] * 2
    for s, n in zip(alone, (10, 5)):
        s.step(n, 1.0, 300.0)
    b.step([5, 0], [1.0] * 2, [300.0] * 2, zero)
    captures = b.stats()["fused_captures"]
    b.set(1, together[1])
    assert S.lib().sl_selftest_batch_switch(b.handle, 1) == S.SL_OK
    b.step([5, 5], [1.0] * 2, [300.0] * 2, zero)
    assert b.stats()["fused_captures"] == captures + 1
    for x, y in zip(alone, together):
        p, q = x.get_state(), y.get_state()
        for k in ("positions", "velocities", "spins", "forces", "fields"):
            assert np.array_equal(p[k], q[k]), k


def test_default_stream_busy_while_a_batch_is_set_up():
    """Work that the caller has queued on the default stream does not delay the clearing of a new batch's tables
    past their use."""
    import torch
    make = lambda: [S.system_from_workload(W.fege_cube(c, T=300.0, seed=c), nep_params.load(),  # noqa: E731
                                           precision=S.SL_PREC_MIXED, seed=c) for c in (4, 6)]
    alone, together = make(), make()
    for s in alone:
        s.step(6, 1.0, 300.0)
    b = S.Batch(together)
    torch.cuda._sleep(200_000_000)   # some 0.1 s
    for _ in range(2):
        b.step([3, 3], [1.0] * 2, [300.0] * 2, [(0.0, 0.0, 0.0)] * 2)
        torch.cuda.synchronize()
    for x, y in zip(alone, together):
        p, q = x.get_state(), y.get_state()
        for k in ("positions", "velocities", "spins", "forces", "fields"):
            assert np.array_equal(p[k], q[k]), k
