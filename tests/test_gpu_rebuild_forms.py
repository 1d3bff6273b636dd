"""Neighbour lists on both sides of the size where a system's own rebuild goes from one cooperative
launch to its kernels one by one (131,072 atoms), and with cells split into parts (few cells)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2606_14073_gb300 import nep_params, spinlat as S, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,drop", [((3, 3, 3), 0), ((3, 3, 3), 5), ((3, 6, 12), 1), ((9, 9, 9), 2),
                                        ((32, 32, 16), 0), ((33, 32, 16), 4095)])
def test_lists_equal_the_oracle(shape, drop):
    rng = np.random.default_rng(shape[0] + drop)
    pos, species, box = W.b20_lattice(*shape)
    per = np.ones(3, np.int32)
    keep = np.sort(rng.permutation(len(pos))[drop:])
    pos = W.wrap(pos + rng.normal(0.0, 0.05, pos.shape), box, per)[keep]
    n = len(pos)
    s = S.System(pos, W.random_unit_vectors(rng, n), box, per, species[keep], nep_params.load(),
                 precision=S.SL_PREC_MIXED)
    s.step(30, 1.0, 300.0)     # builds triggered on the device, too
    pos = s.get_state()["positions"]
    rad, ang = s.get_neighbors()
    builds = s.info()["n_builds"]
    s.destroy()
    method = 0 if n <= 2000 else 1
    for lists, cut in ((rad, 7.0), (ang, 5.0)):
        ref = O.neighbors(pos, box, per, cut, method=method)
        assert all(np.array_equal(a, b) for a, b in zip(lists, ref))
    assert builds >= 2


@pytest.mark.parametrize("cells,prec,then", [(4, S.SL_PREC_FP64, "step"), (12, S.SL_PREC_MIXED, "step"),
                                             (4, S.SL_PREC_MIXED, "energy"), (6, S.SL_PREC_MIXED, "batch"),
                                             (6, S.SL_PREC_FP64, "set_state")])
def test_a_build_that_gives_up(cells, prec, then):
    """A wait of the one-launch build runs out: SL_ETIMEOUT, the build queued behind it does not start, and the
    system then goes on, builds included, bit for bit as one to which nothing happened."""
    make = lambda: S.system_from_workload(W.fege_cube(cells, T=300.0, seed=cells), nep_params.load(),  # noqa: E731
                                          precision=prec, skin=0.1)
    a, b = make(), make()
    builds = b.info()["n_builds"]
    assert S.lib().sl_selftest_rebuild_wait(b.handle) == S.SL_ETIMEOUT
    assert b.info()["n_builds"] == builds
    for s in (a, b):
        if then == "energy":
            s.energy_forces_fields()
        elif then == "set_state":
            st = s.get_state()
            s.set_state(st["positions"], st["velocities"], st["spins"], st["forces"], st["fields"])
        if then == "batch":
            batch = S.Batch([s])
            batch.step([25], [1.0], [300.0], [(0.0, 0.0, 0.0)])
            batch.destroy()
        else:
            s.step(25, 1.0, 300.0)
    assert a.info()["n_builds"] > builds + 1
    p, q = a.get_state(), b.get_state()
    for k in ("positions", "velocities", "spins", "forces", "fields"):
        assert np.array_equal(p[k], q[k]), k
    for x, y in zip(a.get_neighbors(), b.get_neighbors()):
        assert all(np.array_equal(u, v) for u, v in zip(x, y))
    a.destroy()
    b.destroy()


def test_builds_on_several_streams_at_once():
    """Systems stepped by a thread each, a build in nearly every step, so that several one-launch builds
    want the GPU at a time: every system as when it steps alone."""
    from concurrent.futures import ThreadPoolExecutor

    def run(k):
        s = S.system_from_workload(W.fege_cube(6 + 2 * (k % 4), T=300.0, seed=k), nep_params.load(),
                                   precision=S.SL_PREC_MIXED, skin=0.02, seed=k)
        s.step(40, 1.0, 300.0)
        out = s.get_state(), s.info()["n_builds"]
        s.destroy()
        return out

    alone = [run(k) for k in range(8)]
    with ThreadPoolExecutor(8) as ex:
        together = list(ex.map(run, range(8)))
    for (a, na), (b, nb) in zip(alone, together):
        assert na == nb and na > 20
        for k in ("positions", "velocities", "spins", "forces", "fields"):
            assert np.array_equal(a[k], b[k]), k
