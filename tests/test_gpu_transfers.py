"""Results on their way to the host: one piece or many, on one host thread or several, with outputs
left out, and with neighbour capacities too small for the pair records to serve as the buffer."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2606_14073_gb300 import nep_params, spinlat as S, workloads as W

pytestmark = pytest.mark.gpu


def _system(n, prec, **kw):
    rng = np.random.default_rng(n)
    cells = max(3, int(np.ceil((n / 8.0) ** (1.0 / 3.0))))
    pos, species, box = W.b20_lattice(cells, cells, cells)
    per = np.ones(3, np.int32)
    keep = np.sort(rng.permutation(len(pos))[:n])
    pos = W.wrap(pos + rng.normal(0.0, 0.05, pos.shape), box, per)[keep]
    vel = rng.normal(0.0, 0.01, (n, 3))
    spins = W.random_unit_vectors(rng, n)
    return S.System(pos, spins, box, per, species[keep], nep_params.load(), vel, precision=prec, **kw), pos, vel


@pytest.mark.parametrize("n", [1, 33, 1000, 60001])
@pytest.mark.parametrize("prec", [S.SL_PREC_FP64, S.SL_PREC_MIXED])
def test_state_comes_back_in_caller_order(n, prec):
    s, pos, vel = _system(n, prec)
    st = s.get_state()
    assert np.array_equal(st["velocities"], vel)
    assert np.abs(st["positions"] - pos).max() < 1e-12 and np.array_equal(st["ref_positions"], st["positions"])
    again = s.get_state()
    assert all(np.array_equal(st[k], again[k]) for k in ("spins", "forces", "fields"))
    # some of the arrays only
    v, f = np.zeros((n, 3)), np.zeros((n, 3))
    assert S.lib().sl_get_state(s.handle, None, v.ctypes.data, None, f.ctypes.data, None, None, None) == 0
    assert np.array_equal(v, vel) and np.array_equal(f, st["forces"])
    h = np.zeros((n, 3))
    assert S.lib().sl_energy_forces_fields(s.handle, None, None, h.ctypes.data, None) == 0
    r = s.energy_forces_fields(want_virial=False)
    assert np.array_equal(h, r["H"])
    q, e = s.get_descriptors()
    e2 = np.zeros(n)
    assert S.lib().sl_get_descriptors(s.handle, None, e2.ctypes.data) == 0
    assert np.array_equal(e, e2) and np.isfinite(q).all()
    assert abs(r["E"] - e.sum()) <= 1e-9 * np.abs(e).sum()
    s.destroy()


def test_descriptors_with_short_lists():
    """Four atoms in free space and capacities of four: 128 bytes of pair records per atom."""
    pos = np.array([[10.0, 10, 10], [12.3, 10, 10], [10, 12.6, 10], [10, 10, 12.9]])
    rng = np.random.default_rng(1)
    spins, species = W.random_unit_vectors(rng, 4), np.array([0, 1, 1, 0], np.int32)
    box, per = np.array([40.0, 40, 40]), np.zeros(3, np.int32)
    s = S.System(pos, spins, box, per, species, nep_params.load(), precision=S.SL_PREC_MIXED, cap_rad=4, cap_ang=4)
    q, e = s.get_descriptors()
    st = s.get_state()
    s.destroy()
    assert np.array_equal(st["positions"], pos)
    ref = O.descriptors(O.Model(nep_params.load()), pos, spins, species, box, per)
    assert np.abs(q - ref).max() <= 1e-5 * np.abs(ref).max()   # FP32 sums of three pairs
    assert np.isfinite(e).all()
