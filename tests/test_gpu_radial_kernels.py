"""The two radial kernels of mixed precision on both sides of the size where one takes over from
the other, and together in one batch."""
import numpy as np
import pytest

from paper_2606_14073_gb300 import nep_params, spinlat as S, workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def params():
    return nep_params.load()


def _workload(nx, ny, nz, drop, seed):
    rng = np.random.default_rng(seed)
    pos, species, box = W.b20_lattice(nx, ny, nz)
    per = np.ones(3, np.int32)
    pos = W.wrap(pos + rng.normal(0.0, 0.05, pos.shape), box, per)
    keep = np.sort(rng.permutation(len(pos))[drop:])
    n = len(keep)
    return dict(positions=pos[keep], spins=W.random_unit_vectors(rng, n), box=box, periodic=per,
                species=species[keep], velocities=W.maxwell_boltzmann(rng, species[keep], 200.0))


# 16,384 atoms is the largest system of the sixteen-lane kernel; ragged tails on both sides
@pytest.mark.parametrize("shape", [(16, 16, 8, 0), (16, 16, 8, 5), (17, 16, 8, 3), (17, 16, 8, 1019)])
def test_descriptors_and_forces_agree_with_fp64(params, shape):
    w = _workload(*shape, seed=11)
    out = {}
    for prec in (S.SL_PREC_FP64, S.SL_PREC_MIXED):
        s = S.System(params=params, precision=prec, **w)
        q, e = s.get_descriptors()
        out[prec] = (q, e, s.energy_forces_fields())
        s.destroy()
    (q0, e0, r0), (q1, e1, r1) = out[S.SL_PREC_FP64], out[S.SL_PREC_MIXED]
    scale = np.abs(q0).max(0)
    # FP32 coordinates of a box of L = 80 A are off by up to 2^-24 L, so separations by
    # 2 sqrt(3) 2^-24 L = 1.7e-5 A.  Channel slopes reach about sum_k |c_k| k^2 (4/6) / 2 ~ 34 / A where
    # the carrier is largest and a tenth of that over most of the range: over 70 pairs, against
    # descriptors of the order of ten, at most 70 * 3.4 * 1.7e-5 / 10 = 4e-4.
    assert (np.abs(q1 - q0) / scale).max() < 4e-4
    assert np.abs(e1 - e0).max() < 1e-4 * max(1.0, np.abs(e0).max())
    # the parity tests' bounds of mixed precision
    assert np.linalg.norm(r1["F"] - r0["F"], axis=1).max() < 2e-3
    assert np.linalg.norm(r1["H"] - r0["H"], axis=1).max() < 2e-3


@pytest.mark.parametrize("prec", [S.SL_PREC_FP64, S.SL_PREC_MIXED])
def test_batch_of_both_equals_alone(params, prec):
    shapes = [(17, 16, 8, 1), (4, 4, 4, 3), (16, 16, 8, 0)] if prec == S.SL_PREC_MIXED else [(6, 5, 5, 1), (4, 4, 4, 3)]
    ws = [_workload(*sh, seed=20 + k) for k, sh in enumerate(shapes)]
    alone = []
    for k, w in enumerate(ws):
        s = S.System(params=params, precision=prec, replica=k, **w)
        s.step(6, 1.0, 200.0, (0, 0, 0.1))
        alone.append(s.get_state())
        s.destroy()
    systems = [S.System(params=params, precision=prec, replica=k, **w) for k, w in enumerate(ws)]
    batch = S.Batch(systems)
    batch.step(6, 1.0, 200.0, (0, 0, 0.1))
    assert batch.stats()["fused_calls"] == 1
    for s, ref in zip(systems, alone):
        got = s.get_state()
        for key in ("positions", "velocities", "spins", "forces", "fields"):
            assert np.array_equal(got[key], ref[key]), key
    batch.destroy()
    for s in systems:
        s.destroy()
