"""The angular and backward kernels on both sides of the sizes where a warp per atom gives way to
four lanes per atom (3,040 atoms in FP64, 2,048 in mixed precision), against the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2606_14073_gb300 import nep_params, spinlat as S, workloads as W

pytestmark = pytest.mark.gpu


def _system(n, prec):
    rng = np.random.default_rng(n)
    pos, species, box = W.b20_lattice(8, 8, 6)
    per = np.ones(3, np.int32)
    keep = np.sort(rng.permutation(len(pos))[:n])
    pos = W.wrap(pos + rng.normal(0.0, 0.05, pos.shape), box, per)[keep]
    spins = W.random_unit_vectors(rng, n)
    return S.System(pos, spins, box, per, species[keep], nep_params.load(), precision=prec), species[keep], box, per


@pytest.mark.parametrize("prec,n", [(S.SL_PREC_FP64, 3040), (S.SL_PREC_FP64, 3041), (S.SL_PREC_MIXED, 2048),
                                    (S.SL_PREC_MIXED, 2049)])
def test_evaluation_matches_oracle(prec, n):
    s, species, box, per = _system(n, prec)
    st, r = s.get_state(), s.energy_forces_fields()
    q, _ = s.get_descriptors()
    s.destroy()
    model = O.Model(nep_params.load())
    ref = O.evaluate(model, st["positions"], st["spins"], species, box, per)
    if prec == S.SL_PREC_FP64:   # the parity tests' bars
        q_ref = O.descriptors(model, st["positions"], st["spins"], species, box, per)
        assert np.abs(q - q_ref).max() <= 1e-10 * np.abs(q_ref).max()
        for k in ("F", "H", "W"):
            assert np.abs(r[k].reshape(-1) - ref[k].reshape(-1)).max() <= 1e-10 * np.abs(ref[k]).max(), k
    else:
        assert np.linalg.norm(r["F"] - ref["F"], axis=1).max() < 2e-3
        assert np.linalg.norm(r["H"] - ref["H"], axis=1).max() < 2e-3
        assert np.abs(r["W"].reshape(-1) - ref["W"].reshape(-1)).max() <= 1e-4 * np.abs(ref["W"]).max()
