"""The FP64 network kernel (eight atoms per block, two per warp) at partial blocks and warps:
descriptors in, energies and (through the forces) gradients out, against the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2606_14073_gb300 import nep_params, spinlat as S, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 3, 7, 8, 9, 15, 217])
def test_energies_forces_fields_match_oracle(n):
    params = nep_params.load()
    rng = np.random.default_rng(n)
    pos, species, box = W.b20_lattice(3, 3, 4)
    pos, species = (pos + rng.normal(0.0, 0.05, pos.shape))[:n], species[:n]
    pos = W.wrap(pos, box, (1, 1, 1))
    spins, per = W.random_unit_vectors(rng, n), np.ones(3, np.int32)
    s = S.System(pos, spins, box, per, species, params)
    q, e = s.get_descriptors()
    r = s.energy_forces_fields()
    st = s.get_state()
    s.destroy()
    model = O.Model(params)
    ref = O.evaluate(model, st["positions"], st["spins"], species, box, per)
    # the parity tests' bar: sums of some hundred FP64 terms
    assert np.abs(e - ref["Ei"]).max() <= 1e-10 * np.abs(ref["Ei"]).max()
    for k in ("F", "H"):
        assert np.abs(r[k] - ref[k]).max() <= 1e-10 * max(np.abs(ref[k]).max(), 1e-6)
