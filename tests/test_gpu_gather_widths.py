"""The gather on both sides of the sizes where one lane per atom takes over from several (16,384 atoms
in FP64, 65,536 in mixed precision, where up to 16,384 take eight and the others four): forces sum to
zero, and the forces and fields that a system carries from its creation agree with those of the full
evaluation at the same state."""
import numpy as np
import pytest

from paper_2606_14073_gb300 import nep_params, spinlat as S, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,n", [(S.SL_PREC_FP64, 5), (S.SL_PREC_FP64, 16384), (S.SL_PREC_FP64, 16385),
                                    (S.SL_PREC_MIXED, 66), (S.SL_PREC_MIXED, 65536), (S.SL_PREC_MIXED, 65537)])
def test_gathered_forces(prec, n):
    rng = np.random.default_rng(n)
    cells = max(3, int(np.ceil((n / 8.0) ** (1.0 / 3.0))))
    pos, species, box = W.b20_lattice(cells, cells, cells)
    per = np.ones(3, np.int32)
    keep = np.sort(rng.permutation(len(pos))[:n])
    pos = W.wrap(pos + rng.normal(0.0, 0.05, pos.shape), box, per)[keep]
    s = S.System(pos, W.random_unit_vectors(rng, n), box, per, species[keep], nep_params.load(), precision=prec)
    st, r = s.get_state(), s.energy_forces_fields()
    s.destroy()
    # the evaluation takes the backward kernel with the virial, compiled apart: the same some 140
    # terms per atom, each rounded to 2^-53 or 2^-24 of the pair forces (below 10 eV/A)
    eps = 2.0 ** -53 if prec == S.SL_PREC_FP64 else 2.0 ** -24
    for a, b in ((st["forces"], r["F"]), (st["fields"], r["H"])):
        assert np.abs(a - b).max() <= 10.0 * eps * 140.0
    # every pair's two contributions cancel: what is left is that rounding, over the atoms as a walk
    assert np.abs(r["F"].sum(0)).max() <= 10.0 * eps * 140.0 * np.sqrt(n) * 4.0


@pytest.mark.parametrize("n", [7, 16384, 16385])
def test_gathered_forces_eight_and_four_lanes(n):
    """Mixed precision at the line between eight and four lanes: as above."""
    test_gathered_forces(S.SL_PREC_MIXED, n)
