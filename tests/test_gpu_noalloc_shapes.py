"""The no-allocation entry point at the edges of its launch shape: one atom, partial blocks, its
largest size, free axes, atoms many boxes away from the cell, against the FP64 oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2606_14073_gb300 import nep_params, spinlat as S, workloads as W

pytestmark = pytest.mark.gpu

TOL = 1e-10   # FP64 sums of at most 160 terms: rounding near 1e-14, the parity tests' bar


def _lattice(nx, ny, nz, n, seed, periodic=(1, 1, 1), shift=0):
    rng = np.random.default_rng(seed)
    pos, species, box = W.b20_lattice(nx, ny, nz)
    pos = pos + rng.normal(0.0, 0.05, pos.shape)
    if shift:   # whole box lengths, another number for each atom
        pos = pos + box * rng.integers(-shift, shift + 1, pos.shape)
    return pos[:n], W.random_unit_vectors(rng, n), species[:n], box, np.array(periodic, np.int32)


CASES = {
    "one_atom": lambda: _lattice(3, 3, 3, 1, 1),
    "three_atoms_free": lambda: _lattice(3, 3, 3, 3, 2, periodic=(0, 0, 0)),
    "partial_block": lambda: _lattice(3, 3, 4, 285, 3),
    "slab_free_z": lambda: _lattice(4, 3, 5, 479, 4, periodic=(1, 1, 0)),
    "unwrapped": lambda: _lattice(4, 4, 4, 512, 5, shift=3),
    "far_unwrapped": lambda: _lattice(4, 3, 3, 287, 6, shift=2000),
    "largest": lambda: _lattice(4, 8, 8, 2048, 7),
}


@pytest.mark.parametrize("name", list(CASES))
def test_matches_oracle(name):
    torch = pytest.importorskip("torch")
    params = nep_params.load()
    pos, spins, species, box, per = CASES[name]()
    n = len(species)
    pad = lambda a: torch.from_numpy(np.concatenate([a, np.zeros((n, 1))], axis=1)).cuda()  # noqa: E731
    p4, s4, sp = pad(pos), pad(spins), torch.from_numpy(species.astype(np.int32)).cuda()
    q = torch.full((n, 66), np.nan, dtype=torch.float64, device="cuda")
    e = torch.full((n,), np.nan, dtype=torch.float64, device="cuda")
    S.sl_descriptors_energies_noalloc(p4.data_ptr(), s4.data_ptr(), sp.data_ptr(), n, box, per, params, q.data_ptr(),
                                      e.data_ptr(), torch.cuda.current_stream().cuda_stream)
    model = O.Model(params)
    q_ref = O.descriptors(model, pos, spins, species, box, per)
    e_ref = O.evaluate(model, pos, spins, species, box, per)["Ei"]
    # coordinates of thousands of boxes carry 2^-52 of themselves into every separation
    tol = max(TOL, 100.0 * 2.0 ** -52 * np.abs(pos).max())
    assert np.abs(q.cpu().numpy() - q_ref).max() <= tol * max(np.abs(q_ref).max(), 1e-12)
    assert np.abs(e.cpu().numpy() - e_ref).max() <= tol * np.abs(e_ref).max()
