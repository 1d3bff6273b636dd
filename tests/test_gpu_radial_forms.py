"""The wide radial kernel in one kernel and in two (rows, then sums beside the angular kernel), on both
sides of the sizes where the form changes: FP64 against the no-allocation entry point, which
shares neither, mixed precision against FP64; and in one batch, bit for bit as alone."""
import numpy as np
import pytest

from paper_2606_14073_gb300 import nep_params, spinlat as S, workloads as W

pytestmark = pytest.mark.gpu


def _atoms(n, seed):
    rng = np.random.default_rng(seed)
    cells = max(3, int(np.ceil((n / 8.0) ** (1.0 / 3.0))))
    pos, species, box = W.b20_lattice(cells, cells, cells)
    per = np.ones(3, np.int32)
    keep = np.sort(rng.permutation(len(pos))[:n])
    pos = W.wrap(pos + rng.normal(0.0, 0.05, pos.shape), box, per)[keep]
    return pos, W.random_unit_vectors(rng, n), box, per, species[keep], nep_params.load()


@pytest.mark.parametrize("n", [1, 17, 1023, 1024, 1025])
def test_fp64_against_noalloc(n):
    torch = pytest.importorskip("torch")
    pos, spin, box, per, species, params = a = _atoms(n, n)
    s = S.System(*a, precision=S.SL_PREC_FP64)
    q, e = s.get_descriptors()
    s.destroy()
    pad = lambda x: torch.from_numpy(np.concatenate([x, np.zeros((n, 1))], axis=1)).cuda()  # noqa: E731
    p4, s4, sp = pad(pos), pad(spin), torch.from_numpy(species.astype(np.int32)).cuda()
    q0 = torch.zeros((n, 66), dtype=torch.float64, device="cuda")
    e0 = torch.zeros((n,), dtype=torch.float64, device="cuda")
    S.sl_descriptors_energies_noalloc(p4.data_ptr(), s4.data_ptr(), sp.data_ptr(), n, box, per, params, q0.data_ptr(),
                                      e0.data_ptr(), torch.cuda.current_stream().cuda_stream)
    q0, e0 = q0.cpu().numpy(), e0.cpu().numpy()
    # FP64 sums of at most 160 terms in another order: rounding near 1e-14
    assert np.abs(q - q0).max() <= 1e-10 * max(1.0, np.abs(q0).max())
    assert np.abs(e - e0).max() <= 1e-10 * max(1.0, np.abs(e0).max())


@pytest.mark.parametrize("n", [33, 4095, 4096, 4097])
def test_mixed_against_fp64(n):
    a = _atoms(n, n)
    out = []
    for prec in (S.SL_PREC_FP64, S.SL_PREC_MIXED):
        s = S.System(*a, precision=prec)
        out.append(s.get_descriptors())
        s.destroy()
    (q0, e0), (q1, e1) = out
    # FP32 coordinates of a box of up to 40 A: the bound of the radial kernels' test for 80 A
    assert (np.abs(q1 - q0) / np.maximum(np.abs(q0).max(0), 1.0)).max() < 4e-4
    assert np.abs(e1 - e0).max() < 1e-4 * max(1.0, np.abs(e0).max())


@pytest.mark.parametrize("prec,sizes", [(S.SL_PREC_FP64, (1024, 1025, 40)), (S.SL_PREC_MIXED, (4097, 4096, 500))])
def test_batch_of_both_forms(prec, sizes):
    make = lambda: [S.System(*_atoms(n, n), precision=prec, seed=n) for n in sizes]  # noqa: E731
    alone, together = make(), make()
    for s in alone:
        s.step(5, 1.0, 200.0)
    b = S.Batch(together)
    b.step(5, 1.0, 200.0, (0.0, 0.0, 0.0))
    assert b.stats()["fused_calls"] == 1
    for x, y in zip(alone, together):
        p, r = x.get_state(), y.get_state()
        for k in ("positions", "velocities", "spins", "forces", "fields"):
            assert np.array_equal(p[k], r[k]), k
