"""Between two steps of a call the second half of one and the first half of the next share a launch;
a step's bits do not depend on it: one call of several steps, captured or not, against as many
calls of one step, on both sides of the gather's widths, and with what adds terms to the halves."""
import numpy as np
import pytest

from paper_2606_14073_gb300 import nep_params, spinlat as S, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,n,per,extra", [
    (S.SL_PREC_FP64, 5, (1, 1, 1), None), (S.SL_PREC_FP64, 517, (1, 0, 0), "field"),
    (S.SL_PREC_FP64, 16385, (1, 1, 1), None), (S.SL_PREC_MIXED, 33, (1, 1, 1), "longitudinal"),
    (S.SL_PREC_MIXED, 4095, (1, 1, 0), "field"), (S.SL_PREC_FP64, 260, (1, 1, 1), "longitudinal"),
    (S.SL_PREC_MIXED, 16385, (1, 1, 1), "field"), (S.SL_PREC_MIXED, 65537, (1, 1, 1), None)])
def test_one_call_equals_single_steps(prec, n, per, extra):
    rng = np.random.default_rng(n)
    cells = max(3, int(np.ceil((n / 8.0) ** (1.0 / 3.0))))
    pos, species, box = W.b20_lattice(cells, cells, cells)
    keep = np.sort(rng.permutation(len(pos))[:n])
    per = np.array(per, np.int32)
    pos = W.wrap(pos + rng.normal(0.0, 0.05, pos.shape), box, per)[keep]
    vel, spin = W.maxwell_boltzmann(rng, species[keep], 300.0), W.random_unit_vectors(rng, n)
    out = []
    for queue, graph in ((1, 0), (7, 0), (7, 3)):   # steps a call, steps a captured graph
        s = S.System(pos, spin, box, per, species[keep], nep_params.load(), vel, precision=prec, seed=3,
                     steps_per_graph=graph)
        if extra == "field":
            s.set_atom_fields(np.linspace(0.0, 0.3, 3 * n).reshape(n, 3))
        elif extra == "longitudinal":
            s.set_longitudinal(True, 0.1, [[-0.01, 0.005], [0.0, 0.02]])
        for _ in range(7 // queue):
            s.step(queue, 1.0, 300.0, (0.0, 0.0, 0.2))
        out.append(s.get_state())
        s.destroy()
    for o in out[1:]:
        for k in ("positions", "velocities", "spins", "forces", "fields"):
            assert np.array_equal(o[k], out[0][k]), k
