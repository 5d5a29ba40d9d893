"""Batches whose re-optimisations end at any multiple of the graphs' iterations, beside members still in their dual
phase: as each member gets alone."""
import numpy as np
import pytest

import ilpgen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2111_10270_gb300 import build as b

    b.build()
    import paper_2111_10270_gb300 as P

    return P


@pytest.mark.parametrize("reopt", [[0, 1], [3, 20], [4, 33], [20, 20]])
def test_steps_of_any_length(P, reopt):
    import torch

    stream = torch.cuda.Stream()
    ilps = [ilpgen.mrf_grid(12, 10, 4, 1, potts_max=2.0), ilpgen.random_ilp(40, 30, 31, max_row=8, max_coef=2),
            ilpgen.mrf_grid(16, 16, 2, 2)]

    def make(q):
        return P.Instance.from_ilp(ilps[q], rounding_dual_iters=reopt[q % 2], max_rounds=12).build(0, stream)

    def state(inst):
        return inst.solution(), inst.multipliers()[2]

    alone = [make(q) for q in range(3)]
    iters = [a.iterate(130)[0] for a in alone]
    ends = [a.primal_round() for a in alone]
    insts = [make(q) for q in range(3)]
    batch = P.Batch(insts, stream)
    got = batch.solve(130)
    assert got[0].tolist() == iters
    assert [(int(s), int(r)) for r, s in zip(got[1], got[2])] == [(int(s), int(r)) for s, r in ends]
    for a, b in zip(alone, insts):
        (x, objective, feasible), lam = state(a)
        (x2, objective2, feasible2), lam2 = state(b)
        assert np.array_equal(x, x2) and objective == objective2 and feasible == feasible2
        assert np.array_equal(lam, lam2)
