"""Alg. 2's test and perturbation on variables around the limit between a
thread and a warp per variable (8 copies) and around whole warps of copies."""
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


def star(copies, seed):
    """Variables x_0 .. x_2 of `copies` rows each, x_h + y_j <= 1 with a y_j of its own per row."""
    rng = np.random.default_rng(seed)
    m = 3 * copies
    col = np.stack([np.repeat(np.arange(3), copies), 3 + np.arange(m)], 1)[rng.permutation(m)].reshape(-1)
    cost = np.concatenate([rng.standard_normal(3) * copies, rng.standard_normal(m)])
    return ilpgen.ILP(3 + m, cost, np.arange(m + 1, dtype=np.int64) * 2, col.astype(np.int32),
                      np.ones(2 * m, np.int32), np.full(m, -1, np.int8), np.ones(m, np.int64), name="star")


def splitmix(x):
    mask = (1 << 64) - 1
    z = (x + 0x9E3779B97F4A7C15) & mask
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
    return z ^ (z >> 31)


@pytest.mark.parametrize("copies", [1, 7, 8, 9, 31, 32, 33, 64, 65, 300])
def test_one_round_of_perturbation(P, copies):
    """One round without re-optimisation leaves every copy at lambda + p, p from the signs and the FP32 sum of the
    variable's M_ij taken in slot order: the same operations in numpy, compared bit for bit."""
    g = star(copies, copies)
    inst = P.Instance.from_ilp(g, P.capi.default_params(tol=0.0, max_rounds=1, rounding_dual_iters=0, seed=5)).build(0)
    inst.iterate(3)
    inst.finalize()
    var, row, m0, m1 = inst.min_marginals()
    before = inst.multipliers()[2]
    M = m1 - m0
    want = before.copy()
    disagree = False
    for i in range(g.n_vars):
        s = np.flatnonzero(var == i)  # tiles, lanes and layers in order; rows of two layers: slot order below
        # slot order: by tile, then layer, then lane; every row here has the same shape
        order = np.lexsort((s // 2 % 32, s % 2, s // 64))
        m = M[s][order]
        total = np.float32(0)
        for x in m:
            total = np.float32(total + x)
        r = (2.0 * ((splitmix(5 ^ i) >> 11) * 2.0 ** -53) - 1.0)
        if np.all(m > 0):
            p = 1.0
        elif np.all(m < 0):
            p = -1.0
        else:
            disagree = True
            sign = 1.0 if total > 0 else -1.0 if total < 0 else (1.0 if r >= 0 else -1.0)
            p = r if np.all(m == 0) else sign * abs(r)
        want[s] = before[s] + np.float32(p)
    rc, rounds = inst.primal_round()
    assert (rounds >= 1) == disagree
    assert np.array_equal(inst.multipliers()[2], want if disagree else before)
