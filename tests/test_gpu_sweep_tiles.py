"""Sweep kernels at the edges of their tiles: every kernel class (short, long
and wide rows), tiles of 1, 31, 32 and 33 BDDs, rows that end on and beside the
segment and register limits, against the FP64 oracle with the tolerances of the
other parity tests."""
import numpy as np
import pytest

import ilpgen
from parity_util import MM_RTOL, lb_close, rel_err, slot_order

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


def rows_ilp(coef, sense, rhs, count, seed, shared):
    """`count` rows of one pattern.  With `shared`, neighbouring rows have half of their variables in common (all
    copies of those in one tile, or split over two); the other variables lie in one row each."""
    k = len(coef)
    step = max(1, k // 2) if shared else k
    rng = np.random.default_rng(seed)
    n = step * (count - 1) + k
    col = (np.arange(count)[:, None] * step + np.arange(k)).reshape(-1)
    return ilpgen.ILP(n, rng.standard_normal(n), np.arange(count + 1, dtype=np.int64) * k, col.astype(np.int32),
                      np.tile(np.asarray(coef, np.int32), count), np.full(count, sense, np.int8),
                      np.full(count, rhs, np.int64), name="rows")


PATTERNS = {
    # short rows of width 2: at most one, flow, product, marginalisation, at least one
    "amo2": ([1, 1], -1, 1), "amo8": ([1] * 8, -1, 1), "flow5": ([-1, 1, 1, 1, 1], -1, 0),
    "product": ([1, 1, -1], -1, 1), "marg6": ([-1, 1, 1, 1, 1, 1], 0, 0), "cover7": ([1] * 7, 1, 1),
    # short rows of width up to 4
    "card6": ([1] * 6, -1, 3), "knap7": ([2, 1, 1, 2, 1, 1, 1], -1, 3), "exact5": ([1] * 5, 0, 2),
    # long rows: on, one below and one above the segment length
    "amo9": ([1] * 9, -1, 1), "flow16": ([-1] + [1] * 15, -1, 0), "amo17": ([1] * 17, 0, 1),
    "flow24": ([-1] + [1] * 23, -1, 0), "cover25": ([1] * 25, 1, 1), "card16": ([1] * 16, -1, 2),
    "card33": ([1] * 33, -1, 3), "mixed12": ([1, -1] * 6, -1, 1),
    # wide rows
    "knap4": ([3, 5, 7, 6], -1, 11), "knap8": ([3, 1, 2, 3, 1, 2, 3, 2], -1, 8), "knap9": ([1, 2, 3] * 3, -1, 9),
    "card16w": ([1] * 16, -1, 7), "knap12": ([3, 2, 1, 3, 2, 3, 1, 2, 3, 1, 2, 3], 1, 13),
    "exact40": ([1, 2] * 20, 0, 7),
}


@pytest.mark.parametrize("count", [1, 31, 32, 33])
@pytest.mark.parametrize("shared", [False, True], ids=["apart", "shared"])
@pytest.mark.parametrize("name", sorted(PATTERNS))
def test_tile_edges(P, oracle_mod, name, shared, count):
    coef, sense, rhs = PATTERNS[name]
    g = rows_ilp(coef, sense, rhs, count, len(name) * 100 + count, shared)
    inst = P.Instance.from_ilp(g, P.capi.default_params(tol=0.0, jit=-1)).build(0)
    orc = oracle_mod.Problem.from_ilp(g)
    for _ in range(6):
        done, lb = inst.iterate(1)
        olb = orc.iterate(1)[0]
        assert done == 1 and lb_close(lb, olb, scale=np.abs(orc.energies()).sum()), (lb, olb)
    var, row, m0, m1 = inst.min_marginals()
    perm = slot_order(orc, var, row)
    om0, om1 = orc.min_marginals()
    assert rel_err(m0[perm], om0).max() <= MM_RTOL and rel_err(m1[perm], om1).max() <= MM_RTOL
    _, fea = inst.lower_bound()
    assert lb_close(fea, orc.lower_bounds()[1], scale=np.abs(orc.energies()).sum())


CTL_BYTES = 624


@pytest.mark.parametrize("tiles", [1, 255, 256, 257, 512, 2047, 2048, 2049, 2305])
def test_bound_of_any_number_of_chunks(P, oracle_mod, tiles):
    """The bound is reduced by one block up to eight chunks of 256 tiles and by a block per chunk beyond; an
    instance gets the same bound alone and beside one of the other kind."""
    g = rows_ilp(*PATTERNS["product"], 32 * tiles - 5, tiles, False)
    orc = oracle_mod.Problem.from_ilp(g)
    params = P.capi.default_params(tol=0.0, jit=-1, max_rounds=0)
    inst = P.Instance.from_ilp(g, params).build(0)
    for _ in range(3):
        done, lb = inst.iterate(1)
        assert done == 1 and lb_close(lb, orc.iterate(1)[0]), tiles
    other = P.Instance.from_ilp(rows_ilp(*PATTERNS["product"], 32 * (300 if tiles > 2048 else 3000), 7, False),
                                params).build(0)
    inst.reset()
    b = P.Batch([inst, other])
    iters, _, _ = b.solve(3)
    assert list(iters) == [3, 3]
    b.close()
    alone = P.Instance.from_ilp(g, params).build(0)
    alone.iterate(3)
    alone.primal_round()
    # the running bounds of the three iterations: the first entries of the control block that ends a checkpoint
    ring = [np.frombuffer(x.export_state()[-CTL_BYTES:], np.float64, count=3) for x in (inst, alone)]
    assert np.array_equal(ring[0], ring[1]) and np.all(ring[0] != 0)
    assert all(np.array_equal(x, y) for x, y in zip(inst.multipliers(), alone.multipliers()))


@pytest.mark.parametrize("planner", [0, 1], ids=["device plan", "host plan"])
@pytest.mark.parametrize("count", [1, 33, 10921, 10923])
def test_slots_as_listed(P, planner, count):
    """Slots come tile by tile, BDD by BDD and layer by layer, below and above the number (65,536) from which each
    array is copied by itself: six-variable rows in their order after four-variable ones (two shapes)."""
    g = rows_ilp(*PATTERNS["card6"], count, 3, False)
    few = rows_ilp(*PATTERNS["amo2"], 3, 4, False)
    g.cost = np.concatenate([few.cost, g.cost])
    g.row_ptr = np.concatenate([few.row_ptr, g.row_ptr[1:] + len(few.col)])
    g.col = np.concatenate([few.col, g.col + few.n_vars]).astype(np.int32)
    g.coef, g.sense, g.rhs = (np.concatenate([a, b]) for a, b in
                              ((few.coef, g.coef), (few.sense, g.sense), (few.rhs, g.rhs)))
    g.n_vars += few.n_vars
    inst = P.Instance.from_ilp(g, P.capi.default_params(tol=0.0, jit=-1, planner=planner)).build(0)
    inst.iterate(2)
    for again in range(2):
        var, row, m0, m1 = inst.min_marginals()
        assert np.array_equal(var, g.col) and np.array_equal(row, np.repeat(np.arange(g.n_rows), np.diff(g.row_ptr)))
        v2, r2, lam = inst.multipliers()
        assert np.array_equal(v2, var) and np.array_equal(r2, row)
        # rows share no variable: after two iterations a slot's multiplier is its variable's cost again plus what is
        # pending, and the min-marginals of the rows are those of the listed multipliers
        k = 6
        x = lam[len(few.col):].reshape(count, k).astype(np.float64)
        best = np.sort(x, 1)
        base = np.minimum(np.cumsum(best, 1)[:, :3], 0).min(1)
        got = np.minimum(m0, m1)[len(few.col):].reshape(count, k)
        assert np.allclose(got, base[:, None], rtol=1e-5, atol=1e-5)
        if again == 0:
            inst.row_bdd(0)  # brings a device-built plan to the host
            blob = inst.export_state()
            inst.release()
            inst.build(0).import_state(blob)


def join(*parts):
    """The ILPs side by side, without common variables."""
    off = np.cumsum([0] + [p.n_vars for p in parts])
    ptr = np.concatenate([[0], np.cumsum(np.concatenate([np.diff(p.row_ptr) for p in parts]))])
    return ilpgen.ILP(int(off[-1]), np.concatenate([p.cost for p in parts]), ptr.astype(np.int64),
                      np.concatenate([p.col + o for p, o in zip(parts, off)]).astype(np.int32),
                      np.concatenate([p.coef for p in parts]), np.concatenate([p.sense for p in parts]),
                      np.concatenate([p.rhs for p in parts]), name="joined")


# Instances that run bulk sweeps: grids whose edges fill their tiles (4, 2 and 8 labels), and one of them beside
# grids whose edges are cut by the tile's end (slots of one layer of both kinds), rows of variables with one copy,
# partial last tiles and tiles without any local variable; then the smallest, with fewer tiles than resident warps.
BULK = {
    "4 small": lambda: ilpgen.mrf_grid(23, 24, 4, 3, potts_max=2.0),
    "8 small": lambda: ilpgen.mrf_grid(17, 19, 8, 3, potts_max=2.0),
    "4": lambda: ilpgen.mrf_grid(190, 190, 4, 3, potts_max=2.0),
    "2": lambda: ilpgen.mrf_grid(370, 361, 2, 3, potts_max=2.0),
    "8": lambda: ilpgen.mrf_grid(131, 133, 8, 3, potts_max=2.0),
    "mixed": lambda: join(ilpgen.mrf_grid(195, 191, 4, 3), ilpgen.mrf_grid(61, 53, 3, 4), ilpgen.mrf_grid(41, 37, 5, 5),
                          ilpgen.mrf_grid(29, 31, 7, 6), rows_ilp(*PATTERNS["flow5"], 4111, 7, False),
                          rows_ilp(*PATTERNS["marg6"], 4099, 8, True)),
}


@pytest.mark.parametrize("name", sorted(BULK))
def test_bulk_sweeps_match_the_ordinary_ones(P, name):
    """Every state that can be read, bit for bit as without bulk sweeps (block_threads set: never used)."""
    g = BULK[name]()

    def make(**kw):
        return P.Instance.from_ilp(g, P.capi.default_params(tol=0.0, max_rounds=3, jit=1, **kw)).build(0)

    a, b = make(), make(block_threads=128)
    assert a.info()["device_bytes"] > b.info()["device_bytes"]  # the plan of the bulk sweeps

    def arrays(inst):
        blob = inst.export_state()
        assert blob[-4:] == b"\0\0\0\0"
        return blob[:-CTL_BYTES]

    def same():
        assert a.lower_bound() == b.lower_bound()
        assert arrays(a) == arrays(b)

    same()
    assert a.iterate(1) == b.iterate(1)
    same()
    assert a.iterate(9) == b.iterate(9)
    blob = a.export_state()
    same()
    c = make()
    c.import_state(blob)
    assert a.iterate(2) == b.iterate(2) == c.iterate(2)
    assert arrays(a) == arrays(c)
    for inst in (a, b):
        inst.finalize()
    same()
    assert a.iterate(2) == b.iterate(2)
    # a batch runs the ordinary sweeps on what the bulk sweeps left
    small = P.Instance.from_ilp(ilpgen.mrf_grid(9, 9, 3, 1), P.capi.default_params(tol=0.0, max_rounds=3)).build(0)
    batch = P.Batch([a, small])
    batch.solve(3)
    batch.close()
    b.iterate(3)
    b.primal_round()
    same()
    assert np.array_equal(a.solution()[0], b.solution()[0])
    assert a.iterate(2) == b.iterate(2)  # perturbed targets
    same()
    a.reset(), b.reset()
    assert a.iterate(4) == b.iterate(4)
    assert a.primal_round() == b.primal_round()
    same()


@pytest.mark.parametrize("add_back", [False, True])
@pytest.mark.parametrize("name", ["amo2", "amo8", "amo9", "flow16", "product", "marg6", "cover7", "card6", "exact5",
                                  "mixed12"])
def test_evaluation_of_specialised_rows(P, oracle_mod, name, add_back):
    """Rows of width 2 beside wider ones, most in templates of four nodes per layer: the evaluated bound is the
    oracle's."""
    g = join(rows_ilp(*PATTERNS[name], 33, 5, True), rows_ilp(*PATTERNS["card6"], 31, 6, False))
    inst = P.Instance.from_ilp(g, P.capi.default_params(tol=0.0, jit=1)).build(0)
    orc = oracle_mod.Problem.from_ilp(g)
    assert inst.kernel_plan()["jit_tiles"] > 0
    for _ in range(4):
        inst.iterate(1)
        orc.iterate(1)
    if add_back:
        inst.finalize()
        orc.addback()
    _, fea = inst.lower_bound()
    assert lb_close(fea, orc.lower_bounds()[1], scale=np.abs(orc.energies()).sum())
