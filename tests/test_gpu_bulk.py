"""GPU tests of the bulk sweeps' plan and of what instances that run them share."""
import ctypes
import threading

import pytest

import ilpgen
from bulk_view import compile_view
from test_gpu_sweep_tiles import BULK

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2111_10270_gb300 import build as b

    b.build()
    import paper_2111_10270_gb300 as fdog

    return fdog


@pytest.fixture(scope="module")
def view(P, tmp_path_factory):
    return compile_view(P, str(tmp_path_factory.mktemp("view")))


def grid(P, h, w, labels, **kw):
    ilp = ilpgen.mrf_grid(h, w, labels, 3, potts_max=2.0)
    return P.Instance.from_ilp(ilp, P.capi.default_params(tol=0.0, jit=1, **kw))


def test_instances_of_common_kernels_on_two_threads(P):
    """Both run the kernels of the same shapes with shared memory of their own size; profiling launches every pass by
    itself, outside of graphs."""
    import torch

    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    insts = [grid(P, h, w, 4).build(0, s) for (h, w), s in zip([(190, 190), (100, 101)], streams)]
    want = [(i.iterate(800), i.reset())[0] for i in insts]
    errors, got = [], [None, None]

    def work(q):
        try:
            for _ in range(200):
                got[q] = insts[q].iterate(4)
        except Exception as e:
            errors.append(repr(e))

    for i in insts:
        i.set_profiling(True)
    threads = [threading.Thread(target=work, args=(q,)) for q in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert errors == []
    assert [g[1] for g in got] == [w[1] for w in want]


def test_an_instance_back_from_a_server(P, view):
    """A server runs the ordinary sweeps; built again by its owner, the instance runs those it would have without."""
    import numpy as np

    for planner in (0, 1):
        inst = grid(P, 40, 41, 8, planner=planner)
        server = P.Server(max_iters=20)
        ticket = server.submit(inst)
        assert server.wait(ticket)
        inst = server.take(ticket)
        server.close()
        other = grid(P, 40, 41, 8, planner=planner).build(0)
        inst.build(0)
        assert view(other)["ready"] and view(inst)["ready"]
        assert inst.iterate(20) == other.iterate(20)
        assert np.array_equal(inst.multipliers()[2], other.multipliers()[2])


@pytest.mark.parametrize("planner", [0, 1], ids=["device plan", "host plan"])
@pytest.mark.parametrize("size", [(9, 7, 3), (60, 61, 5)])
def test_slots_are_read_on_a_full_device(P, view, size, planner):
    """Without device memory for the listed order the host lists the slots, in the same order."""
    import numpy as np

    inst = grid(P, *size, planner=planner).build(0)
    inst.iterate(7)
    n = inst.info()["n_slots"]
    var, row, lam = np.zeros(n, np.int32), np.zeros(n, np.int32), np.zeros(n, np.float32)
    before = inst.info()["device_bytes"]
    ptr = [ctypes.c_void_p(a.ctypes.data) for a in (var, row, lam)]
    assert view.so.read_on_full_device(inst._h, *ptr) == P.FDOG_OK
    assert inst.info()["device_bytes"] == before
    for got, want in zip((var, row, lam), inst.multipliers()):
        assert np.array_equal(got, want)


@pytest.mark.parametrize("name", sorted(BULK))
def test_the_cases_compared_with_ordinary_sweeps_run_bulk_sweeps(P, view, name):
    """Those of test_bulk_sweeps_match_the_ordinary_ones, which only sees that memory was set aside."""
    ilp = BULK[name]()
    params = dict(tol=0.0, max_rounds=3, jit=1)
    assert view(P.Instance.from_ilp(ilp, P.capi.default_params(**params)).build(0))["ready"]
    assert not view(P.Instance.from_ilp(ilp, P.capi.default_params(block_threads=128, **params)).build(0))["ready"]
