"""CPU tests of the plan of bulk sweeps: which instances have one, what it copies, and what is compiled for it."""
import pytest

import ilpgen
from bulk_view import compile_view


@pytest.fixture(scope="module")
def P():
    from paper_2111_10270_gb300 import build as b

    b.build()
    import paper_2111_10270_gb300 as P

    return P


@pytest.fixture(scope="module")
def view(P, tmp_path_factory):
    return compile_view(P, str(tmp_path_factory.mktemp("view")))


def planned(P, ilp, **kw):
    inst = P.Instance.from_ilp(ilp, P.capi.default_params(jit=1, **kw))
    inst.plan()
    return inst


def test_bulk_kernels_are_compiled_for_instances_that_run_them(P, view):
    # 5 labels: every tile mixed; 6x7 nodes: too few tiles; block_threads: a launch shape of the caller's own
    for ilp, kw in ((ilpgen.mrf_grid(30, 31, 5, 3), {}), (ilpgen.mrf_grid(6, 7, 8, 3), {}),
                    (ilpgen.mrf_grid(17, 19, 8, 3), {"block_threads": 128})):
        v = view(planned(P, ilp, **kw))
        assert v["runs"] == 0 and v["compiled"] and not v["bulk_compiled"], v
    inst = planned(P, ilpgen.mrf_grid(17, 19, 8, 3))
    v = view(inst)
    assert v["runs"] > 0 and v["compiled"] and v["bulk_compiled"], v
