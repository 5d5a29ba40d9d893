"""GPU tests of fdog_bound_reduce_noalloc on values of very different size and on calls after overlapping ones."""
import ctypes
import math
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2111_10270_gb300 import build as b

    b.build()
    import paper_2111_10270_gb300 as P

    torch.cuda.set_device(0)
    return torch, P


def reduce(env, dev, constant, out, stream=None):
    torch, P = env
    s = stream if stream is not None else torch.cuda.current_stream()
    rc = P.lib().fdog_bound_reduce_noalloc(ctypes.c_void_p(dev.data_ptr()), dev.numel(), constant,
                                           ctypes.c_void_p(out.data_ptr()), ctypes.c_void_p(s.cuda_stream))
    assert rc == P.FDOG_OK, rc


def total(env, values, constant=0.0):
    torch = env[0]
    out = torch.full((1,), float("nan"), dtype=torch.float64, device="cuda:0")
    reduce(env, torch.from_numpy(values).to("cuda:0"), constant, out)
    return float(out.item())


# the sum in exact arithmetic, rounded once (int / int division of Fraction rounds correctly)
def exact(values, constant=0.0):
    parts = np.concatenate([values[values != 0.0], [constant]])
    m, e = np.frexp(parts)
    m = np.ldexp(m, 53).astype(np.int64)
    e = e.astype(np.int64) - 53
    s = 0
    for x in np.unique(e):
        s += int(m[e == x].astype(object).sum()) << int(x + 1200)
    return float(Fraction(s, 1 << 1200))


@pytest.mark.parametrize("at", [(0, 1, 2), (2, 0, 1), (0, 300, 700), (0, 5000, 100), (9000, 5000, 20000)])
@pytest.mark.parametrize("big", [1e300, 2.0 ** 112, 2.0 ** 113, 2.0 ** 61, 2.0 ** 60, 1e17])
def test_what_is_left_when_large_values_cancel(env, big, at):
    """Two values that cancel, a small one far below their last place, among zeros, in one block and in several."""
    v = np.zeros(max(at) + 1)
    v[at[0]], v[at[1]], v[at[2]] = big, 1.0 + 2.0 ** -52, -big
    assert total(env, v) == 1.0 + 2.0 ** -52
    assert total(env, v, -1.0) == 2.0 ** -52
    v[at[2]] = 0.0
    assert total(env, v, -big) == 1.0 + 2.0 ** -52
    assert total(env, -v, big) == -1.0 - 2.0 ** -52


@pytest.mark.parametrize("n", [3, 1024, 1025, 4097, (1 << 20) + 1, 4096 * 300 + 17])
@pytest.mark.parametrize("kind", ["noise", "all sizes", "all sizes cancel", "smallest", "largest"])
def test_sums_of_every_size(env, n, kind):
    """The whole range of FP64: the exact sum to one unit in its last place."""
    rng = np.random.default_rng([n, len(kind)])
    v = rng.standard_normal(n)
    if kind == "noise":
        v[::3] *= 1e-25
    elif kind == "all sizes":
        v = np.ldexp(v, rng.integers(-1060, 1000, n).astype(np.int32))
    elif kind == "all sizes cancel":
        v = np.ldexp(v, rng.integers(-1060, 1000, n).astype(np.int32))
        h = n // 2
        v[h:2 * h] = -v[:h][rng.permutation(h)]
        v[0] += 0.0 if n % 2 else 1e-300
    elif kind == "smallest":
        v = rng.integers(-9, 10, n) * 5e-324
        v[n // 3] = -2.5e-308
    else:
        v = np.where(np.arange(n) % 2 == 0, 1.5e308, -1.5e308)
        v[n - 1] = 3.0
    for constant in (0.0, -1.5):
        got, want = total(env, v, constant), exact(v, constant)
        assert abs(got - want) <= math.ulp(want), (got, want)


@pytest.mark.parametrize("apart", [0, 1, 48, 49, 50, 63, 64, 65, 101, 102, 103, 112, 127, 128, 129, 700])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_totals_of_blocks_far_apart(env, sign, apart):
    """The first block's total and the others' at every distance of their exponents that an alignment treats apart."""
    v = np.zeros(3 * 1024)
    v[5], v[1024 + 7], v[2048 + 9] = sign * 2.0 ** apart, 1.0 + 2.0 ** -52, -2.0 ** -30
    for constant in (0.0, -sign * 2.0 ** apart):
        assert abs(total(env, v, constant) - exact(v, constant)) <= math.ulp(exact(v, constant))


def test_totals_beyond_the_range(env):
    assert math.isnan(total(env, np.array([1.7e308, 1.7e308])))
    assert math.isnan(total(env, np.array([1.7e308, 1e-300]), 1.7e308))
    assert math.isnan(total(env, np.array([1.0, 1e-300]), float("inf")))
    assert math.isnan(total(env, np.array([1e300, float("inf"), 1e-300])))
    assert total(env, np.array([1.7e308, 1.7e308, -1.7e308])) == 1.7e308
    assert total(env, np.array([1.0, 1e-300]), 2.0) == 3.0  # and nothing is left over for the next call


def test_overlapping_calls_spoil_no_later_one(env):
    """Calls that overlap race on the common scratch; calls that run alone afterwards are right, also the ones that
    were captured before."""
    torch, P = env
    gen = torch.Generator("cuda").manual_seed(3)
    # grids that fit the GPU side by side
    v = [torch.randn(n, generator=gen, device="cuda", dtype=torch.float64) for n in (400000, 90000)]
    out = torch.zeros(2, device="cuda", dtype=torch.float64)
    graphs = []
    for q in range(2):
        reduce(env, v[q], 0.0, out[q:])  # looks up the scratch
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            for _ in range(256):
                reduce(env, v[q], 0.0, out[q:])
        graphs.append(g)
    s = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    for _ in range(20):
        for q in range(2):
            with torch.cuda.stream(s[q]):
                graphs[q].replay()
    torch.cuda.synchronize()
    for k in range(130):
        # new values each time, so that what an earlier call left does not pass for a result
        q = k % 2
        v[q].mul_(1.01)
        torch.cuda.synchronize()
        if k < 4:
            graphs[q].replay()
        else:
            reduce(env, v[q], 0.0, out[q:])
        torch.cuda.synchronize()
        want = math.fsum(v[q].cpu().numpy())
        assert abs(float(out[q].item()) - want) <= math.ulp(want), k
