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


def test_a_device_without_room_for_bulk_sweeps(P, view):
    """An instance that fits only without their arrays is laid out without."""
    import ctypes

    ilp = ilpgen.mrf_grid(17, 19, 8, 3)
    inst, plain = planned(P, ilp), planned(P, ilp, block_threads=128)
    with_bulk, without = inst.info()["device_bytes"], plain.info()["device_bytes"]
    assert with_bulk > without
    took = ctypes.c_longlong()
    assert view.so.allocate_with_room(inst._h, ctypes.c_longlong(without - 1), ctypes.byref(took)) == P.capi.FDOG_ENOMEM
    inst = planned(P, ilp)
    assert view.so.allocate_with_room(inst._h, ctypes.c_longlong(with_bulk), ctypes.byref(took)) == P.FDOG_OK
    assert took.value == with_bulk and view(inst)["runs"] > 0
    assert view.so.allocate_with_room(inst._h, ctypes.c_longlong(with_bulk - 1), ctypes.byref(took)) == P.FDOG_OK
    assert took.value == without == inst.info()["device_bytes"] and view(inst)["runs"] == 0


# The kernel itself on the CPU: a warp as 32 threads, its PTX replaced by copies and barriers that the test controls.
EMULATION = r"""
#include <algorithm>
#include <atomic>
#include <barrier>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <thread>
#include <vector>
#define __device__
#define __global__
#define __shared__
#define __forceinline__ inline
#define __noinline__
#define __restrict__
#define __launch_bounds__(x)
#define __align__(x)
#define FDOG_FULL 0xffffffffu
struct float2 { float x, y; };
struct int4 { int x, y, z, w; };
static float2 make_float2(float x, float y) { return {x, y}; }
static int4 make_int4(int x, int y, int z, int w) { return {x, y, z, w}; }
static thread_local struct { int x; } threadIdx;
static struct { int x; } blockIdx{0}, blockDim{32}, gridDim{1};
using std::min;
template <class T> T __ldg(const T* p) { return *p; }
static std::barrier<> warp(32);
static float lanes[32];
static void __syncwarp() { warp.arrive_and_wait(); }
static float __shfl_xor_sync(unsigned, float x, int off) {
    lanes[threadIdx.x] = x;
    warp.arrive_and_wait();
    const float y = lanes[threadIdx.x ^ off];
    warp.arrive_and_wait();
    return y;
}
//ABI
float fdog_stages[4096];
struct Bar { long long pending = 0; unsigned phase = 0; };
struct Copy { unsigned dst, bytes, bar; const void* src; };
static std::mutex mu;
static std::map<unsigned, Bar> bar_of;
static std::vector<Copy> held;   // started, not landed
static int hold_from = 1 << 30;  // copies from this one on are held
static int started = 0, started_late = 0, asked = 0;
static std::atomic<bool> given_up{false};  // a wait of the lane that starts the copies has run out
static thread_local int polls = 0;         // of the running wait
static bool land_late = false;
static thread_local unsigned long long now = 1;
static void land(const Copy& c) {
    std::memcpy(reinterpret_cast<char*>(fdog_stages) + c.dst, c.src, c.bytes);
    Bar& b = bar_of[c.bar];
    if ((b.pending -= c.bytes) == 0) b.phase ^= 1u;
}
static void fdog_pdl_trigger() {}
static void fdog_pdl_wait() {}
static void fdog_copies_see_kernels() {}
static unsigned fdog_smem_addr(const void* p) {
    return static_cast<unsigned>(static_cast<const char*>(p) - reinterpret_cast<const char*>(fdog_stages));
}
static void fdog_bar_init(unsigned bars, int n) {
    for (int s = 0; s < n; ++s) bar_of[bars + 8u * s] = Bar();
}
static void fdog_bar_expect(unsigned bar, unsigned bytes) {
    std::lock_guard<std::mutex> lk(mu);
    bar_of[bar].pending += bytes;
}
static void fdog_bulk_copy(unsigned dst, const void* src, unsigned bytes, unsigned bar) {
    std::lock_guard<std::mutex> lk(mu);
    const Copy c{dst, bytes, bar, src};
    if (given_up) ++started_late;
    if (started++ >= hold_from) held.push_back(c);
    else land(c);
}
static InstCtl ctl;
static bool fdog_bar_done(unsigned bar, unsigned parity) {
    std::lock_guard<std::mutex> lk(mu);
    if (given_up && land_late && threadIdx.x == 0 && ++asked == 3) {
        for (const Copy& c : held) land(c);
        held.clear();
    }
    const bool done = bar_of[bar].phase != parity;
    if (done) polls = 0;
    return done;
}
// 0.3 s a poll for the lane that starts the copies, whose waits so end with their fifth; the others' time stands still
// until one of them has
static unsigned long long fdog_now() {
    if (threadIdx.x != 0) return now += given_up ? 300000000ull : 0ull;
    if (++polls == 5) {
        polls = 0;
        given_up = true;
    }
    return now += 300000000ull;
}
static std::atomic<int> wrong{0};
static int k_of[2] = {3, 2};
#define FDOG_BULK_DISPATCH(MODE) \
    for (int t = 0; t < k_of[jit]; ++t) { \
        if (valid && !late && sl[32 * t + lane] != lam[32 * t]) ++wrong; \
        if (valid && !late && sv[32 * t + lane] != 1000 * jit + t) ++wrong; \
        if (valid) lam[32 * t] += 1.f; \
    }
//KERNEL
int main(int argc, char** argv) {
    const int mode = std::atoi(argv[1]);
    hold_from = std::atoi(argv[2]);
    land_late = std::atoi(argv[3]) != 0;
    ctl = InstCtl();
    ctl.iter_limit = 1;
    ctl.error = std::atoi(argv[4]);
    // two runs of tiles: 13 of 3 layers (12 rows of the last valid), 6 of 2 layers
    const int n0 = 13, n1 = 6, n = n0 + n1;
    std::vector<float> lam(32 * (3 * n0 + 2 * n1)), cv(lam.size());
    for (size_t q = 0; q < lam.size(); ++q) lam[q] = 0.5f * q;
    std::vector<TileDev> tiles(n);
    std::vector<float2> lb(n, float2{-1.f, -1.f});
    BulkRun runs[2] = {};
    runs[0].n_bdds = 32 * (n0 - 1) + 12;
    runs[0].k = runs[0].v_n = 3;
    runs[1].tile = n0;
    runs[1].slot_base = runs[1].cv_row = 3 * n0;
    runs[1].slot_base *= 32;
    runs[1].n_bdds = 32 * n1;
    runs[1].k = runs[1].v_n = 2;
    runs[1].jit = 1;
    for (int t = 0; t < n; ++t) tiles[t].pattern = -1;
    for (int q = 0; q < 3 * n0 + 2 * n1; ++q) {
        const int id = q < 3 * n0 ? q % 3 : 1000 + (q - 3 * n0) % 2;
        for (int l = 0; l < 32; ++l) std::memcpy(&cv[32 * q + l], &id, 4);
    }
    InstDev inst{};
    inst.ctl = &ctl;
    inst.lam = lam.data();
    inst.cv = cv.data();
    inst.bulk_runs = runs;
    inst.n_bulk_runs = 2;
    inst.bulk_tiles = n;
    inst.tiles = tiles.data();
    inst.tile_lb = lb.data();
    unsigned pairs[1] = {};
    BulkArgs a{&inst, pairs, 0, n, 6, 2};
    std::vector<std::thread> th;
    for (int l = 0; l < 32; ++l)
        th.emplace_back([&, l] {
            threadIdx.x = l;
            if (mode == 0) fdog_bulk_sweep<0>(a);
            else fdog_bulk_sweep<1>(a);
        });
    for (auto& t : th) t.join();
    int missed = 0;
    for (size_t q = 0; q < lam.size(); ++q) {
        const bool pad = q >= 32 * 3 * (n0 - 1) && q < 32 * 3 * n0 && q % 32 >= 12;
        missed += lam[q] != 0.5f * q + (pad ? 0.f : 1.f);
    }
    std::printf("%d %d %d %d %zu %d\n", ctl.error, started, started_late, (int)wrong, held.size(), missed);
}
"""


@pytest.fixture(scope="module")
def sweep(tmp_path_factory):
    import os
    import subprocess

    from paper_2111_10270_gb300 import build as b

    folder = tmp_path_factory.mktemp("sweep")
    header = open(os.path.join(b.CSRC, "fdog_internal.h")).read()
    abi = header[header.index("// <jit-abi>"):header.index("// </jit-abi>")]
    text = open(os.path.join(b.CSRC, "jit_skeleton.cuh")).read()
    text = text[text.index("#ifdef FDOG_BULK_DISPATCH"):]
    text = text[:text.index("// <ptx>")] + text[text.index("// </ptx>"):text.index('extern "C" __global__')] + "#endif\n"
    src = folder / "sweep.cpp"
    src.write_text(EMULATION.replace("//ABI", abi).replace("//KERNEL", text))
    exe = str(folder / "sweep")
    subprocess.run(["g++", "-std=c++20", "-O1", "-pthread", "-w", str(src), "-o", exe], check=True)

    def run(mode, hold_from=1 << 30, land_late=0, error=0):
        out = subprocess.run([exe, str(mode), str(hold_from), str(land_late), str(error)], capture_output=True, text=True,
                             timeout=60, check=True).stdout.split()
        return dict(zip(("error", "started", "started_late", "wrong", "in_flight", "missed"), map(int, out)))

    return run


@pytest.mark.parametrize("mode", [0, 1])
def test_copy_ahead_reads_every_tile(sweep, mode):
    assert sweep(mode) == {"error": 0, "started": 38, "started_late": 0, "wrong": 0, "in_flight": 0, "missed": 0}


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("hold_from", [0, 9, 10, 30, 37])
def test_a_copy_that_does_not_land_in_time(sweep, mode, hold_from):
    """The pass reports it, starts no further copy, and waits for those on their way before it ends."""
    r = sweep(mode, hold_from, land_late=1)
    assert r["error"] == 1 and r["started_late"] == 0 and r["in_flight"] == 0, r
    r = sweep(mode, hold_from)  # it never lands: every wait ends all the same
    assert r["error"] == 1 and r["started_late"] == 0, r


def test_no_pass_after_an_error(sweep):
    r = sweep(0, error=1)
    assert r["started"] == 0 and r["error"] == 1


@pytest.mark.parametrize("labels,h,w,rows", [(4, 30, 32, 10), (4, 30, 31, 10), (4, 31, 31, 10), (8, 17, 19, 18), (8, 17, 18, 18)])
def test_rows_copied_for_a_partial_last_tile(P, view, labels, h, w, rows):
    """Marginalisation rows of L + 1 layers: L targets and the id of the layer shared with other edges, whether or not
    the edges fill the last tile."""
    inst = planned(P, ilpgen.mrf_grid(h, w, labels, 3), planner=1)
    edges = h * (w - 1) + w * (h - 1)
    v = view(inst)
    assert v["rows"] == rows == (labels + 1) + labels + 1
    tiles = -(-edges * 2 * labels // 32)
    node_tiles = -(-h * w // 32)
    # cv: targets and one id a marginalisation tile; the node rows have no local variable
    assert v["cv_rows"] == tiles * (labels + 1) + node_tiles * labels
