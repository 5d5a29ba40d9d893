"""The library from inside: an instance's plan of bulk sweeps, and calls with a fake allocation.  A few lines of C++
over the internal headers, compiled beside it."""
import ctypes
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cstdlib>
#include "../../include/fastdog.h"
#include "instance.h"
extern "C" void bulk_view(const fdog_instance* inst, long long* v) {
    const fdog::Decomposition& d = inst->dec;
    v[0] = static_cast<long long>(d.bulk_runs.size());
    v[1] = d.bulk_rows;
    v[2] = d.bulk_cv_rows;
    v[3] = inst->batch.bulk.ready;
    std::vector<int> ids;
    for (const auto& s : d.shape_dev)
        if (s.jit >= 0) ids.push_back(s.jit);
    v[4] = fdog::jit_compiled(ids, false);
    v[5] = !ids.empty() && fdog::jit_compiled(ids, true);
}

// one allocation for a planned instance on a device with room for `room` bytes (host memory here); what it took
extern "C" int allocate_with_room(fdog_instance* inst, long long room, long long* bytes) {
    static size_t limit;
    limit = static_cast<size_t>(room);
    const int rc = fdog::allocate_arena(inst, [](void** p, size_t n) {
        if (n > limit) return cudaErrorMemoryAllocation;
        *p = std::calloc(n, 1);
        return cudaSuccess;
    });
    *bytes = rc == FDOG_OK ? static_cast<long long>(inst->arena_bytes) : 0;
    std::free(inst->arena);
    inst->arena = nullptr;
    inst->dev = fdog::DevArrays();
    return rc;
}

// the slots read on a device that has no memory left
extern "C" int read_on_full_device(fdog_instance* inst, int32_t* var, int32_t* row, float* lam) {
    return fdog::read_slots(inst, var, row, inst->dev.lam, lam, nullptr, nullptr,
                            [](void**, size_t) { return cudaErrorMemoryAllocation; });
}
"""


def compile_view(P, folder):
    from paper_2111_10270_gb300 import build as b

    P.lib()
    src, out = os.path.join(folder, "bulk_view.cpp"), os.path.join(folder, "bulk_view.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    cuda = os.path.dirname(os.path.dirname(b.nvcc_path()))
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", src, "-o", out, "-I", b.CSRC, "-I", b.INCLUDE, "-I",
                    os.path.join(cuda, "include"), b.LIB, "-Wl,-rpath," + os.path.dirname(b.LIB)], check=True)
    so = ctypes.CDLL(out)

    def view(inst):
        v = (ctypes.c_longlong * 6)()
        so.bulk_view(inst._h, v)
        return dict(zip(("runs", "rows", "cv_rows", "ready", "compiled", "bulk_compiled"), v))

    view.so = so
    return view
