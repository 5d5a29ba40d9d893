// Slots in the order of the C ABI (tiles in layout order, per tile its BDDs, per
// BDD its layers) read from the interleaved device arrays.
//
// A kernel gathers the asked-for arrays into that order on the device, so that
// the caller's arrays get plain copies.  Copying the padded arrays and walking
// them slot by slot on the host took 5.7 ms for the variables and rows and 2.8
// ms for each value array of 5,484,544 slots, on top of 0.13 ms for the copy
// itself; the gather takes about 16 us an array (it reads and writes 4 bytes a
// slot, the reads of a tile within its own lines).  Up to kFewSlots slots, all
// arrays are gathered by one launch and brought back by one copy, since there
// every launch and copy counts more than the bytes; beyond, one array at a
// time, so that the device holds one listed array only.  On a device without
// room for that one, the padded arrays are copied and listed on the host.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "instance.h"

namespace fdog {

namespace {

constexpr int64_t kFewSlots = 65536;
constexpr int kMaxLists = 4;  // variables, rows and two value arrays

struct SlotArgs {
    const TileDev* tiles;
    const ShapeDev* shapes;
    const int32_t* first;  // first slot of each tile in the listed order
    const int32_t* bdd_row;
    const int32_t* src[kMaxLists];  // padded arrays (32-bit values of any kind); null: the rows of the slots
    int32_t* out;                   // list q of the launch (blockIdx.y) at out + q n_slots
    int32_t n_tiles;
    int32_t n_slots;
};

// a warp per tile, lanes over its slots in the listed order (coalesced writes)
__global__ void __launch_bounds__(256) slot_gather_kernel(SlotArgs a) {
    const int lane = threadIdx.x & 31;
    const int g = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (g >= a.n_tiles) return;
    const TileDev tile = a.tiles[g];
    const int32_t* __restrict__ src = a.src[blockIdx.y];
    const unsigned k = static_cast<unsigned>(a.shapes[tile.shape].k);
    const unsigned n = k * static_cast<unsigned>(tile.n_valid);
    int32_t* __restrict__ out = a.out + static_cast<int64_t>(blockIdx.y) * a.n_slots + a.first[g];
    for (unsigned s = lane; s < n; s += kTile) {
        const unsigned l = s / k, t = s - l * k;
        out[s] = src ? src[tile.slot_base + t * kTile + l] : a.bdd_row[tile.bdd_base + l];
    }
}

// Writes a byte of every page of host memory that is about to be overwritten.
// A copy from the device into pages that the process has not touched yet takes
// their faults one by one from the GPU's side (37 ms for 88 MB, against 2 ms
// into touched ones); host threads take them in parallel.
void touch_pages(void* const* dst, int lists, size_t bytes) {
    constexpr size_t kPage = 4096;
    constexpr int64_t kItems = 64;  // items a page counts for, so that every thread gets some
    const int64_t pages = static_cast<int64_t>(bytes / kPage) + 1;  // the last one also where dst is not aligned
    parallel_chunks(lists * pages * kItems, [&](int64_t b, int64_t e) {
        for (int64_t q = (b + kItems - 1) / kItems; q * kItems < e; ++q) {
            volatile char* const c = static_cast<char*>(dst[q / pages]);
            if (c) c[std::min<size_t>(static_cast<size_t>(q % pages) * kPage, bytes - 1)] = 0;
        }
    });
}

int make_slots(fdog_instance* inst, DeviceAlloc alloc) {
    if (inst->slot_first) return FDOG_OK;
    const Decomposition& d = inst->dec;
    const size_t nt = d.tiles.size(), nb = static_cast<size_t>(d.n_bdds);
    const size_t ns = static_cast<size_t>(d.n_slots) * (d.n_slots <= kFewSlots ? kMaxLists : 1);
    auto up = [](size_t n) { return (std::max<size_t>(n, 1) * sizeof(int32_t) + 255) / 256 * 256; };
    std::vector<int32_t> first;
    try {
        first.resize(nt);
    } catch (const std::bad_alloc&) {
        return FDOG_ENOMEM;
    }
    int32_t at = 0;
    for (size_t t = 0; t < nt; ++t) {
        first[t] = at;
        at += d.tiles[t].n_valid * d.shapes[d.tiles[t].shape].k;
    }
    void* at_dev = nullptr;
    const size_t bytes = up(nt) + up(nb) + up(ns);
    if (alloc(&at_dev, bytes) != cudaSuccess) {
        cudaGetLastError();
        return FDOG_ENOMEM;
    }
    char* const p = static_cast<char*>(at_dev);
    int32_t* const d_first = reinterpret_cast<int32_t*>(p);
    int32_t* const d_row = reinterpret_cast<int32_t*>(p + up(nt));
    // a device-built plan's rows are on the device until a host call downloads the plan; from here on in slot_row
    cudaError_t e = copy_async(inst, d_first, first.data(), sizeof(int32_t) * nt, cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = d.on_device ? cudaMemcpyAsync(d_row, d.d_bdd_row, sizeof(int32_t) * nb, cudaMemcpyDeviceToDevice, inst->stream)
                        : copy_async(inst, d_row, d.bdd_row.data(), sizeof(int32_t) * nb, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaStreamSynchronize(inst->stream);  // `first` goes out of scope
    if (e != cudaSuccess) {
        cudaFree(p);
        return fail_cuda(inst, e, "slot order");
    }
    if (d.on_device) {
        cudaFreeAsync(inst->dec.d_bdd_row, inst->stream);
        inst->dec.d_bdd_row = nullptr;
    }
    inst->slot_first = d_first;
    inst->slot_row = d_row;
    inst->slot_out = reinterpret_cast<int32_t*>(p + up(nt) + up(nb));
    inst->slot_bytes = bytes;
    return FDOG_OK;
}

// The same without device memory.
int read_slots_on_host(fdog_instance* inst, int32_t* var, int32_t* row, const float* const (&dev)[2],
                       float* const (&out)[2]) {
    const int rc = ensure_host_plan(inst);
    if (rc != FDOG_OK) return rc;
    const Decomposition& d = inst->dec;
    // each slot's place in the listed order and in the padded arrays, and its BDD
    auto each = [&](auto&& put) {
        int64_t q = 0;
        for (const TileDev& t : d.tiles) {
            const int k = d.shapes[t.shape].k;
            for (int l = 0; l < t.n_valid; ++l)
                for (int layer = 0; layer < k; ++layer)
                    put(q++, t.slot_base + static_cast<int64_t>(layer) * kTile + l, t.bdd_base + l);
        }
    };
    if (var) each([&](int64_t q, int64_t p, int32_t) { var[q] = d.var[p]; });
    if (row) each([&](int64_t q, int64_t, int32_t b) { row[q] = d.bdd_row[b]; });
    std::vector<float> h;
    for (int a = 0; a < 2; ++a) {
        if (!out[a]) continue;
        try {
            h.resize(static_cast<size_t>(d.slots_pad));
        } catch (const std::bad_alloc&) {
            return FDOG_ENOMEM;
        }
        cudaError_t e = copy_async(inst, h.data(), dev[a], sizeof(float) * h.size(), cudaMemcpyDeviceToHost);
        if (e == cudaSuccess) e = cudaStreamSynchronize(inst->stream);
        if (e != cudaSuccess) return fail_cuda(inst, e, "copy slots");
        each([&](int64_t q, int64_t p, int32_t) { out[a][q] = h[p]; });
    }
    return FDOG_OK;
}

}  // namespace

int read_slots(fdog_instance* inst, int32_t* var, int32_t* row, const float* dev0, float* out0, const float* dev1,
               float* out1, DeviceAlloc alloc) {
    const Decomposition& d = inst->dec;
    if (d.n_slots == 0) return FDOG_OK;
    int rc = make_slots(inst, alloc);
    if (rc == FDOG_ENOMEM) return read_slots_on_host(inst, var, row, {dev0, dev1}, {out0, out1});
    if (rc != FDOG_OK) return rc;
    const int32_t n = static_cast<int32_t>(d.n_slots);
    const size_t bytes = sizeof(int32_t) * static_cast<size_t>(n);
    SlotArgs a{inst->dev.tiles, inst->dev.shapes, inst->slot_first, inst->slot_row, {}, inst->slot_out,
               static_cast<int32_t>(d.tiles.size()), n};
    const void* src[kMaxLists] = {inst->dev.var, nullptr, dev0, dev1};
    void* dst[kMaxLists] = {var, row, out0, out1};
    auto gather = [&](int lists) {
        inst->cfg.count();
        slot_gather_kernel<<<dim3((a.n_tiles + 7) / 8, lists), 256, 0, inst->stream>>>(a);
        return cudaGetLastError();
    };
    cudaError_t e = cudaSuccess;
    if (n <= kFewSlots) {
        int lists = 0;
        for (int q = 0; q < kMaxLists; ++q)
            if (dst[q]) a.src[lists++] = static_cast<const int32_t*>(src[q]);
        std::vector<int32_t> all;
        try {
            all.resize(static_cast<size_t>(lists) * n);
        } catch (const std::bad_alloc&) {
            return FDOG_ENOMEM;
        }
        if (lists > 0) e = gather(lists);
        if (lists > 0 && e == cudaSuccess)
            e = copy_async(inst, all.data(), inst->slot_out, lists * bytes, cudaMemcpyDeviceToHost);
        if (e == cudaSuccess) e = cudaStreamSynchronize(inst->stream);
        const int32_t* from = all.data();
        for (int q = 0; q < kMaxLists && e == cudaSuccess; ++q)
            if (dst[q]) {
                std::memcpy(dst[q], from, bytes);
                from += n;
            }
    } else {
        bool touched = false;
        for (int q = 0; q < kMaxLists && e == cudaSuccess; ++q) {
            if (!dst[q]) continue;
            a.src[0] = static_cast<const int32_t*>(src[q]);
            e = gather(1);
            if (!touched) {  // all arrays at once, while the first gather runs
                touched = true;
                try {
                    touch_pages(dst, kMaxLists, bytes);
                } catch (...) {  // the copies take the faults
                }
            }
            if (e == cudaSuccess) e = copy_async(inst, dst[q], inst->slot_out, bytes, cudaMemcpyDeviceToHost);
        }
        if (e == cudaSuccess) e = cudaStreamSynchronize(inst->stream);
    }
    return e == cudaSuccess ? FDOG_OK : fail_cuda(inst, e, "copy slots");
}

void free_slots(fdog_instance* inst) {
    if (inst->slot_first) cudaFree(inst->slot_first);
    inst->slot_first = inst->slot_row = inst->slot_out = nullptr;
    inst->slot_bytes = 0;
}

}  // namespace fdog
