// Plan and launch of the bulk sweeps (jit_skeleton.cuh) of one instance.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <new>
#include <vector>

#include "instance.h"
#include "kernels.h"
#include "sweep.cuh"

namespace fdog {

namespace {

constexpr int kBulkWarps = 8;
constexpr int kBulkStages = 2;
// The rule for bulk sweeps: three quarters of the tiles plain, and at least this many of them.  200 iterations on grids,
// ms, ordinary and bulk sweeps: 4 labels, 0.27 k tiles 3.13 and 3.07, 2.1 k 4.11 and 3.75, 8.6 k 5.10 and 4.81, 19 k 6.85
// and 5.94, 48 k 12.1 and 10.1; 8 labels, 0.31 k tiles 3.50 and 3.33, 4.2 k 5.65 and 4.48.  Rows of three layers (2
// labels) leave little to form from a copied tile: 4.8 k tiles 4.11 and 3.99, 11 k 4.87 and 4.91, 25 k 6.56 and 6.21,
// 37 k 7.91 and 7.58, 74 k 12.9 and 11.7.  With 3 labels the edges that a tile's end cuts make every tile a mixed one,
// whose slots all need ids and whose layers take both ways: 16 k tiles 6.32 and 6.43, 65 k 14.4 and 15.4 (and once 26).
// So they do with 5 to 7 labels, where the longer rows can pay for it (9.8 k tiles of 5 labels 5.63 and 5.69, 26 k 9.65
// and 8.89; 7.8 k of 6 labels 6.05 and 5.66): the rule leaves them on the ordinary sweeps.  Other families of this
// repository have no tile-local variables in regular tiles.
constexpr int32_t kBulkMinTiles = 256, kBulkMinShortTiles = 16384;
constexpr int64_t kBulkMaxPatterns = 64;  // a tile's table entry has 8 bits for its pattern; more would be large tables

size_t smem_of(int stages, int rows) {
    return sizeof(float) * kTile * kBulkWarps * FDOG_BULK_WARP_ROWS(stages, rows);
}

// Targets and ids of the tiles of the members that run bulk sweeps (InstDev::cv), a warp per tile: the targets after
// every change of C, the ids with them (they never change).
__global__ void __launch_bounds__(256) bulk_targets_kernel(const InstDev* insts, const int32_t* prefix, int n_inst,
                                                           int total) {
    const int lane = threadIdx.x & 31;
    const int warps = (gridDim.x * blockDim.x) >> 5;
    for (int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < total; w += warps) {
        const int ii = dev::find_inst_warp(prefix, n_inst, w, lane);
        const InstDev* __restrict__ I = insts + ii;
        const int g = w - __ldg(prefix + ii) - I->bulk_first;
        if (!I->cv || g < 0 || g >= I->bulk_tiles) continue;
        int q = I->n_bulk_runs - 1;
        while (q > 0 && I->bulk_runs[q].tile > g) --q;
        const BulkRun r = I->bulk_runs[q];
        const int j = g - r.tile;
        const int32_t* __restrict__ var = I->var + r.slot_base + j * r.k * kTile + lane;
        float* __restrict__ out = I->cv + static_cast<size_t>(r.cv_row + j * (r.c_n + r.v_n)) * kTile + lane;
        for (int t = 0; t < r.c_n; ++t) {
            const int v = var[(r.c_lo + t) * kTile];
            out[t * kTile] = v >= 0 ? I->C[v] : 0.f;
        }
        for (int t = 0; t < r.v_n; ++t) out[(r.c_n + t) * kTile] = __int_as_float(var[(r.v_lo + t) * kTile]);
    }
}

}  // namespace

bool bulk_possible(const Decomposition& d) {
    const int64_t np = static_cast<int64_t>(d.patterns.size() / 2);
    const int32_t t0 = d.cls_tile_begin[kJitClass], n = d.cls_tile_begin[kJitClass + 1] - t0;
    if (np < 1 || np > kBulkMaxPatterns || !d.cls_has_local[kJitClass] || n < kBulkMinTiles) return false;
    if (n < kBulkMinShortTiles) {
        int64_t layers = 0;
        for (int32_t t = 0; t < n; ++t) layers += d.shapes[d.tiles[t0 + t].shape].k;
        if (2 * layers < 9 * static_cast<int64_t>(n)) return false;  // fewer than 4.5 a row
    }
    int shapes = 0;
    for (int c : d.shape_cls) shapes += c == kJitClass;
    return shapes <= FDOG_BULK_RUNS;
}

// Without memory for it the instance runs the ordinary sweeps.
void plan_bulk(Decomposition& d, const uint16_t* local_ent) try {
    d.bulk_planned = true;
    d.bulk_runs.clear();
    d.bulk_pairs.clear();
    const size_t np = d.patterns.size() / 2;
    std::vector<uint32_t> pairs(np * 257, 0xFFFFFFFFu), rest(np * kEpiMaxK, 0xFFFFFFFFu);
    auto set = [&](size_t p, uint32_t at, uint32_t value) {
        uint32_t& w = pairs[(p * 8 + at / kTile / 2) * kTile + at % kTile];
        const int shift = at / kTile % 2 ? 16 : 0;
        w = (w & ~(0xFFFFu << shift)) | value << shift;
        rest[p * kEpiMaxK + at / kTile] &= ~(1u << at % kTile);
    };
    for (size_t p = 0; p < np; ++p) {
        bool pairs_only = true;
        for (int32_t e = 0; e < d.patterns[2 * p + 1]; ++e) {
            const uint16_t* o = local_ent + 4 * (static_cast<size_t>(d.patterns[2 * p]) + e);
            if (o[2] != 0xFFFFu) return;  // a variable with more than two copies
            if (o[1] != 0xFFFFu) {
                set(p, o[0], o[1] * 4u);
                set(p, o[1], o[0] * 4u);
            } else {
                set(p, o[0], FDOG_PAIR_ONE);
                pairs_only = false;
            }
        }
        uint32_t local = 0;
        for (int l = 0; l < kEpiMaxK; ++l) {
            const uint32_t m = rest[p * kEpiMaxK + l];
            if (m == 0u) local |= 1u << l;
            else if (m != 0xFFFFFFFFu) pairs_only = false;
        }
        pairs[np * 256 + p] = pairs_only ? FDOG_PAIR_PLAIN | local : 0u;
    }
    // runs, and the layers whose targets or ids some tile of the run needs
    const int32_t t0 = d.cls_tile_begin[kJitClass], t1 = d.cls_tile_begin[kJitClass + 1];
    int64_t row = 0;
    int rows = 0;
    for (int32_t t = t0; t < t1;) {
        const int shape = d.tiles[t].shape, k = d.shapes[shape].k;
        BulkRun r{};
        r.tile = t - t0;
        r.slot_base = d.tiles[t].slot_base;
        r.k = k;
        r.jit = d.shape_dev[shape].jit;
        uint32_t local = 0, other = 0;  // layers
        std::vector<uint8_t> seen(np + 1, 0);
        for (; t < t1 && d.tiles[t].shape == shape; ++t) {
            const int p = d.tiles[t].pattern, valid = d.tiles[t].n_valid;
            r.n_bdds += valid;
            if (valid == kTile) {
                if (seen[p + 1]) continue;
                seen[p + 1] = 1;
            }
            // lanes without a BDD, in a run's last tile, need neither
            const uint32_t lanes = valid == kTile ? 0xFFFFFFFFu : (1u << valid) - 1u;
            for (int l = 0; l < k; ++l) {
                const uint32_t m = p < 0 ? 0xFFFFFFFFu : rest[static_cast<size_t>(p) * kEpiMaxK + l];
                if (m & lanes) other |= 1u << l;
                if (~m & lanes) local |= 1u << l;
            }
        }
        auto range = [&](uint32_t m, int32_t& lo, int32_t& n) {
            lo = n = 0;
            for (int l = 0; l < k; ++l)
                if (m >> l & 1u) {
                    if (n == 0) lo = l;
                    n = l + 1 - lo;
                }
        };
        range(local, r.c_lo, r.c_n);
        range(other, r.v_lo, r.v_n);
        if (r.jit >= 1 << 22 || row > (int64_t(1) << 25)) {  // beyond a table entry
            d.bulk_runs.clear();
            return;
        }
        r.cv_row = static_cast<int32_t>(row);
        row += static_cast<int64_t>(t - t0 - r.tile) * (r.c_n + r.v_n);
        rows = std::max(rows, r.k + r.c_n + r.v_n);
        d.bulk_runs.push_back(r);
    }
    int64_t plain = 0;
    for (int32_t t = t0; t < t1; ++t)
        plain += d.tiles[t].pattern < 0 || pairs[np * 256 + d.tiles[t].pattern] != 0u;
    // cv is addressed in 32 bits
    if (row > (int64_t(1) << 25) || 4 * plain < 3 * static_cast<int64_t>(t1 - t0)) {
        d.bulk_runs.clear();
        return;
    }
    d.bulk_rows = rows;
    d.bulk_cv_rows = row;
    d.bulk_pairs = std::move(pairs);
} catch (const std::bad_alloc&) {
    d.bulk_runs.clear();
}

std::vector<int> bulk_ids(const fdog_instance* inst) {
    std::vector<int> ids;
    if (bulk_wanted(inst))
        for (const BulkRun& r : inst->dec.bulk_runs) ids.push_back(r.jit);
    return ids;
}

int setup_bulk(fdog_instance* inst) {
    BulkPlan& plan = inst->batch.bulk;
    plan = BulkPlan();
    const Decomposition& d = inst->dec;
    if (!inst->hdesc.cv) return FDOG_OK;
    const DevArrays& a = inst->dev;
    cudaError_t e = copy_async(inst, a.bulk_runs, d.bulk_runs.data(), sizeof(BulkRun) * d.bulk_runs.size(),
                               cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = copy_async(inst, a.bulk_pairs, d.bulk_pairs.data(), sizeof(uint32_t) * d.bulk_pairs.size(),
                       cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return fail_cuda(inst, e, "bulk sweep plan");
    plan.args = BulkArgs{a.inst, a.bulk_pairs, static_cast<int32_t>(d.patterns.size() / 2),
                         d.cls_tile_begin[kJitClass + 1] - d.cls_tile_begin[kJitClass], d.bulk_rows, kBulkStages};
    const size_t smem = smem_of(kBulkStages, d.bulk_rows);
    int most = 1 << 30;
    for (int m = 0; m < 2; ++m) {
        int n = 0;
        plan.fn[m] = inst->bulk_jit.fn[m];
        if (allow_smem(plan.fn[m], smem) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, plan.fn[m], 32 * kBulkWarps, smem) != cudaSuccess) {
            cudaGetLastError();
            n = 0;
        }
        most = std::min(most, n);
    }
    plan.blocks_per_sm = most;
    plan.ready = most > 0;
    return FDOG_OK;
}

cudaError_t launch_bulk(const DevBatch& b, int mode, const LaunchCfg& cfg, cudaStream_t s) {
    BulkArgs args = b.bulk.args;
    args.inst = b.insts;
    const size_t smem = smem_of(args.stages, args.rows);
    const void* fn = b.bulk.fn[mode];
    const cudaError_t e = allow_smem(fn, smem);
    if (e != cudaSuccess) return e;
    const int blocks = std::min(b.bulk.blocks_per_sm * cfg.num_sms, (args.total + kBulkWarps - 1) / kBulkWarps);
    void* kargs[] = {&args};
    return launch_windowed(fn, blocks, 32 * kBulkWarps, kargs, smem, s, b.l2);
}

cudaError_t launch_bulk_targets(const DevBatch& b, const LaunchCfg& cfg, cudaStream_t s) {
    if (!b.any_cv || b.tiles_all_total == 0) return cudaSuccess;
    cfg.count();
    const int blocks = std::min((b.tiles_all_total + 7) / 8, cfg.num_sms * 8);
    bulk_targets_kernel<<<blocks, 256, 0, s>>>(b.insts, b.tile_all_prefix, b.n_inst, b.tiles_all_total);
    return cudaGetLastError();
}

}  // namespace fdog
