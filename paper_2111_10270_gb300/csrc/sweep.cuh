// Sweep kernel template (included by the per-width translation units).
//
// One warp per tile of 32 BDDs of one shape, one thread per BDD.  All
// per-layer loads/stores of a warp are single 128-byte transactions
// (interleaved slots); the shape template is read with warp-uniform loads.
// Shortest-path labels of the direction opposite to the pass are recomputed
// on chip at the start of each pass, so no per-node state goes to HBM: the
// per-slot multipliers are the only state the sweeps stream.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "kernels.h"

namespace fdog {
namespace dev {

// Programmatic dependent launch.  The iteration kernels are launched with
// programmatic stream serialization: a kernel may be scheduled while the one
// before it on its stream drains.  pdl_wait() returns once that kernel has
// completed and its writes are visible (at once for a launch without the
// attribute), so every such kernel calls it before it touches memory;
// pdl_trigger() lets the next kernel be scheduled once every block of this
// one has started.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ float finf() { return __int_as_float(0x7f800000); }

// largest instance index i with prefix[i] <= g (empty instances are skipped)
__device__ __forceinline__ int find_inst(const int32_t* __restrict__ prefix, int n, int g) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(prefix + mid) <= g) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// The same by a whole warp, g the same in every lane: one load for up to 32
// instances instead of one after the other.
__device__ __forceinline__ int find_inst_warp(const int32_t* __restrict__ prefix, int n, int g, int lane) {
    if (n == 1) return 0;
    int at = 0;
    for (int b = 0; b < n; b += 32) {
        const unsigned m = __ballot_sync(kFull, b + lane < n && __ldg(prefix + b + lane) <= g);
        at += __popc(m);
        if (m != kFull) break;
    }
    return at - 1;
}

template <int W>
__device__ __forceinline__ void load_codes(const uint16_t* __restrict__ p, uint32_t (&c)[W]) {
    if constexpr (W == 2) {
        const uint32_t u = __ldg(reinterpret_cast<const unsigned int*>(p));
        c[0] = u & 0xFFFFu; c[1] = u >> 16;
    } else if constexpr (W == 4) {
        const uint2 u = __ldg(reinterpret_cast<const uint2*>(p));
        c[0] = u.x & 0xFFFFu; c[1] = u.x >> 16; c[2] = u.y & 0xFFFFu; c[3] = u.y >> 16;
    } else {
#pragma unroll
        for (int q = 0; q < W / 8; ++q) {
            const uint4 u = __ldg(reinterpret_cast<const uint4*>(p) + q);
            c[8 * q + 0] = u.x & 0xFFFFu; c[8 * q + 1] = u.x >> 16;
            c[8 * q + 2] = u.y & 0xFFFFu; c[8 * q + 3] = u.y >> 16;
            c[8 * q + 4] = u.z & 0xFFFFu; c[8 * q + 5] = u.z >> 16;
            c[8 * q + 6] = u.w & 0xFFFFu; c[8 * q + 7] = u.w >> 16;
        }
    }
}

// label of the successor with the given code: a node of the next layer, TOP (0) or BOT (inf)
template <int W>
__device__ __forceinline__ float pick(const float (&x)[W], uint32_t code) {
    float r = (code == kCodeTop) ? 0.f : finf();
#pragma unroll
    for (int w = 0; w < W; ++w) r = (code == static_cast<uint32_t>(w)) ? x[w] : r;
    return r;
}

template <int W>
__device__ __forceinline__ void push(float (&x)[W], uint32_t code, float val) {
#pragma unroll
    for (int w = 0; w < W; ++w)
        if (code == static_cast<uint32_t>(w)) x[w] = fminf(x[w], val);
}

// Codes of one layer, two arcs (lo | hi << 8) to a word.
template <int W>
struct LayerCodes {
    uint32_t w[W / 2];
    __device__ __forceinline__ uint32_t lo(int v) const { return (w[v / 2] >> (16 * (v % 2))) & 0xFFu; }
    __device__ __forceinline__ uint32_t hi(int v) const { return (w[v / 2] >> (16 * (v % 2) + 8)) & 0xFFu; }
};

// Codes of the kRegK layers from layer t0 on (a multiple of kRegK), all loads
// issued together: templates start on 16 bytes and a layer takes 2 W bytes.
// Beyond the shape's last layer the words are whatever follows it in memory
// (the template array has room for them) and are not used.
template <int W>
__device__ __forceinline__ void load_segment_codes(const uint16_t* __restrict__ tpl, int t0, LayerCodes<W> (&c)[kRegK]) {
    const uint4* __restrict__ p = reinterpret_cast<const uint4*>(tpl + static_cast<size_t>(t0) * W);
#pragma unroll
    for (int q = 0; q < kRegK * W / 8; ++q) {
        const uint4 u = __ldg(p + q);
        const uint32_t x[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) c[(4 * q + j) / (W / 2)].w[(4 * q + j) % (W / 2)] = x[j];
    }
}

// Inner layers of 0/1 rows have one of two width-2 structures, equal up to
// the order of the nodes: one node that may still take a 1 (which leads to
// the other) and one that may not.  Most layers of matching, flow and
// marginalisation rows are these; they take a handful of instructions where
// the general step selects every successor among four.  The code is the same
// for the whole warp, so the choice costs one uniform branch.
constexpr uint32_t kStepUp = 0xFF010100u;    // node 0: 0 -> 0, 1 -> 1; node 1: 0 -> 1, 1 -> BOT
constexpr uint32_t kStepDown = 0x0001FF00u;  // node 0: 0 -> 0, 1 -> BOT; node 1: 0 -> 1, 1 -> 0

// labels SP(v, TOP) of a layer from those of the next one (Alg. 4)
template <int W>
__device__ __forceinline__ void pull_labels(float (&x)[W], const LayerCodes<W>& c, float l) {
    if (W == 2 && c.w[0] == kStepUp) {
        x[0] = fminf(x[0], x[1] + l);
    } else if (W == 2 && c.w[0] == kStepDown) {
        x[1] = fminf(x[1], x[0] + l);
    } else {
        float cur[W];
#pragma unroll
        for (int v = 0; v < W; ++v) cur[v] = fminf(pick<W>(x, c.lo(v)), pick<W>(x, c.hi(v)) + l);
#pragma unroll
        for (int v = 0; v < W; ++v) x[v] = cur[v];
    }
}

// labels SP(r, v) of the next layer from those of this one (Alg. 3)
template <int W>
__device__ __forceinline__ void push_labels(float (&x)[W], const LayerCodes<W>& c, float l) {
    if (W == 2 && c.w[0] == kStepUp) {
        x[1] = fminf(x[0] + l, x[1]);
    } else if (W == 2 && c.w[0] == kStepDown) {
        x[0] = fminf(x[0], x[1] + l);
    } else {
        float nx[W];
#pragma unroll
        for (int v = 0; v < W; ++v) nx[v] = finf();
#pragma unroll
        for (int v = 0; v < W; ++v) {
            push<W>(nx, c.lo(v), x[v]);
            push<W>(nx, c.hi(v), x[v] + l);
        }
#pragma unroll
        for (int v = 0; v < W; ++v) x[v] = nx[v];
    }
}

// Eq. 6 of a layer without the layer's own multiplier in m1: f its labels
// SP(r, .), b the next layer's SP(., TOP)
template <int W>
__device__ __forceinline__ void layer_marginals(const float (&f)[W], const float (&b)[W], const LayerCodes<W>& c,
                                                float& m0, float& m1) {
    if (W == 2 && c.w[0] == kStepUp) {
        m0 = fminf(f[0] + b[0], f[1] + b[1]);
        m1 = f[0] + b[1];
    } else if (W == 2 && c.w[0] == kStepDown) {
        m0 = fminf(f[0] + b[0], f[1] + b[1]);
        m1 = f[1] + b[0];
    } else {
        m0 = finf();
        m1 = finf();
#pragma unroll
        for (int v = 0; v < W; ++v) {
            m0 = fminf(m0, f[v] + pick<W>(b, c.lo(v)));
            m1 = fminf(m1, f[v] + pick<W>(b, c.hi(v)));
        }
    }
}

// 1 / c rounded to FP32 for a copy count c <= 8 (constants folded at compile
// time); the deferred term of a variable is (C_i - sum_j lambda^j_i) times it
// in every kernel that forms one, so all of them agree bit for bit
__device__ __forceinline__ float inv_copies(int c) {
    return c == 1 ? 1.f : c == 2 ? 0.5f : c == 3 ? 1.f / 3.f : c == 4 ? 0.25f
         : c == 5 ? 1.f / 5.f : c == 6 ? 1.f / 6.f : c == 7 ? 1.f / 7.f : 0.125f;
}

// Deferred terms of the tile-local variables (every copy in this tile),
// formed right after the pass from the staged multipliers: the same sum, in
// the same ascending slot order, as the deferred-sum kernel uses.
// ep_lam / ep_var: this warp's staging, layer t lane l at [32 t + l].
__device__ __forceinline__ void tile_local_sums(const InstDev* __restrict__ I, int pattern, const float* ep_lam,
                                                const int* ep_var, int lane) {
    const int2 pat = reinterpret_cast<const int2*>(I->patterns)[pattern];
    for (int e = lane; e < pat.y; e += 32) {
        const ushort4 o = reinterpret_cast<const ushort4*>(I->local_ent)[pat.x + e];
        float s = 0.f + ep_lam[o.x];
        int c = 1;
        if (o.y != 0xFFFFu) { s += ep_lam[o.y]; ++c; }
        if (o.z != 0xFFFFu) { s += ep_lam[o.z]; ++c; }
        if (o.w != 0xFFFFu) { s += ep_lam[o.w]; ++c; }
        const int v = ep_var[o.x];
        I->T[v] = (I->C[v] - s) * inv_copies(c);
    }
}

// L2 prefetch of the multiplier and variable rows of the tile this warp
// visits next (lane t takes layer t), issued before the current tile is
// computed so that the next tile's first loads hit L2.
__device__ __forceinline__ void prefetch_tile(const SweepArgs& a, int g, int lane) {
    if (g >= a.total) return;
    const int ii = find_inst_warp(a.prefix, a.n_inst, g, lane);
    const InstDev* __restrict__ I = a.insts + ii;
    const TileDev tile = I->tiles[__ldg(a.first + ii) + (g - __ldg(a.prefix + ii))];
    const int k = I->shapes[tile.shape].k;
    for (int t = lane; t < k; t += kTile) {
        const long long p = static_cast<long long>(tile.slot_base) + static_cast<long long>(kTile) * t;
        asm volatile("prefetch.global.L2 [%0];" ::"l"(I->lam + p));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(I->var + p));
    }
}

// Loops over the layers of a register-held BDD.  The trip count is the
// constant kRegK and the loops unroll completely, so every index is a
// compile-time constant and the arrays stay in registers.
#define FD_UP(t) _Pragma("unroll") for (int t = 0; t < kRegK; ++t) if (t < k)
#define FD_DOWN(t) _Pragma("unroll") for (int t = kRegK - 1; t >= 0; --t) if (t < k)

// compensated FP32 butterfly of the lanes' shares of the bound (all lanes end equal)
__device__ __forceinline__ float2 tile_bound(float s) {
    float comp = 0.f;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const float o = __shfl_xor_sync(kFull, s, off);
        const float oc = __shfl_xor_sync(kFull, comp, off);
        const float sum = s + o;
        const float bp = sum - s;
        const float err = (s - (sum - bp)) + (o - bp);
        s = sum;
        comp = comp + oc + err;
    }
    return make_float2(s, comp);
}

// shared-memory floats one warp of reg_tile uses
__host__ __device__ __forceinline__ size_t reg_warp_floats(const SweepArgs& a) {
    return static_cast<size_t>(a.epi) * kTile * 2;
}

// Short rows (at most kRegK layers) of narrow BDDs (W <= kRegW): everything in
// registers.  One tile g of a class (lane = BDD), the warp's shared memory at
// wsm; the tile this warp visits next (g_next, if below a.total) is
// prefetched into L2.  A lone instance has about one tile per warp, so the
// kernel's time is its chain of dependent loads: the codes of all layers, the
// multipliers and the variable ids are each loaded at once, then all terms T
// (interleaved layer by layer, every layer waited for its own id before the
// next one's loads were issued).
template <int W, int MODE>
__device__ __forceinline__ void reg_tile(const SweepArgs& a, int g, int g_next, float* wsm, int lane) {
    constexpr bool update = MODE == kFwdUpdate || MODE == kBwdUpdate;
    prefetch_tile(a, g_next, lane);
    const int ii = find_inst_warp(a.prefix, a.n_inst, g, lane);
    const InstDev* __restrict__ I = a.insts + ii;
    if (update && FDOG_INACTIVE(I->ctl)) return;  // stopped, or out of iterations
    const int ti = __ldg(a.first + ii) + (g - __ldg(a.prefix + ii));
    const TileDev tile = I->tiles[ti];
    const ShapeDev sh = I->shapes[tile.shape];
    const int k = sh.k;
    const bool valid = lane < tile.n_valid;
    const float omega = I->omega;
    const size_t base = static_cast<size_t>(tile.slot_base) + lane;
    float* __restrict__ lam = I->lam;
    float* ep_lam = wsm;
    int* ep_var = reinterpret_cast<int*>(ep_lam + static_cast<size_t>(a.epi) * kTile);
    const bool local = update && a.epi > 0 && tile.pattern >= 0;

    // padding lanes hold multiplier 0 and variable -1
    LayerCodes<W> c[kRegK];
    load_segment_codes<W>(I->tpl + sh.tpl_off, 0, c);
    float L[kRegK], T[kRegK], S[kRegK][W];
    int V[kRegK];
    FD_UP(t) L[t] = lam[base + static_cast<size_t>(t) * kTile];
    if constexpr (update) {
        FD_UP(t) V[t] = __ldcs(I->var + base + static_cast<size_t>(t) * kTile);  // streamed once per pass
        const float* Tv = I->T;
        FD_UP(t) T[t] = V[t] >= 0 ? Tv[V[t]] : 0.f;
        if (local) {
            FD_UP(t) ep_var[t * kTile + lane] = V[t];
        }
    }

    float term = 0.f;  // this BDD's share of the lower bound
    float x[W];        // the running labels
    if constexpr (MODE == kFwdUpdate || MODE == kMinMarg || MODE == kEval) {
        // SP(v, TOP) of every node at the current multipliers (Alg. 4 without updates);
        // S[t] the labels of layer t + 1 (the last layer's arcs lead to terminals: unused)
#pragma unroll
        for (int v = 0; v < W; ++v) x[v] = finf();
        FD_DOWN(t) {
#pragma unroll
            for (int v = 0; v < W; ++v) S[t][v] = x[v];
            pull_labels<W>(x, c[t], L[t]);
        }
        if constexpr (MODE == kEval) term = x[0];
    } else {
        // SP(r, v) of every node at the current multipliers (Alg. 3 without updates)
#pragma unroll
        for (int v = 0; v < W; ++v) x[v] = v == 0 ? 0.f : finf();
        FD_UP(t) {
#pragma unroll
            for (int v = 0; v < W; ++v) S[t][v] = x[v];
            push_labels<W>(x, c[t], L[t]);
        }
    }

    if constexpr (MODE == kFwdUpdate || MODE == kMinMarg) {
        // ascending pass: SP(r, .) incrementally (Alg. 3) and Eq. 6 per layer
#pragma unroll
        for (int v = 0; v < W; ++v) x[v] = v == 0 ? 0.f : finf();
        float* __restrict__ mm0 = I->mm0;
        float* __restrict__ mm1 = I->mm1;
        FD_UP(t) {
            float m0, m1;
            layer_marginals<W>(x, S[t], c[t], m0, m1);
            m1 += L[t];
            if constexpr (MODE == kFwdUpdate) {
                L[t] = fmaf(-omega, m1 - m0, L[t]) + T[t];  // Eq. 5
            } else if (valid) {
                const size_t p = base + static_cast<size_t>(t) * kTile;
                if (a.flags & kMMBoth) { mm0[p] = m0; mm1[p] = m1; }
                else mm0[p] = m1 - m0;
            }
            push_labels<W>(x, c[t], L[t]);
        }
    }

    if constexpr (MODE == kBwdUpdate) {
        // descending pass: SP(., TOP) incrementally (Alg. 4) and Eq. 6 per layer
#pragma unroll
        for (int v = 0; v < W; ++v) x[v] = finf();
        float negsum = 0.f;
        FD_DOWN(t) {
            float m0, m1;
            layer_marginals<W>(S[t], x, c[t], m0, m1);
            m1 += L[t];
            const float d = m1 - m0;
            L[t] = fmaf(-omega, d, L[t]) + T[t];  // Eq. 5
            negsum += fmaxf(-d, 0.f);
            pull_labels<W>(x, c[t], L[t]);
        }
        term = fmaf(-omega, negsum, x[0]);
    }

    if constexpr (update) {
        if (valid) {
            FD_UP(t) lam[base + static_cast<size_t>(t) * kTile] = L[t];
        }
        if (local) {
            FD_UP(t) ep_lam[t * kTile + lane] = L[t];
            __syncwarp();
            tile_local_sums(I, tile.pattern, ep_lam, ep_var, lane);
            __syncwarp();
        }
    }
    // only the descending update pass and the energy sweep feed a bound reduction
    if constexpr (MODE == kBwdUpdate || MODE == kEval) {
        const float2 p = tile_bound(valid ? term : 0.f);
        if (lane == 0) I->tile_lb[ti] = p;
    }
}

// Wide BDDs (W > kRegW): per-layer state in shared memory, one column per lane
// (so no bank conflicts), rows of 32 floats: the multipliers and terms of
// every layer, one row per node for the stored labels (a.nodes: most nodes of
// a shape of the launch), two layers of running labels and two constant rows
// for the terminals.  A layer's nodes are visited one by one up to the number
// it has, and a successor's label is read from the row its code names, the
// same for the whole warp.  Holding all W labels in registers and selecting
// among them for every arc took some 500 selects per layer at W = 16 whatever
// its nodes (99 us a sweep of 368 tiles of at most 12 layers).
// shared-memory floats one warp of wide_tile uses
template <int W>
__host__ __device__ __forceinline__ size_t wide_warp_floats(const SweepArgs& a) {
    return (static_cast<size_t>(a.kstride) * 2 + a.nodes + 2 * W + 2) * kTile + static_cast<size_t>(a.epi) * kTile * 2;
}

template <int W, int MODE>
__device__ __forceinline__ void wide_tile(const SweepArgs& a, int g, int g_next, float* wsm, int lane) {
    constexpr bool update = MODE == kFwdUpdate || MODE == kBwdUpdate;
    constexpr bool asc = MODE != kBwdUpdate;  // labels SP(., TOP) first, then the layers in ascending order
    prefetch_tile(a, g_next, lane);
    const int ii = find_inst_warp(a.prefix, a.n_inst, g, lane);
    const InstDev* __restrict__ I = a.insts + ii;
    if (update && FDOG_INACTIVE(I->ctl)) return;
    const int ti = __ldg(a.first + ii) + (g - __ldg(a.prefix + ii));
    const TileDev tile = I->tiles[ti];
    const ShapeDev sh = I->shapes[tile.shape];
    const int k = sh.k;
    const uint16_t* __restrict__ tpl = I->tpl + sh.tpl_off;
    const bool valid = lane < tile.n_valid;
    const float omega = I->omega;
    const size_t base = static_cast<size_t>(tile.slot_base) + lane;
    float* __restrict__ lam = I->lam;
    const bool local = update && a.epi > 0 && tile.pattern >= 0;

    float* Lr = wsm + lane;                                   // multipliers, row t
    float* Tr = Lr + static_cast<size_t>(a.kstride) * kTile;  // terms, row t
    float* X = Tr + static_cast<size_t>(a.kstride) * kTile;   // TOP (0), BOT (inf)
    float* R0 = X + 2 * kTile;                                // running labels of two neighbouring layers
    float* S = R0 + 2 * W * kTile;                            // stored labels, layer after layer as they are formed
    float* ep_lam = wsm + (static_cast<size_t>(a.kstride) * 2 + a.nodes + 2 * W + 2) * kTile;
    int* ep_var = reinterpret_cast<int*>(ep_lam + static_cast<size_t>(a.epi) * kTile);

    // codes of layer t: lane v < W holds node v's; padding nodes have code 0xFFFF
    auto codes_of = [&](int t) -> uint32_t { return lane < W && t >= 0 && t < k ? __ldg(tpl + t * W + lane) : 0xFFFFu; };
    auto count_of = [&](uint32_t c) { return __popc(__ballot_sync(kFull, c != 0xFFFFu)); };
    // row of a successor: a node of the layer at `next`, or a terminal's constant row
    auto row_of = [&](float* next, uint32_t code) -> float* {
        return code < kCodeTop ? next + code * kTile : X + (code - kCodeTop) * kTile;
    };

    X[0] = 0.f;
    X[kTile] = finf();
#pragma unroll 4
    for (int t = 0; t < k; ++t) {
        const size_t p = base + static_cast<size_t>(t) * kTile;
        Lr[t * kTile] = lam[p];
        if (update) Tr[t * kTile] = __int_as_float(__ldcs(I->var + p));  // streamed once per pass
    }
    if constexpr (update) {
        const float* Tv = I->T;
        if (local)
            for (int t = 0; t < k; ++t) ep_var[t * kTile + lane] = __float_as_int(Tr[t * kTile]);
#pragma unroll 4
        for (int t = 0; t < k; ++t) {
            const int v = __float_as_int(Tr[t * kTile]);
            Tr[t * kTile] = v >= 0 ? Tv[v] : 0.f;
        }
    }

    // labels of the direction opposite to the pass, at the current multipliers.
    // asc: SP(v, TOP), from the last layer (Alg. 4); each layer's rows follow the next layer's.
    // else: SP(r, v), from the root (Alg. 3); each layer's rows follow the one before.
    float* at = S;  // rows of the layer last completed
    float term = 0.f;
    {
        uint32_t c = codes_of(asc ? k - 1 : 0);
        int n = count_of(c);
        if constexpr (asc) {
            float* next = X;  // the last layer has terminal codes only
            for (int t = k - 1; t >= 0; --t) {
                const uint32_t cp = codes_of(t - 1);  // in flight while this layer is formed
                const float lt = Lr[t * kTile];
                for (int v = 0; v < n; ++v) {
                    const uint32_t cv = __shfl_sync(kFull, c, v);
                    at[v * kTile] = fminf(*row_of(next, cv & 0xFFu), *row_of(next, cv >> 8) + lt);
                }
                next = at;
                at += n * kTile;
                c = cp;
                n = count_of(c);
            }
            at = next;  // layer 0
            if constexpr (MODE == kEval) term = at[0];
        } else {
            at[0] = 0.f;
            for (int t = 0; t + 1 < k; ++t) {
                const uint32_t cn = codes_of(t + 1);
                const int nn = count_of(cn);
                float* next = at + n * kTile;
                for (int v = 0; v < nn; ++v) next[v * kTile] = finf();
                const float lt = Lr[t * kTile];
                for (int v = 0; v < n; ++v) {
                    const uint32_t cv = __shfl_sync(kFull, c, v);
                    const uint32_t lo = cv & 0xFFu, hi = cv >> 8;
                    const float f = at[v * kTile];
                    if (lo < kCodeTop) next[lo * kTile] = fminf(next[lo * kTile], f);
                    if (hi < kCodeTop) next[hi * kTile] = fminf(next[hi * kTile], f + lt);
                }
                at = next;
                c = cn;
                n = nn;
            }
        }
    }

    if constexpr (MODE == kFwdUpdate || MODE == kMinMarg) {
        // ascending pass: SP(r, .) incrementally (Alg. 3) and Eq. 6 per layer
        float* f = R0;
        float* fn = R0 + W * kTile;
        f[0] = 0.f;
        float* __restrict__ mm0 = I->mm0;
        float* __restrict__ mm1 = I->mm1;
        uint32_t c = codes_of(0);
        int n = count_of(c);
        for (int t = 0; t < k; ++t) {
            const uint32_t cn = codes_of(t + 1);
            const int nn = count_of(cn);
            float* next = at - nn * kTile;  // SP(., TOP) of layer t + 1
            float m0 = finf(), m1 = finf();
            for (int v = 0; v < n; ++v) {
                const uint32_t cv = __shfl_sync(kFull, c, v);
                const float fv = f[v * kTile];
                m0 = fminf(m0, fv + *row_of(next, cv & 0xFFu));
                m1 = fminf(m1, fv + *row_of(next, cv >> 8));
            }
            float lt = Lr[t * kTile];
            m1 += lt;
            if constexpr (MODE == kFwdUpdate) {
                lt = fmaf(-omega, m1 - m0, lt) + Tr[t * kTile];  // Eq. 5
                Lr[t * kTile] = lt;
            } else if (valid) {
                const size_t p = base + static_cast<size_t>(t) * kTile;
                if (a.flags & kMMBoth) { mm0[p] = m0; mm1[p] = m1; }
                else mm0[p] = m1 - m0;
            }
            for (int v = 0; v < nn; ++v) fn[v * kTile] = finf();
            for (int v = 0; v < n; ++v) {
                const uint32_t cv = __shfl_sync(kFull, c, v);
                const uint32_t lo = cv & 0xFFu, hi = cv >> 8;
                const float fv = f[v * kTile];
                if (lo < kCodeTop) fn[lo * kTile] = fminf(fn[lo * kTile], fv);
                if (hi < kCodeTop) fn[hi * kTile] = fminf(fn[hi * kTile], fv + lt);
            }
            float* h = f;
            f = fn;
            fn = h;
            at = next;
            c = cn;
            n = nn;
        }
    }

    if constexpr (MODE == kBwdUpdate) {
        // descending pass: SP(., TOP) incrementally (Alg. 4) and Eq. 6 per layer
        float* b = R0;
        float* bn = R0 + W * kTile;
        float negsum = 0.f;
        uint32_t c = codes_of(k - 1);
        int n = count_of(c);
        for (int t = k - 1; t >= 0; --t) {
            const uint32_t cp = codes_of(t - 1);
            float m0 = finf(), m1 = finf();
            for (int v = 0; v < n; ++v) {
                const uint32_t cv = __shfl_sync(kFull, c, v);
                const float fv = at[v * kTile];
                m0 = fminf(m0, fv + *row_of(b, cv & 0xFFu));
                m1 = fminf(m1, fv + *row_of(b, cv >> 8));
            }
            float lt = Lr[t * kTile];
            m1 += lt;
            const float d = m1 - m0;
            lt = fmaf(-omega, d, lt) + Tr[t * kTile];  // Eq. 5
            Lr[t * kTile] = lt;
            negsum += fmaxf(-d, 0.f);
            for (int v = 0; v < n; ++v) {
                const uint32_t cv = __shfl_sync(kFull, c, v);
                bn[v * kTile] = fminf(*row_of(b, cv & 0xFFu), *row_of(b, cv >> 8) + lt);
            }
            float* h = b;
            b = bn;
            bn = h;
            c = cp;
            n = count_of(c);
            at -= n * kTile;
        }
        term = fmaf(-omega, negsum, b[0]);
    }

    if constexpr (update) {
#pragma unroll 4
        for (int t = 0; t < k; ++t) {
            if (valid) lam[base + static_cast<size_t>(t) * kTile] = Lr[t * kTile];
        }
        if (local) {
            for (int t = 0; t < k; ++t) ep_lam[t * kTile + lane] = Lr[t * kTile];
            __syncwarp();
            tile_local_sums(I, tile.pattern, ep_lam, ep_var, lane);
            __syncwarp();
        }
    }
    if constexpr (MODE == kBwdUpdate || MODE == kEval) {
        const float2 p = tile_bound(valid ? term : 0.f);
        if (lane == 0) I->tile_lb[ti] = p;
    }
}

// the register and the shared-memory tiles behind one name
template <int W, bool REG, int MODE>
__global__ void __launch_bounds__(256) sweep_kernel(SweepArgs a) {
    extern __shared__ float smem[];
    pdl_trigger();
    pdl_wait();
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    const int wpb = blockDim.x >> 5;
    float* wsm = smem + static_cast<size_t>(wib) * (REG ? reg_warp_floats(a) : wide_warp_floats<W>(a));
    for (int g = blockIdx.x * wpb + wib; g < a.total; g += gridDim.x * wpb) {
        if constexpr (REG) reg_tile<W, MODE>(a, g, g + gridDim.x * wpb, wsm, lane);
        else wide_tile<W, MODE>(a, g, g + gridDim.x * wpb, wsm, lane);
    }
}


// Long rows (more than kRegK layers) of narrow BDDs (W <= kRegW).  Staging
// every layer in shared memory would size each warp's region by the longest
// row of the launch and starve the SM of warps, so the layers are processed
// in segments of kRegK held in registers instead.  A first sweep over the
// whole row keeps only the labels at segment ends (checkpoints, in shared
// memory); the update sweep then visits the segments in its own direction,
// reloads each one's multipliers and recomputes its labels from its
// checkpoint.  Every label and update is formed by the same operations in the
// same order as in reg_tile, so results are identical; the cost is one extra
// label sweep over data the warp has just read.  As in reg_tile a segment's
// codes, multipliers and ids are each loaded at once, and one segment (of the
// ids: two) ahead of their use, so that no walk waits for memory in the middle.
// A lone cell-tracking sequence (160 tiles) went from 25.7 and 20.7 us
// (ascending, descending) to 20.1 and 16.4; what is left of a warp's 1,920 and
// 1,720 instructions is a chain: 9.6 and 10.5 cycles each, 3.4 and 3.8 of them
// memory, 3 the latency of the operation before, 1.6 instruction fetch.
// Without AHEAD a segment is loaded when the one before it is done: the
// persistent kernel (persist.cu), whose passes share 128 registers a thread,
// spilled 816 bytes with the look-ahead and 484 without (39.8 instances/s in
// place of 35.4 on 64 cell-tracking sequences).
// Shared memory per warp: a.kstride checkpoints x W labels x 32 lanes, then
// the tile-local staging (a.epi layers).
// shared-memory floats one warp of seg_tile uses
template <int W>
__host__ __device__ __forceinline__ size_t seg_warp_floats(const SweepArgs& a) {
    return static_cast<size_t>(a.kstride) * W * kTile + static_cast<size_t>(a.epi) * kTile * 2;
}

template <int W, int MODE, bool AHEAD = true>
__device__ __forceinline__ void seg_tile(const SweepArgs& a, int g, int g_next, float* wsm, int lane) {
    constexpr int C = kRegK;
    constexpr bool update = MODE == kFwdUpdate || MODE == kBwdUpdate;
    constexpr bool asc = MODE != kBwdUpdate;  // the update sweep's direction
    float* cp = wsm + lane;  // checkpoint of segment s, label v at cp[(s * W + v) * kTile]
    float* ep_lam = wsm + static_cast<size_t>(a.kstride) * W * kTile;
    int* ep_var = reinterpret_cast<int*>(ep_lam + static_cast<size_t>(a.epi) * kTile);
    prefetch_tile(a, g_next, lane);
    const int ii = find_inst_warp(a.prefix, a.n_inst, g, lane);
    const InstDev* __restrict__ I = a.insts + ii;
    if (update && FDOG_INACTIVE(I->ctl)) return;
    const int ti = __ldg(a.first + ii) + (g - __ldg(a.prefix + ii));
    const TileDev tile = I->tiles[ti];
    const ShapeDev sh = I->shapes[tile.shape];
    const int k = sh.k;
    const int nseg = (k + C - 1) / C;
    const uint16_t* __restrict__ tpl = I->tpl + sh.tpl_off;
    const bool valid = lane < tile.n_valid;
    const float omega = I->omega;
    const size_t base = static_cast<size_t>(tile.slot_base) + lane;
    float* __restrict__ lam = I->lam;
    const int32_t* __restrict__ varp = I->var;
    const float* Tv = I->T;
    const bool local = update && a.epi > 0 && tile.pattern >= 0;

    // loads of one segment; padding lanes hold multiplier 0 and variable -1
    auto fetch_lam = [&](int s, float (&L)[C]) {
#pragma unroll
        for (int j = 0; j < C; ++j)
            if (s * C + j < k) L[j] = lam[base + static_cast<size_t>(s * C + j) * kTile];
    };
    auto fetch_var = [&](int s, int (&V)[C]) {
#pragma unroll
        for (int j = 0; j < C; ++j)
            V[j] = s * C + j < k ? __ldcs(varp + base + static_cast<size_t>(s * C + j) * kTile) : -1;  // streamed
    };
    // terms of a segment's variables; ids staged for the tile-local sums
    auto fetch_terms = [&](int s, const int (&V)[C], float (&T)[C]) {
#pragma unroll
        for (int j = 0; j < C; ++j) T[j] = V[j] >= 0 ? Tv[V[j]] : 0.f;
        if (local) {
#pragma unroll
            for (int j = 0; j < C; ++j)
                if (s * C + j < k) ep_var[(s * C + j) * kTile + lane] = V[j];
        }
    };
    // segments in the order of the update sweep are u = 0 .. nseg - 1, the label sweep visits them from the last
    auto seg_of = [&](int u) { return asc ? u : nseg - 1 - u; };

    float x[W];
    float L[C], T[C], Ln[C], Tn[C];
    int V[C];
    LayerCodes<W> c[C], cn[C];
    // Label sweep: SP(v, TOP) over the whole row from its end (asc), SP(r, v) from its root (else); checkpoint of
    // a segment: the labels it starts from.  The last segment visited is the update sweep's first, its
    // multipliers and codes stay in L and c.
#pragma unroll
    for (int v = 0; v < W; ++v) x[v] = !asc && v == 0 ? 0.f : finf();
    fetch_lam(seg_of(nseg - 1), L);
    load_segment_codes<W>(tpl, seg_of(nseg - 1) * C, c);
    if constexpr (update) fetch_var(seg_of(0), V);
    for (int u = nseg - 1; u >= 0; --u) {
        const int s = seg_of(u);
        const int kk = min(k - s * C, C);
        if (AHEAD && u > 0) {  // in flight while this segment is swept
            fetch_lam(seg_of(u - 1), Ln);
            load_segment_codes<W>(tpl, seg_of(u - 1) * C, cn);
        }
#pragma unroll
        for (int v = 0; v < W; ++v) cp[(s * W + v) * kTile] = x[v];
        if (u > 0 || MODE == kEval) {  // the first segment's own labels are formed by the update sweep
            if constexpr (asc) {
#pragma unroll
                for (int j = C - 1; j >= 0; --j)
                    if (j < kk) pull_labels<W>(x, c[j], L[j]);
            } else {
#pragma unroll
                for (int j = 0; j < C; ++j)
                    if (j < kk) push_labels<W>(x, c[j], L[j]);
            }
        }
        if (AHEAD && u > 0) {
#pragma unroll
            for (int j = 0; j < C; ++j) { L[j] = Ln[j]; c[j] = cn[j]; }
        } else if (u > 0) {
            fetch_lam(seg_of(u - 1), L);
            load_segment_codes<W>(tpl, seg_of(u - 1) * C, c);
        }
    }
    float term = 0.f;
    if constexpr (MODE == kEval) {
        term = x[0];
    } else {
        if constexpr (update) {
            fetch_terms(seg_of(0), V, T);
            if (AHEAD && nseg > 1) fetch_var(seg_of(1), V);
        }
        float* __restrict__ mm0 = I->mm0;
        float* __restrict__ mm1 = I->mm1;
        float negsum = 0.f;
#pragma unroll
        for (int v = 0; v < W; ++v) x[v] = asc && v == 0 ? 0.f : finf();
        for (int u = 0; u < nseg; ++u) {
            const int s = seg_of(u);
            const int kk = min(k - s * C, C);
            if (AHEAD && u + 1 < nseg) {  // in flight while this segment is swept
                fetch_lam(seg_of(u + 1), Ln);
                load_segment_codes<W>(tpl, seg_of(u + 1) * C, cn);
                if constexpr (update) {
                    fetch_terms(seg_of(u + 1), V, Tn);
                    if (u + 2 < nseg) fetch_var(seg_of(u + 2), V);
                }
            }
            // opposite labels of the segment's layers, from its checkpoint: S[j] holds those of the layer after j
            // (asc) or of layer j (else)
            float S[C][W], y[W];
#pragma unroll
            for (int v = 0; v < W; ++v) y[v] = cp[(s * W + v) * kTile];
            if constexpr (asc) {
#pragma unroll
                for (int j = C - 1; j >= 0; --j) {
                    if (j < kk) {
#pragma unroll
                        for (int v = 0; v < W; ++v) S[j][v] = y[v];
                        if (j > 0) pull_labels<W>(y, c[j], L[j]);
                    }
                }
            } else {
#pragma unroll
                for (int j = 0; j < C; ++j) {
                    if (j < kk) {
#pragma unroll
                        for (int v = 0; v < W; ++v) S[j][v] = y[v];
                        if (j + 1 < C) push_labels<W>(y, c[j], L[j]);
                    }
                }
            }
            if constexpr (asc) {
#pragma unroll
                for (int j = 0; j < C; ++j) {
                    if (j < kk) {
                        float m0, m1;
                        layer_marginals<W>(x, S[j], c[j], m0, m1);
                        m1 += L[j];
                        if constexpr (MODE == kFwdUpdate) {
                            L[j] = fmaf(-omega, m1 - m0, L[j]) + T[j];  // Eq. 5
                        } else if (valid) {
                            const size_t p = base + static_cast<size_t>(s * C + j) * kTile;
                            if (a.flags & kMMBoth) { mm0[p] = m0; mm1[p] = m1; }
                            else mm0[p] = m1 - m0;
                        }
                        push_labels<W>(x, c[j], L[j]);
                    }
                }
            } else {
#pragma unroll
                for (int j = C - 1; j >= 0; --j) {
                    if (j < kk) {
                        float m0, m1;
                        layer_marginals<W>(S[j], x, c[j], m0, m1);
                        m1 += L[j];
                        const float d = m1 - m0;
                        L[j] = fmaf(-omega, d, L[j]) + T[j];  // Eq. 5
                        negsum += fmaxf(-d, 0.f);
                        pull_labels<W>(x, c[j], L[j]);
                    }
                }
            }
            if constexpr (update) {
#pragma unroll
                for (int j = 0; j < C; ++j) {
                    if (j < kk) {
                        if (valid) lam[base + static_cast<size_t>(s * C + j) * kTile] = L[j];
                        if (local) ep_lam[(s * C + j) * kTile + lane] = L[j];
                    }
                }
            }
            if (AHEAD && u + 1 < nseg) {
#pragma unroll
                for (int j = 0; j < C; ++j) { L[j] = Ln[j]; T[j] = Tn[j]; c[j] = cn[j]; }
            } else if (u + 1 < nseg) {
                fetch_lam(seg_of(u + 1), L);
                load_segment_codes<W>(tpl, seg_of(u + 1) * C, c);
                if constexpr (update) {
                    fetch_var(seg_of(u + 1), V);
                    fetch_terms(seg_of(u + 1), V, T);
                }
            }
        }
        if constexpr (!asc) term = fmaf(-omega, negsum, x[0]);
    }

    if constexpr (update) {
        if (local) {
            __syncwarp();
            tile_local_sums(I, tile.pattern, ep_lam, ep_var, lane);
            __syncwarp();
        }
    }
    if constexpr (MODE == kBwdUpdate || MODE == kEval) {  // the passes whose bound is reduced
        const float2 p = tile_bound(valid ? term : 0.f);
        if (lane == 0) I->tile_lb[ti] = p;
    }
}

template <int W, int MODE>
__global__ void __launch_bounds__(256) sweep_seg_kernel(SweepArgs a) {
    extern __shared__ float smem[];
    pdl_trigger();
    pdl_wait();
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    const int wpb = blockDim.x >> 5;
    float* wsm = smem + static_cast<size_t>(wib) * seg_warp_floats<W>(a);
    for (int g = blockIdx.x * wpb + wib; g < a.total; g += gridDim.x * wpb)
        seg_tile<W, MODE>(a, g, g + gridDim.x * wpb, wsm, lane);
}

#undef FD_UP
#undef FD_DOWN

}  // namespace dev

// host-side dispatch of one width's instantiations (defined in sweep_w<W>.cu)
template <int W>
cudaError_t launch_sweep_width(bool reg, int mode, int blocks, int threads, size_t smem, cudaStream_t s,
                               const SweepArgs& a, const L2Window& l2);

namespace dev {
template <int W, bool REG>
inline auto sweep_fn(int mode) -> void (*)(SweepArgs) {
    return mode == kFwdUpdate ? sweep_kernel<W, REG, kFwdUpdate>
         : mode == kBwdUpdate ? sweep_kernel<W, REG, kBwdUpdate>
         : mode == kMinMarg   ? sweep_kernel<W, REG, kMinMarg>
                              : sweep_kernel<W, REG, kEval>;
}
template <int W>
inline auto seg_fn(int mode) -> void (*)(SweepArgs) {
    return mode == kFwdUpdate ? sweep_seg_kernel<W, kFwdUpdate>
         : mode == kBwdUpdate ? sweep_seg_kernel<W, kBwdUpdate>
         : mode == kMinMarg   ? sweep_seg_kernel<W, kMinMarg>
                              : sweep_seg_kernel<W, kEval>;
}
}  // namespace dev

// narrow widths have the register and the segmented kernels, wide ones the shared-memory kernel
#define FDOG_DEFINE_SWEEP_WIDTH(W)                                                                             \
    template <>                                                                                                \
    cudaError_t launch_sweep_width<W>(bool reg, int mode, int blocks, int threads, size_t smem, cudaStream_t s, \
                                      const SweepArgs& a, const L2Window& l2) {                                \
        void (*fn)(SweepArgs);                                                                                 \
        if constexpr (W <= kRegW) fn = reg ? dev::sweep_fn<W, true>(mode) : dev::seg_fn<W>(mode);              \
        else fn = dev::sweep_fn<W, false>(mode);                                                               \
        const cudaError_t e = allow_smem(reinterpret_cast<const void*>(fn), smem);                             \
        if (e != cudaSuccess) return e;                                                                        \
        void* args[] = {const_cast<SweepArgs*>(&a)};                                                           \
        return launch_windowed(reinterpret_cast<const void*>(fn), blocks, threads, args, smem, s, l2);         \
    }

}  // namespace fdog
