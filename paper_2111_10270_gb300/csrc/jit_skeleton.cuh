// Skeleton of the shape-specialised sweep kernels.  This file is not compiled
// by nvcc: the build embeds it as text, and at plan time jit.cpp appends the
// generated per-shape functions and dispatch tables and compiles the result
// for sm_103a with NVRTC.
//
// The tile loop, instance lookup and per-tile bound reduction are the same as
// in the static sweep kernels (sweep.cuh); only the per-BDD work differs: it
// is straight-line code for one known shape, with every successor choice
// resolved when the code was generated, so a thread spends its instructions
// on the min-plus arithmetic itself.

#define FDOG_INF __int_as_float(0x7f800000)
#define FDOG_FULL 0xffffffffu

#ifdef FDOG_DISPATCH
// largest instance index i with prefix[i] <= g, g the same in every lane
__device__ __forceinline__ int fdog_find_inst(const int32_t* __restrict__ prefix, int n, int g, int lane) {
    if (n == 1) return 0;
    int at = 0;
    for (int b = 0; b < n; b += 32) {
        const unsigned m = __ballot_sync(FDOG_FULL, b + lane < n && __ldg(prefix + b + lane) <= g);
        at += __popc(m);
        if (m != FDOG_FULL) break;
    }
    return at - 1;
}

// Deferred terms of the tile-local variables, formed right after an update
// pass from the staged multipliers (same sum and order as the deferred-sum
// kernel); staging: layer t lane l at [32 t + l].
__device__ __forceinline__ void fdog_tile_local_sums(const InstDev* __restrict__ I, int pattern,
                                                     const float* ep_lam, const int* ep_var, int lane) {
    const int2 pat = reinterpret_cast<const int2*>(I->patterns)[pattern];
    for (int e = lane; e < pat.y; e += 32) {
        const ushort4 o = reinterpret_cast<const ushort4*>(I->local_ent)[pat.x + e];
        float s = 0.f + ep_lam[o.x];
        int c = 1;
        if (o.y != 0xFFFFu) { s += ep_lam[o.y]; ++c; }
        if (o.z != 0xFFFFu) { s += ep_lam[o.z]; ++c; }
        if (o.w != 0xFFFFu) { s += ep_lam[o.w]; ++c; }
        const int v = ep_var[o.x];
        // (C - sum) times 1 / c rounded to FP32, as in the deferred-sum kernel
        const float inv = c == 1 ? 1.f : c == 2 ? 0.5f : c == 3 ? 1.f / 3.f : 0.25f;
        I->T[v] = (I->C[v] - s) * inv;
    }
}

// L2 prefetch of the multiplier and variable rows of the tile this warp
// visits next (lane t takes layer t), issued before the current tile is
// computed so that the next tile's first loads hit L2.
__device__ __forceinline__ void fdog_prefetch_tile(const SweepArgs& a, int g, int lane) {
    if (g >= a.total) return;
    const int ii = fdog_find_inst(a.prefix, a.n_inst, g, lane);
    const InstDev* __restrict__ I = a.insts + ii;
    const TileDev tile = I->tiles[__ldg(a.first + ii) + (g - __ldg(a.prefix + ii))];
    const int k = I->shapes[tile.shape].k;
    if (lane < k) {
        const long long p = (long long)tile.slot_base + 32LL * lane;
        asm volatile("prefetch.global.L2 [%0];" ::"l"(I->lam + p));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(I->var + p));
    }
}

// MODE: 0 ascending pass with updates, 1 descending pass with updates,
//       2 min-marginals, 3 energies only
template <int MODE>
__device__ __forceinline__ void fdog_jit_sweep(const SweepArgs& a) {
    extern __shared__ float fdog_smem[];
    // programmatic dependent launch (the launches allow it): let the next kernel be scheduled once every
    // block has started, and touch memory only after the kernel before this one has completed
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    const int wpb = blockDim.x >> 5;
    float* ep_lam = fdog_smem + (long long)wib * a.epi * 32 * 2;
    int* ep_var = (int*)(ep_lam + (long long)a.epi * 32);
    for (int g = blockIdx.x * wpb + wib; g < a.total; g += gridDim.x * wpb) {
        fdog_prefetch_tile(a, g + gridDim.x * wpb, lane);
        const int ii = fdog_find_inst(a.prefix, a.n_inst, g, lane);
        const InstDev* __restrict__ I = a.insts + ii;
        if (MODE <= 1 && FDOG_INACTIVE(I->ctl)) continue;
        const int ti = __ldg(a.first + ii) + (g - __ldg(a.prefix + ii));
        const TileDev tile = I->tiles[ti];
        const int jit = I->shapes[tile.shape].jit;
        const bool valid = lane < tile.n_valid;
        const long long base = (long long)tile.slot_base + lane;
        const bool local = MODE <= 1 && a.epi > 0 && tile.pattern >= 0;
        float term = 0.f;
        FDOG_DISPATCH(MODE)
        if (local) {
            __syncwarp();
            fdog_tile_local_sums(I, tile.pattern, ep_lam, ep_var, lane);
            __syncwarp();
        }
        if (MODE == 1 || MODE == 3) {  // only the descending pass and the energy sweep feed a bound reduction
            float s = valid ? term : 0.f, comp = 0.f;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                const float o = __shfl_xor_sync(FDOG_FULL, s, off);
                const float oc = __shfl_xor_sync(FDOG_FULL, comp, off);
                const float sum = s + o;
                const float bp = sum - s;
                const float err = (s - (sum - bp)) + (o - bp);
                s = sum;
                comp = comp + oc + err;
            }
            if (lane == 0) I->tile_lb[ti] = make_float2(s, comp);
        }
    }
}

extern "C" __global__ void __launch_bounds__(256) fdog_jit_fwd(SweepArgs a) { fdog_jit_sweep<0>(a); }
extern "C" __global__ void __launch_bounds__(256) fdog_jit_bwd(SweepArgs a) { fdog_jit_sweep<1>(a); }
extern "C" __global__ void __launch_bounds__(256) fdog_jit_mm(SweepArgs a) { fdog_jit_sweep<2>(a); }
extern "C" __global__ void __launch_bounds__(256) fdog_jit_eval(SweepArgs a) { fdog_jit_sweep<3>(a); }
#endif

#ifdef FDOG_BULK_DISPATCH
// ---- bulk sweeps -------------------------------------------------------------
// Update passes of one large instance.  In the sweeps above a warp waits in
// turn for its tile's descriptor, its multipliers and ids, the terms they
// name, and at the end for the targets C of its tile-local variables; with
// every warp slot of the GPU taken they run at 62 and 70 us a pass on the
// 512x512 grid with four labels, for 374 MB, and no part of that chain can be
// moved forward because registers are all in use.  Here the warps stay and
// walk many tiles each, and what a tile reads is copied ahead into shared
// memory by bulk copies (cp.async.bulk, one mbarrier per stage of a warp),
// which hold no registers:
//   * its multipliers, one run of k rows;
//   * one block with the targets of its layers with tile-local slots, in slot
//     order (so a variable's target is there for each of its copies), and the
//     ids of its other layers.
// The term of a tile-local variable (all of whose at most two copies lie in
// the tile) is formed here, from the multipliers the last pass left in the
// tile, instead of at the end of that pass: T is neither written nor gathered
// for it, and its slots need no ids.  The same FP32 operations in the same
// order, so the same terms.  A pass moves 274 MB, in about 48 us: the 500
// iterations and two roundings of that grid went from 88.2 to 69.2 ms.  What
// bounds it now is instructions, 265 and 310 a tile (ascending, descending)
// with 66 and 69% of the issue slots taken, before memory latency (3 to 4 of
// the 10 to 11 cycles between two instructions of a warp).  Tiles are looked
// up 16 at a time, both copies of a pair by one bulk copy, and plain patterns
// have a path without choices per slot.  Two
// stages (69.5 ms; three 70.3, four 74.5): at 62 registers four blocks of eight
// warps fit an SM, and more stages take L1 from the gathers of T.  Capping the
// registers at 48 for a fifth block made them spill (74.9 ms).  The L2 window
// on T is worth 1 ms.
// <ptx>
__device__ __forceinline__ void fdog_pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void fdog_pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// the bulk copies that follow read what kernels wrote
__device__ __forceinline__ void fdog_copies_see_kernels() { asm volatile("fence.proxy.async.global;" ::: "memory"); }

__device__ __forceinline__ unsigned fdog_smem_addr(const void* p) {
    return (unsigned)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void fdog_bar_init(unsigned bars, int n) {
    for (int s = 0; s < n; ++s)
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bars + 8u * s) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void fdog_bar_expect(unsigned bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool fdog_bar_done(unsigned bar, unsigned parity) {
    unsigned done;
    asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
                 : "=r"(done) : "r"(bar), "r"(parity) : "memory");
    return done != 0;
}

__device__ __forceinline__ unsigned long long fdog_now() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void fdog_bulk_copy(unsigned dst, const void* src, unsigned bytes, unsigned bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar) : "memory");
}
// </ptx>

// waits for a stage's copies; gives up (false) after a second
__device__ __forceinline__ bool fdog_bulk_wait(unsigned bar, unsigned parity) {
    unsigned long long t0 = 0;
    while (!fdog_bar_done(bar, parity)) {
        const unsigned long long t = fdog_now();
        if (t0 == 0) t0 = t;
        else if (t - t0 > 1000000000ull) return false;
    }
    return true;
}

// waits once more for up to `stages` of the `left` tiles' copies, from stage s of phase `parity` on
__device__ __noinline__ void fdog_bulk_drain(unsigned bars, int stages, int s, unsigned parity, int left) {
    for (int q = 0; q < stages && q < left; ++q) {
        fdog_bulk_wait(bars + 8u * s, parity);
        if (++s == stages) {
            s = 0;
            parity ^= 1u;
        }
    }
}

// (s, c) <- (s, c) + (x, y) for compensated FP32 pairs, as the butterflies above form them
__device__ __forceinline__ void fdog_pair_add(float& s, float& c, float x, float y) {
    const float sum = s + x;
    const float bp = sum - s;
    const float err = (s - (sum - bp)) + (x - bp);
    s = sum;
    c = c + y + err;
}

template <int MODE>
__device__ __forceinline__ void fdog_bulk_sweep(const BulkArgs& a) {
    extern __shared__ __align__(128) float fdog_stages[];
    const int lane = threadIdx.x & 31;
    const int wpb = blockDim.x >> 5;
    fdog_pdl_trigger();
    // this warp's rows: stages; a table of the 32 tiles around the current one (16 ahead are filled in at a time, a
    // lane per tile, so that finding a tile costs next to nothing); the terms of four tiles; the barriers
    float* const stage0 = fdog_stages + (threadIdx.x >> 5) * FDOG_BULK_WARP_ROWS(a.stages, a.rows) * 32;
    int4* const tab = (int4*)(stage0 + a.stages * a.rows * 32);
    float* const terms = (float*)(tab + 32);
    const unsigned bars = fdog_smem_addr(terms + 136);
    if (lane == 0) fdog_bar_init(bars, a.stages);
    __syncwarp();
    fdog_pdl_wait();
    fdog_copies_see_kernels();
    const InstDev* __restrict__ I = a.inst;
    InstCtl* const ctl = I->ctl;
    // all of it asked for at once; after an error no later pass waits again
    const int done = ctl->done, iter = ctl->iter, limit = ctl->iter_limit, error = ctl->error, t_zero = ctl->t_zero;
    if ((done != 0) | (iter >= limit) | (error != 0)) return;
    const bool zero = MODE == 0 && t_zero;  // a descending pass follows an ascending one
    const float omega = I->omega;
    float* const lam0 = I->lam;
    const float* const cv0 = I->cv;
    const float* const T = I->T;
    const int first = I->bulk_first;
    const int stride = gridDim.x * wpb;
    const int g0 = blockIdx.x * wpb + (threadIdx.x >> 5);
    const int n = g0 < a.total ? (a.total - g0 + stride - 1) / stride : 0;  // tiles of this warp

    auto fill = [&](int block) {
        const int it = 16 * block + lane;
        if (lane < 16 && it < n) {
            const int g = g0 + it * stride;
            const BulkRun* r = I->bulk_runs;
            for (int q = I->n_bulk_runs - 1; q > 0; --q)
                if (I->bulk_runs[q].tile <= g) {
                    r = I->bulk_runs + q;
                    break;
                }
            const int j = g - r->tile;
            const int n_valid = min(32, r->n_bdds - 32 * j);
            tab[it & 31] = make_int4(r->slot_base + j * r->k * 32, r->cv_row + j * (r->c_n + r->v_n),
                                     r->k | r->c_n << 5 | r->v_n << 10 | r->c_lo << 15 | r->v_lo << 19 | n_valid << 23,
                                     r->jit << 8 | (I->tiles[first + g].pattern + 1));
        }
        __syncwarp();
    };
    bool late = false;
    auto issue = [&](int it, int s) {
        if (it < n && lane == 0 && !late) {
            const int4 e = tab[it & 31];
            const unsigned rows = e.z & 31, more = (e.z >> 5 & 31) + (e.z >> 10 & 31);
            const unsigned bar = bars + 8u * s;
            const unsigned dst = fdog_smem_addr(stage0 + s * a.rows * 32);
            fdog_bar_expect(bar, (rows + more) * 128u);
            fdog_bulk_copy(dst, lam0 + e.x, rows * 128u, bar);
            fdog_bulk_copy(dst + rows * 128u, cv0 + e.y * 32, more * 128u, bar);
        }
    };
    fill(0);
    for (int s = 0; s < a.stages; ++s) issue(s, s);
    unsigned pk[8], plain_of = 0;
    int have = -1, s = 0;
    unsigned parity = 0;
    for (int i = 0; i < n; ++i) {
        if ((i & 15) == 0) fill((i >> 4) + 1);
        const int4 e = tab[i & 31];
        const int pat = e.w & 255;
        if (pat != have) {  // most neighbouring tiles have the same pattern
            have = pat;
#pragma unroll
            for (int q = 0; q < 8; ++q)
                pk[q] = pat > 0 ? __ldg(a.pairs + ((pat - 1) * 8 + q) * 32 + lane) : 0xFFFFFFFFu;
            plain_of = pat > 0 ? __ldg(a.pairs + a.n_pat * 256 + pat - 1) : FDOG_PAIR_PLAIN;
        }
        const int k = e.z & 31, n_valid = e.z >> 23;
        const unsigned plain = n_valid == 32 && !zero ? plain_of : 0u;
        const int jit = e.w >> 8;
        const bool valid = lane < n_valid;
        float* const lam = lam0 + (e.x + lane);
        const float* const sl = stage0 + s * a.rows * 32;
        const float* const sc = sl + (k - (e.z >> 15 & 15)) * 32;
        const int* const sv = (const int*)(sl + (k + (e.z >> 5 & 31) - (e.z >> 19 & 15)) * 32);
        // a lane that has waited in vain reports it (the host then returns an error) and waits no more; every lane
        // goes on, so that the warp stays together.  No copy is started any more, and the lane that starts them waits
        // once more for each that may still be on its way into this block's shared memory.
        if (!late && !fdog_bulk_wait(bars + 8u * s, parity)) {
            late = true;
            ctl->error = 1;
            if (lane == 0) fdog_bulk_drain(bars, a.stages, s, parity, n - i);
        }
        float term = 0.f;
        FDOG_BULK_DISPATCH(MODE)
        __syncwarp();  // every lane has read the stage
        issue(i + a.stages, s);
        if (++s == a.stages) {
            s = 0;
            parity ^= 1u;
        }
        if (MODE == 1) {
            // Partials of the bound, four tiles at a time: eight lanes reduce one tile, in the order of the
            // butterflies above (lane l + 16, l + 8, then 4, 2, 1).  A butterfly per tile took 45 instructions,
            // this takes 16.
            terms[(i & 3) * 33 + lane] = valid ? term : 0.f;
            if ((i & 3) == 3 || i == n - 1) {
                __syncwarp();
                const int q = lane >> 3, j = lane & 7;
                const float* const t = terms + q * 33 + j;
                float x = t[0], xc = 0.f, y = t[8], yc = 0.f;
                fdog_pair_add(x, xc, t[16], 0.f);
                fdog_pair_add(y, yc, t[24], 0.f);
                fdog_pair_add(x, xc, y, yc);
#pragma unroll
                for (int off = 4; off > 0; off >>= 1) {
                    const float o = __shfl_xor_sync(FDOG_FULL, x, off);
                    const float oc = __shfl_xor_sync(FDOG_FULL, xc, off);
                    fdog_pair_add(x, xc, o, oc);
                }
                if (j == 0 && q <= (i & 3)) I->tile_lb[first + g0 + (i - (i & 3) + q) * stride] = make_float2(x, xc);
                __syncwarp();
            }
        }
    }
}

extern "C" __global__ void __launch_bounds__(256) fdog_bulk_fwd(BulkArgs a) { fdog_bulk_sweep<0>(a); }
extern "C" __global__ void __launch_bounds__(256) fdog_bulk_bwd(BulkArgs a) { fdog_bulk_sweep<1>(a); }
#endif
