// fdog_bound_reduce_noalloc: the lower-bound reduction for callers that
// cannot allocate device memory.
//
// Some callers cannot call cudaMalloc where they need a bound: plug-ins that
// live inside a host framework which owns every device allocation through its
// own pool (a direct cudaMalloc would bypass its accounting), and real-time
// loops that forbid allocation after start-up (cudaMalloc may synchronise the
// device and has no latency bound).  They already hold the per-subproblem
// energies E_j in their own device buffer and only need the deterministic
// sum.  The sum is formed in integers, so that it is exact whatever the order:
// a block aligns its values to the largest exponent among them and adds them as
// 128-bit fixed-point numbers; a second launch of one block adds the blocks'
// totals in the same way.  Bits that such a window has no place for (2^-101 of
// the largest value and below: values of very different size, which may be all
// that is left once the large ones cancel) go through windows of their own into
// an accumulator of the whole FP64 range.  What bounds it is
// the read of the values and what a call takes at least, two launches of about 3
// us: FP64 additions run at two per clock and SM on this part, so that the
// compensated FP64 tree over 256 values per block that stood here took 144 us a
// call for 4,000,037 values and 47 us for 2^20; integer shifts and additions run
// at the full rate (18.4 and 10.3 us; 2,000 values 6.2, with the tree 11.2).  The
// blocks' totals travel as integers too: as pairs of doubles they and a second
// launch that handles every case in line took 3 us more.
// Scratch -- the blocks' totals and that accumulator -- is one file-scope static
// device array instead of memory owned by an instance.  A call leaves nothing in
// it that a later one reads: the second launch needs no counter of finished
// blocks, which overlapping calls could leave off zero, and clears the accumulator.
#include <cuda.h>  // CUcontext / CUresult types of the two driver calls fetched at run time
#include <cuda_runtime.h>

#include <cstdint>
#include <mutex>

#include "../../include/fastdog.h"
#include "kernels.h"

namespace {

constexpr int kThreads = 256;
// values per thread: up to 2^20 values with few, so that they spread over all SMs (977 blocks of 1,024), more with
// many, so that the blocks' totals stay few (608 blocks of 4,096 values are resident)
constexpr int kFewPer = 4, kManyPer = 16;
constexpr int64_t kFewMax = int64_t(1) << 20;
constexpr int64_t kMaxValues = int64_t(1) << 23;  // 8,388,608 values per call
constexpr int kMaxBlocks = static_cast<int>(kMaxValues / (kThreads * kManyPer));
static_assert(kFewMax / (kThreads * kFewPer) <= kMaxBlocks, "scratch holds the totals of either kind");
constexpr int kMaxDevices = 64;

// Fixed-point sums.  A value of biased exponent e (1 for subnormal numbers) is
// m 2^(e - 1075) with a 53-bit m; beside values of largest exponent emax it is
// added as m 2^(kUp - (emax - e)), without the bits below the last place.  2^23
// such terms (4,096 values a block, 2,048 blocks) and the sign fit 128 bits.
constexpr int kUp = 49;
struct __align__(16) Fixed {
    unsigned long long lo, hi;  // two's complement
};

constexpr int kDigits = 70;
struct Scratch {
    Fixed part[kMaxBlocks];  // total of each block, zero if it went into digit
    int exponent[kMaxBlocks];  // the exponent it is aligned to; 2047: a value was not finite
    // The blocks' totals that a window cannot hold, as digits of 32 bits in 64 from bit 2^-1123 (2^(1 - 1075 - kUp))
    // on, summed by integer atomics.  Zero between calls: the finishing block, which runs after every block of its
    // call, clears them, so the last call to finish does whatever overlapped before it.
    unsigned long long digit[kDigits];
};

// Held by every GPU that loads this library until the process exits.  In host
// code this name is only a host-side stand-in: the device address comes from
// cudaGetSymbolAddress, once per device, with that device current.
static __device__ __align__(256) Scratch g_scratch;

std::mutex g_mu;
// per device: the scratch address and the id of the context it was looked up in
Scratch* g_addr[kMaxDevices] = {};
unsigned long long g_ctx[kMaxDevices] = {};

__device__ __forceinline__ int exponent_of(double v) {
    const int e = (__double2hiint(v) >> 20) & 0x7FF;
    return e ? e : 1;
}

__device__ __forceinline__ void add(Fixed& a, const Fixed& b) {
    a.lo += b.lo;
    a.hi += b.hi + (a.lo < b.lo ? 1u : 0u);
}

__device__ __forceinline__ bool is_zero(double v) { return (__double_as_longlong(v) << 1) == 0; }

// v into a, except the bits below the last place, which it returns.  ALL: there are none.
template <bool ALL>
__device__ __forceinline__ double add_value(Fixed& a, double v, int emax) {
    const unsigned long long bits = __double_as_longlong(v);
    const bool normal = (bits >> 52) & 0x7FFu;
    const unsigned long long m = (bits & 0xFFFFFFFFFFFFFull) | (normal ? 1ull << 52 : 0ull);
    const int up = kUp - (emax - exponent_of(v));
    Fixed t;
    if (ALL) {  // 0 to kUp, but for zeros
        t.lo = m << (up & 63);
        t.hi = (m >> 1) >> ((63 - up) & 63);
    } else {
        t.lo = up >= 0 ? m << up : (up > -64 ? m >> -up : 0ull);
        t.hi = up > 0 ? m >> (64 - up) : 0ull;
    }
    const unsigned long long neg = 0ull - (bits >> 63);  // all ones for a negative value
    t.lo ^= neg;
    t.hi ^= neg;
    t.lo -= neg;
    t.hi += neg && t.lo == 0ull ? 1u : 0u;
    add(a, t);
    if (ALL || up >= 0) return 0.0;
    if (up <= -53) return v;
    const double kept = __longlong_as_double(bits & ~((1ull << -up) - 1));
    return (m >> -up) ? v - kept : v;  // exact: the low bits of v (of a subnormal kept, too)
}

// a in units of 2^(emax - 1075 - kUp) into digits
__device__ __forceinline__ void add_digits(unsigned long long* digit, const Fixed& a, int emax) {
    const int q = (emax - 1) >> 5, sh = (emax - 1) & 31;
    const unsigned long long w0 = a.lo << sh;
    const unsigned long long w1 = sh ? a.hi << sh | a.lo >> (64 - sh) : a.hi;
    const long long w2 = static_cast<long long>(a.hi) >> (sh ? 64 - sh : 63);  // the top, with the sign
    const unsigned long long d[5] = {w0 & 0xFFFFFFFFull, w0 >> 32, w1 & 0xFFFFFFFFull, w1 >> 32,
                                     static_cast<unsigned long long>(w2)};
#pragma unroll
    for (int i = 0; i < 5; ++i)
        if (d[i]) atomicAdd(digit + q + i, d[i]);
}

// the digits' number rounded to the nearest double; NaN beyond the largest
__device__ __noinline__ double round_digits(unsigned long long* digit) {
    constexpr unsigned long long mask = 0xFFFFFFFFull;
    long long carry = 0;
    for (int i = 0; i < kDigits; ++i) {
        carry += static_cast<long long>(digit[i]);
        digit[i] = static_cast<unsigned long long>(carry) & mask;
        carry >>= 32;
    }
    const bool neg = carry < 0;
    if (neg) {
        unsigned long long c = 1;
        for (int i = 0; i < kDigits; ++i) {
            c += ~digit[i] & mask;
            digit[i] = c & mask;
            c >>= 32;
        }
    }
    int top = kDigits - 1;
    while (top >= 0 && digit[top] == 0) --top;
    if (top < 0) return 0.0;
    auto at = [&](int i) { return i >= 0 ? digit[i] : 0ull; };
    const int lz = __clz(static_cast<int>(digit[top]));
    unsigned long long m = (digit[top] << 32 | at(top - 1)) << lz;
    const unsigned long long below = at(top - 2) << lz;
    m |= below >> 32;
    bool more = (below & mask) != 0;
    for (int i = top - 3; i >= 0 && !more; --i) more = digit[i] != 0;
    const int e = 32 * top + 31 - lz - 1074 - kUp;  // m 2^(e - 63)
    const unsigned long long low = m & 0x7FFu;
    m >>= 11;
    if (low > 0x400u || (low == 0x400u && (more || (m & 1u)))) ++m;
    const double r = scalbn(static_cast<double>(m), e - 52);  // a result below 2^-1022 has no bits to round
    if (isinf(r)) return __longlong_as_double(0x7ff8000000000000ll);
    return neg ? -r : r;
}

// the block's total in thread 0
__device__ __forceinline__ void block_sum(Fixed& a) {
    __shared__ Fixed sh[kThreads / 32];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        Fixed o;
        o.lo = __shfl_down_sync(0xffffffffu, a.lo, off);
        o.hi = __shfl_down_sync(0xffffffffu, a.hi, off);
        add(a, o);
    }
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = a;
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < kThreads / 32; ++w) add(a, sh[w]);
}

// Keys of the threads' values: twice the high word, which has the exponent on top, for the largest, and that with
// the low word as one bit, less one, for the smallest that is not zero (a zero is the largest key).
struct Keys {
    unsigned lo = 0xFFFFFFFFu, hi = 0;
};

__device__ __forceinline__ void add_key(Keys& k, double v) {
    const unsigned h = static_cast<unsigned>(__double2hiint(v)) << 1;
    k.hi = max(k.hi, h);
    k.lo = min(k.lo, h + min(static_cast<unsigned>(__double2loint(v)), 1u) - 1u);
}

// smallest exponent of the block's values that are not zero (2047 or more without any) and largest of all, in every
// thread
__device__ __forceinline__ int2 block_exponents(Keys k) {
    __shared__ uint2 sh[kThreads / 32];
    k.lo = __reduce_min_sync(0xffffffffu, k.lo);
    k.hi = __reduce_max_sync(0xffffffffu, k.hi);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = make_uint2(k.lo, k.hi);
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) {
        const uint2 o = sh[w];
        k.lo = min(k.lo, o.x);
        k.hi = max(k.hi, o.y);
    }
    return make_int2(max(static_cast<int>(((k.lo >> 1) + (k.lo & 1u)) >> 20), 1), max(static_cast<int>(k.hi >> 21), 1));
}

// The block's total of what a window below the values' largest exponent holds, in thread 0; x keeps the bits below.
// Returns whether there are any, the same in every thread.
template <int N>
__device__ __forceinline__ bool window_sum(double (&x)[N], int emax, Fixed& a) {
    a = Fixed{0, 0};
    bool rest = false;
#pragma unroll
    for (int q = 0; q < N; ++q) {
        x[q] = add_value<false>(a, x[q], emax);
        rest = rest || !is_zero(x[q]);
    }
    block_sum(a);
    return __syncthreads_or(rest);
}

// the block's values into digits, window by window (each takes 102 bits of exponent at least: at most 21)
template <int N>
__device__ __forceinline__ void digits_of(double (&x)[N], unsigned long long* digit) {
    bool more = true;
    while (more) {
        Keys k;
#pragma unroll
        for (int q = 0; q < N; ++q) add_key(k, x[q]);
        const int emax = block_exponents(k).y;
        Fixed a;
        more = window_sum(x, emax, a);
        if (threadIdx.x == 0) add_digits(digit, a, emax);
    }
}

// a as a leading double and a remainder; whether they are all of it
__device__ __forceinline__ bool to_pair(Fixed a, int emax, double2& p) {
    const bool neg = a.hi >> 63;
    if (neg) {
        a.lo = 0ull - a.lo;
        a.hi = ~a.hi + (a.lo == 0ull ? 1u : 0u);
    }
    // three parts of at most 43 bits, each exact as a double
    constexpr unsigned long long mask = (1ull << 43) - 1;
    const int e0 = emax - 1075 - kUp;
    const double p0 = scalbn(static_cast<double>(a.lo & mask), e0);
    const double p1 = scalbn(static_cast<double>((a.lo >> 43 | a.hi << 21) & mask), e0 + 43);
    const double p2 = scalbn(static_cast<double>(a.hi >> 22), e0 + 86);
    const double s = p2 + p1;  // p2 is zero or the larger
    const double t = p1 - (s - p2);
    const double low = t + p0;
    const double b = low - t;
    const double lost = (t - (low - b)) + (p0 - b);
    const double top = s + low, rest = low - (top - s);
    p = neg ? make_double2(-top, -rest) : make_double2(top, rest);
    return lost == 0.0 && !isinf(top);
}

template <int PER>
__device__ __forceinline__ void load_values(double (&x)[PER], const double* __restrict__ v, int64_t n) {
    const int64_t first = static_cast<int64_t>(blockIdx.x) * (kThreads * PER) + threadIdx.x;
#pragma unroll
    for (int q = 0; q < PER; ++q) x[q] = first + q * kThreads < n ? v[first + q * kThreads] : 0.0;
}

// a block whose values need more than one window: all of it through digits (whose sum may well be short). Out of
// line, with the values read again, so that it takes no registers from the usual path.
template <int PER>
__device__ __noinline__ void spread_block(const double* __restrict__ v, int64_t n, unsigned long long* digit) {
    double x[PER];
    load_values(x, v, n);
    digits_of(x, digit);
}

// Four blocks to an SM with 16 values a thread (64 registers), eight with 4.
template <int PER>
__global__ void __launch_bounds__(kThreads, PER > 4 ? 4 : 8) bound_reduce_noalloc_kernel(const double* __restrict__ v, int64_t n,
                                                                         Scratch* scr) {
    // the finishing block is scheduled while these run and waits for their end
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    double x[PER];
    load_values(x, v, n);
    Keys k;
#pragma unroll
    for (int q = 0; q < PER; ++q) add_key(k, x[q]);
    const int2 e = block_exponents(k);
    Fixed a{0, 0};
    if (e.y < 0x7FF && e.y - e.x <= kUp) {
#pragma unroll
        for (int q = 0; q < PER; ++q) add_value<true>(a, x[q], e.y);
        block_sum(a);
    } else if (e.y < 0x7FF) {
        spread_block<PER>(v, n, scr->digit);
    }
    if (threadIdx.x == 0) {
        scr->part[blockIdx.x] = a;
        scr->exponent[blockIdx.x] = e.y;
    }
}

// The rest of a sum that the finishing block could not form in one window: the blocks' totals, read again, and the
// constant into digits, rounded once.  Out of line: the usual path is a few hundred instructions, which a lone block
// waits for.
__device__ __noinline__ void finish_digits(const Scratch* scr, int blocks, double constant, double* out,
                                           unsigned long long* digit) {
    for (int b = threadIdx.x; b < blocks; b += kThreads) add_digits(digit, scr->part[b], scr->exponent[b]);
    __syncthreads();
    if (threadIdx.x == 0) {
        const int e = exponent_of(constant);
        if (e == 0x7FF) {
            *out = __longlong_as_double(0x7ff8000000000000ll);
        } else {
            Fixed c{0, 0};
            add_value<true>(c, constant, e);
            add_digits(digit, c, e);
            *out = round_digits(digit);
        }
    }
}

// the blocks' totals and the constant, by one block
__global__ void __launch_bounds__(kThreads) bound_finish_noalloc_kernel(Scratch* scr, int blocks, double constant,
                                                                         double* __restrict__ out) {
    __shared__ unsigned long long digit[kDigits];
    __shared__ int most[kThreads / 32];
    __shared__ bool done;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const unsigned long long d = threadIdx.x < kDigits ? scr->digit[threadIdx.x] : 0ull;
    int e = 1;
#pragma unroll 4
    for (int b = threadIdx.x; b < blocks; b += kThreads) {
        const Fixed a = scr->part[b];
        const int eb = scr->exponent[b];
        if ((a.lo | a.hi) != 0ull || eb == 0x7FF) e = max(e, eb);
    }
    e = __reduce_max_sync(0xffffffffu, e);
    if ((threadIdx.x & 31) == 0) most[threadIdx.x >> 5] = e;
    if (d) scr->digit[threadIdx.x] = 0;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) e = max(e, most[w]);
    if (e == 0x7FF) {
        if (threadIdx.x == 0) *out = __longlong_as_double(0x7ff8000000000000ll);
        return;
    }
    // totals aligned to the largest exponent; what that would cut off goes another way
    Fixed t{0, 0};
    bool rest = d != 0;
#pragma unroll 4
    for (int b = threadIdx.x; b < blocks; b += kThreads) {
        Fixed a = scr->part[b];
        const int down = min(max(e - scr->exponent[b], 0), 127);  // less than 0: a zero
        const int part = down & 63;
        const unsigned long long sign = static_cast<long long>(a.hi) < 0 ? ~0ull : 0ull;
        if (down >= 64) {
            rest = rest || a.lo != 0;
            a.lo = a.hi;
            a.hi = sign;
        }
        rest = rest || (a.lo & ((1ull << part) - 1)) != 0;
        a.lo = a.lo >> part | (a.hi << 1) << (63 - part);
        a.hi = static_cast<unsigned long long>(static_cast<long long>(a.hi) >> part);
        add(t, a);
    }
    block_sum(t);
    rest = __syncthreads_or(rest);
    if (threadIdx.x == 0) {
        double2 p;
        done = to_pair(t, e, p) && !rest;
        // (p.x + constant) with its rounding error added to the remainder
        const double s = p.x + constant;
        const double err = fabs(p.x) >= fabs(constant) ? (p.x - s) + constant : (constant - s) + p.x;
        if (done) *out = s + (err + p.y);
    }
    if (threadIdx.x < kDigits) digit[threadIdx.x] = d;
    __syncthreads();
    if (!done) finish_digits(scr, blocks, constant, out, digit);
}

// Unique id of the calling thread's current CUDA context (0 if there is
// none), from cuCtxGetCurrent / cuCtxGetId fetched through the runtime, so
// the library needs no link against the driver library.  The id changes when
// cudaDeviceReset destroys a device's primary context and a later call
// creates a new one, in which the module -- and g_scratch -- may be loaded at
// another address.
unsigned long long current_context_id() {
    using GetCurrent = CUresult (*)(CUcontext*);
    using GetId = CUresult (*)(CUcontext, unsigned long long*);
    static GetCurrent get_current = nullptr;
    static GetId get_id = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_current = reinterpret_cast<GetCurrent>(f);
        f = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_id = reinterpret_cast<GetId>(f);
        cudaGetLastError();
    });
    CUcontext ctx = nullptr;
    unsigned long long id = 0;
    if (!get_current || !get_id || get_current(&ctx) != CUDA_SUCCESS || !ctx || get_id(ctx, &id) != CUDA_SUCCESS)
        return 0;
    return id;
}

// Device address of g_scratch on the current device.  Set-up (the
// cudaGetSymbolAddress lookup, with the device current) runs on the first
// call on a device and again whenever the current context is not the one the
// cached address was looked up in (after cudaDeviceReset).
Scratch* scratch_for_current_device(int* status) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        cudaGetLastError();
        *status = FDOG_ECUDA;
        return nullptr;
    }
    std::lock_guard<std::mutex> lk(g_mu);
    const unsigned long long ctx = current_context_id();
    if (!g_addr[dev] || ctx == 0 || ctx != g_ctx[dev]) {
        void* p = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&p, g_scratch);  // creates the primary context if needed
        if (e != cudaSuccess || !p) {
            cudaGetLastError();
            g_addr[dev] = nullptr;
            *status = FDOG_ECUDA;
            return nullptr;
        }
        g_addr[dev] = static_cast<Scratch*>(p);
        g_ctx[dev] = current_context_id();
    }
    *status = FDOG_OK;
    return g_addr[dev];
}

}  // namespace

extern "C" int fdog_bound_reduce_noalloc(const double* dev_values, int64_t n, double constant, double* dev_out,
                                         void* cuda_stream) {
    if (n < 0 || n > kMaxValues || (n > 0 && !dev_values) || !dev_out) return FDOG_EINVAL;
    int status = FDOG_OK;
    Scratch* scr = scratch_for_current_device(&status);
    if (!scr) return status;
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    const bool few = n <= kFewMax;
    const int64_t per_block = kThreads * (few ? kFewPer : kManyPer);
    const unsigned blocks = n > 0 ? static_cast<unsigned>((n + per_block - 1) / per_block) : 1u;
    if (few) bound_reduce_noalloc_kernel<kFewPer><<<blocks, kThreads, 0, s>>>(dev_values, n, scr);
    else bound_reduce_noalloc_kernel<kManyPer><<<blocks, kThreads, 0, s>>>(dev_values, n, scr);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) {
        // programmatic launch: its block waits on the device for the end of the launch above
        int n_blocks = static_cast<int>(blocks);
        void* args[] = {&scr, &n_blocks, &constant, &dev_out};
        e = fdog::launch_windowed(reinterpret_cast<const void*>(bound_finish_noalloc_kernel), 1, kThreads, args, 0, s,
                                  fdog::L2Window());
        if (e != cudaSuccess) cudaGetLastError();
    }
    return e == cudaSuccess ? FDOG_OK : FDOG_ECUDA;
}
