// fdog_bound_reduce_noalloc: the lower-bound reduction for callers that
// cannot allocate device memory.
//
// Some callers cannot call cudaMalloc where they need a bound: plug-ins that
// live inside a host framework which owns every device allocation through its
// own pool (a direct cudaMalloc would bypass its accounting), and real-time
// loops that forbid allocation after start-up (cudaMalloc may synchronise the
// device and has no latency bound).  They already hold the per-subproblem
// energies E_j in their own device buffer and only need the deterministic
// sum.  The sum is formed in integers: a block aligns its values to the
// largest exponent among them and adds them as 128-bit fixed-point numbers,
// which is exact down to 2^-112 of the largest value whatever the order, and
// the last block adds the blocks' totals in the same way.  What bounds it is
// the read of the values: FP64 additions run at two per clock and SM on this
// part, so that the compensated FP64 tree over 256 values per block that
// stood here took 142 us for 4,000,037 values; integer shifts and additions
// run at the full rate (18.5 us).  Scratch -- the block totals and the last-block
// tickets -- is one file-scope static device array instead of memory owned by an
// instance.
#include <cuda.h>  // CUcontext / CUresult types of the two driver calls fetched at run time
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>
#include <mutex>

#include "../../include/fastdog.h"

namespace {

constexpr int kThreads = 256;
// values per thread: up to 2^20 values with few, so that they spread over all SMs (977 blocks of 1,024), more with
// many, so that the blocks' totals stay few and one wave holds them up to 4.9 million values
constexpr int kFewPer = 4, kManyPer = 16;
constexpr int64_t kFewMax = int64_t(1) << 20;
constexpr int64_t kMaxValues = int64_t(1) << 23;  // 8,388,608 values per call
constexpr int kMaxBlocks = static_cast<int>(kMaxValues / (kThreads * kManyPer));
static_assert(kFewMax / (kThreads * kFewPer) <= kMaxBlocks, "scratch holds the totals of either kind");
constexpr int kMaxDevices = 64;
constexpr unsigned kTickets = 64;

struct Scratch {
    double part[2 * kMaxBlocks];  // total of each block: leading part, remainder
    // A call's last-block ticket, which wraps to zero with its last block.  Calls take them in turn, so that calls
    // that overlapped, with wrong sums in `part`, leave every ticket at zero all the same, and no memset is needed.
    unsigned ticket[kTickets];
};

// Held by every GPU that loads this library until the process exits.  In host
// code this name is only a host-side stand-in: the device address comes from
// cudaGetSymbolAddress, once per device, with that device current.
static __device__ __align__(256) Scratch g_scratch;

std::mutex g_mu;
// per device: the scratch address and the id of the context it was looked up in
Scratch* g_addr[kMaxDevices] = {};
unsigned long long g_ctx[kMaxDevices] = {};
std::atomic<unsigned> g_calls{0};

// Fixed-point sums.  A value of biased exponent e (1 for subnormal numbers) is
// m 2^(e - 1075) with a 53-bit m; beside values of largest exponent emax it is
// added as m 2^(kUp - (emax - e)), bits below the last place dropped.  2^14
// such terms and the sign fit 128 bits.
constexpr int kUp = 60;
struct Fixed {
    unsigned long long lo, hi;  // two's complement
};

__device__ __forceinline__ int exponent_of(double v) {
    const int e = (__double2hiint(v) >> 20) & 0x7FF;
    return e ? e : 1;
}

__device__ __forceinline__ void add(Fixed& a, const Fixed& b) {
    a.lo += b.lo;
    a.hi += b.hi + (a.lo < b.lo ? 1u : 0u);
}

__device__ __forceinline__ void add_value(Fixed& a, double v, int emax) {
    const unsigned long long bits = __double_as_longlong(v);
    const bool normal = (bits >> 52) & 0x7FFu;
    const unsigned long long m = (bits & 0xFFFFFFFFFFFFFull) | (normal ? 1ull << 52 : 0ull);
    const int up = kUp - (emax - exponent_of(v));
    Fixed t;
    t.lo = up >= 0 ? m << up : (up > -64 ? m >> -up : 0ull);
    t.hi = up > 0 ? m >> (64 - up) : 0ull;
    const unsigned long long neg = 0ull - (bits >> 63);  // all ones for a negative value
    t.lo ^= neg;
    t.hi ^= neg;
    t.lo -= neg;
    t.hi += neg && t.lo == 0ull ? 1u : 0u;
    add(a, t);
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

// largest of the threads' exponents, in every thread
__device__ __forceinline__ int block_max(int e) {
    __shared__ int sh[kThreads / 32];
    e = __reduce_max_sync(0xffffffffu, e);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = e;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) e = max(e, sh[w]);
    return e;
}

// a as a leading double and a remainder; NaN if a value was not finite (emax 2047)
__device__ __forceinline__ double2 to_pair(Fixed a, int emax) {
    if (emax == 0x7FF) return make_double2(__longlong_as_double(0x7ff8000000000000ll), 0.0);
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
    const double s = p2 + p1;                // p2 is zero or the larger
    const double low = (p1 - (s - p2)) + p0;
    const double top = s + low, rest = low - (top - s);
    return neg ? make_double2(-top, -rest) : make_double2(top, rest);
}

template <int PER>
__global__ void __launch_bounds__(kThreads) bound_reduce_noalloc_kernel(const double* __restrict__ v, int64_t n,
                                                                         double constant, double* __restrict__ out,
                                                                         Scratch* scr, unsigned call) {
    __shared__ bool last;
    const int64_t first = static_cast<int64_t>(blockIdx.x) * (kThreads * PER) + threadIdx.x;
    double x[PER];
    int e = 1;
#pragma unroll
    for (int q = 0; q < PER; ++q) x[q] = first + q * kThreads < n ? v[first + q * kThreads] : 0.0;
#pragma unroll
    for (int q = 0; q < PER; ++q) e = max(e, exponent_of(x[q]));
    e = block_max(e);
    Fixed a{0, 0};
#pragma unroll
    for (int q = 0; q < PER; ++q) add_value(a, x[q], e);
    block_sum(a);
    if (threadIdx.x == 0) {
        const double2 p = to_pair(a, e);
        scr->part[2 * blockIdx.x] = p.x;
        scr->part[2 * blockIdx.x + 1] = p.y;
        __threadfence();
        last = atomicInc(scr->ticket + call % kTickets, gridDim.x - 1) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    const int parts = 2 * static_cast<int>(gridDim.x);
    int el = 1;
    for (int q = threadIdx.x; q < parts; q += kThreads) el = max(el, exponent_of(__ldcg(scr->part + q)));
    __syncthreads();
    el = block_max(el);
    Fixed t{0, 0};
    for (int q = threadIdx.x; q < parts; q += kThreads) add_value(t, __ldcg(scr->part + q), el);
    __syncthreads();
    block_sum(t);
    if (threadIdx.x == 0) {
        const double2 p = to_pair(t, el);
        // (p.x + constant) with its rounding error added to the remainder
        const double s = p.x + constant;
        const double err = fabs(p.x) >= fabs(constant) ? (p.x - s) + constant : (constant - s) + p.x;
        *out = s + (err + p.y);
    }
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
    const unsigned call = g_calls.fetch_add(1, std::memory_order_relaxed);
    if (few) bound_reduce_noalloc_kernel<kFewPer><<<blocks, kThreads, 0, s>>>(dev_values, n, constant, dev_out, scr, call);
    else bound_reduce_noalloc_kernel<kManyPer><<<blocks, kThreads, 0, s>>>(dev_values, n, constant, dev_out, scr, call);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? FDOG_OK : FDOG_ECUDA;
}
