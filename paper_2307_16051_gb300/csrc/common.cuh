// common.cuh — shared device/host helpers for the sm_103a kernels.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <cstdio>
#include <string>

namespace nl {

// ---------------------------------------------------------------- host side --

// Thread-local last-error text, surfaced by nl_last_error().
void set_error(const char* fmt, ...);
const char* get_error();

#define NL_CUDA_OK(expr)                                                                   \
    do {                                                                                   \
        cudaError_t _e = (expr);                                                           \
        if (_e != cudaSuccess) {                                                           \
            ::nl::set_error("%s:%d %s: %s", __FILE__, __LINE__, #expr, cudaGetErrorString(_e)); \
            return NL_ECUDA;                                                               \
        }                                                                                  \
    } while (0)

#define NL_TRY(expr)                    \
    do {                                \
        nl_status _s = (expr);          \
        if (_s != NL_OK) return _s;     \
    } while (0)

inline int64_t round_up(int64_t a, int64_t b) { return (a + b - 1) / b * b; }
inline int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }

int num_sms();

// cudaMalloc that gives the workspaces kept by ws_malloc_async's pool back and
// tries again before it reports that the device is full: every device allocation
// of the library that is not from that pool.
cudaError_t trim_malloc(void** p, size_t bytes);
// The same for the handles' device pools; fails on purpose while the test
// hook nl_debug_fail_allocs has allocations left to fail.
cudaError_t dev_malloc(void** p, size_t bytes);

// Whether the next stream creation fails on purpose (the test hook nl_debug_fail_streams).
bool debug_fail_stream();

// Stream-ordered workspace of a kernel-level entry point, released with
// cudaFreeAsync: from the library's own memory pool on the current device,
// which keeps up to kWsKeep bytes of released memory across synchronisations
// (the default pool returns all of it to the system at each one and maps it
// again at the next call: 190 us of a call that synchronises).  trim_malloc gives
// the kept memory back, and so does this when the device is full.
constexpr size_t kWsKeep = (size_t)256 << 20;
cudaError_t ws_malloc_async(void** p, size_t bytes, cudaStream_t st);

// Carves 256-byte aligned sub-buffers out of one device allocation (a null
// base only measures: off is the size needed).
struct Carver {
    char* base;
    size_t off = 0;
    explicit Carver(void* b) : base((char*)b) {}
    template <typename T>
    T* take(size_t n)
    {
        off = (off + 255) & ~(size_t)255;
        T* p = (T*)(base + off);
        off += n * sizeof(T);
        return p;
    }
};

// Optional per-kernel-class timing (nl_kernel_timing): when enabled for a
// class, every launch of it is bracketed by CUDA events on its stream.
void prof_begin(const char* kernel_class, cudaStream_t st);
void prof_end(const char* kernel_class, cudaStream_t st);

// Raise a kernel's dynamic shared-memory limit to the device's opt-in maximum
// minus the kernel's static shared memory.  Clears the runtime error state on
// failure and reports it as NL_ECUDA.
int set_max_dynamic_smem(const void* func);

// Device-side error word bits (solver status block).
enum : unsigned {
    ERR_TIMEOUT_TRSV = 1u << 0,  // a triangular-solve block gave up waiting on a predecessor
    ERR_TIMEOUT_OTHER = 1u << 1,
    ERR_NONFINITE = 1u << 2,
};

// Bounded spin limit for inter-CTA waits: about a second at the spin period.
constexpr long long kSpinLimit = 1LL << 24;

// -------------------------------------------------------------- device side --

__device__ __forceinline__ float round_h(float v) { return __half2float(__float2half_rn(v)); }

// The multipliers of the binary16 factorisations, l = fl16(fl32(a / u)) for a
// binary16 pivot u != 0, with no division and no branch.  With y = -1/|u| from
// the hardware's approximate reciprocal (relative error at most 2^-23) and a
// given the sign of u (a'),
//   q = fl(a' y),  e = fl(q |u| + a'),  q' = fl(e y + q)
// is -fl32(a / u) exactly:
//   * q is within a few units of -a'/|u|, so e is exact (a 24-bit times an
//     11-bit significand, cancelled to a few units), and
//     q + e y = -a'/|u| (1 + d) with |d| < 2^-44;
//   * a quotient of a 24-bit by an 11-bit significand is never within 2^-36
//     (relative) of a midpoint of two binary32 values without being one (a' - m |u|
//     is a multiple of 2^-34 for a 25-bit m), and it is never a midpoint
//     (that m |u| has more than 24 bits); so q' rounds as the quotient does.
// Results below binary32's normal range round to a binary16 zero either way.
// y negative makes the sign of a zero result right: e is then +0.
__device__ __forceinline__ float rcp_neg_abs(float u)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(-fabsf(u)));
    return y;
}
// -fl32(a / u), u finite and not zero: us carries u's sign, y = rcp_neg_abs(u), den = |u|
__device__ __forceinline__ float div_neg(float a, float us, float y, float den)
{
    const float as = __uint_as_float(__float_as_uint(a) ^ (__float_as_uint(us) & 0x80000000u));
    const float q = __fmul_rn(as, y);
    return __fmaf_rn(__fmaf_rn(q, den, as), y, q);
}
__device__ __forceinline__ float div_round_h(float a, float u)
{
    return -round_h(div_neg(a, u, rcp_neg_abs(u), fabsf(u)));
}

// s / u, bit for bit, by u's reciprocal r = rcp_in_range(u), for chains of quotients by
// divisors known beforehand: the quotient corrected once by its exact remainder
// (P. Markstein, IBM J. Res. Dev. 34, 1990), three dependent instructions on the
// chain instead of a division's (and none of its slow paths: a zero numerator
// takes one).  With 2^-100 < |u| < 2^100 and 2^-900 <= |s| < 2^900 quotient, reciprocal
// and remainder are normal numbers and the remainder is exact; the product s r
// is within 1.5 units, and the corrected quotient rounds as the division does
// (for every pair of significands of 5 to 12 bits; more bits only make the
// exceptions rarer).  A zero numerator's product has the quotient's sign.  Every other
// numerator (huge, tiny, infinite, NaN) and every u with r = 0 takes the
// division.  The range tests are on the exponent bits, off the double-precision pipe.
__device__ __forceinline__ double rcp_in_range(double u)
{
    return fabs(u) >= 1e-30 && fabs(u) <= 1e30 ? 1.0 / u : 0.0;
}
__device__ __forceinline__ float rcp_in_range(float) { return 0.0f; }
__device__ __forceinline__ double div_by(double s, double u, double r)
{
    const unsigned hi = (unsigned)__double2hiint(s) & 0x7fffffffu;
    const double q = __dmul_rn(s, r);
    if (__double2hiint(r) == 0 || (hi >> 20) - 123u >= 1800u)  // biased exponents 123 .. 1922
        return __double2hiint(r) != 0 && (hi | (unsigned)__double2loint(s)) == 0u ? q : s / u;
    return __fma_rn(__fma_rn(-q, u, s), r, q);
}
__device__ __forceinline__ float div_by(float s, float u, float) { return s / u; }

template <typename T>
__device__ __forceinline__ T warp_sum(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Deterministic block-wide sum (fixed reduction tree).  `red` needs
// blockDim.x/32 entries.  Result valid in every thread.
template <typename T>
__device__ __forceinline__ T block_sum(T v, T* red)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    v = warp_sum(v);
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    T s = T(0);
    for (int w = 0; w < nw; ++w) s += red[w];
    return s;
}

// The sum of part[0 .. n), by every thread of the last block of a grid-wide
// reduction: each thread adds every blockDim.x-th partial in order, then the
// fixed tree of block_sum (red: blockDim.x / 32 entries; valid in every
// thread).  One thread adding all of them takes a dependent double addition
// each, the whole of a small kernel's tail: 2048 partials took 75 us of the
// residual's 263 us at N = 16384, and 512 about 10 of 29 us at N = 4096.
__device__ __forceinline__ double partials_sum(const double* part, int n, double* red)
{
    double t = 0.0;
    for (int q = threadIdx.x; q < n; q += blockDim.x) t += __ldcg(part + q);
    return block_sum(t, red);
}

__device__ __forceinline__ int ld_acquire_gpu(const int* p)
{
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release_gpu(int* p, int v)
{
    asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Element loads/stores for the three factor storage types.
__device__ __forceinline__ float ld_elem(const __half* p) { return __half2float(*p); }
__device__ __forceinline__ float ld_elem(const float* p) { return *p; }
__device__ __forceinline__ double ld_elem(const double* p) { return *p; }
__device__ __forceinline__ void st_elem(__half* p, float v) { *p = __float2half_rn(v); }
__device__ __forceinline__ void st_elem(float* p, float v) { *p = v; }
__device__ __forceinline__ void st_elem(double* p, double v) { *p = v; }

}  // namespace nl
