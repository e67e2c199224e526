// trsv.cu — z = U^{-1} L^{-1} P v with the factors of the LU (Algorithm IR's
// correction d = U^{-1} L^{-1} r, Section 2.2; the preconditioner-vector
// product of GMRES-IR).  For the half-precision factors the binary16 entries
// are promoted to single as they are loaded and all arithmetic is single
// (interprecision transfer on the fly, eq. (2.16), Section 2.3).
//
// Blocked substitution with block size T.  The inverses of the T x T
// diagonal blocks of L and U are formed once per factorisation (in the
// solve precision), so each block step is a small matrix-vector product.
// One cooperative launch per triangle: CTA g owns block rows g, g+G, ...;
// a block row accumulates the contributions of the finished blocks as their
// readiness flags appear (epoch-tagged, acquire/release), then multiplies by
// the diagonal inverse and publishes its slice.  Every wait is bounded: after
// about a second the CTA records a timeout in the error word and all CTAs
// return, leaving the context usable.
#include <cooperative_groups.h>

#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace nl {

namespace cg = cooperative_groups;

constexpr int T_ = kTrsvT;
constexpr int kTrsvThreads = 256;           // 64 rows x 4 column quarters
constexpr long long kWaitCycles = 2000000000LL;  // ~1 s at 2 GHz

template <typename T>
__device__ __forceinline__ T ldcg(const T* p) { return __ldcg(p); }

// ---------------------------------------------------------------- prepare --

// Final row permutation from the LAPACK-style interchanges:
// perm[i] = original index of the entry that ends up at position i.
__global__ void __launch_bounds__(1024) k_perm(int N, const int* __restrict__ ipiv, int* __restrict__ perm,
                                               int* __restrict__ list)
{
    extern __shared__ int ps[];
    __shared__ int cnt[1024];
    const int tid = threadIdx.x, nt = blockDim.x;
    for (int i = tid; i < N; i += nt) ps[i] = i;
    // compact the non-trivial interchanges, keeping their order
    const int seg = (N + nt - 1) / nt, a = tid * seg, e = min(N, a + seg);
    int c = 0;
    for (int k = a; k < e; ++k) c += (ipiv[k] != k);
    cnt[tid] = c;
    if (!__syncthreads_or(c)) {  // no interchanges (every factorisation of the H-equation): no serial pass
        for (int i = tid; i < N; i += nt) perm[i] = i;
        if (tid == 0) list[N] = 0;
        return;
    }
    if (tid == 0) {
        int s = 0;
        for (int q = 0; q < nt; ++q) {
            int v = cnt[q];
            cnt[q] = s;
            s += v;
        }
        list[N] = s;
    }
    __syncthreads();
    int o = cnt[tid];
    for (int k = a; k < e; ++k)
        if (ipiv[k] != k) list[o++] = k;
    __syncthreads();
    if (tid == 0) {
        const int m = list[N];
        for (int q = 0; q < m; ++q) {
            int k = list[q], p = ipiv[k];
            int t = ps[k];
            ps[k] = ps[p];
            ps[p] = t;
        }
    }
    __syncthreads();
    for (int i = tid; i < N; i += nt) perm[i] = ps[i];
}

// ------------------------------------------------------------------ solve --

__device__ __forceinline__ bool wait_flag(const int* flag, int epoch, unsigned* err)
{
    long long t0 = clock64();
    while (ld_acquire_gpu(flag) != epoch) {
        if (*((volatile unsigned*)err) != 0u) return false;
        if (clock64() - t0 > kWaitCycles) {
            atomicOr(err, (unsigned)ERR_TIMEOUT_TRSV);
            return false;
        }
        __nanosleep(20);
    }
    return true;
}

// LOWER: forward solve y = L^{-1} P v (block rows in increasing order).
// !LOWER: back solve z = U^{-1} y (block rows in decreasing order).
template <typename S, typename T, bool LOWER>
__global__ void __launch_bounds__(kTrsvThreads) k_trsv(int N, int nblk, const S* __restrict__ LU, int64_t ld,
                                                      const T* __restrict__ v, const int* __restrict__ perm,
                                                      const T* __restrict__ dinv, T* __restrict__ out,
                                                      int* __restrict__ flags, int epoch, unsigned* __restrict__ err)
{
    __shared__ T xs[T_];
    __shared__ T acc[T_];
    __shared__ int abort_s;
    const int tid = threadIdx.x, r = tid >> 2, qq = tid & 3;
    const T* Dinv = dinv + (LOWER ? 0 : (int64_t)nblk * T_ * T_);
    for (int g = blockIdx.x; g < nblk; g += gridDim.x) {
        const int b = LOWER ? g : nblk - 1 - g;
        const int r0 = b * T_, row = r0 + r;
        if (tid < T_) {
            int i = r0 + tid;
            T x = T(0);
            if (i < N) x = LOWER ? v[perm[i]] : ldcg(v + i);
            acc[tid] = x;
        }
        T part = T(0);
        const S* Lrow = LU + (int64_t)min(row, N - 1) * ld;
        const int c_begin = LOWER ? 0 : nblk - 1, c_end = LOWER ? b : b, c_step = LOWER ? 1 : -1;
        for (int c = c_begin; c != c_end; c += c_step) {
            if (tid == 0) abort_s = wait_flag(flags + c, epoch, err) ? 0 : 1;
            __syncthreads();
            if (abort_s) return;
            if (tid < T_) {
                int i = c * T_ + tid;
                xs[tid] = (i < N) ? ldcg(out + i) : T(0);
            }
            __syncthreads();
            if (row < N) {
                const int cb = c * T_ + qq * 16;
#pragma unroll
                for (int k = 0; k < 16; ++k) {
                    int col = cb + k;
                    T a = (col < N) ? (T)ld_elem(Lrow + col) : T(0);
                    part = fma(a, xs[qq * 16 + k], part);
                }
            }
        }
        part += __shfl_xor_sync(0xffffffffu, part, 1);
        part += __shfl_xor_sync(0xffffffffu, part, 2);
        __syncthreads();
        if (qq == 0) acc[r] -= part;
        __syncthreads();
        // slice = Dinv_b * acc
        const T* D = Dinv + (int64_t)b * T_ * T_ + r * T_ + qq * 16;
        T s = T(0);
#pragma unroll
        for (int k = 0; k < 16; ++k) s = fma(D[k], acc[qq * 16 + k], s);
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        if (qq == 0 && row < N) {
            out[row] = s;
            __threadfence();
        }
        __syncthreads();
        if (tid == 0) {
            __threadfence();
            st_release_gpu(flags + b, epoch);
        }
    }
}

// ---------------------------------------------- single-precision mailbox --
// For the single-precision solve each solved entry is published as one 64-bit
// word {value bits, epoch} with a release store; a consumer polls the word of
// the entry it needs with an acquire load, so readiness and data arrive
// together in one memory round trip.  Block size 128: the diagonal inverse
// (64 KB) is staged in shared memory and each thread prefetches its 64
// binary16 entries of the next tile before polling.
constexpr int T2 = 128;

// A published word carries its own readiness (the epoch) and its value, and a
// consumer reads nothing else the producer wrote, so relaxed GPU-scope accesses
// suffice (no acquire / release, hence no cache invalidation per poll).
__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long* p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed_u64(unsigned long long* p, unsigned long long v)
{
    asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// A 128 x 128 tile times a vector by 512 threads, as both half-precision solves
// do it: lane cg = lane & 15 of a half warp takes eight columns of the four rows
// 4 (2 warp + lane / 16).., so a row is read by 16 neighbouring lanes (whole lines),
// a thread reads eight of the vector's entries for four rows, and the 16 lanes'
// sums are reduced with five shuffles, which leave row e(lane) in the lane.
// (A row quarter per thread read the whole vector from shared memory for one
// row and every matrix line in eight pieces: twice the time per tile.)
// Vectors of 128 floats are padded to 144 (column c at c + 4 (c / 32)).
constexpr int kTvThreads = 512;
constexpr int kTvPad = 144;
__device__ __forceinline__ int tv_pos(int c) { return c + 4 * (c >> 5); }
// rows i0 .. i0 + 3, columns c0 .. c0 + 7 (zeros outside the matrix)
template <bool STREAM>
__device__ __forceinline__ void tv_load_tile(const __half* __restrict__ LU, int64_t ld, int N, int i0, int c0, bool vecld,
                                             uint4 (&t)[4])
{
    const bool vec = vecld && c0 + 8 <= N;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const __half* src = LU + (int64_t)(i0 + e) * ld + c0;
        if (vec && i0 + e < N) {
            t[e] = STREAM ? __ldcs(reinterpret_cast<const uint4*>(src)) : *reinterpret_cast<const uint4*>(src);
        } else {
            __half h[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) h[k] = (i0 + e < N && c0 + k < N) ? src[k] : __float2half_rn(0.0f);
            memcpy(&t[e], h, 16);
        }
    }
}
// p[e] += row e of the tile times z (the padded vector's entries 8 cg .. 8 cg + 7)
__device__ __forceinline__ void tv_dot_tile(const uint4 (&t)[4], const float* __restrict__ z, float (&p)[4])
{
    const float4 a = *reinterpret_cast<const float4*>(z), b = *reinterpret_cast<const float4*>(z + 4);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const __half2* h = reinterpret_cast<const __half2*>(&t[e]);
        const float2 f0 = __half22float2(h[0]), f1 = __half22float2(h[1]), f2 = __half22float2(h[2]),
                     f3 = __half22float2(h[3]);
        p[e] = fmaf(f0.x, a.x, p[e]);
        p[e] = fmaf(f0.y, a.y, p[e]);
        p[e] = fmaf(f1.x, a.z, p[e]);
        p[e] = fmaf(f1.y, a.w, p[e]);
        p[e] = fmaf(f2.x, b.x, p[e]);
        p[e] = fmaf(f2.y, b.y, p[e]);
        p[e] = fmaf(f3.x, b.z, p[e]);
        p[e] = fmaf(f3.y, b.w, p[e]);
    }
}
// rows i0 .. i0 + 3 of a 128 x 128 inverse: columns 4 cg .. and 64 + 4 cg ..
__device__ __forceinline__ void tv_load_inv(const float* __restrict__ D, int i0, int cg, float4 (&dq)[8])
{
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        dq[2 * e] = *reinterpret_cast<const float4*>(D + (i0 + e) * T2 + 4 * cg);
        dq[2 * e + 1] = *reinterpret_cast<const float4*>(D + (i0 + e) * T2 + 64 + 4 * cg);
    }
}
__device__ __forceinline__ void tv_dot_inv(const float4 (&dq)[8], const float* __restrict__ acc, int cg, float (&p)[4])
{
    const float4 a = *reinterpret_cast<const float4*>(acc + tv_pos(4 * cg)),
                 b = *reinterpret_cast<const float4*>(acc + tv_pos(64 + 4 * cg));
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        p[e] = dq[2 * e].x * a.x;
        p[e] = fmaf(dq[2 * e].y, a.y, p[e]);
        p[e] = fmaf(dq[2 * e].z, a.z, p[e]);
        p[e] = fmaf(dq[2 * e].w, a.w, p[e]);
        p[e] = fmaf(dq[2 * e + 1].x, b.x, p[e]);
        p[e] = fmaf(dq[2 * e + 1].y, b.y, p[e]);
        p[e] = fmaf(dq[2 * e + 1].z, b.z, p[e]);
        p[e] = fmaf(dq[2 * e + 1].w, b.w, p[e]);
    }
}
// The sum over the 16 lanes of row e(lane) = 2 (lane & 1) + (lane / 2 & 1).
__device__ __forceinline__ int tv_row(int lane) { return 2 * (lane & 1) + ((lane >> 1) & 1); }
__device__ __forceinline__ float tv_reduce(const float (&p)[4], int lane)
{
    const bool b0 = lane & 1, b1 = lane & 2;
    const float s0 = __shfl_xor_sync(0xffffffffu, b0 ? p[0] : p[2], 1), s1 = __shfl_xor_sync(0xffffffffu, b0 ? p[1] : p[3], 1);
    const float q0 = (b0 ? p[2] : p[0]) + s0, q1 = (b0 ? p[3] : p[1]) + s1;
    float v = (b1 ? q1 : q0) + __shfl_xor_sync(0xffffffffu, b1 ? q0 : q1, 2);
    v += __shfl_xor_sync(0xffffffffu, v, 4);
    v += __shfl_xor_sync(0xffffffffu, v, 8);
    return v;
}

// Bounded poll of one published entry: false once `limit` cycles have passed
// (a negative limit gives up before the first poll: the test of the timeout
// path, a wait that runs out whatever the producer does).
__device__ __forceinline__ bool poll_value(const unsigned long long* p, unsigned epoch, float* out,
                                           const unsigned* err, long long limit)
{
    if (limit < 0) return false;
    long long t0 = clock64();
    for (;;) {
        unsigned long long w = ld_relaxed_u64(p);
        if ((unsigned)(w >> 32) == epoch) {
            *out = __uint_as_float((unsigned)w);
            return true;
        }
        if (*((volatile const unsigned*)err) != 0u) return false;
        if (clock64() - t0 > limit) return false;
    }
}

template <bool LOWER>
__global__ void __launch_bounds__(kTvThreads, 1) k_trsv_mb(int N, int nblk, const __half* __restrict__ LU, int64_t ld,
                                                       const float* __restrict__ v,
                                                       const unsigned long long* __restrict__ vin_mb,
                                                       const int* __restrict__ perm, const float* __restrict__ dinv,
                                                       unsigned long long* __restrict__ mb, float* __restrict__ out,
                                                       unsigned epoch, unsigned* __restrict__ err, long long wait_cycles,
                                                       const float* __restrict__ rs)
{
    __shared__ __align__(16) float ys[2][kTvPad];  // the tile's vector, alternating
    __shared__ __align__(16) float acc[kTvPad];
    const int tid = threadIdx.x, lane = tid & 31, cg = lane & 15;
    const int row4 = 4 * (2 * (tid >> 5) + (lane >> 4));  // this thread's four rows of a block
    const bool vecld = ((((uintptr_t)LU) & 15) == 0) && (ld % 8 == 0);
    const float* Dinv = dinv + (LOWER ? 0 : (int64_t)nblk * T2 * T2);
    for (int g = blockIdx.x; g < nblk; g += gridDim.x) {
        const int b = LOWER ? g : nblk - 1 - g;
        const int r0 = b * T2;
        __syncthreads();
        float4 dq[8];  // this thread's part of the block's diagonal inverse (independent of the waits)
        tv_load_inv(Dinv + (int64_t)b * T2 * T2, row4, cg, dq);
        if (tid < T2) {
            const int i = r0 + tid;
            float x = 0.0f;
            if (i < N)
                x = LOWER ? (rs ? v[perm[i]] * rs[perm[i]] : v[perm[i]]) : __uint_as_float((unsigned)vin_mb[i]);
            acc[tv_pos(tid)] = x;
        }
        float p[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        const int cnt = LOWER ? b : nblk - 1 - b;
        // tile (b, c): its entries are loaded one tile ahead of their use, streamed once (not kept in the caches).
        // Two ahead needs more than the 128 registers (44 bytes spilled) and takes 96 us a pair of triangles
        // at N = 4096 and 283 at 12000, one ahead 86 and 261.
        auto fetch = [&](int s, uint4 (&t)[4]) {
            const int c = LOWER ? s : nblk - 1 - s;
            tv_load_tile<true>(LU, ld, N, r0 + row4, c * T2 + 8 * cg, vecld, t);
        };
        auto poll = [&](int s) -> bool {  // threads 0..127: the vector of tile s
            if (tid >= T2) return true;
            const int i = (LOWER ? s : nblk - 1 - s) * T2 + tid;
            float y = 0.0f;
            const bool okp = i >= N || poll_value(mb + i, epoch, &y, err, wait_cycles);
            ys[s & 1][tv_pos(tid)] = y;
            return okp;
        };
        uint4 t0[4], t1[4];
        if (cnt > 0) fetch(0, t0);
        for (int s = 0; s < cnt; ++s) {
            if (s + 1 < cnt) fetch(s + 1, t1);
            if (__syncthreads_or(!poll(s))) {  // (the other buffer's readers are at most one tile behind)
                if (tid == 0) atomicOr(err, (unsigned)ERR_TIMEOUT_TRSV);
                return;
            }
            tv_dot_tile(t0, ys[s & 1] + tv_pos(8 * cg), p);
#pragma unroll
            for (int q = 0; q < 4; ++q) t0[q] = t1[q];
        }
        const float part = tv_reduce(p, lane);
        if (cnt == 0) __syncthreads();  // (acc was written by other threads; with tiles the loop's barriers passed)
        if (cg < 4) acc[tv_pos(row4 + tv_row(lane))] -= part;
        __syncthreads();
        tv_dot_inv(dq, acc, cg, p);
        const float sum = tv_reduce(p, lane);
        const int row = r0 + row4 + tv_row(lane);
        if (cg < 4 && row < N) {
            if (out) out[row] = sum;
            st_relaxed_u64(mb + row, ((unsigned long long)epoch << 32) | __float_as_uint(sum));
        }
    }
}

// ------------------------------------------------ cluster triangular solve --
// One thread-block cluster of C CTAs (C <= 16) solves both triangles in one
// launch.  Block b of 128 rows belongs to CTA (step of b) mod C, which keeps the
// running right-hand side of its blocks in shared memory.  The owner of step
// s forms z_b = Dinv_b acc_b and stores z_b into every CTA's shared memory
// with st.async (16 bytes a lane: one instruction per warp for all 16 CTAs),
// each store completing a transaction count on that CTA's mbarrier for step s
// (one mbarrier per block and triangle, used once).  A CTA waits
// only for the z it needs next; the owner of step s+1 first subtracts
// L(b(s+1), b(s)) z_s, with the tile already in registers, then publishes
// z_{b(s+1)} before it applies z_s to its other blocks, so the chain from
// one block to the next is one shared-memory signal and two 128 x 128
// products (tile and inverse, both held in registers).  The tiles off the chain are loaded one ahead of their use.
// Every row of the factor is read by exactly one CTA.  Bound by the chain
// (2 N / 128 steps) up to N = 4096 or so, above it by the 16 SMs' share of L2 and
// HBM bandwidth.  Measured per solve pair: N = 256 12.5, 1024 26, 2048 49, 4096 102 us
// (two launches, each element stored to each CTA by itself, and tiles loaded
// when used: 20, 35, 58, 124).
constexpr int kClThreads = kTvThreads;
constexpr int kClPad = kTvPad;
constexpr int kClMaxSmem = 220 * 1024;
constexpr long long kClWaitIters = 1LL << 24;

// Dynamic shared memory: 2 nblk mbarriers, then nblk + nown padded vectors.
__host__ __device__ inline int trsv_cl_bar_bytes(int nblk) { return nblk * 16; }
inline size_t trsv_cl_smem(int nblk, int nown)
{
    return (size_t)trsv_cl_bar_bytes(nblk) + (size_t)(nblk + nown) * kClPad * sizeof(float);
}

__device__ __forceinline__ uint32_t cl_smem_u32(const void* p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ uint32_t cl_mapa(uint32_t a, int rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void cl_st_async4(uint32_t addr, const float (&v)[4], uint32_t bar)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr),
                 "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])),
                 "r"(__float_as_uint(v[3])), "r"(bar)
                 : "memory");
}
// Bounded wait for phase 0 of a local mbarrier; false after `iters` polls
// (kClWaitIters by default; 0 gives up at once, the test of the timeout path).
__device__ __forceinline__ bool cl_wait(uint32_t bar, long long iters = kClWaitIters)
{
    for (long long it = 0; it < iters; ++it) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0;\n"
            " selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(bar)
            : "memory");
        if (done) return true;
    }
    return false;
}

struct ClState {
    int N, nblk, C, rank, nown;
    const __half* LU;
    int64_t ld;
    bool vecld;
    float *yv, *acc;
    int* abort_cta;
    unsigned* err;
    long long wait_iters;
};

// One triangle: acc holds the right-hand side of this CTA's blocks (in the
// triangle's block order), bar its nblk mbarriers; the solution is left in
// every CTA's yv and, if out is given, written there.
template <bool LOWER>
__device__ __forceinline__ void cl_triangle(const ClState& S, const float* __restrict__ Dinv, uint64_t* bar,
                                            float* __restrict__ out)
{
    const int tid = threadIdx.x, lane = tid & 31, cg = lane & 15;
    const int row4 = 4 * (2 * (tid >> 5) + (lane >> 4));  // this thread's four rows of a block
    const int prow = tv_pos(row4 + tv_row(lane));         // padded position of the row whose sum it gets
    const int C = S.C, rank = S.rank, nblk = S.nblk, nown = S.nown, N = S.N;
    float* yv = S.yv;
    float* acc = S.acc;
    auto blk = [&](int s) { return LOWER ? s : nblk - 1 - s; };
    float4 dq[8];  // this thread's part of the inverse of the next block it publishes
    uint4 ct[4];   // its factor entries of the next tile on its chain
    uint4 nt[4];   // and of the next tile off the chain
    auto load_D = [&](int b) { tv_load_inv(Dinv + (int64_t)b * T2 * T2, row4, cg, dq); };
    auto load_tile = [&](int sb, int sc, uint4 (&t)[4]) {  // rows of step sb's block, columns of step sc's
        tv_load_tile<false>(S.LU, S.ld, N, blk(sb) * T2 + row4, blk(sc) * T2 + 8 * cg, S.vecld, t);
    };
    // this CTA's first block off the chain at step s (the chain's is step s + 1's)
    auto first_off = [&](int s) {
        const int j = (s < rank) ? 0 : (s - rank) / C + 1;  // its blocks solved after step s
        return (j < nown && rank + j * C == s + 1) ? j + 1 : j;
    };
    // acc of its block j minus a tile times z
    auto apply = [&](int j, const uint4 (&t)[4], const float* z) {
        float p[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        tv_dot_tile(t, z + tv_pos(8 * cg), p);
        const float part = tv_reduce(p, lane);
        if (cg < 4) acc[j * kClPad + prow] -= part;
    };
    // z_b = Dinv_b acc_b for the step s this CTA owns, stored into every CTA
    auto publish = [&](int s) {
        const int b = blk(s);
        float p[4];
        tv_dot_inv(dq, acc + (s / C) * kClPad, cg, p);
        const float sum = tv_reduce(p, lane);
        // lane: its half warp's four rows to CTA cg
        float v[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] = __shfl_sync(0xffffffffu, sum, (lane & 0x1c) | (e >> 1) | ((e & 1) << 1));
        if (cg < C)
            cl_st_async4(cl_mapa(cl_smem_u32(yv + (size_t)b * kClPad + tv_pos(row4)), cg), v,
                         cl_mapa(cl_smem_u32(bar + s), cg));
        if (out && cg < 4) {
            const int i = b * T2 + row4 + tv_row(lane);
            if (i < N) out[i] = sum;
        }
        if (s + C < nblk) {
            // inverse and chain tile for this CTA's next step s + C
            load_D(blk(s + C));
            load_tile(s + C, s + C - 1, ct);
        }
    };
    if (rank < nblk) load_D(blk(rank));
    if (rank >= 1 && rank < nblk) load_tile(rank, rank - 1, ct);
    if (rank == 0) publish(0);
    if (first_off(0) < nown) load_tile(rank + first_off(0) * C, 0, nt);
    for (int s = 0; s < nblk; ++s) {
        const int b = blk(s);
        bool ok = false;
        if (!*((volatile int*)S.abort_cta)) {
            ok = cl_wait(cl_smem_u32(bar + s), S.wait_iters);
            if (!ok) {
                *S.abort_cta = 1;
                atomicOr(S.err, (unsigned)ERR_TIMEOUT_TRSV);
            }
        }
        // one answer per warp (apply's shuffles name all lanes): lanes may see the bound or the abort word differently
        __syncwarp();
        ok = __all_sync(0xffffffffu, ok);
        const float* z = yv + (size_t)b * kClPad;
        int j = (s < rank) ? 0 : (s - rank) / C + 1;  // this CTA's blocks solved after step s
        if (j < nown && rank + j * C == s + 1) {
            // next block on the chain: update with the tile already in registers, then publish it
            if (ok) apply(j, ct, z);
            __syncthreads();
            publish(s + 1);
            ++j;
        }
        const int jn = s + 1 < nblk ? first_off(s + 1) : nown;  // the next step's first tile
        for (; j < nown; ++j) {
            uint4 t[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) t[q] = nt[q];
            if (j + 1 < nown) load_tile(rank + (j + 1) * C, s, nt);
            else if (jn < nown) load_tile(rank + jn * C, s + 1, nt);
            if (ok) apply(j, t, z);
        }
    }
    // After a wait gave up, the owners of the later steps still publish them
    // (their values unused), so every mbarrier of this CTA still completes:
    // wait for all of them (the default bound) before leaving, so that no
    // st.async into this CTA's shared memory is still in flight when it exits.
    __syncthreads();
    if (*((volatile int*)S.abort_cta))
        for (int s = 0; s < nblk; ++s) cl_wait(cl_smem_u32(bar + s));
}

__global__ void __launch_bounds__(kClThreads, 1) k_trsv_cl(int N, int nblk, const __half* __restrict__ LU, int64_t ld,
                                                       const float* __restrict__ v, const int* __restrict__ perm,
                                                       const float* __restrict__ dinv, float* __restrict__ out,
                                                       unsigned* __restrict__ err, long long wait_iters,
                                                       const float* __restrict__ rs)
{
    cg::cluster_group cl = cg::this_cluster();
    extern __shared__ __align__(16) unsigned char cl_raw[];
    __shared__ int abort_cta;
    uint64_t* bar = reinterpret_cast<uint64_t*>(cl_raw);
    ClState S;
    S.N = N;
    S.nblk = nblk;
    S.C = (int)cl.num_blocks();
    S.rank = (int)cl.block_rank();
    S.nown = (nblk - S.rank + S.C - 1) / S.C;
    S.LU = LU;
    S.ld = ld;
    S.vecld = ((((uintptr_t)LU) & 15) == 0) && ((ld * 2) % 16 == 0);
    S.yv = reinterpret_cast<float*>(cl_raw + trsv_cl_bar_bytes(nblk));  // solved blocks, padded
    S.acc = S.yv + (size_t)nblk * kClPad;                                // this CTA's blocks, padded
    S.abort_cta = &abort_cta;
    S.err = err;
    S.wait_iters = wait_iters;
    const int tid = threadIdx.x;
    for (int j = 0; j < S.nown; ++j)
        for (int t = tid; t < T2; t += kClThreads) {
            const int i = (S.rank + j * S.C) * T2 + t;
            S.acc[j * kClPad + tv_pos(t)] = (i < N) ? (rs ? v[perm[i]] * rs[perm[i]] : v[perm[i]]) : 0.0f;
        }
    if (tid == 0) abort_cta = 0;
    for (int s = tid; s < 2 * nblk; s += kClThreads) {
        const uint32_t a = cl_smem_u32(bar + s);
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(a));
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(a), "r"(T2 * 4) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    cl.sync();  // barriers initialised and every CTA running before the first remote store
    cl_triangle<true>(S, dinv, bar, nullptr);
    // every CTA holds all of y and has used it: the blocks' right-hand sides of the
    // upper triangle, whose solution overwrites it
    cl.sync();
    for (int j = 0; j < S.nown; ++j)
        for (int t = tid; t < T2; t += kClThreads) {
            const int p = tv_pos(t), b = nblk - 1 - (S.rank + j * S.C);
            S.acc[j * kClPad + p] = (b * T2 + t < N) ? S.yv[(size_t)b * kClPad + p] : 0.0f;
        }
    cl.sync();  // (read before any CTA publishes into yv)
    cl_triangle<false>(S, dinv + (int64_t)nblk * T2 * T2, bar + nblk, out);
    cl.sync();  // no CTA leaves before every CTA has passed all of its waits
}

// ------------------------------------------------------------------- host --

static int trsv_block(bool fp64) { return fp64 ? T_ : T2; }

size_t trsv_work_bytes(int N, bool fp64)
{
    const int tb = trsv_block(fp64);
    int nblk = (int)cdiv(N, tb);
    size_t el = fp64 ? 8 : 4;
    return round_up((size_t)N * 4, 256) + round_up((size_t)2 * nblk * tb * tb * el, 256) +
           round_up((size_t)2 * nblk * 4, 256) + round_up((size_t)N * 8 * 2, 256) + 256 +
           round_up((size_t)(N + 1) * 4, 256);
}

void trsv_work_carve(void* base, int N, bool fp64, TrsvWork* w)
{
    const int tb = trsv_block(fp64);
    int nblk = (int)cdiv(N, tb);
    size_t el = fp64 ? 8 : 4;
    char* p = (char*)base;
    w->perm = (int*)p;
    p += round_up((size_t)N * 4, 256);
    w->dinv = p;
    p += round_up((size_t)2 * nblk * tb * tb * el, 256);
    w->flags = (int*)p;
    p += round_up((size_t)2 * nblk * 4, 256);
    w->y = p;  // double: N elements; float: 2 x N 64-bit mailbox words
    p += round_up((size_t)N * 8 * 2, 256);
    w->err = (unsigned*)p;
    p += 256;
    w->scan = (int*)p;
}

// Diagonal-block inverses for block size TB, right-looking: once X's row t of
// a column is final, it is applied to every later row, so the rows have no
// dependence chain among them.  L (unit lower): entry i of column c is
// -sum_{t=c}^{i-1} l_it x_t with the terms added in increasing t, x_c = 1.  U:
// x_t = s_t / u_tt with s_i = [i == c] - sum_{t>i} u_it x_t, the terms added in
// decreasing t.  Entries outside the block (a ragged last block) are zero.
//
// A CTA takes one triangle of one block and kInvC columns, eight threads per
// column: thread (c, g) keeps the rows i = g mod 8 in registers, and the owner
// of row t hands x_t to the others through shared memory, one barrier per step.
// Bound in double precision: an instruction occupies its warp for about 65
// cycles until four warps keep the SM's few units busy (then 19 each), so the
// work is spread over all SMs, four warps each.  One thread per column and both
// triangles in one CTA of two warps took 162 us at N = 1001; this takes 38 (41 at N = 2048).
constexpr int kInvC = 16, kInvG = 8;

template <typename S, typename T, int TB>
__global__ void __launch_bounds__(kInvC * kInvG) k_invdiag_t(int N, const S* __restrict__ LU, int64_t ld,
                                                             T* __restrict__ dinv, int nblk)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* At = reinterpret_cast<T*>(smem_raw);  // At[t * (TB + 1) + i]: entry (i, t)
    __shared__ T xs[2][kInvC], rd[TB];
    constexpr int R = TB / kInvG, kGroups = TB / kInvC, W = TB + 1;
    const int b = blockIdx.x / (2 * kGroups), tri = (blockIdx.x / kGroups) & 1, c0 = (blockIdx.x % kGroups) * kInvC;
    const int r0 = b * TB, nb_ = min(TB, N - r0), tid = threadIdx.x;
    const int c = tid % kInvC, g = tid / kInvC, col = c0 + c;
    for (int e = tid; e < TB * TB; e += kInvC * kInvG) {
        const int i = e / TB, j = e % TB;
        At[j * W + i] = (i < nb_ && j < nb_) ? (T)ld_elem(LU + (int64_t)(r0 + i) * ld + r0 + j) : T(0);
    }
    __syncthreads();
    T acc[R];  // rows g + 8 r
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r] = T(0);
    if (tri == 0) {
#pragma unroll
        for (int tb = 0; tb < R; ++tb)
            for (int tg = (8 * tb < c0 ? 8 : 0); tg < 8; ++tg) {  // (c0: a multiple of eight)
                const int t = 8 * tb + tg;
                if (t >= nb_) break;
                if (g == tg) {
                    if (t >= col) acc[tb] = t == col ? T(1) : -acc[tb];
                    xs[t & 1][c] = acc[tb];
                }
                __syncthreads();
                const T xt = xs[t & 1][c];
                if (t >= col) {
                    const T* a = At + t * W + g;
                    if (g > tg) acc[tb] = fma(a[8 * tb], xt, acc[tb]);
#pragma unroll
                    for (int r = tb + 1; r < R; ++r) acc[r] = fma(a[8 * r], xt, acc[r]);
                }
            }
    } else {
        if (tid < TB) {
            rd[tid] = rcp_in_range(At[tid * W + tid]);
        }
#pragma unroll
        for (int r = 0; r < R; ++r) acc[r] = g + 8 * r == col && col < nb_ ? T(1) : T(0);
        __syncthreads();
#pragma unroll
        for (int tb = R - 1; tb >= 0; --tb)
            for (int tg = 7; tg >= 0; --tg) {
                const int t = 8 * tb + tg;
                if (t >= nb_ || t >= c0 + kInvC) continue;
                if (g == tg) {
                    if (t <= col && col < nb_) acc[tb] = div_by(acc[tb], At[t * W + t], rd[t]);
                    xs[t & 1][c] = acc[tb];
                }
                __syncthreads();
                const T xt = -xs[t & 1][c];
                if (t <= col && col < nb_) {
                    const T* a = At + t * W + g;
                    if (g < tg) acc[tb] = fma(a[8 * tb], xt, acc[tb]);
#pragma unroll
                    for (int r = 0; r < tb; ++r) acc[r] = fma(a[8 * r], xt, acc[r]);
                }
            }
    }
    T* out = dinv + (int64_t)(tri * nblk + b) * TB * TB;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = g + 8 * r;
        out[i * TB + col] = i < nb_ && col < nb_ ? acc[r] : T(0);
    }
}

// The binary16 factors' 128 x 128 diagonal-block inverses, the recurrences of
// k_invdiag_t with the terms of every entry in the same order, one thread per
// column.  The rows are taken in chunks of 32 (from the last one up for U):
// the chunk's 32 accumulators stay in registers while the finished rows t are
// applied (the block's column t, staged transposed, is the same for every
// thread: eight broadcast loads for 32 fused multiply-adds), then the chunk is
// solved against its own 32 x 32 triangle.  Bound by the multiply-adds of the
// column with the most rows (192 t of 32 and four triangles).  A warp skips the
// rows t before (U: after) its 32 columns, where x_t is zero.  Four threads per
// column, right-looking, each re-reading its 32 entries of column t at every
// step, took 50 us; this takes 27 us (N <= 2048, launch included).
constexpr int kInvThreads = 128;
constexpr int kInvS = 132;  // stride of the transposed block (floats)
constexpr size_t kInvSmem = (size_t)T2 * kInvS * sizeof(float) + (size_t)T2 * T2 * sizeof(float) + T2 * sizeof(float);

template <bool UPPER>
__device__ __forceinline__ void invdiag16_pass(const __half* __restrict__ LU, int64_t ld, float* __restrict__ D, int r0,
                                               int nb_)
{
    extern __shared__ __align__(16) float inv_sm[];
    float* At = inv_sm;              // At[t * kInvS + i]: entry (i, t), U's negated
    float* X = At + T2 * kInvS;      // X[t * T2 + column]
    float* dg = X + T2 * T2;
    const int col = threadIdx.x, warp = threadIdx.x >> 5;
    {
        const int i = threadIdx.x;  // a row of the block
        const __half* src = LU + (int64_t)(r0 + min(i, nb_ - 1)) * ld + r0;
        const bool vec = nb_ == T2 && ((((uintptr_t)(LU + r0)) & 15) == 0) && (ld % 8 == 0);
#pragma unroll 4
        for (int t0 = 0; t0 < T2; t0 += 8) {
            __align__(16) __half h[8];
            if (vec) {
                *reinterpret_cast<uint4*>(h) = *reinterpret_cast<const uint4*>(src + t0);
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e) h[e] = (i < nb_ && t0 + e < nb_) ? src[t0 + e] : __float2half_rn(0.0f);
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float v = __half2float(h[e]);
                At[(t0 + e) * kInvS + i] = UPPER ? -v : v;
                if (t0 + e == i) dg[i] = v;
            }
        }
    }
    __syncthreads();
    const bool live = col < nb_;
    for (int s = 0; s < T2 / 32; ++s) {
        const int R = UPPER ? 3 - s : s, i0 = 32 * R;
        float acc[32];
#pragma unroll
        for (int r = 0; r < 32; ++r) acc[r] = (UPPER && i0 + r == col && live) ? 1.0f : 0.0f;
        if (UPPER ? R <= warp : R >= warp) {
            // finished rows: for L the chunks warp .. R-1 in increasing order, for U warp .. R+1 in decreasing order
            const int n = 32 * (UPPER ? warp - R : R - warp);
            int t = UPPER ? 32 * warp + 31 : 32 * warp;
#pragma unroll 2
            for (int m = 0; m < n; ++m, t += UPPER ? -1 : 1) {
                const float xt = X[t * T2 + col];
                const float4* a4 = reinterpret_cast<const float4*>(At + t * kInvS + i0);
#pragma unroll
                for (int g = 0; g < 8; ++g) {
                    const float4 v = a4[g];
                    acc[4 * g] = fmaf(v.x, xt, acc[4 * g]);
                    acc[4 * g + 1] = fmaf(v.y, xt, acc[4 * g + 1]);
                    acc[4 * g + 2] = fmaf(v.z, xt, acc[4 * g + 2]);
                    acc[4 * g + 3] = fmaf(v.w, xt, acc[4 * g + 3]);
                }
            }
#pragma unroll
            for (int k = 0; k < 32; ++k) {
                const int tt = UPPER ? 31 - k : k, t = i0 + tt;
                float xt = 0.0f;
                if (live && t < nb_) {
                    if (UPPER) xt = (t > col) ? 0.0f : acc[tt] / dg[t];
                    else xt = (t < col) ? 0.0f : ((t == col) ? 1.0f : -acc[tt]);
                }
                acc[tt] = xt;
                const float4* a4 = reinterpret_cast<const float4*>(At + t * kInvS + i0);
#pragma unroll
                for (int g = 0; g < 8; ++g) {
                    if (UPPER ? 4 * g >= tt : 4 * g + 3 <= tt) continue;
                    const float4 v = a4[g];
                    const float a[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int i = 4 * g + e;
                        if (UPPER ? i < tt : i > tt) acc[i] = fmaf(a[e], xt, acc[i]);
                    }
                }
            }
        }
#pragma unroll
        for (int r = 0; r < 32; ++r) {
            X[(i0 + r) * T2 + col] = acc[r];  // (read back by this thread only)
            D[(i0 + r) * T2 + col] = acc[r];
        }
    }
}

// CTA b < nblk: L^{-1} of block b; CTA nblk + b: U^{-1} of block b (U's
// entries are staged negated, so both updates are fma(a, x_t, acc)).
__global__ void __launch_bounds__(kInvThreads) k_invdiag16(int N, const __half* __restrict__ LU, int64_t ld,
                                                           float* __restrict__ dinv, int nblk)
{
    const bool upper = (int)blockIdx.x >= nblk;
    const int b = upper ? (int)blockIdx.x - nblk : (int)blockIdx.x;
    const int r0 = b * T2, nb_ = min(T2, N - r0);
    float* D = dinv + (int64_t)blockIdx.x * T2 * T2;
    if (upper)
        invdiag16_pass<true>(LU, ld, D, r0, nb_);
    else
        invdiag16_pass<false>(LU, ld, D, r0, nb_);
}

template <typename S, typename T>
static nl_status prepare_impl(int N, const S* LU, int64_t ld, const int* ipiv, const TrsvWork& w, cudaStream_t st,
                              int* launches)
{
    constexpr bool half = std::is_same<S, __half>::value;
    constexpr int TB = half ? T2 : T_;  // the block size of the solve that follows
    const int nblk = (int)cdiv(N, TB);
    static bool attr = false;
    if (!attr) {
        const void* inv;
        if constexpr (half) inv = (const void*)k_invdiag16;
        else inv = (const void*)k_invdiag_t<S, T, TB>;
        if (set_max_dynamic_smem((const void*)k_perm) != NL_OK || set_max_dynamic_smem(inv) != NL_OK) return NL_ECUDA;
        attr = true;
    }
    if ((size_t)N * 4 > 200 * 1024) {
        set_error("trsv: N=%d too large for the permutation kernel", N);
        return NL_EINVAL;
    }
    k_perm<<<1, 1024, (size_t)N * 4, st>>>(N, ipiv, w.perm, w.scan);
    prof_begin("k_invdiag", st);
    if constexpr (half)
        k_invdiag16<<<2 * nblk, kInvThreads, kInvSmem, st>>>(N, LU, ld, (float*)w.dinv, nblk);
    else
        k_invdiag_t<S, T, TB><<<2 * nblk * (TB / kInvC), kInvC * kInvG, (size_t)TB * (TB + 1) * sizeof(T), st>>>(
            N, LU, ld, (T*)w.dinv, nblk);
    prof_end("k_invdiag", st);
    NL_CUDA_OK(cudaGetLastError());
    if (launches) *launches += 2;
    return NL_OK;
}

nl_status trsv_prepare16(int N, const __half* LU, int64_t ld, const int* ipiv, const TrsvWork& w, cudaStream_t st,
                         int* launches)
{
    return prepare_impl<__half, float>(N, LU, ld, ipiv, w, st, launches);
}

nl_status trsv_prepare64(int N, const double* LU, int64_t ld, const int* ipiv, const TrsvWork& w, cudaStream_t st,
                         int* launches)
{
    return prepare_impl<double, double>(N, LU, ld, ipiv, w, st, launches);
}

nl_status trsv_prepare32(int N, const float* LU, int64_t ld, const int* ipiv, const TrsvWork& w, cudaStream_t st,
                         int* launches)
{
    return prepare_impl<float, float>(N, LU, ld, ipiv, w, st, launches);
}

template <typename S, typename T, bool LOWER>
static nl_status launch_trsv(int N, const S* LU, int64_t ld, const T* v, T* out, const TrsvWork& w, int epoch,
                             int* flags, cudaStream_t st)
{
    const int nblk = (int)cdiv(N, T_);
    auto kern = k_trsv<S, T, LOWER>;
    static int max_grid = 0;
    if (max_grid == 0) {
        int per_sm = 0;
        NL_CUDA_OK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kTrsvThreads, 0));
        max_grid = std::max(1, per_sm) * num_sms();
    }
    int grid = std::min(nblk, max_grid);
    const int* perm = w.perm;
    const T* dinv = (const T*)w.dinv;
    unsigned* err = w.err;
    void* args[] = {(void*)&N, (void*)&nblk, (void*)&LU, (void*)&ld, (void*)&v, (void*)&perm, (void*)&dinv,
                    (void*)&out, (void*)&flags, (void*)&epoch, (void*)&err};
    NL_CUDA_OK(cudaLaunchCooperativeKernel((const void*)kern, dim3(grid), dim3(kTrsvThreads), args, 0, st));
    return NL_OK;
}

template <typename S, typename T>
static nl_status solve_impl(int N, const S* LU, int64_t ld, const T* v, T* z, const TrsvWork& w, int epoch,
                            cudaStream_t st, int* launches)
{
    const int nblk = (int)cdiv(N, T_);
    T* y = (T*)w.y;
    nl_status s = launch_trsv<S, T, true>(N, LU, ld, v, y, w, epoch, w.flags, st);
    if (s != NL_OK) return s;
    s = launch_trsv<S, T, false>(N, LU, ld, y, z, w, epoch, w.flags + nblk, st);
    if (launches) *launches += 2;
    return s;
}

template <bool LOWER>
static nl_status launch_trsv_mb(int N, const __half* LU, int64_t ld, const float* v, const unsigned long long* vin_mb,
                                unsigned long long* mb, float* out, const TrsvWork& w, unsigned epoch, cudaStream_t st)
{
    const int nblk = (int)cdiv(N, T2);
    auto kern = k_trsv_mb<LOWER>;
    static int max_grid = 0;
    if (max_grid == 0) {
        int per_sm = 0;
        NL_CUDA_OK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kTvThreads, 0));
        max_grid = std::max(1, per_sm) * num_sms();
    }
    int grid = std::min(nblk, max_grid);
    const int* perm = w.perm;
    const float* dinv = (const float*)w.dinv;
    unsigned* err = w.err;
    long long wait = w.wait_limit == 0 ? kWaitCycles : (w.wait_limit < 0 ? -1LL : (long long)w.wait_limit);
    const float* rs = w.rs;
    void* args[] = {(void*)&N,   (void*)&nblk, (void*)&LU,  (void*)&ld,    (void*)&v,   (void*)&vin_mb, (void*)&perm,
                    (void*)&dinv, (void*)&mb, (void*)&out, (void*)&epoch, (void*)&err, (void*)&wait, (void*)&rs};
    prof_begin("k_trsv_mb", st);
    cudaError_t le = cudaLaunchCooperativeKernel((const void*)kern, dim3(grid), dim3(kTvThreads), args, 0, st);
    prof_end("k_trsv_mb", st);
    NL_CUDA_OK(le);
    return NL_OK;
}

// Whether a cluster of C CTAs of the cluster triangular solve can be
// co-scheduled on this device (cached per process; C in {4, 8, 16}).
static bool trsv_cluster_ok(int C)
{
    static int avail[3] = {-1, -1, -1};
    const int slot = C == 16 ? 2 : (C == 8 ? 1 : 0);
    if (avail[slot] < 0) {
        bool ok = true;
        do {
            const void* kern = (const void*)k_trsv_cl;
            if (cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
                cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kClMaxSmem) != cudaSuccess) {
                ok = false;
                break;
            }
            cudaLaunchConfig_t cfg = {};
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = C;
            attr[0].val.clusterDim.y = 1;
            attr[0].val.clusterDim.z = 1;
            cfg.gridDim = dim3(C);
            cfg.blockDim = dim3(kClThreads);
            cfg.dynamicSmemBytes = kClMaxSmem;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess || n < 1) ok = false;
        } while (false);
        cudaGetLastError();
        avail[slot] = ok ? 1 : 0;
    }
    return avail[slot] == 1;
}

// Cluster size for nblk blocks under the request req (0 = largest available,
// -1 = none, else the largest available <= req); 0 = use the mailbox solve.
// Automatic choice: the cluster's 16 SMs stream the whole factor, so beyond
// 24 blocks (N > 3072) the mailbox solve over all SMs is faster (measured on
// GB300 per solve pair, cluster / mailbox: 26 / 29 us at N = 1024, 49 / 49 at 2048, 77 / 69 at
// 3072, 90 / 79 at 3584, 103 / 90 at 4096, 299 / 173 at 8192; mailbox alone 261 us at
// 12000, 347 at 16384, where a row half per thread with its inverse in shared memory took
// 600 and 980).  The line lies between the sizes where a mailbox that loaded two tiles
// ahead lost and won (54 us at 2048, 96 at 4096); with one ahead it is level at 2048.
constexpr int kClAutoMaxBlocks = 24;
static int trsv_cluster_size(int nblk, int req)
{
    if (req < 0 || (req == 0 && nblk > kClAutoMaxBlocks)) return 0;
    for (int C : {16, 8, 4})
        if ((req == 0 || C <= req) && trsv_cluster_ok(C)) {
            const int Cn = std::min(C, nblk);
            if (trsv_cl_smem(nblk, (int)cdiv(nblk, Cn)) > (size_t)kClMaxSmem) return 0;
            return Cn;
        }
    return 0;
}

static nl_status launch_trsv_cl(int N, const __half* LU, int64_t ld, const float* v, float* out, const TrsvWork& w,
                                int C, cudaStream_t st)
{
    const int nblk = (int)cdiv(N, T2);
    const int nown = (int)cdiv(nblk, C);
    const size_t smem = trsv_cl_smem(nblk, nown);
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(C);
    cfg.blockDim = dim3(kClThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const int* perm = w.perm;
    const float* dinv = (const float*)w.dinv;
    prof_begin("k_trsv_cl", st);
    const long long wait = w.wait_limit == 0 ? kClWaitIters : (w.wait_limit < 0 ? 0LL : (long long)w.wait_limit);
    cudaError_t le = cudaLaunchKernelEx(&cfg, k_trsv_cl, N, nblk, LU, ld, v, perm, dinv, out, w.err, wait, w.rs);
    prof_end("k_trsv_cl", st);
    NL_CUDA_OK(le);
    return NL_OK;
}

nl_status trsv_solve16(int N, const __half* LU, int64_t ld, const float* v, float* z, const TrsvWork& w, int epoch,
                       cudaStream_t st, int* launches)
{
    const int C = trsv_cluster_size((int)cdiv(N, T2), w.cluster);
    if (C > 0) {
        if (launches) *launches += 1;
        return launch_trsv_cl(N, LU, ld, v, z, w, C, st);
    }
    unsigned long long* mbf = (unsigned long long*)w.y;
    unsigned long long* mbb = mbf + N;
    nl_status s = launch_trsv_mb<true>(N, LU, ld, v, nullptr, mbf, nullptr, w, (unsigned)epoch, st);
    if (s != NL_OK) return s;
    s = launch_trsv_mb<false>(N, LU, ld, nullptr, mbf, mbb, z, w, (unsigned)epoch, st);
    if (launches) *launches += 2;
    return s;
}

nl_status trsv_solve64(int N, const double* LU, int64_t ld, const double* v, double* z, const TrsvWork& w, int epoch,
                       cudaStream_t st, int* launches)
{
    return solve_impl<double, double>(N, LU, ld, v, z, w, epoch, st, launches);
}

nl_status trsv_solve32(int N, const float* LU, int64_t ld, const float* v, float* z, const TrsvWork& w, int epoch,
                       cudaStream_t st, int* launches)
{
    return solve_impl<float, float>(N, LU, ld, v, z, w, epoch, st, launches);
}

// The binary16 factors promoted to a single-precision copy (exact), for the
// GMRES-IR preconditioner that solves with single-precision factors.
__global__ void __launch_bounds__(256) k_promote16(int N, const __half* __restrict__ A, int64_t lda,
                                                   float* __restrict__ B, int64_t ldb)
{
    const int64_t i = blockIdx.y;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < N; j += gridDim.x * blockDim.x)
        B[i * ldb + j] = __half2float(A[i * lda + j]);
}

nl_status launch_promote16(int N, const __half* A, int64_t lda, float* B, int64_t ldb, cudaStream_t st)
{
    if (N < 1 || N > 32768) return NL_EINVAL;
    k_promote16<<<dim3((unsigned)std::min<int64_t>(cdiv(N, 256), 8), (unsigned)N), 256, 0, st>>>(N, A, lda, B, ldb);
    NL_CUDA_OK(cudaGetLastError());
    return NL_OK;
}

// ------------------------------------------------- binary16 arithmetic --
// Both triangular solves with every product and difference rounded to
// binary16: the step of the two-precision F16 Newton method (Section 1.3),
// computed in the precision of its factorisation.  Column-oriented in one
// CTA: at step t the final entry x_t is applied to every later row (forward)
// or earlier row (backward), so row i takes its updates in increasing t in
// the forward solve and in decreasing t in the backward one.  The product of
// two binary16 numbers is exact in binary32 and is rounded once, to binary16;
// the difference and the backward quotient are formed in binary32 (IEEE
// round to nearest) and then rounded to binary16, which gives the correctly
// rounded binary16 result because 24 >= 2 * 11 + 2 (rounding twice is
// innocuous when the wider format has at least 2p + 2 bits, Figueroa 1995).
// All in single precision: binary64 here would run on the SM's few FP64
// units and dominate the sweep.
constexpr int kH16Threads = 1024;

__device__ __forceinline__ __half h16_sub_prod(__half b, __half l, __half x)
{
    const float p = __half2float(__float2half_rn(__half2float(l) * __half2float(x)));
    return __float2half_rn(__half2float(b) - p);
}

__device__ __forceinline__ __half h16_div(__half a, __half b)
{
    return __float2half_rn(__fdiv_rn(__half2float(a), __half2float(b)));
}

// Register-pipelined sweep for N <= 4096 (R <= 4 rows per thread, row
// i = tid + k * 1024): the factor is read in chunks of eight columns, one
// 16-byte load per row and chunk, issued a chunk ahead of its use, so the
// loads overlap the previous chunk's eight barrier steps.  Same operations in
// the same order as the scalar sweep.
__device__ __forceinline__ __half h16_lane(const uint4& v, int s)
{
    const unsigned w = (s >> 1) == 0 ? v.x : (s >> 1) == 1 ? v.y : (s >> 1) == 2 ? v.z : v.w;
    return __ushort_as_half((unsigned short)(w >> (16 * (s & 1))));
}

template <int R>
__device__ __forceinline__ void h16_load_chunk(const __half* __restrict__ LU, int64_t ld, int N, int c, int tid,
                                               uint4 (&v)[R])
{
#pragma unroll
    for (int k = 0; k < R; ++k) {
        const int i = tid + k * kH16Threads;
        v[k] = (i < N && c >= 0 && 8 * c < N) ? __ldg(reinterpret_cast<const uint4*>(LU + (int64_t)i * ld + 8 * c))
                                              : make_uint4(0u, 0u, 0u, 0u);
    }
}

// u_tt for t in [8c, 8c + 8) (1 beyond N), packed as one 16-byte value.
__device__ __forceinline__ uint4 h16_load_diag(const __half* __restrict__ LU, int64_t ld, int N, int c)
{
    unsigned w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int t0 = 8 * c + 2 * q, t1 = t0 + 1;
        const unsigned short lo = (c >= 0 && t0 < N) ? __half_as_ushort(LU[(int64_t)t0 * ld + t0]) : (unsigned short)0x3c00;
        const unsigned short hi = (c >= 0 && t1 < N) ? __half_as_ushort(LU[(int64_t)t1 * ld + t1]) : (unsigned short)0x3c00;
        w[q] = (unsigned)lo | ((unsigned)hi << 16);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

template <int R>
__device__ void lusolve16h_vec(int N, const __half* __restrict__ LU, int64_t ld, __half* b, __half* zout,
                               float* __restrict__ u, float scale, int tid)
{
    const int nch = (N + 7) / 8;
    uint4 cur[R], nxt[R];
    h16_load_chunk<R>(LU, ld, N, 0, tid, cur);
    for (int c = 0; c < nch; ++c) {  // L y = P b, unit diagonal
        h16_load_chunk<R>(LU, ld, N, c + 1, tid, nxt);
#pragma unroll
        for (int s = 0; s < 8; ++s) {
            const int t = 8 * c + s;
            if (t < N - 1) {
                const __half xt = b[t];
#pragma unroll
                for (int k = 0; k < R; ++k) {
                    const int i = tid + k * kH16Threads;
                    if (i > t && i < N) b[i] = h16_sub_prod(b[i], h16_lane(cur[k], s), xt);
                }
                __syncthreads();
            }
        }
#pragma unroll
        for (int k = 0; k < R; ++k) cur[k] = nxt[k];
    }
    // the chunk's diagonal entries u_tt, packed eight binary16 to 16 bytes
    uint4 dcur = h16_load_diag(LU, ld, N, nch - 1), dnxt;
    h16_load_chunk<R>(LU, ld, N, nch - 1, tid, cur);
    for (int c = nch - 1; c >= 0; --c) {  // U z = y
        h16_load_chunk<R>(LU, ld, N, c - 1, tid, nxt);
        dnxt = h16_load_diag(LU, ld, N, c - 1);
#pragma unroll
        for (int s = 7; s >= 0; --s) {
            const int t = 8 * c + s;
            if (t < N) {
                const __half xt = h16_div(b[t], h16_lane(dcur, s));
                if (tid == 0) {
                    if (zout) zout[t] = xt;
                    if (u) u[t] = scale * __half2float(xt);
                }
#pragma unroll
                for (int k = 0; k < R; ++k) {
                    const int i = tid + k * kH16Threads;
                    if (i < t) b[i] = h16_sub_prod(b[i], h16_lane(cur[k], s), xt);
                }
                __syncthreads();
            }
        }
#pragma unroll
        for (int k = 0; k < R; ++k) cur[k] = nxt[k];
        dcur = dnxt;
    }
}

__global__ void __launch_bounds__(kH16Threads) k_lusolve16h(int N, const __half* __restrict__ LU, int64_t ld,
                                                           const int* __restrict__ ipiv, const int* __restrict__ perm,
                                                           const double* __restrict__ F, const float* __restrict__ r,
                                                           const double* __restrict__ nrm, const __half* vin,
                                                           __half* zout, float* __restrict__ u)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __half* b = reinterpret_cast<__half*>(smem_raw);  // N entries
    const int tid = threadIdx.x;
    float scale = 1.0f;
    if (F) {
        const double fn = *nrm;
        for (int i = tid; i < N; i += kH16Threads) {
            const int j = perm ? perm[i] : i;
            b[i] = __double2half(-F[j] / fn);
        }
    } else if (r) {
        scale = (float)*nrm;
        for (int i = tid; i < N; i += kH16Threads) {
            const int j = perm ? perm[i] : i;
            b[i] = __float2half_rn(r[j] / scale);
        }
    } else {
        for (int i = tid; i < N; i += kH16Threads) b[i] = vin[perm ? perm[i] : i];
    }
    __syncthreads();
    if (!perm && tid == 0) {  // P b, the interchanges in factorisation order
        for (int k = 0; k < N; ++k) {
            const int p = ipiv[k];
            if (p != k && (unsigned)p < (unsigned)N) {
                const __half t = b[k];
                b[k] = b[p];
                b[p] = t;
            }
        }
    }
    __syncthreads();
    const bool vec = N <= 4 * kH16Threads && (ld % 8) == 0 && (((uintptr_t)LU) & 15) == 0;
    if (vec) {
        const int R = (N + kH16Threads - 1) / kH16Threads;
        if (R == 1) lusolve16h_vec<1>(N, LU, ld, b, zout, u, scale, tid);
        else if (R == 2) lusolve16h_vec<2>(N, LU, ld, b, zout, u, scale, tid);
        else lusolve16h_vec<4>(N, LU, ld, b, zout, u, scale, tid);
        return;
    }
    for (int t = 0; t + 1 < N; ++t) {  // L y = P b, unit diagonal
        const __half xt = b[t];
        for (int i = t + 1 + tid; i < N; i += kH16Threads) b[i] = h16_sub_prod(b[i], LU[(int64_t)i * ld + t], xt);
        __syncthreads();
    }
    for (int t = N - 1; t >= 0; --t) {  // U z = y
        const __half xt = h16_div(b[t], LU[(int64_t)t * ld + t]);
        if (tid == 0) {
            if (zout) zout[t] = xt;
            if (u) u[t] = scale * __half2float(xt);
        }
        for (int i = tid; i < t; i += kH16Threads) b[i] = h16_sub_prod(b[i], LU[(int64_t)i * ld + t], xt);
        __syncthreads();
    }
}

nl_status lusolve16h(int N, const __half* LU, int64_t ld, const int* ipiv, const int* perm, const double* F,
                     const float* r, const double* nrm, const __half* vin, __half* zout, float* u, cudaStream_t st)
{
    if (N < 1 || N > 32768 || !LU || !(ipiv || perm) || ld < N || ((F || r) ? !nrm : !vin)) {
        set_error("binary16 solve: bad argument");
        return NL_EINVAL;
    }
    static bool attr = false;
    if (!attr) {
        if (set_max_dynamic_smem((const void*)k_lusolve16h) != NL_OK) return NL_ECUDA;
        attr = true;
    }
    prof_begin("k_lusolve16h", st);
    k_lusolve16h<<<1, kH16Threads, (size_t)N * sizeof(__half), st>>>(N, LU, ld, ipiv, perm, F, r, nrm, vin, zout, u);
    prof_end("k_lusolve16h", st);
    NL_CUDA_OK(cudaGetLastError());
    return NL_OK;
}

}  // namespace nl
