// lu.cu — blocked right-looking LU with partial pivoting (Section 1.3:
// Gaussian elimination; Section 2: the half-precision factorisation of J_h).
//
// Two-level blocking.  The matrix is processed in outer panels of NB columns.
// Each outer panel is copied into a working array P (binary32 for the
// half-precision LU, binary64 for the double LU) and factored leaf by leaf
// (leaf = kLeaf columns):
//   * k_leaf: one thread-block cluster holds the leaf's rows in registers.
//     Per column, each CTA finds its best pivot candidate (warp shuffles),
//     broadcasts the candidate row to every CTA of the cluster through
//     distributed shared memory, and after one cluster barrier every CTA
//     picks the same pivot (largest |a|, first in the current row order)
//     and eliminates.  Rows stay in place; positions are tracked, and the
//     rows are written to their final positions at the end.  The epilogue
//     applies the leaf's interchanges to the other panel columns and forms
//     the leaf's U rows for the remaining panel columns.
//   * k_panel_gemm: the rest of the panel below the leaf is updated.
// After the panel: interchanges on the other columns of the matrix (k_laswp),
// U12 = L11^{-1} A12 (k_trsm_u12), and the trailing update
// A22 <- A22 - L21 U12 (SIMT here, or tcgen05 in gemm_tc.cu).
//
// Half-precision arithmetic model: binary32 arithmetic on binary16 data; the
// multipliers and the pivot rows' entries are rounded to binary16 as soon as
// they are formed, and everything not yet eliminated is rounded to binary16
// once per outer panel (when P is written back and when the trailing update
// is stored).  With the SIMT trailing update this reproduces, operation for
// operation, Gaussian elimination with that rounding schedule.
#include <atomic>
#include <cooperative_groups.h>

#include <algorithm>
#include <climits>
#include <queue>
#include <type_traits>

#include "common.cuh"
#include "internal.h"
#include "tcgen05.cuh"

namespace cg = cooperative_groups;

namespace nl {

constexpr int kLeafThreads = 256;
constexpr int kMaxCluster = 16;

template <typename T, int NBL>
struct alignas(16) LeafRec {
    T abs;      // |candidate|, -1 when the CTA has no live row
    int pos;    // candidate's current position (relative to the leaf's first row)
    int pad;
    T v[NBL];   // candidate row over the leaf's columns
};

template <typename T>
__device__ __forceinline__ bool better(T a, int pa, T b, int pb)
{
    return a > b || (a == b && pa < pb);
}

template <typename T>
__device__ __forceinline__ T maybe_round(T v, bool r)
{
    return v;
}
template <>
__device__ __forceinline__ float maybe_round<float>(float v, bool r)
{
    return r ? round_h(v) : v;
}

// Register-array element at a runtime index, by static selects (keeps the
// array in registers).
template <int NBL, typename T>
__device__ __forceinline__ T pick(const T (&row)[NBL], int j)
{
    T r = row[0];
#pragma unroll
    for (int t = 1; t < NBL; ++t)
        if (t == j) r = row[t];
    return r;
}
template <int NBL, typename T>
__device__ __forceinline__ void place(T (&row)[NBL], int j, T v)
{
#pragma unroll
    for (int t = 0; t < NBL; ++t)
        if (t == j) row[t] = v;
}

// P: working panel, row r (relative to the panel's first row K), column t
// (relative to K), leading dimension ldp.  The leaf covers columns
// [k0, k0+wl) and rows [k0, M).  ipiv_out points at ipiv[K + k0].
template <typename T, int NBL, int R, bool RND>
__global__ void __launch_bounds__(kLeafThreads, 1) k_leaf(T* __restrict__ P, int ldp, int k0, int M, int w, int wl,
                                                       int* __restrict__ ipiv_out, int piv_base,
                                                       int* __restrict__ info, int C, int rows_per_cta)
{
    using Rec = LeafRec<T, NBL>;
    __shared__ Rec inbox[2][kMaxCluster];
    __shared__ Rec outbox;
    __shared__ Rec prow_save[NBL];  // pivot row of each step: L11 (below diag) and U11
    __shared__ T wabs[kLeafThreads / 32];
    __shared__ int wpos[kLeafThreads / 32];
    __shared__ int piv_s[NBL];

    const int rank = (C > 1) ? (int)cg::this_cluster().block_rank() : 0;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int Ml = M - k0;
    const int lo = rank * rows_per_cta, hi = min(Ml, lo + rows_per_cta);

    T v[R][NBL];
    int pos[R];
    bool live[R];
#pragma unroll
    for (int s = 0; s < R; ++s) {
        int lr = lo + tid + s * kLeafThreads;
        live[s] = lr < hi;
        pos[s] = lr;
#pragma unroll
        for (int t = 0; t < NBL; ++t)
            v[s][t] = (live[s] && t < wl) ? P[(int64_t)(k0 + lr) * ldp + k0 + t] : T(0);
    }

    for (int j = 0; j < wl; ++j) {
        // ---- local and CTA-wide candidate: largest |a_ij|, then smallest position
        T babs = T(-1);
        int bpos = INT_MAX, bs = -1;
#pragma unroll
        for (int s = 0; s < R; ++s) {
            if (live[s]) {
                T a = pick<NBL>(v[s], j);
                a = a < T(0) ? -a : a;
                if (!(a == a)) a = T(-0.5);  // NaN never wins over a number
                if (better(a, pos[s], babs, bpos)) {
                    babs = a;
                    bpos = pos[s];
                    bs = s;
                }
            }
        }
        T wa = babs;
        int wp = bpos;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            T oa = __shfl_xor_sync(0xffffffffu, wa, o);
            int op = __shfl_xor_sync(0xffffffffu, wp, o);
            if (better(oa, op, wa, wp)) {
                wa = oa;
                wp = op;
            }
        }
        if (lane == 0) {
            wabs[warp] = wa;
            wpos[warp] = wp;
        }
        __syncthreads();
        T ca = T(-1);
        int cp = INT_MAX;
        for (int q = 0; q < kLeafThreads / 32; ++q)
            if (better(wabs[q], wpos[q], ca, cp)) {
                ca = wabs[q];
                cp = wpos[q];
            }
        if (bs >= 0 && bpos == cp) {
            outbox.abs = ca;
            outbox.pos = cp;
#pragma unroll
            for (int s = 0; s < R; ++s)
                if (s == bs) {
#pragma unroll
                    for (int t = 0; t < NBL; ++t) outbox.v[t] = v[s][t];
                }
        }
        if (cp == INT_MAX && tid == 0) {
            outbox.abs = T(-1);
            outbox.pos = INT_MAX;
        }
        __syncthreads();

        // ---- exchange candidates across the cluster
        const Rec* recs;
        int nrec;
        if (C > 1) {
            cg::cluster_group cl = cg::this_cluster();
            constexpr int kWords = sizeof(Rec) / 16;
            for (int q = tid; q < C * kWords; q += kLeafThreads) {
                int peer = q / kWords, wd = q % kWords;
                float4* dst = reinterpret_cast<float4*>(cl.map_shared_rank(&inbox[j & 1][rank], peer));
                dst[wd] = reinterpret_cast<const float4*>(&outbox)[wd];
            }
            cl.sync();
            recs = inbox[j & 1];
            nrec = C;
        } else {
            recs = &outbox;
            nrec = 1;
        }
        T ga = T(-1);
        int gp = INT_MAX, gsrc = 0;
        for (int q = 0; q < nrec; ++q)
            if (better(recs[q].abs, recs[q].pos, ga, gp)) {
                ga = recs[q].abs;
                gp = recs[q].pos;
                gsrc = q;
            }
        const Rec& pr = recs[gsrc];
        T u[NBL];
#pragma unroll
        for (int t = 0; t < NBL; ++t) u[t] = (t >= j) ? maybe_round(pr.v[t], RND) : T(0);
        if (tid == 0) {
            piv_s[j] = gp;
            if (rank == 0) ipiv_out[j] = piv_base + gp;
            // keep the pivot row: entries left of j are its multipliers
#pragma unroll
            for (int t = 0; t < NBL; ++t) prow_save[j].v[t] = (t >= j) ? u[t] : pr.v[t];
        }

        // ---- interchange bookkeeping: the pivot row moves to position j,
        //      the row at position j moves to the pivot's old position
#pragma unroll
        for (int s = 0; s < R; ++s) {
            if (live[s]) {
                if (pos[s] == gp) {
                    live[s] = false;
                    pos[s] = j;
#pragma unroll
                    for (int t = 0; t < NBL; ++t)
                        if (t >= j) v[s][t] = u[t];
                } else if (pos[s] == j) {
                    pos[s] = gp;
                }
            }
        }

        // ---- elimination of column j in the live rows
        const T ukk = pick<NBL>(u, j);
        if (ukk != T(0)) {
#pragma unroll
            for (int s = 0; s < R; ++s) {
                if (live[s]) {
                    T l = maybe_round(pick<NBL>(v[s], j) / ukk, RND);
                    place<NBL>(v[s], j, l);
#pragma unroll
                    for (int t = 0; t < NBL; ++t)
                        if (t > j) v[s][t] = fma(-l, u[t], v[s][t]);
                }
            }
        } else if (tid == 0 && rank == 0) {
            atomicCAS(info, 0, piv_base + j + 1);
        }
    }

    // ---- rows to their final positions (leaf columns)
#pragma unroll
    for (int s = 0; s < R; ++s) {
        int lr = lo + tid + s * kLeafThreads;
        if (lr < hi) {
#pragma unroll
            for (int t = 0; t < NBL; ++t)
                if (t < wl) P[(int64_t)(k0 + pos[s]) * ldp + k0 + t] = v[s][t];
        }
    }
    if (rank != 0) return;
    __syncthreads();

    // ---- epilogue (one CTA): interchanges on the other panel columns, then
    //      the leaf's U rows for the panel columns right of the leaf
    const int nother = w - wl;
    for (int q = tid; q < nother; q += kLeafThreads) {
        int col = (q < k0) ? q : q + wl;
        for (int jj = 0; jj < wl; ++jj) {
            int p = piv_s[jj];
            if (p != jj) {
                T* a = P + (int64_t)(k0 + jj) * ldp + col;
                T* b = P + (int64_t)(k0 + p) * ldp + col;
                T tmp = *a;
                *a = *b;
                *b = tmp;
            }
        }
        if (col >= k0 + wl) {
            T uu[NBL];
#pragma unroll
            for (int kk = 0; kk < NBL; ++kk) {
                if (kk < wl) {
                    T a = P[(int64_t)(k0 + kk) * ldp + col];
#pragma unroll
                    for (int t = 0; t < NBL; ++t)
                        if (t < kk) a = fma(-prow_save[kk].v[t], uu[t], a);
                    a = maybe_round(a, RND);
                    uu[kk] = a;
                    P[(int64_t)(k0 + kk) * ldp + col] = a;
                } else {
                    uu[kk] = T(0);
                }
            }
        }
    }
}

// Rest of the panel below a leaf: P[i][c] -= sum_t P[i][k0+t] P[k0+t][c],
// rows i in [k0+wl, M), columns c in [k0+wl, w), t in [0, wl) in order,
// kept in the working precision (no rounding).
template <typename T, int NBL>
__global__ void __launch_bounds__(256) k_panel_gemm(T* __restrict__ P, int ldp, int k0, int wl, int M, int w)
{
    __shared__ T Us[NBL][64];
    const int c0 = k0 + wl;
    const int tx = threadIdx.x & 63, ty = threadIdx.x >> 6;
    const int rbase = c0 + blockIdx.x * 64;
    for (int cc = 0; cc < w - c0; cc += 64) {
        const int c = c0 + cc + tx;
        __syncthreads();
        for (int q = threadIdx.x; q < NBL * 64; q += 256) {
            int t = q / 64, x = q % 64;
            Us[t][x] = (t < wl && c0 + cc + x < w) ? P[(int64_t)(k0 + t) * ldp + c0 + cc + x] : T(0);
        }
        __syncthreads();
        if (c < w) {
            for (int rr = ty; rr < 64; rr += 4) {
                int i = rbase + rr;
                if (i >= M) break;
                const T* Li = P + (int64_t)i * ldp + k0;
                T acc = P[(int64_t)i * ldp + c];
#pragma unroll
                for (int t = 0; t < NBL; ++t)
                    if (t < wl) acc = fma(-Li[t], Us[t][tx], acc);
                P[(int64_t)i * ldp + c] = acc;
            }
        }
    }
}

template <typename T, typename S>
__global__ void k_panel_load(const S* __restrict__ A, int64_t lda, int K, int M, int w, T* __restrict__ P, int ldp)
{
    const int i = blockIdx.x;
    for (int t = threadIdx.x; t < w; t += blockDim.x) P[(int64_t)i * ldp + t] = (T)ld_elem(A + (int64_t)(K + i) * lda + K + t);
}

template <typename T, typename S>
__global__ void k_panel_store(S* __restrict__ A, int64_t lda, int K, int M, int w, const T* __restrict__ P, int ldp)
{
    const int i = blockIdx.x;
    for (int t = threadIdx.x; t < w; t += blockDim.x) st_elem(A + (int64_t)(K + i) * lda + K + t, P[(int64_t)i * ldp + t]);
}

// Row interchanges of panel [K, K+w) on all other columns, in order.
template <typename S>
__global__ void __launch_bounds__(256) k_laswp(S* __restrict__ A, int64_t lda, int K, int w, int N,
                                               const int* __restrict__ ipiv)
{
    __shared__ int ps[256];
    for (int q = threadIdx.x; q < w; q += blockDim.x) ps[q] = ipiv[K + q];
    __syncthreads();
    int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= N - w) return;
    const int col = (q < K) ? q : q + w;
    for (int jj = 0; jj < w; ++jj) {
        int p = ps[jj];
        if (p != K + jj) {
            S* a = A + (int64_t)(K + jj) * lda + col;
            S* b = A + (int64_t)p * lda + col;
            S t = *a;
            *a = *b;
            *b = t;
        }
    }
}

// U12 = L11^{-1} A12 for rows [K, K+w), columns [K+w, N); each thread forms
// one column by forward substitution, rounding each entry when formed (half
// LU).  Rows are taken eight at a time so that the eight running sums are
// independent (instruction-level parallelism); each entry still accumulates
// its terms t = 0, 1, ..., k-1 in order.  Optionally also writes U12^T
// (binary16, ldut) for the tensor-core update.  flag: skip when set.
constexpr int kTrsmThreads = 64;

template <typename T, typename S, bool RND>
__global__ void __launch_bounds__(kTrsmThreads) k_trsm_u12(S* __restrict__ A, int64_t lda, int K, int w, int N,
                                                          __half* __restrict__ Ut, int ldut,
                                                          const int* __restrict__ flag)
{
    if (flag && *(volatile const int*)flag) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* L = reinterpret_cast<T*>(smem_raw);  // w x w, strictly lower part
    T* us = L + w * w;                       // w x kTrsmThreads (column per thread)
    for (int q = threadIdx.x; q < w * w; q += blockDim.x) {
        int r = q / w, t = q % w;
        L[q] = (t < r) ? (T)ld_elem(A + (int64_t)(K + r) * lda + K + t) : T(0);
    }
    __syncthreads();
    const int c0 = K + w + blockIdx.x * kTrsmThreads;
    const int c = c0 + threadIdx.x;
    const int tid = threadIdx.x;
    if (c < N) {
        for (int k0 = 0; k0 < w; k0 += 8) {
            T acc[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) acc[q] = (k0 + q < w) ? (T)ld_elem(A + (int64_t)(K + k0 + q) * lda + c) : T(0);
            for (int t = 0; t < k0; ++t) {
                const T ut = us[t * kTrsmThreads + tid];
#pragma unroll
                for (int q = 0; q < 8; ++q) acc[q] = fma(-L[(k0 + q) * w + t], ut, acc[q]);
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int k = k0 + q;
                if (k < w) {
                    T a = acc[q];
                    for (int t = k0; t < k; ++t) a = fma(-L[k * w + t], us[t * kTrsmThreads + tid], a);
                    a = maybe_round(a, RND);
                    us[k * kTrsmThreads + tid] = a;
                    st_elem(A + (int64_t)(K + k) * lda + c, a);
                }
            }
        }
    }
    if (Ut) {
        __syncthreads();
        const int ncol = min(kTrsmThreads, N - c0);
        for (int q = threadIdx.x; q < ncol * w; q += blockDim.x) {
            int col = q / w, kk = q % w;
            Ut[(int64_t)(c0 - K - w + col) * ldut + kk] = __float2half_rn((float)us[kk * kTrsmThreads + col]);
        }
    }
}

// ------------------------------------------------ no-interchange fast path --
// Partial pivoting picks the diagonal row at step j exactly when no row
// below holds a larger |a_ij| (ties go to the diagonal, which comes first).
// The fast path factors each panel without interchanges and checks that
// condition on every pre-division value; the elimination arithmetic is the
// same, so when no check fails the factors and pivots (ipiv[k] = k) are
// exactly those of partial pivoting.  Any failure (or a zero / NaN pivot)
// sets *flag; the remaining fast-path kernels then return at once and the
// caller refactors with the interchanging path.

// ------------------------------------------------ 32-wide chunk routines --
// All routines below apply to each entry the elimination's updates
// a <- a - l_t u_t in increasing t (one rounding each: the product of two
// binary16 numbers is exact in binary32), round multipliers and U entries to
// binary16 when they are formed, and check each pre-division value against
// its pivot (|a_it| <= |u_tt|: partial pivoting keeps the diagonal).

__device__ __forceinline__ float absT(float x) { return fabsf(x); }
__device__ __forceinline__ double absT(double x) { return fabs(x); }

// Diagonal block [K, K+w)^2 (w <= 128) in one CTA, held in shared memory
// (double precision: the F64 baseline).  Right-looking with look-ahead, one
// barrier per column: at step k the first wp / 32 warps (a row per thread) take
// column k + 1 alone (update, pivot check, division), while the others apply
// column k's multipliers to the columns right of it (lanes along a row).  The
// bound is the double-precision pipe (two multiply-adds per SM and cycle: w^3 / 3
// of them, 22 us at w = 64, and the divisions, about 13 us).  Measured, w = 64:
// 64 us; a warp per 32 x 32 sub-block with the pivot row by shuffles and solves by
// groups of eight lanes took 243.
constexpr int kDiagThreads = 512;

// Block [K, K+w)^2 of A into shared memory W (ld ldw), identity-padded to
// wp; 16-byte vector loads when the row segments allow them.
template <typename T, typename S, int NT>
__device__ __forceinline__ void load_block(const S* __restrict__ A, int64_t lda, int K, int w, int wp, T* W, int ldw,
                                           int tid)
{
    constexpr int V = 16 / sizeof(S);  // elements per 16-byte vector
    const bool vec = (w % V == 0) && ((((uintptr_t)(A + (int64_t)K * lda + K)) & 15) == 0) && ((lda * sizeof(S)) % 16 == 0);
    if (vec) {
        const int vpr = w / V;
#pragma unroll 4
        for (int q = tid; q < w * vpr; q += NT) {
            const int i = q / vpr, tv = q - i * vpr;
            uint4 raw = *reinterpret_cast<const uint4*>(A + (int64_t)(K + i) * lda + K + tv * V);
            const S* e = reinterpret_cast<const S*>(&raw);
#pragma unroll
            for (int k = 0; k < V; ++k) W[i * ldw + tv * V + k] = (T)ld_elem(e + k);
        }
    } else {
#pragma unroll 4
        for (int q = tid; q < w * w; q += NT) {
            const int i = q / w, t = q - i * w;
            W[i * ldw + t] = (T)ld_elem(A + (int64_t)(K + i) * lda + K + t);
        }
    }
    for (int q = tid; q < wp * wp; q += NT) {
        const int i = q / wp, t = q - i * wp;
        if (i >= w || t >= w) W[i * ldw + t] = (i == t) ? T(1) : T(0);
    }
}

template <typename T, typename S, int NT>
__device__ __forceinline__ void store_block(S* __restrict__ A, int64_t lda, int K, int w, const T* W, int ldw, int tid)
{
    constexpr int V = 16 / sizeof(S);
    const bool vec = (w % V == 0) && ((((uintptr_t)(A + (int64_t)K * lda + K)) & 15) == 0) && ((lda * sizeof(S)) % 16 == 0);
    if (vec) {
        const int vpr = w / V;
#pragma unroll 4
        for (int q = tid; q < w * vpr; q += NT) {
            const int i = q / vpr, tv = q - i * vpr;
            uint4 raw;
            S* e = reinterpret_cast<S*>(&raw);
#pragma unroll
            for (int k = 0; k < V; ++k) st_elem(e + k, W[i * ldw + tv * V + k]);
            *reinterpret_cast<uint4*>(A + (int64_t)(K + i) * lda + K + tv * V) = raw;
        }
    } else {
        for (int q = tid; q < w * w; q += NT) {
            const int i = q / w, t = q - i * w;
            st_elem(A + (int64_t)(K + i) * lda + K + t, W[i * ldw + t]);
        }
    }
}

template <typename T, typename S, bool RND>
__device__ __forceinline__ void diag_lu_body(S* __restrict__ A, int64_t lda, int K, int w,
                                                             int* __restrict__ ipiv, int* __restrict__ flag,
                                                             void* __restrict__ stage)
{
    if (*(volatile int*)flag) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* W = reinterpret_cast<T*>(smem_raw);
    const int wp = (w + 31) & ~31, ldw = wp + 1;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wa = wp / 32;  // warps that take the next column
    __shared__ T piv[2];     // the pivots, alternating
    load_block<T, S, kDiagThreads>(A, lda, K, w, wp, W, ldw, tid);
    __syncthreads();
    bool bad = false;
    for (int k = -1; k < w - 1; ++k) {
        const T* Wk = W + k * ldw;  // row k: U from the diagonal on (k = -1: nothing to apply)
        if (warp < wa) {
            const int i = tid, c = k + 1;
            T x = T(0);
            if (i > k) x = W[i * ldw + c];
            if (k >= 0 && i > k) x = fma(-W[i * ldw + k], Wk[c], x);
            if (i == c) {
                x = maybe_round(x, RND);
                piv[c & 1] = x;
                W[c * ldw + c] = x;
            }
            __syncwarp();
            asm volatile("bar.sync 1, %0;" ::"r"(32 * wa) : "memory");
            const T u = piv[c & 1];
            if (i > c) {  // (padding rows too: zero against a zero pivot is left to the interchanging path)
                if (!(absT(x) <= absT(u)) || !(u != T(0))) bad = true;
                W[i * ldw + c] = maybe_round(x / u, RND);
            }
        } else if (k >= 0) {
            const int nv = kDiagThreads / 32 - wa;
            for (int j = k + 2 + lane; j < w; j += 32) {
                const T u = Wk[j];
                for (int i = k + 1 + warp - wa; i < w; i += nv) {
                    T x = fma(-W[i * ldw + k], u, W[i * ldw + j]);
                    if (RND && i == k + 1) x = maybe_round(x, RND);  // row k + 1 is final
                    W[i * ldw + j] = x;
                }
            }
        }
        __syncthreads();
    }
    // every pivot (the last one has no row below it that would have checked it)
    if (tid < w && !(absT(W[tid * ldw + tid]) > T(0))) bad = true;
    if (__syncthreads_or(bad)) {
        if (tid == 0) atomicOr(flag, 1);
        return;
    }
    store_block<T, S, kDiagThreads>(A, lda, K, w, W, ldw, tid);
    // staged copies for k_offdiag: U11 (row role) and L11^T (column role),
    // wp x wp each, identity / zero padded, in its shared-memory layout
    using H = typename std::conditional<std::is_same<S, __half>::value, __half, T>::type;
    H* SU = reinterpret_cast<H*>(stage);
    H* SL = SU + wp * wp;
    for (int q = tid; q < wp * wp; q += kDiagThreads) {
        const int r = q / wp, t = q - r * wp;
        const T wv = W[r * ldw + t], wt = W[t * ldw + r];
        SU[q] = (H)((r < w && t < w) ? ((t >= r) ? wv : T(0)) : ((r == t) ? T(1) : T(0)));
        SL[q] = (H)((r < w && t < w && t > r) ? wt : T(0));
    }
    if (tid < w) ipiv[K + tid] = K + tid;
}

template <typename T, typename S, bool RND>
__global__ void __launch_bounds__(kDiagThreads, 1) k_diag_lu(S* __restrict__ A, int64_t lda, int K, int w,
                                                             int* __restrict__ ipiv, int* __restrict__ flag,
                                                             void* __restrict__ stage)
{
    diag_lu_body<T, S, RND>(A, lda, K, w, ipiv, flag, stage);
}

// Off-diagonal blocks of a panel of width w (double precision), one launch: L21 =
// A21 U11^{-1} (row role) and U12 = L11^{-1} A12 (column role), 32 rows (columns,
// a lane each) per CTA, so that a small panel still spreads over the SMs (the
// bound is the double-precision pipe, which takes a warp's instruction whole
// however few lanes are on).  As in the diagonal block, warp 0 takes entry t + 1
// of every line (update, check, division) while the other warps apply entry t to
// the later ones: one barrier per step, every entry's terms in increasing t.
// U11 / L11^T as staged by k_diag_lu.  The quotients are products with the
// pivots' reciprocals, made once and corrected (div_by): three dependent
// instructions of a step instead of a division's dozen.  Measured, w = 64: 39 us a
// panel at N = 1001 and 2048 (with divisions 70 and 43: the empty lines of a
// ragged last CTA divide zeros, which is the division's slow path; groups of
// eight lanes per row, four of 32 lanes dividing, took 85 at N = 1001; one thread
// per row with its entries in registers, 137).
constexpr int kOffThreads = 256;
constexpr int kOffLines = 32;

template <typename T, typename S>
__device__ __forceinline__ void offdiag_body(S* __restrict__ A, int64_t lda, int K, int w, int N, int nrow_blocks,
                                             int* __restrict__ flag, const void* __restrict__ stage, int bid)
{
    if (flag && *(volatile int*)flag) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int XS = kOffLines + 1;
    __shared__ T rd[128];  // row role: rcp_in_range(u_tt)
    const int wp = (w + 31) & ~31;
    T* D = reinterpret_cast<T*>(smem_raw);  // wp x wp: U11 (row role) or L11^T (column role), identity-padded
    T* X = D + wp * wp;                     // X[t * XS + line]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool row_role = bid < nrow_blocks;
    const int line0 = K + w + (row_role ? bid : bid - nrow_blocks) * kOffLines, n = min(kOffLines, N - line0);
    {
        const uint4* src = reinterpret_cast<const uint4*>(reinterpret_cast<const T*>(stage) + (row_role ? 0 : wp * wp));
        uint4* dst = reinterpret_cast<uint4*>(D);
        const int nv = wp * wp * (int)sizeof(T) / 16;
#pragma unroll 4
        for (int q = tid; q < nv; q += kOffThreads) dst[q] = src[q];
    }
    if (row_role) {
        for (int q = tid; q < kOffLines * w; q += kOffThreads) {
            const int r = q / w, t = q - r * w;
            X[t * XS + r] = r < n ? (T)ld_elem(A + (int64_t)(line0 + r) * lda + K + t) : T(0);
        }
    } else {
        for (int q = tid; q < kOffLines * w; q += kOffThreads) {
            const int t = q / kOffLines, c = q - t * kOffLines;
            X[t * XS + c] = c < n ? (T)ld_elem(A + (int64_t)(K + t) * lda + line0 + c) : T(0);
        }
    }
    __syncthreads();
    if (row_role && tid < w) rd[tid] = rcp_in_range(D[tid * wp + tid]);
    __syncthreads();
    bool bad = false;
    for (int t = -1; t < w - 1; ++t) {
        const T* Dt = D + t * wp;
        const T l = t >= 0 ? X[t * XS + lane] : T(0);
        if (warp == 0) {
            const int c = t + 1;
            T x = X[c * XS + lane];
            if (t >= 0) x = fma(-l, Dt[c], x);
            if (row_role) {
                const T u = D[c * wp + c];
                if (lane < n && (!(absT(x) <= absT(u)) || !(u != T(0)))) bad = true;
                x = div_by(x, u, rd[c]);
            }
            X[c * XS + lane] = x;
        } else if (t >= 0) {
            for (int j = t + 1 + warp; j < w; j += kOffThreads / 32 - 1) X[j * XS + lane] = fma(-l, Dt[j], X[j * XS + lane]);
        }
        __syncthreads();
    }
    if (__syncthreads_or(bad) && tid == 0 && flag) atomicOr(flag, 1);
    if (row_role) {
        for (int q = tid; q < n * w; q += kOffThreads) {
            const int r = q / w, t = q - r * w;
            st_elem(A + (int64_t)(line0 + r) * lda + K + t, X[t * XS + r]);
        }
    } else {
        for (int q = tid; q < kOffLines * w; q += kOffThreads) {
            const int t = q / kOffLines, c = q - t * kOffLines;
            if (c < n) st_elem(A + (int64_t)(K + t) * lda + line0 + c, X[t * XS + c]);
        }
    }
}

template <typename T, typename S>
__global__ void __launch_bounds__(kOffThreads) k_offdiag(S* __restrict__ A, int64_t lda, int K, int w, int N,
                                                         int nrow_blocks, int* __restrict__ flag,
                                                         const void* __restrict__ stage)
{
    offdiag_body<T, S>(A, lda, K, w, N, nrow_blocks, flag, stage, (int)blockIdx.x);
}
__host__ __device__ constexpr size_t offdiag_smem(int wp, size_t el) { return ((size_t)wp * wp + (size_t)wp * (kOffLines + 1)) * el; }

// ------------------------------------------ fast path, binary16 factors --
// The stage buffer holds, for the off-diagonal solves of one panel: U11 and
// -L11^T (wp x wp binary16 each, identity / zero padded) and the unrounded
// pivots a_tt (kStagePivOff floats in).
constexpr int kStagePivOff = 2 * 128 * 128;

// k_diag_lu16: the diagonal block [K, K+w)^2 (w <= 128) in one CTA, right-looking
// over blocks of eight columns.  It is bound by its dependent chain (128
// columns), so the chain runs in one warp and everything else beside it.
// Step q (C0 = 8 q), between two CTA barriers:
//   warp 0: the multipliers of the next 32 rows (a row per lane; the diagonal
//     block's U and pivots are in registers), block q applied to the next
//     diagonal block, and that block factored in registers (lane r holds
//     row r; the pivot row by shuffles, about 90 cycles a column);
//   the others: U's next columns (warp 4, for warp 0's next block) and those
//     further right, the multipliers of the rows further below; step q
//     published; then (the warps off warp 0's scheduler) block q applied to the
//     rest of the trailing matrix, four columns of every few rows per thread.
// The working copy S is binary32 in shared memory; final entries go to Hs as
// binary16, the multipliers negated (so updates are fused multiply-adds
// without a sign).  Products use fma.rn.f32.f16 (binary16 x binary16 +
// binary32, one rounding), which equals the binary32 fused multiply-add of the
// promoted values and saves the promotions.  Multipliers: div_neg
// (common.cuh).  Every entry takes its updates in increasing k, one fused
// multiply-add each, exactly as in right-looking elimination; partial pivoting
// keeps the diagonal iff |a_it| <= |a_tt| for all rows below (ties go to the
// diagonal, which comes first), checked on every pre-division value; a pivot
// that is zero or not finite in binary16 is left to the interchanging path
// too.  There are no spin waits.
// Measured (GB300, w = 128, one launch alone): 28.7 us, of which about 19 are the
// steps and 5 the stage; the former column pipeline (a hand-off between warps
// per column, 16 warps competing for the issue slots of the chain) took 57 us.
// NT threads; WMAX = 64 or 128, the largest w.
constexpr int kD16Threads = 512;
template <int WMAX>
struct Diag16 {
    static constexpr int LD = WMAX + 4;   // floats; LDS.128 of one row per lane is conflict-free
    static constexpr int HLD = WMAX + 8;  // binary16
    static constexpr size_t smem = (size_t)WMAX * LD * 4 + (size_t)WMAX * HLD * 2;
};
constexpr size_t kDiag16Smem = Diag16<128>::smem;
// k_panel16x: the operand slabs of the update's tile, behind what the CTA holds otherwise
constexpr size_t kCrossOpsOff = 103 * 1024;
constexpr size_t kCrossSmem = kCrossOpsOff + 1024 + 4 * 16384;
static_assert(kDiag16Smem <= kCrossOpsOff, "the block lies before the operands");

// fl32(a b + c), a and b binary16 (bits)
__device__ __forceinline__ float fma_h(unsigned short a, unsigned short b, float c)
{
    float d;
    asm("fma.rn.f32.f16 %0, %1, %2, %3;" : "=f"(d) : "h"(a), "h"(b), "f"(c));
    return d;
}
__device__ __forceinline__ unsigned short h_lo(unsigned v) { return (unsigned short)(v & 0xffffu); }
__device__ __forceinline__ unsigned short h_hi(unsigned v) { return (unsigned short)(v >> 16); }
__device__ __forceinline__ unsigned short h_bits(float v) { return __half_as_ushort(__float2half_rn(v)); }
__device__ __forceinline__ float h_val(unsigned short v) { return __half2float(__ushort_as_half(v)); }
__device__ __forceinline__ unsigned h_pack(unsigned short lo, unsigned short hi) { return (unsigned)lo | ((unsigned)hi << 16); }
// entry e (0..7, a constant after unrolling) of eight packed binary16 values
__device__ __forceinline__ unsigned short h_at(const uint4& v, int e)
{
    const unsigned w = (e < 2) ? v.x : (e < 4) ? v.y : (e < 6) ? v.z : v.w;
    return (e & 1) ? h_hi(w) : h_lo(w);
}

// Eight consecutive entries (16-byte aligned) as binary32, and back: binary16
// storage (the factorised matrix) rounds on store; binary32 storage (the
// single-precision shadow of an outer block, two-level LU) keeps the value.
__device__ __forceinline__ void load8(const __half* p, float* v)
{
    const uint4 raw = *reinterpret_cast<const uint4*>(p);
    const __half* e = reinterpret_cast<const __half*>(&raw);
#pragma unroll
    for (int c = 0; c < 8; ++c) v[c] = __half2float(e[c]);
}
__device__ __forceinline__ void load8(const float* p, float* v)
{
    const float4 a = reinterpret_cast<const float4*>(p)[0], b = reinterpret_cast<const float4*>(p)[1];
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
__device__ __forceinline__ void store8(__half* p, const float* v)
{
    __align__(16) __half h[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) h[c] = __float2half_rn(v[c]);
    *reinterpret_cast<uint4*>(p) = *reinterpret_cast<const uint4*>(h);
}
__device__ __forceinline__ void store8(float* p, const float* v)
{
    reinterpret_cast<float4*>(p)[0] = make_float4(v[0], v[1], v[2], v[3]);
    reinterpret_cast<float4*>(p)[1] = make_float4(v[4], v[5], v[6], v[7]);
}

// The look-ahead's part of a trailing update inside the next panel's own CTAs
// (k_panel16x): a CTA's tile C - L21 U12, rounded to binary16, where the tile has
// already been loaded into shared memory as binary32 (X[r * 132 + c] by rows, or
// X[c * 132 + r] for a column CTA): the same tcgen05 products in the same order as
// the update kernel's tile, so bitwise the same entries, which need not go
// through memory before they are factored.  Two 64-wide slabs of each operand by
// TMA into ops (64 KB, 1024-byte aligned), eight MMAs of K = 16 into 128 TMEM
// columns, then every thread takes 32 columns of one row.  cross_begin starts the
// loads (before the CTA loads its tile), cross_end applies the product.  It takes
// about 2 us of a panel; as a launch of its own between the panels it took 6 us
// and a second launch gap of 3.
struct CrossTile {
    const CUtensorMap *a, *b;  // L21 from the panel's first row on; U12^T from its first column on
    int arow, brow;            // this CTA's tile
};
constexpr long long kCrossWait = 2000000000LL;  // cycles: about a second
__device__ __forceinline__ void cross_begin(const CrossTile& T, uint32_t ops, uint64_t* bar, uint32_t* tslot)
{
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)), "r"(128u));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (threadIdx.x == 32) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&bar[0])));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&bar[1])));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        const uint32_t bl = smem_u32(&bar[0]);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bl), "r"(4u * 16384u) : "memory");
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            tma_load_2d(ops + q * 16384u, T.a, 64 * q, T.arow, bl);
            tma_load_2d(ops + 32768u + q * 16384u, T.b, 64 * q, T.brow, bl);
        }
    }
}

// COLS: X holds columns (rows of 128 t each), else rows; n: lines held.  False after a timeout.
template <bool COLS>
__device__ __forceinline__ bool cross_end(uint32_t ops, uint64_t* bar, const uint32_t* tslot, float* X, int n, unsigned* err)
{
    __shared__ int dead;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) dead = 0;
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();  // the tile is in X, the TMEM address and the barriers are set
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *(volatile const uint32_t*)tslot, bl = smem_u32(&bar[0]), bm = smem_u32(&bar[1]);
    if (threadIdx.x == 32) {
        if (!mbar_wait(bl, 0, kCrossWait)) {
            atomicOr(err, (unsigned)ERR_TIMEOUT_OTHER);
            *(volatile int*)&dead = 1;
            mbar_wait(bl, 0, kCrossWait);  // let copies in flight land
        } else {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            constexpr uint32_t idesc = tc_idesc_mn(128, 128);
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const uint32_t off = (uint32_t)(k >> 2) * 16384u + (uint32_t)(k & 3) * 32u;
                const uint64_t ad = sw128_desc(ops + off), bd = sw128_desc(ops + 32768u + off);
                const uint32_t acc = k ? 1u : 0u;
                asm volatile(
                    "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                    " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
                    "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bm) : "memory");
        }
    }
    __syncwarp();
    __syncthreads();
    bool good = !*(volatile int*)&dead;  // CTA-uniform
    const bool waited = good ? mbar_wait(bm, 0, kCrossWait) : true;
    if (__syncthreads_or(!waited)) {
        if (threadIdx.x == 0) {
            atomicOr(err, (unsigned)ERR_TIMEOUT_OTHER);
            mbar_wait(bm, 0, kCrossWait);  // let the MMAs in flight finish
        }
        good = false;
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const int q = warp & 3, c0 = (warp >> 2) * 32, row = q * 32 + lane;  // TMEM lane, first column
    if (good && (COLS ? c0 < n : q * 32 < n)) {  // (n: a multiple of 32)
        uint32_t r[32];
        const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)c0;
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
            "%14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
              "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
              "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]),
              "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]),
              "=r"(r[30]), "=r"(r[31])
            : "r"(taddr));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (COLS) {
#pragma unroll
            for (int e = 0; e < 32; ++e) {
                float* x = X + (c0 + e) * 132 + row;
                *x = round_h(*x - __uint_as_float(r[e]));
            }
        } else {
            float4* x = reinterpret_cast<float4*>(X + row * 132 + c0);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float4 v = x[e];
                x[e] = make_float4(round_h(v.x - __uint_as_float(r[4 * e])), round_h(v.y - __uint_as_float(r[4 * e + 1])),
                                   round_h(v.z - __uint_as_float(r[4 * e + 2])), round_h(v.w - __uint_as_float(r[4 * e + 3])));
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(128u));
    }
    return good;
}

// The published copy of a factored diagonal block (k_panel16): 64-bit words
// {epoch, two binary16 values}; a word is its own ready flag.
//   word k * 64 + e / 2, e > k even:           u_ke, u_k(e+1)
//   word kPubL + k * 64 + e / 2, e > k even:   -l_ek, -l_(e+1)k
//   word kPubP + t:                            the unrounded pivot a_tt (binary32)
// Step s publishes U's rows and L's columns 8 s..8 s + 7 and their pivots.
constexpr int kPubL = 128 * 64;
constexpr int kPubP = 2 * 128 * 64;
constexpr size_t kPubWords = (size_t)kPubP + 128;

__device__ __forceinline__ void pub_store2(unsigned long long* dst, unsigned epoch, unsigned v0, unsigned v1)
{
    const unsigned long long t = (unsigned long long)epoch << 32;
    asm volatile("st.volatile.global.v2.u64 [%0], {%1, %2};" ::"l"(dst), "l"(t | v0), "l"(t | v1) : "memory");
}

// One warp per k (k = 0..7, warp v of 8).
template <int HLD>
__device__ __forceinline__ void diag16_publish(int s, int w8, const unsigned short* Hs, const float4* rc,
                                               unsigned long long* pub, unsigned epoch, int v, int lane)
{
    const int C = 8 * s, k = C + v, e = C + 4 * lane;
    if (e < w8) {
        const unsigned short* h = Hs + e * HLD + k;
        const uint2 u = *reinterpret_cast<const uint2*>(Hs + k * HLD + e);
        pub_store2(pub + kPubL + k * 64 + (e >> 1), epoch, h_pack(h[0], h[HLD]), h_pack(h[2 * HLD], h[3 * HLD]));
        pub_store2(pub + k * 64 + (e >> 1), epoch, u.x, u.y);
    }
    if (lane == 0 && v < 4)
        pub_store2(pub + kPubP + C + 2 * v, epoch, __float_as_uint(rc[C + 2 * v].z), __float_as_uint(rc[C + 2 * v + 1].z));
}

// PUB: also publish the block as it is factored, for the streaming solves of
// k_panel16.  stage (may be null): U11, -L11^T and the pivots for k_offdiag16.
// CROSS: the block first takes its part of the last update (ct).
template <bool PUB = false, typename S_ = __half, int WMAX = 128, int NT = kD16Threads, bool CROSS = false>
__device__ __forceinline__ void diag_lu16_body(S_* __restrict__ A, int64_t lda, int K, int w,
                                               int* __restrict__ ipiv, int* __restrict__ flag,
                                               float* __restrict__ stage,
                                               unsigned long long* __restrict__ pub = nullptr, unsigned epoch = 0,
                                               const CrossTile* ct = nullptr, unsigned* err = nullptr)
{
    if (*(volatile int*)flag) return;
    using G = Diag16<WMAX>;
    constexpr int LD = G::LD, HLD = G::HLD, NW = NT / 32, NU = 24 * NW;  // NU: threads of the warps off scheduler 0
    constexpr int RW = WMAX / 32;  // warps 0..RW-1 take the rows below a block, warps 4..RW+3 the columns right of it
    static_assert(!PUB || NW == 16, "eight publishing warps");
    extern __shared__ __align__(16) float lsh[];
    float* S = lsh;                                                            // S[i * LD + j]: the working copy
    unsigned short* Hs = reinterpret_cast<unsigned short*>(S + WMAX * LD);     // U, and L negated
    __shared__ float4 rc[WMAX];  // per pivot: rcp_neg_abs, |u|, the unrounded value
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int w8 = (w + 7) & ~7, nq = w8 >> 3;
    const bool vec = (w % 8 == 0) && ((((uintptr_t)(A + (int64_t)K * lda + K)) & 15) == 0) && (lda % 8 == 0);
    __shared__ __align__(8) uint64_t xbar[2];
    __shared__ uint32_t xslot;
    const uint32_t ops = (smem_u32(lsh) + (uint32_t)kCrossOpsOff + 1023u) & ~1023u;
    if constexpr (CROSS) cross_begin(*ct, ops, xbar, &xslot);
    // load, eight columns per thread, padded with the identity to w8
    for (int p = tid; p < w8 * nq; p += NT) {
        const int i = p / nq, C = 8 * (p - i * nq);
        const S_* src = A + (int64_t)(K + min(i, w - 1)) * lda + K + C;
        float v[8];
        if (vec) {
            load8(src, v);
        } else {
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const int j = C + c;
                v[c] = (i < w && j < w) ? ld_elem(src + c) : ((i == j) ? 1.0f : 0.0f);
            }
        }
        store8(S + i * LD + C, v);
    }
    bool bad = false;
    if constexpr (CROSS) bad = !cross_end<false>(ops, xbar, &xslot, S, 128, err);
    __syncthreads();
    const int r = lane & 7;
    const int pubv = wid - 8;  // warps 8..15 publish
    const bool pubw = wid >= 8;
    float d[8];  // warp 0, lane r < 8: row r of the diagonal block (the other lanes' values are not used)
    if (wid == 0) {
        *reinterpret_cast<float4*>(d) = *reinterpret_cast<const float4*>(S + r * LD);
        *reinterpret_cast<float4*>(d + 4) = *reinterpret_cast<const float4*>(S + r * LD + 4);
    }
    for (int q = 0; q < nq; ++q) {
        const int C0 = 8 * q, C1 = C0 + 8;
        unsigned um[8][4];            // warp 0: U's rows of the diagonal block, packed from the diagonal on
        float cp[8], cy[8], cu[8];    // and its pivots, rcp_neg_abs, |u|
        if (wid == 0) {
            unsigned hw[4];  // row r's multipliers, packed
            unsigned viol = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                // the pivot row's shuffles run beside the division
                const float p = __shfl_sync(0xffffffffu, d[k], k);
                float us[8];
                us[k] = p;
#pragma unroll
                for (int e = k + 1; e < 8; ++e) us[e] = __shfl_sync(0xffffffffu, d[e], k);
                const float ut = round_h(p), y = rcp_neg_abs(ut);
#pragma unroll
                for (int e = k & ~1; e < 8; e += 2) {
                    const __half2 v = __floats2half2_rn(e < k ? 0.0f : us[e], us[e + 1]);
                    um[k][e / 2] = *reinterpret_cast<const unsigned*>(&v);
                }
                cp[k] = p;
                cy[k] = y;
                cu[k] = fabsf(ut);
                const unsigned short l = h_bits(div_neg(d[k], p, y, cu[k]));
                if (!(fabsf(d[k]) <= fabsf(p))) viol |= 1u << k;
#pragma unroll
                for (int e = k + 1; e < 8; ++e)
                    d[e] = fma_h(l, (e & 1) ? h_hi(um[k][e / 2]) : h_lo(um[k][e / 2]), d[e]);
                rc[C0 + k] = make_float4(y, cu[k], p, 0.0f);
                unsigned row[4];  // row k is final in lane k: its multipliers, then U
#pragma unroll
                for (int e = 0; e < 4; ++e) row[e] = 2 * e < k ? hw[e] : um[k][e];
                if (k & 1) {
                    hw[k / 2] |= (unsigned)l << 16;
                    row[k / 2] = (um[k][k / 2] & 0xffff0000u) | (hw[k / 2] & 0xffffu);
                } else {
                    hw[k / 2] = l;
                }
                if (lane == k)
                    *reinterpret_cast<uint4*>(Hs + (C0 + k) * HLD + C0) = make_uint4(row[0], row[1], row[2], row[3]);
            }
            // rows below row k (lane r > k)
            if (lane < 8 && (viol & ((1u << r) - 1u))) bad = true;
        } else if ((wid & 3) && q > 0) {
            // block q-1 applied right of and below itself, but for the diagonal block (warp 0's)
            const int B0 = C0 - 8, n4 = (w8 - C0) >> 2, t = ((wid >> 2) * 3 + (wid & 3) - 1) * 32 + lane;
            float rn4;
            asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rn4) : "f"((float)n4));
            const int sl = (int)(((float)t + 0.5f) * rn4), ns = (int)(((float)NU + 0.5f) * rn4);
            const int J = C0 + 4 * (t - sl * n4);
            if (sl < ns) {
                unsigned short u[8][4];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const uint2 v = *reinterpret_cast<const uint2*>(Hs + (B0 + k) * HLD + J);
                    u[k][0] = h_lo(v.x); u[k][1] = h_hi(v.x); u[k][2] = h_lo(v.y); u[k][3] = h_hi(v.y);
                }
                // two rows at a time (a thread of the diagonal block's columns starts below it)
                int i = C0 + sl;
                if (J < C1)
                    while (i < C1) i += ns;
                const int step = ns * LD, hstep = ns * HLD;
                float* Si = S + i * LD + J;
                const unsigned short* Hi = Hs + i * HLD + B0;
                for (; i + ns < w8; i += 2 * ns, Si += 2 * step, Hi += 2 * hstep) {
                    float4 v = *reinterpret_cast<const float4*>(Si), z = *reinterpret_cast<const float4*>(Si + step);
                    const uint4 L = *reinterpret_cast<const uint4*>(Hi), M = *reinterpret_cast<const uint4*>(Hi + hstep);
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const unsigned short l = h_at(L, k), m = h_at(M, k);
                        v.x = fma_h(l, u[k][0], v.x);
                        v.y = fma_h(l, u[k][1], v.y);
                        v.z = fma_h(l, u[k][2], v.z);
                        v.w = fma_h(l, u[k][3], v.w);
                        z.x = fma_h(m, u[k][0], z.x);
                        z.y = fma_h(m, u[k][1], z.y);
                        z.z = fma_h(m, u[k][2], z.z);
                        z.w = fma_h(m, u[k][3], z.w);
                    }
                    *reinterpret_cast<float4*>(Si) = v;
                    *reinterpret_cast<float4*>(Si + step) = z;
                }
                if (i < w8) {
                    float4 v = *reinterpret_cast<const float4*>(Si);
                    const uint4 L = *reinterpret_cast<const uint4*>(Hi);
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const unsigned short l = h_at(L, k);
                        v.x = fma_h(l, u[k][0], v.x);
                        v.y = fma_h(l, u[k][1], v.y);
                        v.z = fma_h(l, u[k][2], v.z);
                        v.w = fma_h(l, u[k][3], v.w);
                    }
                    *reinterpret_cast<float4*>(Si) = v;
                }
            }
        }
        __syncthreads();
        if (C1 >= w8) break;
        if (wid == 0) {
            // row C1 + lane, with the diagonal block's U and pivots in registers
            const int i = min(C1 + lane, w8 - 1);
            const float* Si = S + i * LD + C0;
            float x[8];
            *reinterpret_cast<float4*>(x) = *reinterpret_cast<const float4*>(Si);
            *reinterpret_cast<float4*>(x + 4) = *reinterpret_cast<const float4*>(Si + 4);
            unsigned short h[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                h[k] = h_bits(div_neg(x[k], cp[k], cy[k], cu[k]));
                bad |= !(fabsf(x[k]) <= fabsf(cp[k]));
#pragma unroll
                for (int e = k + 1; e < 8; ++e)
                    x[e] = fma_h(h[k], (e & 1) ? h_hi(um[k][e / 2]) : h_lo(um[k][e / 2]), x[e]);
            }
            if (C1 + lane < w8)
                *reinterpret_cast<uint4*>(Hs + i * HLD + C0) =
                    make_uint4(h_pack(h[0], h[1]), h_pack(h[2], h[3]), h_pack(h[4], h[5]), h_pack(h[6], h[7]));
            __syncwarp();
            asm volatile("bar.arrive 2, %0;" ::"n"(NT) : "memory");
            asm volatile("bar.sync 3, 64;" ::: "memory");  // U's next columns (warp 4)
            const float* Sd = S + (C1 + r) * LD + C1;
            *reinterpret_cast<float4*>(d) = *reinterpret_cast<const float4*>(Sd);
            *reinterpret_cast<float4*>(d + 4) = *reinterpret_cast<const float4*>(Sd + 4);
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const uint4 U = *reinterpret_cast<const uint4*>(Hs + (C0 + k) * HLD + C1);
#pragma unroll
                for (int e = 0; e < 8; ++e) d[e] = fma_h(h[k], h_at(U, e), d[e]);
            }
        } else {
            const int F0 = C1 + 32;  // first row below and column right that are not warp 0's and warp 4's
            if (wid >= 1 && wid < RW) {
                const int i = F0 + (wid - 1) * 32 + lane;
                if (i < w8) {
                    float x[8];
                    const float* Si = S + i * LD + C0;
                    *reinterpret_cast<float4*>(x) = *reinterpret_cast<const float4*>(Si);
                    *reinterpret_cast<float4*>(x + 4) = *reinterpret_cast<const float4*>(Si + 4);
                    unsigned short h[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const uint4 U = *reinterpret_cast<const uint4*>(Hs + (C0 + k) * HLD + C0);
                        const float4 c = rc[C0 + k];
                        bad |= !(fabsf(x[k]) <= fabsf(c.z));
                        h[k] = h_bits(div_neg(x[k], c.z, c.x, c.y));
#pragma unroll
                        for (int e = k + 1; e < 8; ++e) x[e] = fma_h(h[k], h_at(U, e), x[e]);
                    }
                    *reinterpret_cast<uint4*>(Hs + i * HLD + C0) =
                        make_uint4(h_pack(h[0], h[1]), h_pack(h[2], h[3]), h_pack(h[4], h[5]), h_pack(h[6], h[7]));
                }
            } else if (wid >= 4 && wid < 4 + RW) {
                const int j = (wid == 4 ? C1 : F0 + (wid - 5) * 32) + lane;  // a column right
                if (j < w8) {
                    float x[8];
                    uint4 L[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        x[k] = S[(C0 + k) * LD + j];
                        L[k] = *reinterpret_cast<const uint4*>(Hs + (C0 + k) * HLD + C0);
                    }
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const unsigned short u = h_bits(x[k]);
                        Hs[(C0 + k) * HLD + j] = u;
#pragma unroll
                        for (int e = k + 1; e < 8; ++e) x[e] = fma_h(h_at(L[e], k), u, x[e]);
                    }
                }
                __syncwarp();
                if (wid == 4) asm volatile("bar.arrive 3, 64;" ::: "memory");
            }
            __syncwarp();
            asm volatile("bar.sync 2, %0;" ::"n"(NT) : "memory");
            if (PUB && pubw) diag16_publish<HLD>(q, w8, Hs, rc, pub, epoch, pubv, lane);
        }
    }
    if (PUB && pubw) diag16_publish<HLD>(nq - 1, w8, Hs, rc, pub, epoch, pubv, lane);
    if (tid < w8) bad |= !(rc[tid].y > 0.0f && rc[tid].y <= 65504.0f);
    if (__syncthreads_or(bad)) {
        if (tid == 0) atomicOr(flag, 1);
        return;
    }
    // the factors to A (the sign of L's entries restored)
    for (int p = tid; p < w * nq; p += NT) {
        const int i = p / nq, C = 8 * (p - i * nq);
        const uint4 h = *reinterpret_cast<const uint4*>(Hs + i * HLD + C);
        unsigned hw[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
        for (int c = 0; c < 8; c += 2) {
            if (C + c < i) hw[c / 2] ^= 0x8000u;
            if (C + c + 1 < i) hw[c / 2] ^= 0x80000000u;
        }
        S_* dst = A + (int64_t)(K + i) * lda + K + C;
        if constexpr (std::is_same<S_, __half>::value) {
            if (vec) {
                *reinterpret_cast<uint4*>(dst) = make_uint4(hw[0], hw[1], hw[2], hw[3]);
                continue;
            }
        }
#pragma unroll
        for (int c = 0; c < 8; ++c)
            if (C + c < w) st_elem(dst + c, h_val((c & 1) ? h_hi(hw[c / 2]) : h_lo(hw[c / 2])));
    }
    if (stage) {
        // U11 and -L11^T (binary16, identity / zero padded to wp) and the pivots
        const int wp = (w + 31) & ~31;
        unsigned short* SU = reinterpret_cast<unsigned short*>(stage);
        unsigned short* SL = SU + wp * wp;
        for (int i = wid; i < wp; i += NW)
            for (int j = lane; j < wp; j += 32) {
                const bool in = i < w && j < w;
                SU[i * wp + j] = in ? (j >= i ? Hs[i * HLD + j] : (unsigned short)0) : (unsigned short)(i == j ? 0x3c00 : 0);
                SL[i * wp + j] = (in && j > i) ? Hs[j * HLD + i] : (unsigned short)0;
            }
        if (tid < w) stage[kStagePivOff + tid] = rc[tid].z;
    }
    if (tid < w) ipiv[K + tid] = K + tid;
}

template <typename S>
__global__ void __launch_bounds__(kD16Threads, 1) k_diag_lu16(S* __restrict__ A, int64_t lda, int K, int w,
                                                             int* __restrict__ ipiv, int* __restrict__ flag,
                                                             float* __restrict__ stage)
{
    diag_lu16_body<false, S>(A, lda, K, w, ipiv, flag, stage);
}

// k_panel16: the diagonal block and the off-diagonal solves of one panel in
// one launch.  One CTA factors the diagonal block (above) and publishes each
// block column of eight as it is finished; the other CTAs stream behind it,
// one step per block column: a CTA owns up to 256 rows of L21 or columns of
// U12 ("lines"), their not-yet-solved entries X in binary32 in shared memory.
// At step q
//   * a solver thread per line applies block q-1 to its block q (64 fused
//     multiply-adds), and solves it: for a row, l_it = fl16(x_it / u_tt) with
//     the pivot check; for a column, u_tj = fl16(x_tj);
//   * the helper warps apply block q-1 to the lines' blocks q+1, q+2, ...;
//   * two warps fetch the published words of later steps into M (binary16,
//     M[k][e] = u_ke for rows, -l_ek for columns), an mbarrier per step;
// and one barrier of the solvers and helpers joins them.  So what is left
// after the last published block is one block solve: a step of the stream
// (about 500 cycles) is shorter than a step of the diagonal block, and the
// launch takes the diagonal block's time plus a tail of one step (N = 4096:
// 30.5 us a panel on average, 67.9 us with the column pipeline and left-looking
// streams; one pair of words in flight per fetching lane and a step published
// only in the next one: 36.6 us).  Eight
// lines' multipliers of a solved block overwrite the first half of its place
// in X.  Every entry takes its fused multiply-adds in increasing k, so the
// results are bitwise those of k_diag_lu16 followed by k_offdiag16.  Every
// wait is bounded and also ends when the fast path has been abandoned: the
// warps then run their steps without waiting, so no barrier is missed.
constexpr int kPnlThreads = 512;
constexpr int kPnlRows = 256;   // at most this many lines per streaming CTA
constexpr int kPnlFetchW = 14;  // warps 14 and 15 fetch the published words
constexpr int kPnlXld = 132;    // floats
constexpr int kPnlMld = 136;    // binary16
constexpr size_t kPnlSmem = (size_t)kPnlRows * kPnlXld * 4 + (size_t)128 * kPnlMld * 2 + 128 * 4 + 16 * 8;
static_assert(kPnlSmem >= kDiag16Smem, "the diagonal block's CTA uses the same launch");
static_assert((size_t)128 * kPnlXld * 4 + (size_t)128 * kPnlMld * 2 + 128 * 4 + 16 * 8 <= kCrossOpsOff,
              "a streaming CTA of 128 lines lies before the operands");
constexpr long long kPnlSpin = 1LL << 22;

// Fetch lane: up to five pairs of published words (16 bytes each; bit v of todo:
// pair v), all loads in flight at once, until both words of every pair carry
// this launch's epoch.
template <typename Src, typename Dst>
__device__ __forceinline__ bool pnl_fetch(unsigned todo, Src src, Dst dst, unsigned epoch, const int* flag,
                                          const int* gave_up)
{
    for (long long it = 0; todo && it < kPnlSpin; ++it) {
        unsigned long long a[5], b[5];
#pragma unroll
        for (int v = 0; v < 5; ++v)
            if (todo >> v & 1u)
                asm volatile("ld.volatile.global.v2.u64 {%0, %1}, [%2];" : "=l"(a[v]), "=l"(b[v]) : "l"(src(v)) : "memory");
#pragma unroll
        for (int v = 0; v < 5; ++v)
            if ((todo >> v & 1u) && (unsigned)(a[v] >> 32) == epoch && (unsigned)(b[v] >> 32) == epoch) {
                dst(v, (unsigned)a[v], (unsigned)b[v]);
                todo &= ~(1u << v);
            }
        if (todo && (it & 63) == 63 && (*(volatile const int*)flag || *(volatile const int*)gave_up)) return false;
    }
    return !todo;
}

__device__ __forceinline__ void pnl_wait_ready(uint32_t bar, int* gave_up)
{
    if (*(volatile int*)gave_up) return;
    for (long long it = 0; it < kPnlSpin; ++it) {
        uint32_t done;
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n selp.u32 %0, 1, 0, p;\n}\n"
                     : "=r"(done)
                     : "r"(bar)
                     : "memory");
        if (done || *(volatile int*)gave_up) return;
    }
    *(volatile int*)gave_up = 1;
}

// x[e] += h_k M[k][e], k = 0..7 in order: a block's finished eight (hist) applied to eight later entries
__device__ __forceinline__ void pnl_apply(const uint4& hist, const unsigned short* __restrict__ M, int ldm, float (&x)[8])
{
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const uint4 m = *reinterpret_cast<const uint4*>(M + k * ldm);
        const unsigned short h = h_at(hist, k);
#pragma unroll
        for (int e = 0; e < 8; ++e) x[e] = fma_h(h, h_at(m, e), x[e]);
    }
}

// One streaming CTA: ROWS = rows of L21, else columns of U12; rpc lines (a multiple of 32).
template <bool ROWS, typename S = __half, bool CROSS = false>
__device__ __forceinline__ void panel16_stream(S* __restrict__ A, int64_t lda, int K, int w, int N, int blk,
                                               int rpc, __half* __restrict__ Ut, int ldut, int ut_col0, int ut_k0,
                                               int* __restrict__ flag, const unsigned long long* __restrict__ pub,
                                               unsigned epoch, unsigned* __restrict__ err, const CrossTile* ct = nullptr)
{
    extern __shared__ __align__(16) float psm[];
    float* X = psm;                                                                   // X[line * kPnlXld + t]
    unsigned short* M = reinterpret_cast<unsigned short*>(X + (CROSS ? 128 : kPnlRows) * kPnlXld);  // M[k * kPnlMld + e]
    float* pv = reinterpret_cast<float*>(M + 128 * kPnlMld);                          // unrounded pivots (rows)
    uint64_t* ready = reinterpret_cast<uint64_t*>(pv + 128);
    __shared__ int gave_up;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int w8 = (w + 7) & ~7, nq = w8 >> 3;
    const int line0 = K + w + blk * rpc, nlive = min(rpc, N - line0);
    if (tid == 0) gave_up = 0;
    if (tid < 16) asm volatile("mbarrier.init.shared::cta.b64 [%0], 2;" ::"r"((unsigned)__cvta_generic_to_shared(&ready[tid])));
    const bool vec = (w % 8 == 0) && (lda % 8 == 0) && ((((uintptr_t)(A + K)) & 15) == 0);
    const bool cvec = (lda % 8 == 0) && ((((uintptr_t)(A + line0)) & 15) == 0);  // eight columns at a time
    __shared__ __align__(8) uint64_t xbar[2];
    __shared__ uint32_t xslot;
    const uint32_t ops = (smem_u32(psm) + (uint32_t)kCrossOpsOff + 1023u) & ~1023u;
    if constexpr (CROSS) cross_begin(*ct, ops, xbar, &xslot);
    if (ROWS) {
        for (int p = tid; p < rpc * nq; p += kPnlThreads) {
            const int r = p / nq, C = 8 * (p - r * nq);
            float v[8];
            const S* src = A + (int64_t)(line0 + min(r, nlive - 1)) * lda + K + C;
            if (vec) {
                load8(src, v);
            } else {
#pragma unroll
                for (int c = 0; c < 8; ++c) v[c] = (C + c < w) ? ld_elem(src + c) : 0.0f;
            }
            store8(X + r * kPnlXld + C, v);
        }
    } else if (cvec) {
        const int g8 = rpc >> 3;
        for (int p = tid; p < g8 * w8; p += kPnlThreads) {
            const int t = p / g8, c = 8 * (p - t * g8);
            float v[8];
            if (t < w && c + 8 <= nlive) {
                load8(A + (int64_t)(K + t) * lda + line0 + c, v);
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    v[e] = (t < w) ? ld_elem(A + (int64_t)(K + t) * lda + line0 + min(c + e, nlive - 1)) : 0.0f;
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) X[(c + e) * kPnlXld + t] = v[e];
        }
    } else {
        for (int p = tid; p < rpc * w8; p += kPnlThreads) {
            const int t = p / rpc, c = p - t * rpc;
            X[c * kPnlXld + t] = (t < w) ? ld_elem(A + (int64_t)(K + t) * lda + line0 + min(c, nlive - 1)) : 0.0f;
        }
    }
    bool bad = false, dead = false;
    if constexpr (CROSS) dead = !cross_end<!ROWS>(ops, xbar, &xslot, X, rpc, err);
    __syncthreads();
    if (warp >= kPnlFetchW) {
        bool ok = true;
        for (int q = 0; q < nq; ++q) {
            // warp v: every second of the step's eight rows of M from the v-th, four entries per lane;
            // lanes 0 and 1 of a row CTA also four pivots
            const int C = 8 * q, f = warp - kPnlFetchW, e = C + 4 * lane, kp = C + 4 * f + 2 * lane;
            const unsigned long long* src = pub + (ROWS ? 0 : kPubL) + (C + f) * 64 + (e >> 1);
            unsigned short* dst = M + (C + f) * kPnlMld + e;
            const unsigned todo = (e < w8 ? 15u : 0u) | (ROWS && lane < 2 ? 16u : 0u);
            ok = ok && pnl_fetch(
                           todo, [&](int v) { return v < 4 ? src + v * 128 : pub + kPubP + kp; },
                           [&](int v, unsigned v0, unsigned v1) {
                               if (v < 4) *reinterpret_cast<uint2*>(dst + 2 * v * kPnlMld) = make_uint2(v0, v1);
                               else *reinterpret_cast<float2*>(pv + kp) = make_float2(__uint_as_float(v0), __uint_as_float(v1));
                           },
                           epoch, flag, &gave_up);
            if (!ok) *(volatile int*)&gave_up = 1;
            __syncwarp();
            if (lane == 0)
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"((unsigned)__cvta_generic_to_shared(&ready[q]))
                             : "memory");
        }
    } else {
        const int nsol = rpc >> 5;  // solver warps; the rest help
        for (int q = 0; q < nq; ++q) {
            const int C0 = 8 * q, B0 = C0 - 8;
            pnl_wait_ready((unsigned)__cvta_generic_to_shared(&ready[q]), &gave_up);
            __syncwarp();
            if (warp < nsol) {
                float* xl = X + tid * kPnlXld + C0;
                float x[8];
                *reinterpret_cast<float4*>(x) = *reinterpret_cast<const float4*>(xl);
                *reinterpret_cast<float4*>(x + 4) = *reinterpret_cast<const float4*>(xl + 4);
                if (q > 0) pnl_apply(*reinterpret_cast<const uint4*>(xl - 8), M + B0 * kPnlMld + C0, kPnlMld, x);
                unsigned short h[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const uint4 m = *reinterpret_cast<const uint4*>(M + (C0 + k) * kPnlMld + C0);
                    if (ROWS) {
                        const float p = pv[C0 + k], ut = h_val(h_at(m, k));
                        if (!(fabsf(x[k]) <= fabsf(p))) bad = true;
                        h[k] = h_bits(div_neg(x[k], p, rcp_neg_abs(ut), fabsf(ut)));
                    } else {
                        h[k] = h_bits(x[k]);
                    }
#pragma unroll
                    for (int e = k + 1; e < 8; ++e) x[e] = fma_h(h[k], h_at(m, e), x[e]);
                }
                *reinterpret_cast<uint4*>(xl) =
                    make_uint4(h_pack(h[0], h[1]), h_pack(h[2], h[3]), h_pack(h[4], h[5]), h_pack(h[6], h[7]));
            } else if (q > 0) {
                const int nitem = nsol * (nq - q - 1);
                for (int it = warp - nsol; it < nitem; it += kPnlFetchW - nsol) {
                    const int b = it / nsol, ln = 32 * (it - b * nsol) + lane, C = C0 + 8 + 8 * b;
                    float* xl = X + ln * kPnlXld;
                    float x[8];
                    *reinterpret_cast<float4*>(x) = *reinterpret_cast<const float4*>(xl + C);
                    *reinterpret_cast<float4*>(x + 4) = *reinterpret_cast<const float4*>(xl + C + 4);
                    pnl_apply(*reinterpret_cast<const uint4*>(xl + B0), M + B0 * kPnlMld + C, kPnlMld, x);
                    *reinterpret_cast<float4*>(xl + C) = make_float4(x[0], x[1], x[2], x[3]);
                    *reinterpret_cast<float4*>(xl + C + 4) = make_float4(x[4], x[5], x[6], x[7]);
                }
            }
            asm volatile("bar.sync 1, %0;" ::"n"(32 * kPnlFetchW) : "memory");
        }
        if (tid >= nlive) bad = false;
    }
    if (__syncthreads_or(bad || dead) && tid == 0) atomicOr(flag, 1);
    if (gave_up) {
        if (tid == 0) {
            // a timeout (not an abandoned fast path) is an error; either way the
            // caller refactors with interchanges
            if (!*(volatile const int*)flag) atomicOr(err, (unsigned)ERR_TIMEOUT_OTHER);
            atomicOr(flag, 1);
        }
        return;
    }
    // the solved blocks: eight binary16 values (multipliers negated) at X[line][8 q]
    if (ROWS) {
        for (int p = tid; p < nlive * nq; p += kPnlThreads) {
            const int r = p / nq, C = 8 * (p - r * nq);
            uint4 h = *reinterpret_cast<const uint4*>(X + r * kPnlXld + C);
            h.x ^= 0x80008000u; h.y ^= 0x80008000u; h.z ^= 0x80008000u; h.w ^= 0x80008000u;
            S* dst = A + (int64_t)(line0 + r) * lda + K + C;
            if constexpr (std::is_same<S, __half>::value) {
                if (vec) {
                    *reinterpret_cast<uint4*>(dst) = h;
                    continue;
                }
            }
            if (vec) {
                float v[8];
#pragma unroll
                for (int c = 0; c < 8; ++c) v[c] = h_val(h_at(h, c));
                store8(dst, v);
            } else {
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    if (C + c < w) st_elem(dst + c, h_val(h_at(h, c)));
            }
        }
    } else {
        // U12 by rows, then U12^T for the tensor-core update: row idx - ut_col0, columns
        // ut_k0 .. ut_k0 + w - 1 (columns left of ut_col0 are not part of that update)
        const unsigned short* Xh = reinterpret_cast<const unsigned short*>(X);
        const int g8 = cvec ? nlive >> 3 : 0;  // whole groups of eight columns
        for (int p = tid; p < g8 * w; p += kPnlThreads) {
            const int t = p / g8, c = 8 * (p - t * g8);
            unsigned short h[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) h[e] = Xh[2 * ((c + e) * kPnlXld + (t & ~7)) + (t & 7)];
            S* dst = A + (int64_t)(K + t) * lda + line0 + c;
            if constexpr (std::is_same<S, __half>::value) {
                *reinterpret_cast<uint4*>(dst) =
                    make_uint4(h_pack(h[0], h[1]), h_pack(h[2], h[3]), h_pack(h[4], h[5]), h_pack(h[6], h[7]));
            } else {
                float v[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) v[e] = h_val(h[e]);
                store8(dst, v);
            }
        }
        for (int p = tid; p < (rpc - 8 * g8) * w; p += kPnlThreads) {
            const int t = p / (rpc - 8 * g8), c = 8 * g8 + p - t * (rpc - 8 * g8);
            if (c < nlive)
                st_elem(A + (int64_t)(K + t) * lda + line0 + c,
                        h_val(Xh[2 * (c * kPnlXld + (t & ~7)) + (t & 7)]));
        }
        if (Ut) {
            const bool uvec = (w % 8 == 0) && (ldut % 8 == 0) && (ut_k0 % 8 == 0) && ((((uintptr_t)Ut) & 15) == 0);
            for (int p = tid; p < nlive * nq; p += kPnlThreads) {
                const int c = p / nq, C = 8 * (p - c * nq), idx = line0 + c;
                if (idx < ut_col0) continue;
                const uint4 h = *reinterpret_cast<const uint4*>(X + c * kPnlXld + C);
                __half* u0 = Ut + (int64_t)(idx - ut_col0) * ldut + ut_k0 + C;
                if (uvec) {
                    *reinterpret_cast<uint4*>(u0) = h;
                } else {
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        if (C + e < w) u0[e] = __ushort_as_half(h_at(h, e));
                }
            }
        }
    }
}

// S: the storage the panel is read from and written to: the binary16 matrix,
// or (two-level LU) its single-precision shadow over the current outer block.
// Ut: U12^T in binary16 for the columns from ut_col0 (at K offset ut_k0).
// Roles are handed out in the order the CTAs start (an atomic ticket; panel p
// of a factorisation counts in word p % 2, its first CTA clears the other word
// and its last one its own; both are cleared when the factorisation starts): ticket 0
// factors the diagonal block and publishes its columns, tickets 1..nrb stream
// rows, the rest stream columns.  A CTA only ever waits on the diagonal CTA,
// which took its ticket before any waiting CTA existed and so is running: the
// launch needs no co-residency.
template <typename S>
__global__ void __launch_bounds__(kPnlThreads, 1) k_panel16(S* __restrict__ A, int64_t lda, int K, int w, int N,
                                                           int nrb, int rpc, int* __restrict__ ipiv, int* __restrict__ flag,
                                                           __half* __restrict__ Ut,
                                                           int ldut, int ut_col0, int ut_k0,
                                                           unsigned long long* __restrict__ pub, unsigned epoch,
                                                           unsigned* __restrict__ err, int* __restrict__ tickets,
                                                           int slot)
{
    __shared__ int role;
    if (threadIdx.x == 0) {
        const int t = atomicAdd(&tickets[slot], 1);
        if (t == 0) tickets[slot ^ 1] = 0;                // for the next panel (launched after this one ends)
        if (t == (int)gridDim.x - 1) tickets[slot] = 0;  // every ticket is taken: this launch's word is free
        role = t;
    }
    __syncthreads();
    const int r = role;
    if (r == 0)
        diag_lu16_body<true, S>(A, lda, K, w, ipiv, flag, nullptr, pub, epoch);
    else if (r <= nrb)
        panel16_stream<true, S>(A, lda, K, w, N, r - 1, rpc, Ut, ldut, ut_col0, ut_k0, flag, pub, epoch, err);
    else
        panel16_stream<false, S>(A, lda, K, w, N, r - 1 - nrb, rpc, Ut, ldut, ut_col0, ut_k0, flag, pub, epoch, err);
}

// k_panel16 for a panel of 128 columns after a panel of 128 whose update has not
// touched the panel's rows and columns yet: every CTA first applies it to its own
// tile (cross_begin / cross_end).  mA: L21 of the last panel from row K on, mB: its
// U12^T from column K on.  rpc: 64, 96 or 128.
__global__ void __launch_bounds__(kPnlThreads, 1) k_panel16x(const __grid_constant__ CUtensorMap mA,
                                                            const __grid_constant__ CUtensorMap mB,
                                                            __half* __restrict__ A, int64_t lda, int K, int w, int N,
                                                            int nrb, int rpc, int* __restrict__ ipiv, int* __restrict__ flag,
                                                            __half* __restrict__ Ut, int ldut,
                                                            unsigned long long* __restrict__ pub, unsigned epoch,
                                                            unsigned* __restrict__ err, int* __restrict__ tickets, int slot)
{
    __shared__ int role;
    if (threadIdx.x == 0) {
        const int t = atomicAdd(&tickets[slot], 1);
        if (t == 0) tickets[slot ^ 1] = 0;
        if (t == (int)gridDim.x - 1) tickets[slot] = 0;
        role = t;
    }
    __syncthreads();
    const int r = role;
    if (r == 0) {
        const CrossTile ct{&mA, &mB, 0, 0};
        diag_lu16_body<true, __half, 128, kD16Threads, true>(A, lda, K, w, ipiv, flag, nullptr, pub, epoch, &ct, err);
    } else if (r <= nrb) {
        const CrossTile ct{&mA, &mB, w + (r - 1) * rpc, 0};
        panel16_stream<true, __half, true>(A, lda, K, w, N, r - 1, rpc, Ut, ldut, K + w, 0, flag, pub, epoch, err, &ct);
    } else {
        const CrossTile ct{&mA, &mB, 0, w + (r - 1 - nrb) * rpc};
        panel16_stream<false, __half, true>(A, lda, K, w, N, r - 1 - nrb, rpc, Ut, ldut, K + w, 0, flag, pub, epoch, err, &ct);
    }
}

// k_offdiag16: L21 = A21 U11^{-1} (row role) and U12 = L11^{-1} A12 (column
// role) for a panel of width w, one thread per row (or column), 128 per CTA.
// A thread takes its row in blocks of eight, left-looking: the block is first
// updated with the row's earlier blocks (kept in shared memory as binary16, the
// multipliers negated), then solved against its diagonal 8 x 8 block of U11: at
// step t the thread checks its pre-division value against the unrounded pivot and
// forms l = fl16(x_t / u_tt).  The column role is the same with -L11 and no
// division (U entries rounded to binary16 as they are formed), and also writes
// U12^T for the tensor-core update.  U11 / -L11^T come from the stage as
// binary16 and are read by all threads at once (broadcast), eight entries a
// load, for fma.rn.f32.f16.  Every entry takes its updates in increasing t, as in
// right-looking elimination.  Bound by the multiply-adds where a launch fills the
// GPU, else by one CTA's time; the loops are short on purpose: the former
// straight-line solve of 32 entries ran from instruction memory once per chunk,
// and a line's entries are all loaded at the start (loaded block by block they
// were the longest stall).  A launch of a few CTAs at w = 64 takes 16 us (42
// before); the 512-instance batch's grouped factorisation 3.4 ms (4.2).
constexpr int kO16Threads = 128;
constexpr int kO16Rows = 128;  // rows or columns per CTA

// R: rows (columns) per CTA, one thread each: 128, or 256 for wide launches of
// 128-column panels (twice the warps per SM at one CTA per SM)
__host__ __device__ size_t offdiag16_smem(int wp, int R = kO16Rows)
{
    return ((size_t)wp * wp + (size_t)wp * R) * 2 + 2 * wp * sizeof(float);
}

template <typename S = __half, int ROWS = kO16Rows>
__device__ __forceinline__ void offdiag16_body(S* __restrict__ A, int64_t lda, int K, int w, int N,
                                               int nrow_blocks, __half* __restrict__ Ut, int ldut,
                                               int* __restrict__ flag, const float* stage, int bid,
                                               int ut_col0 = -1, int ut_k0 = 0, int tid_in = -1,
                                               float* smem = nullptr)
{
    if (ut_col0 < 0) ut_col0 = K + w;
    if (tid_in < 0 && *(volatile int*)flag) return;  // (a group of a larger CTA: its caller checked)
    extern __shared__ __align__(16) float osm[];
    const int wp = (w + 31) & ~31;
    // tid_in / smem: a group of 128 threads of a larger CTA and its own shared region (the
    // persistent grouped factorisation runs four such groups side by side)
    unsigned short* D = reinterpret_cast<unsigned short*>(smem ? smem : osm);  // U11 (rows) or -L11^T (columns), wp x wp
    unsigned short* X = D + wp * wp;   // every thread's finished blocks: multipliers (negated) / U entries
    float* pv = reinterpret_cast<float*>(X + wp * ROWS);  // a_tt, unrounded
    float* rinv = pv + wp;             // rcp_neg_abs(u_tt)
    const int tid = tid_in >= 0 ? tid_in : (int)threadIdx.x;
    const bool row_role = bid < nrow_blocks;
    {
        const uint4* s4 = reinterpret_cast<const uint4*>(reinterpret_cast<const unsigned short*>(stage) +
                                                         (row_role ? 0 : wp * wp));
        uint4* d4 = reinterpret_cast<uint4*>(D);
        const int nv = wp * wp / 8;
#pragma unroll 4
        for (int v = tid; v < nv; v += ROWS) d4[v] = s4[v];
        if (tid < wp) pv[tid] = tid < w ? stage[kStagePivOff + tid] : 1.0f;
    }
    __syncthreads();
    if (row_role && tid < wp) rinv[tid] = rcp_neg_abs(h_val(D[tid * wp + tid]));
    __syncthreads();
    const int idx = K + w + (row_role ? bid : bid - nrow_blocks) * ROWS + tid;
    const bool live = idx < N;
    uint4* H = reinterpret_cast<uint4*>(X) + tid;     // H[q * ROWS]: block q of this thread
    S* R = A + (int64_t)min(idx, N - 1) * lda + K;    // the row, or
    S* Cl = A + (int64_t)K * lda + min(idx, N - 1);   // the column
    const bool vec = (w % 8 == 0) && ((((uintptr_t)(A + K)) & 15) == 0) && (lda % 8 == 0);
    const bool uvec = Ut && idx >= ut_col0 && (w % 8 == 0) && (ldut % 8 == 0) && (ut_k0 % 8 == 0) && ((((uintptr_t)Ut) & 15) == 0);
    __half* ut = Ut + (Ut ? (int64_t)(idx - ut_col0) * ldut + ut_k0 : 0);
    const int nq = (w + 7) >> 3;
    bool bad = false;
    constexpr bool kHalf = std::is_same<S, __half>::value;
    if constexpr (kHalf) {
        // every block's entries first, all loads in flight, to where its solved ones will stand
#pragma unroll 4
        for (int q = 0; q < nq; ++q) {
            uint4 v;
            if (row_role && vec) {
                v = *reinterpret_cast<const uint4*>(R + 8 * q);
            } else {
                unsigned short e[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int t = 8 * q + k;
                    e[k] = t < w ? __half_as_ushort(row_role ? R[t] : Cl[(int64_t)t * lda]) : (unsigned short)0;
                }
                v = make_uint4(h_pack(e[0], e[1]), h_pack(e[2], e[3]), h_pack(e[4], e[5]), h_pack(e[6], e[7]));
            }
            H[q * ROWS] = v;
        }
    }
#pragma unroll 1
    for (int q = 0; q < nq; ++q) {
        const int C = 8 * q;
        float x[8];
        if constexpr (kHalf) {
            const uint4 v = H[q * ROWS];
#pragma unroll
            for (int k = 0; k < 8; ++k) x[k] = h_val(h_at(v, k));
        } else {
#pragma unroll
            for (int k = 0; k < 8; ++k)
                x[k] = (C + k < w) ? ld_elem(row_role ? R + C + k : Cl + (int64_t)(C + k) * lda) : 0.0f;
        }
#pragma unroll 1
        for (int b = 0; b < q; ++b) pnl_apply(H[b * ROWS], D + 8 * b * wp + C, wp, x);
        unsigned short h[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const uint4 m = *reinterpret_cast<const uint4*>(D + (C + k) * wp + C);
            if (row_role) {
                const float p = pv[C + k];
                bad |= live && C + k < w && !(fabsf(x[k]) <= fabsf(p));
                h[k] = h_bits(div_neg(x[k], p, rinv[C + k], fabsf(h_val(h_at(m, k)))));
            } else {
                h[k] = h_bits(x[k]);
            }
#pragma unroll
            for (int e = k + 1; e < 8; ++e) x[e] = fma_h(h[k], h_at(m, e), x[e]);
        }
        uint4 hv = make_uint4(h_pack(h[0], h[1]), h_pack(h[2], h[3]), h_pack(h[4], h[5]), h_pack(h[6], h[7]));
        H[q * ROWS] = hv;
        if (!live) continue;
        if (row_role) {
            hv.x ^= 0x80008000u; hv.y ^= 0x80008000u; hv.z ^= 0x80008000u; hv.w ^= 0x80008000u;
            if (vec) {
                if constexpr (std::is_same<S, __half>::value) {
                    *reinterpret_cast<uint4*>(R + C) = hv;
                } else {
                    float v[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) v[e] = h_val(h_at(hv, e));
                    store8(R + C, v);
                }
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    if (C + e < w) st_elem(R + C + e, h_val(h_at(hv, e)));
            }
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e)
                if (C + e < w) st_elem(Cl + (int64_t)(C + e) * lda, h_val(h_at(hv, e)));
            if (uvec) {
                *reinterpret_cast<uint4*>(ut + C) = hv;  // U12^T row (the tensor-core B operand)
            } else if (Ut && idx >= ut_col0) {
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    if (C + e < w) ut[C + e] = __ushort_as_half(h_at(hv, e));
            }
        }
    }
    if (row_role) {  // (the groups of a larger CTA share a role)
        if (__syncthreads_or(bad) && tid == 0) atomicOr(flag, 1);
    }
}

template <typename S, int ROWS = kO16Rows>
__global__ void __launch_bounds__(ROWS) k_offdiag16(S* __restrict__ A, int64_t lda, int K, int w, int N,
                                                 int nrow_blocks, __half* __restrict__ Ut, int ldut,
                                                 int* __restrict__ flag, const float* __restrict__ stage,
                                                 int ut_col0, int ut_k0)
{
    offdiag16_body<S, ROWS>(A, lda, K, w, N, nrow_blocks, Ut, ldut, flag, stage, (int)blockIdx.x, ut_col0, ut_k0);
}

// The off-diagonal solves of one panel: 128 rows (columns) per CTA, or 256 for a
// panel of 128 columns whose 128-row CTAs would not all fit at once (one CTA per
// SM either way at that width, so twice the warps per SM).  Bitwise the same
// results: every row (column) is solved by one thread in the same order.
template <typename S>
static nl_status launch_offdiag16(S* A, int64_t ld, int K, int wd, int N, __half* ut, int ldut, int* flag,
                                  const float* stage, int ut_col0, int ut_k0, cudaStream_t st)
{
    const int rest = N - K - wd, wp = (int)round_up(wd, 32);
    const bool wide = wp > 64 && 2 * (int)cdiv(rest, kO16Rows) > num_sms();
    prof_begin("k_offdiag16", st);
    if (wide) {
        const int nrb = (int)cdiv(rest, 256);
        k_offdiag16<S, 256><<<2 * nrb, 256, offdiag16_smem(wp, 256), st>>>(A, ld, K, wd, N, nrb, ut, ldut, flag, stage,
                                                                         ut_col0, ut_k0);
    } else {
        const int nrb = (int)cdiv(rest, kO16Rows);
        k_offdiag16<S><<<2 * nrb, kO16Threads, offdiag16_smem(wp), st>>>(A, ld, K, wd, N, nrb, ut, ldut, flag, stage,
                                                                        ut_col0, ut_k0);
    }
    prof_end("k_offdiag16", st);
    NL_CUDA_OK(cudaGetLastError());
    return NL_OK;
}

// C <- C - A B with per-element sequential fused multiply-adds over k in
// order, accumulated in T and stored once (rounded to binary16 for __half).
// BT x BT tiles (64 or 32), 256 threads.
template <typename S, typename T, int BT = 64>
__device__ __forceinline__ void gemm_simt_body(int M, int Nc, int K, const S* __restrict__ A, int64_t lda,
                                                   const S* __restrict__ B, int64_t ldb, S* __restrict__ C,
                                                   int64_t ldc, const int* __restrict__ flag, int m0, int n0)
{
    if (flag && *(volatile const int*)flag) return;
    constexpr int BM = BT, BN = BT, BK = 16, R = BT / 16;
    __shared__ T As[BK][BM + 1];
    __shared__ T Bs[BK][BN];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    T acc[R][R];
#pragma unroll
    for (int a = 0; a < R; ++a)
#pragma unroll
        for (int b = 0; b < R; ++b) {
            int i = m0 + ty + 16 * a, j = n0 + tx + 16 * b;
            acc[a][b] = (i < M && j < Nc) ? (T)ld_elem(C + (int64_t)i * ldc + j) : T(0);
        }
    for (int k0 = 0; k0 < K; k0 += BK) {
        __syncthreads();
        for (int q = threadIdx.x; q < BM * BK; q += 256) {
            int r = q / BK, kk = q % BK;
            int i = m0 + r, k = k0 + kk;
            As[kk][r] = (i < M && k < K) ? (T)ld_elem(A + (int64_t)i * lda + k) : T(0);
        }
        for (int q = threadIdx.x; q < BK * BN; q += 256) {
            int kk = q / BN, x = q % BN;
            int k = k0 + kk, j = n0 + x;
            Bs[kk][x] = (k < K && j < Nc) ? (T)ld_elem(B + (int64_t)k * ldb + j) : T(0);
        }
        __syncthreads();
        const int kmax = min(BK, K - k0);
        for (int kk = 0; kk < kmax; ++kk) {
            T av[R], bv[R];
#pragma unroll
            for (int a = 0; a < R; ++a) av[a] = As[kk][ty + 16 * a];
#pragma unroll
            for (int b = 0; b < R; ++b) bv[b] = Bs[kk][tx + 16 * b];
#pragma unroll
            for (int a = 0; a < R; ++a)
#pragma unroll
                for (int b = 0; b < R; ++b) acc[a][b] = fma(-av[a], bv[b], acc[a][b]);
        }
    }
#pragma unroll
    for (int a = 0; a < R; ++a)
#pragma unroll
        for (int b = 0; b < R; ++b) {
            int i = m0 + ty + 16 * a, j = n0 + tx + 16 * b;
            if (i < M && j < Nc) st_elem(C + (int64_t)i * ldc + j, acc[a][b]);
        }
}

template <typename S, typename T, int BT>
__global__ void __launch_bounds__(256) k_gemm_simt(int M, int Nc, int K, const S* __restrict__ A, int64_t lda,
                                                   const S* __restrict__ B, int64_t ldb, S* __restrict__ C,
                                                   int64_t ldc, const int* __restrict__ flag)
{
    gemm_simt_body<S, T, BT>(M, Nc, K, A, lda, B, ldb, C, ldc, flag, (int)blockIdx.y * BT, (int)blockIdx.x * BT);
}

// ------------------------------------------------------------------ host --

// Workspace layout: the interchanging path's working panel (N x min(nb, 128)),
// U12^T for the tensor-core update (N x nb binary16), info/flag words, the
// diagonal-block stage, the published columns, and for an outer block above
// 128 (two-level LU, binary16 only) the single-precision shadow N x ld, else
// (binary16) the look-ahead's second U12^T buffer.
size_t lu_work_bytes(int N, int nb, bool fp64)
{
    size_t el = fp64 ? 8 : 4;
    size_t pnl = (size_t)N * std::min(nb, 128) * el;
    size_t ut = fp64 ? 0 : (size_t)round_up(N, 128) * nb * 2;
    size_t shadow = fp64 ? 0 : (nb > 128 ? (size_t)N * round_up(N, 64) * 4 + 256 : round_up(ut, 256));
    return round_up(pnl, 256) + round_up(ut, 256) + 256 + (size_t)2 * 128 * 128 * 8 + 128 * 8 +
           round_up(kPubWords * 8, 256) + shadow;
}

void lu_work_carve(void* base, int N, int nb, bool fp64, LuWork* w)
{
    char* p = (char*)base;
    size_t el = fp64 ? 8 : 4;
    w->pnl = p;
    p += round_up((size_t)N * std::min(nb, 128) * el, 256);
    size_t ut = fp64 ? 0 : (size_t)round_up(N, 128) * nb * 2;
    w->ut = fp64 ? nullptr : (__half*)p;
    p += round_up(ut, 256);
    w->info = (int*)p;
    w->flag = w->info + 1;
    p += 256;
    w->stage = p;
    p += (size_t)2 * 128 * 128 * 8 + 128 * 8;
    w->pub = (unsigned long long*)p;
    p += round_up(kPubWords * 8, 256);
    w->ut2 = nullptr;
    if (!fp64 && nb > 128) {
        w->p32 = (float*)p;
        w->ldp32 = round_up(N, 64);
    } else {
        w->p32 = nullptr;
        w->ldp32 = 0;
        if (!fp64) w->ut2 = (__half*)p;
    }
}

nl_status lu_side_prepare(LuWork* w, cudaStream_t st)
{
    // one step below st's priority (lower priority = larger number): the rest of an update has
    // a panel's time of slack, so it yields SMs to the latency-bound panels of concurrent solves
    int prio = 0, least = 0, greatest = 0;
    NL_CUDA_OK(cudaStreamGetPriority(st, &prio));
    NL_CUDA_OK(cudaDeviceGetStreamPriorityRange(&least, &greatest));
    prio = std::min(prio + 1, least);
    if (w->side) {
        int have = 0;
        NL_CUDA_OK(cudaStreamGetPriority(w->side, &have));
        if (have == prio) return NL_OK;
        NL_CUDA_OK(cudaStreamSynchronize(w->side));
        NL_CUDA_OK(cudaStreamDestroy(w->side));
        w->side = nullptr;
    }
    if (debug_fail_stream()) {
        set_error("LU look-ahead: stream creation failed (test hook)");
        return NL_ECUDA;
    }
    NL_CUDA_OK(cudaStreamCreateWithPriority(&w->side, cudaStreamNonBlocking, prio));
    if (!w->ev_fork) NL_CUDA_OK(cudaEventCreateWithFlags(&w->ev_fork, cudaEventDisableTiming));
    for (auto& e : w->ev_join)
        if (!e) NL_CUDA_OK(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    return NL_OK;
}

void lu_side_release(LuWork* w)
{
    if (w->side) cudaStreamDestroy(w->side);
    if (w->ev_fork) cudaEventDestroy(w->ev_fork);
    for (auto& e : w->ev_join)
        if (e) cudaEventDestroy(e);
    w->side = nullptr;
    w->ev_fork = w->ev_join[0] = w->ev_join[1] = nullptr;
}

template <typename T, int NBL, int R, bool RND>
static nl_status launch_leaf_r(T* P, int ldp, int k0, int M, int w, int wl, int* ipiv_out, int piv_base, int* info,
                               int C, int rows_per_cta, cudaStream_t st)
{
    auto kern = k_leaf<T, NBL, R, RND>;
    if (C > 1) {
        static bool attr_done = false;
        if (!attr_done) {
            NL_CUDA_OK(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
            attr_done = true;
        }
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = C;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(C);
        cfg.blockDim = dim3(kLeafThreads);
        cfg.dynamicSmemBytes = 0;
        cfg.stream = st;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        NL_CUDA_OK(cudaLaunchKernelEx(&cfg, kern, P, ldp, k0, M, w, wl, ipiv_out, piv_base, info, C, rows_per_cta));
    } else {
        kern<<<1, kLeafThreads, 0, st>>>(P, ldp, k0, M, w, wl, ipiv_out, piv_base, info, 1, rows_per_cta);
        NL_CUDA_OK(cudaGetLastError());
    }
    return NL_OK;
}

// Cluster size and rows per thread for a leaf of Ml rows: the fewest CTAs
// (cheapest exchange) with at most 4 (8 beyond 16384 rows) rows per thread.
template <typename T, int NBL, bool RND>
static nl_status launch_leaf(T* P, int ldp, int k0, int M, int w, int wl, int* ipiv_out, int piv_base, int* info,
                             cudaStream_t st)
{
    const int Ml = M - k0;
    // at most 4 rows per thread (spill-free) unless the leaf needs more than
    // 16 CTAs at that density
    int C = (int)cdiv(Ml, 4 * kLeafThreads);
    if (C > kMaxCluster) C = (int)cdiv(Ml, 8 * kLeafThreads);
    if (C > kMaxCluster) {
        set_error("LU leaf: %d rows exceed the register-resident limit", Ml);
        return NL_EINVAL;
    }
    if (C > 8) C = 16;
    else if (C > 4) C = 8;
    else if (C > 2) C = 4;
    const int rows_per_cta = (int)cdiv(Ml, C);
    const int R = (int)cdiv(rows_per_cta, kLeafThreads);
    if (R <= 1) return launch_leaf_r<T, NBL, 1, RND>(P, ldp, k0, M, w, wl, ipiv_out, piv_base, info, C, rows_per_cta, st);
    if (R <= 2) return launch_leaf_r<T, NBL, 2, RND>(P, ldp, k0, M, w, wl, ipiv_out, piv_base, info, C, rows_per_cta, st);
    if (R <= 4) return launch_leaf_r<T, NBL, 4, RND>(P, ldp, k0, M, w, wl, ipiv_out, piv_base, info, C, rows_per_cta, st);
    return launch_leaf_r<T, NBL, 8, RND>(P, ldp, k0, M, w, wl, ipiv_out, piv_base, info, C, rows_per_cta, st);
}

template <typename S, typename T>
static nl_status launch_gemm_simt(int M, int Nc, int K, const S* A, int64_t lda, const S* B, int64_t ldb, S* C,
                                  int64_t ldc, cudaStream_t st, const int* flag = nullptr)
{
    if (M <= 0 || Nc <= 0 || K <= 0) return NL_OK;
    // Double precision is bound by its pipe (a 64 x 64 tile of depth 64 takes an SM 66 us), so the
    // tile follows the work of the busiest SM; single precision keeps 64.
    const int64_t sms = num_sms(), t64 = cdiv(Nc, 64) * cdiv(M, 64), t32 = cdiv(Nc, 32) * cdiv(M, 32);
    bool small = false;
    if constexpr (sizeof(T) == 8) small = cdiv(t32, sms) < 4 * cdiv(t64, sms);
    if constexpr (sizeof(T) == 8) {
        if (small)
            k_gemm_simt<S, T, 32><<<dim3((unsigned)cdiv(Nc, 32), (unsigned)cdiv(M, 32)), 256, 0, st>>>(M, Nc, K, A, lda, B, ldb,
                                                                                                C, ldc, flag);
    }
    if (!small)
        k_gemm_simt<S, T, 64><<<dim3((unsigned)cdiv(Nc, 64), (unsigned)cdiv(M, 64)), 256, 0, st>>>(M, Nc, K, A, lda, B, ldb,
                                                                                                C, ldc, flag);
    NL_CUDA_OK(cudaGetLastError());
    return NL_OK;
}

__global__ void k_transpose16(int R, int Cc, const __half* __restrict__ in, int64_t ldi, __half* __restrict__ out,
                              int64_t ldo)
{
    __shared__ __half tile[32][33];
    int c = blockIdx.x * 32 + threadIdx.x, r = blockIdx.y * 32 + threadIdx.y;
    for (int k = 0; k < 32; k += 8)
        if (r + k < R && c < Cc) tile[threadIdx.y + k][threadIdx.x] = in[(int64_t)(r + k) * ldi + c];
    __syncthreads();
    c = blockIdx.y * 32 + threadIdx.x;
    r = blockIdx.x * 32 + threadIdx.y;
    for (int k = 0; k < 32; k += 8)
        if (r + k < Cc && c < R) out[(int64_t)(r + k) * ldo + c] = tile[threadIdx.x][threadIdx.y + k];
}

nl_status launch_transpose16(int R, int Cc, const __half* in, int64_t ldi, __half* out, int64_t ldo, cudaStream_t st)
{
    dim3 grid((unsigned)cdiv(Cc, 32), (unsigned)cdiv(R, 32));
    k_transpose16<<<grid, dim3(32, 8), 0, st>>>(R, Cc, in, ldi, out, ldo);
    NL_CUDA_OK(cudaGetLastError());
    return NL_OK;
}

nl_status gemm16_update(int M, int Nc, int K, const __half* A, int64_t lda, const __half* B, int64_t ldb, __half* C,
                        int64_t ldc, int gemm, cudaStream_t st)
{
    if (gemm == 2 || gemm == 3) {
        // the tensor-core path takes B transposed (K-major): build it
        __half* Bt = nullptr;
        NL_CUDA_OK(ws_malloc_async((void**)&Bt, (size_t)round_up(Nc, 128) * K * 2, st));
        nl_status s = launch_transpose16(K, Nc, B, ldb, Bt, K, st);
        if (s == NL_OK) s = tc_gemm16_update(M, Nc, K, A, lda, Bt, K, C, ldc, st, nullptr, gemm == 3);
        cudaFreeAsync(Bt, st);
        return s;
    }
    return launch_gemm_simt<__half, float>(M, Nc, K, A, lda, B, ldb, C, ldc, st);
}

// A22 <- A22 - L21 U12 for the panel [K, K+wd): tcgen05 when possible.
template <typename T, typename S>
static nl_status trailing_update(int N, S* A, int64_t ld, int K, int wd, int nb, bool tc, const __half* ut,
                                 const int* flag, cudaStream_t st)
{
    const int rest = N - K - wd;
    S* L21 = A + (int64_t)(K + wd) * ld + K;
    S* U12 = A + (int64_t)K * ld + K + wd;
    S* A22 = A + (int64_t)(K + wd) * ld + K + wd;
    if (tc) {
        if constexpr (std::is_same<S, __half>::value) return tc_gemm16_update(rest, rest, wd, L21, ld, ut, nb, A22, ld, st, flag);
    }
    return launch_gemm_simt<S, T>(rest, rest, wd, L21, ld, U12, ld, A22, ld, st, flag);
}

// The streaming panel (k_panel16): one CTA for the diagonal block plus
// ceil(rest / rpc) CTAs for the rows of L21 and as many for the columns of U12.
static nl_status panel16_setup()
{
    static std::atomic<bool> done{false};
    if (done.load(std::memory_order_acquire)) return NL_OK;
    if (set_max_dynamic_smem((const void*)k_panel16<__half>) != NL_OK ||
        set_max_dynamic_smem((const void*)k_panel16<float>) != NL_OK ||
        set_max_dynamic_smem((const void*)k_panel16x) != NL_OK)
        return NL_ECUDA;
    done.store(true, std::memory_order_release);
    return NL_OK;
}

// Lines (rows, columns) per streaming CTA, one CTA per SM: 64 while they take
// at most half of the SMs (the rest is for the look-ahead's update and for other
// streams' solves), then 96 while all fit on the GPU at once, else 128 (a
// launch of several waves keeps going: a CTA that starts after the diagonal
// block is done finds every word published).  Few lines make the tail after the
// last published block short, few CTAs leave SMs to the work beside it.  Measured
// with 64 as long as all fit, with 96 (128) from half of the SMs on: a solve at
// N = 4096 9.60, 9.44 (9.96) ms, five at once 24.0, 22.6 (22.5) ms, one
// factorisation at N = 8192 3.04, 2.97 ms; 96 at every size: 9.58, 22.5, 2.97 ms.
static int panel16_rows_per_cta(int rest, int pref = 0)
{
    if (pref == kPnlRows) return kPnlRows;
    if (1 + 2 * (int)cdiv(rest, 64) <= num_sms() / 2) return 64;
    return 1 + 2 * (int)cdiv(rest, 96) <= num_sms() ? 96 : 128;
}

static std::atomic<unsigned> g_panel_epoch{0};

template <typename S>
static nl_status launch_panel16(S* A, int64_t ld, int K, int wd, int N, int* ipiv, const LuWork& w, __half* Ut,
                                int ldut, cudaStream_t st, int slot, int ut_col0 = -1, int ut_k0 = 0,
                                const __half* ut_prev = nullptr)
{
    // ut_prev: U12^T of the last panel (128 columns), whose update of this panel's tiles is still to be done
    if (ut_col0 < 0) ut_col0 = K + wd;
    const int rest = N - K - wd;
    int rpc = panel16_rows_per_cta(rest, w.stream);
    int nrb = (int)cdiv(rest, rpc);
    unsigned epoch = ++g_panel_epoch;
    if (epoch == 0) epoch = ++g_panel_epoch;  // 0 is the cleared buffer's tag
    int* flag = w.flag;
    unsigned long long* pub = w.pub;
    NL_TRY(panel16_setup());
    unsigned* err = tc_error_word();
    if (!err) err = (unsigned*)(w.info + 2);  // (a word of the info block nobody else uses)
    int* tickets = w.info + 8;  // two counters (+8, +9) of the info block; slot: the panel's index mod 2
    if constexpr (std::is_same<S, __half>::value) {
        if (ut_prev) {
            TmapBytes mA, mB;
            if (!tc_encode_operand(A + (int64_t)K * ld + K - 128, N - K, ld, &mA) ||
                !tc_encode_operand(ut_prev, N - K, ldut, &mB)) {
                set_error("panel: cuTensorMapEncodeTiled failed");
                return NL_ECUDA;
            }
            prof_begin("k_panel16", st);
            k_panel16x<<<1 + 2 * nrb, kPnlThreads, kCrossSmem, st>>>(
                reinterpret_cast<const CUtensorMap&>(mA), reinterpret_cast<const CUtensorMap&>(mB), A, ld, K, wd, N, nrb, rpc,
                ipiv, flag, Ut, ldut, pub, epoch, err, tickets, slot);
            prof_end("k_panel16", st);
            NL_CUDA_OK(cudaGetLastError());
            return NL_OK;
        }
    }
    prof_begin("k_panel16", st);
    k_panel16<S><<<1 + 2 * nrb, kPnlThreads, kPnlSmem, st>>>(A, ld, K, wd, N, nrb, rpc, ipiv, flag, Ut, ldut,
                                                            ut_col0, ut_k0, pub, epoch, err, tickets, slot);
    prof_end("k_panel16", st);
    NL_CUDA_OK(cudaGetLastError());
    return NL_OK;
}

template <typename T, typename S, int NBL, bool RND>
static nl_status lu_factor_impl(int N, S* A, int64_t ld, int* ipiv, int nb, int gemm, bool fast, const LuWork& w,
                                cudaStream_t st, int* launches)
{
    T* P = (T*)w.pnl;
    const int ldp = nb;
    int nl = 0;
    NL_CUDA_OK(cudaMemsetAsync(w.info, 0, 10 * sizeof(int), st));  // info, flag, ..., the panel's role ticket
    constexpr bool kHalf = std::is_same<S, __half>::value;
    static bool smem_set = false;
    if (!smem_set) {
        if (set_max_dynamic_smem((const void*)k_trsm_u12<T, S, RND>) != NL_OK) return NL_ECUDA;
        if constexpr (kHalf) {
            if (set_max_dynamic_smem((const void*)k_offdiag16<__half>) != NL_OK ||
                set_max_dynamic_smem((const void*)k_offdiag16<float>) != NL_OK ||
                set_max_dynamic_smem((const void*)k_offdiag16<__half, 256>) != NL_OK ||
                set_max_dynamic_smem((const void*)k_offdiag16<float, 256>) != NL_OK ||
                set_max_dynamic_smem((const void*)k_diag_lu16<__half>) != NL_OK ||
                set_max_dynamic_smem((const void*)k_diag_lu16<float>) != NL_OK)
                return NL_ECUDA;
        } else {
            if (set_max_dynamic_smem((const void*)k_offdiag<T, S>) != NL_OK ||
                set_max_dynamic_smem((const void*)k_diag_lu<T, S, RND>) != NL_OK)
                return NL_ECUDA;
        }
        smem_set = true;
    }
    bool pub_cleared = false;
    // Look-ahead (fast path, tensor-core update): the update after panel q is split into the
    // cross (the first 128-row and 128-column tile strips of the trailing matrix, which hold
    // panel q + 1), one launch on st, and the rest on w.side, which then runs in the shadow of
    // panel q + 1 and is joined back (ev_join[q % 2]) before the cross of update q + 1.  The
    // tiles are the same tcgen05 tiles as in one update, so the factors are bitwise the same.
    // Panels alternate U12^T buffers.
    constexpr int kLaTile = 128;  // the tcgen05 update's tile (M = N = 128)
    const bool la = kHalf && fast && lu_looks_ahead(nb, gemm) && w.side && w.ut2 && w.ev_fork && w.ev_join[0] &&
                    w.ev_join[1];
    struct Join {
        const LuWork& w;
        cudaStream_t st;
        int pending = 0;  // bit q % 2: the rest of update q is recorded on ev_join[q % 2], not yet joined
        bool wait(int q)
        {
            if (q < 0 || !((pending >> (q & 1)) & 1)) return true;
            pending &= ~(1 << (q & 1));
            return cudaStreamWaitEvent(st, w.ev_join[q & 1], 0) == cudaSuccess;
        }
        bool all() { return wait(0) && wait(1); }
        ~Join() { all(); }
    } join{w, st};
    auto join_ok = [&](bool ok) -> nl_status {
        if (ok) return NL_OK;
        set_error("LU look-ahead: cudaStreamWaitEvent failed");
        return NL_ECUDA;
    };
    auto ut_of = [&](int K) { return (la && ((K / nb) & 1)) ? w.ut2 : w.ut; };
    // With panels of 128 the next panel's own CTAs take the cross (k_panel16x), while it has
    // rows below it and its CTAs hold at most 128 lines; cross_ut: U12^T of the panel whose cross is left to the next.
    const __half* cross_ut = nullptr;
    const bool merge = la && nb == kLaTile && w.stream == 0;
    // the update after the panel at K (width wd)
    auto update = [&](int K, int wd, bool tc, const __half* utp) -> nl_status {
        const int rest = N - K - wd, q = K / nb;
        if (!(la && tc)) {
            NL_TRY(join_ok(join.all()));
            return trailing_update<T, S>(N, A, ld, K, wd, nb, tc, utp, w.flag, st);
        }
        if constexpr (kHalf) {
            S* L21 = A + (int64_t)(K + wd) * ld + K;
            S* A22 = A + (int64_t)(K + wd) * ld + K + wd;
            const bool side_now = rest > kLaTile;
            if (side_now) NL_CUDA_OK(cudaEventRecord(w.ev_fork, st));
            NL_TRY(join_ok(join.wait(q - 1)));  // the rest of update q - 1 wrote the cross's tiles
            if (merge && wd == kLaTile && side_now) {
                cross_ut = utp;
                --nl;
            } else NL_TRY(tc_gemm16_update(rest, rest, wd, L21, ld, utp, nb, A22, ld, st, w.flag, false, true));
            if (side_now) {
                const int m2 = rest - kLaTile;
                NL_TRY(join_ok(join.wait(q - 2)));  // ev_join[q % 2] is free again
                NL_CUDA_OK(cudaStreamWaitEvent(w.side, w.ev_fork, 0));
                // (a panel's time of slack: a quarter of the SMs, the rest left to concurrent solves' panels)
                NL_TRY(tc_gemm16_update(m2, m2, wd, L21 + (int64_t)kLaTile * ld, ld, utp + (int64_t)kLaTile * nb, nb,
                                        A22 + (int64_t)kLaTile * ld + kLaTile, ld, w.side, w.flag, false, false,
                                        std::max(1, num_sms() / 4)));
                NL_CUDA_OK(cudaEventRecord(w.ev_join[q & 1], w.side));
                join.pending |= 1 << (q & 1);
                ++nl;
            }
        }
        return NL_OK;
    };
    for (int K = 0; K < N; K += nb) {
        const int wd = std::min(nb, N - K), M = N - K;
        const int rest = N - K - wd;
        const bool tc = (gemm == 2) && std::is_same<S, __half>::value && (wd % 64 == 0);
        const size_t trsm_smem = (size_t)wd * wd * sizeof(T) + (size_t)wd * kTrsmThreads * sizeof(T);
        if (fast) {
            const int wp = (int)round_up(wd, 32);
            if constexpr (kHalf) {
                if (rest > 0 && w.stream >= 0) {
                    if (!pub_cleared) {
                        NL_CUDA_OK(cudaMemsetAsync(w.pub, 0, kPubWords * 8, st));
                        pub_cleared = true;
                    }
                    __half* utp = tc ? ut_of(K) : nullptr;
                    const __half* cu = cross_ut;
                    cross_ut = nullptr;
                    NL_TRY(launch_panel16(A, ld, K, wd, N, ipiv, w, utp, nb, st, (K / nb) & 1, -1, 0, cu));
                    NL_TRY(update(K, wd, tc, utp));
                    nl += 2;
                    continue;
                }
                prof_begin("k_diag_lu16", st);
                k_diag_lu16<__half><<<1, kD16Threads, kDiag16Smem, st>>>(A, ld, K, wd, ipiv, w.flag,
                                                                      rest > 0 ? (float*)w.stage : nullptr);
                prof_end("k_diag_lu16", st);
            } else {
                prof_begin("k_diag_lu", st);
                k_diag_lu<T, S, RND><<<1, kDiagThreads, (size_t)wp * (wp + 1) * sizeof(T), st>>>(A, ld, K, wd, ipiv,
                                                                                            w.flag, w.stage);
                prof_end("k_diag_lu", st);
            }
            ++nl;
            if (rest > 0) {
                if constexpr (kHalf) {
                    NL_TRY(launch_offdiag16<__half>(A, ld, K, wd, N, tc ? ut_of(K) : nullptr, nb, w.flag,
                                                    (const float*)w.stage, -1, 0, st));
                } else {
                    const int nrb = (int)cdiv(rest, kOffLines);
                    prof_begin("k_offdiag", st);
                    k_offdiag<T, S><<<2 * nrb, kOffThreads, offdiag_smem(wp, sizeof(T)), st>>>(A, ld, K, wd, N, nrb, w.flag,
                                                                                            w.stage);
                    prof_end("k_offdiag", st);
                }
                NL_TRY(update(K, wd, tc, ut_of(K)));
                nl += 2;
            }
            NL_CUDA_OK(cudaGetLastError());
            continue;
        }
        k_panel_load<T, S><<<M, 128, 0, st>>>(A, ld, K, M, wd, P, ldp);
        ++nl;
        for (int k0 = 0; k0 < wd; k0 += NBL) {
            const int wl = std::min(NBL, wd - k0);
            nl_status s = launch_leaf<T, NBL, RND>(P, ldp, k0, M, wd, wl, ipiv + K + k0, K + k0, w.info, st);
            if (s != NL_OK) return s;
            ++nl;
            if (k0 + wl < wd && M > k0 + wl) {
                unsigned g = (unsigned)cdiv(M - k0 - wl, 64);
                k_panel_gemm<T, NBL><<<g, 256, 0, st>>>(P, ldp, k0, wl, M, wd);
                ++nl;
            }
        }
        k_panel_store<T, S><<<M, 128, 0, st>>>(A, ld, K, M, wd, P, ldp);
        ++nl;
        if (N - wd > 0) {
            k_laswp<S><<<(unsigned)cdiv(N - wd, 256), 256, 0, st>>>(A, ld, K, wd, N, ipiv);
            ++nl;
        }
        if (rest > 0) {
            k_trsm_u12<T, S, RND><<<(unsigned)cdiv(rest, kTrsmThreads), kTrsmThreads, trsm_smem, st>>>(
                A, ld, K, wd, N, tc ? w.ut : nullptr, nb, nullptr);
            nl_status s = trailing_update<T, S>(N, A, ld, K, wd, nb, tc, w.ut, nullptr, st);
            if (s != NL_OK) return s;
            nl += 2;
        }
        NL_CUDA_OK(cudaGetLastError());
    }
    NL_TRY(join_ok(join.all()));
    if (launches) *launches += nl;
    return NL_OK;
}

// ------------------------------------------------------ two-level LU --
// Outer block W (a multiple of 128 up to 512), inner panels of 128, for the
// binary16 fast path: the arithmetic of rounding period W, i.e. the oracle's
// binary16-storage / binary32-arithmetic elimination with nb = W.  Per outer
// block [K0, K0 + W):
//   * its row and column strips (rows K0.. x columns K0..K0+W-1, and rows
//     K0..K0+W-1 x the columns right of it) are copied to a single-precision
//     shadow P;
//   * each inner panel is factored on P by the streaming panel (or the two
//     launches) exactly as the one-level path factors A: multipliers and U
//     entries rounded to binary16 as they are formed, U12^T of the columns
//     right of the outer block written in binary16 for the update below;
//   * the inner panel's update is applied in single precision, unrounded, to
//     the rest of the two strips only: with the SIMT update one fused
//     multiply-add per term in increasing k (the oracle's sequence exactly);
//     with the tensor-core update on the tcgen05 kernel for binary32 C (the
//     operands are binary16 values, so the K products are exact and their
//     sum is applied with one binary32 rounding);
//   * the strips go back to A (their entries are now binary16 values), and
//     the rest of the matrix receives one update of depth W,
//     A22 <- fl16(A22 - L21 U12), on the tensor cores (K streamed through the
//     persistent kernel's operand ring) or SIMT.
// So the trailing matrix is read and written once per W columns instead of
// once per 128.
template <bool TO32>
__global__ void __launch_bounds__(256) k_strip_copy(__half* __restrict__ A, int64_t lda, float* __restrict__ P,
                                                    int64_t ldp, int r0, int c0, int ncols)
{
    const int i = r0 + blockIdx.y;
    const int j = c0 + (blockIdx.x * 256 + threadIdx.x) * 8;
    if (j >= c0 + ncols) return;
    __half* a = A + (int64_t)i * lda + j;
    float* q = P + (int64_t)i * ldp + j;
    const int n = min(8, c0 + ncols - j);
    if (n == 8 && ((((uintptr_t)a) & 15) == 0) && ((((uintptr_t)q) & 15) == 0)) {
        float v[8];
        if (TO32) {
            load8(a, v);
            store8(q, v);
        } else {
            load8(q, v);
            store8(a, v);
        }
    } else {
        for (int e = 0; e < n; ++e) {
            if (TO32) q[e] = __half2float(a[e]);
            else a[e] = __float2half_rn(q[e]);
        }
    }
}

template <bool TO32>
static nl_status copy_block(__half* A, int64_t lda, float* P, int64_t ldp, int r0, int c0, int nrows, int ncols,
                            cudaStream_t st)
{
    if (nrows <= 0 || ncols <= 0) return NL_OK;
    for (int y0 = 0; y0 < nrows; y0 += 65535) {
        const int ny = std::min(65535, nrows - y0);
        k_strip_copy<TO32><<<dim3((unsigned)cdiv(ncols, 256 * 8), (unsigned)ny), 256, 0, st>>>(A, lda, P, ldp, r0 + y0,
                                                                                              c0, ncols);
    }
    NL_CUDA_OK(cudaGetLastError());
    return NL_OK;
}

static nl_status lu16_factor_2lvl(int N, __half* A, int64_t ld, int* ipiv, int W, int gemm, const LuWork& w,
                                  cudaStream_t st, int* launches)
{
    float* P = w.p32;
    const int64_t ldp = w.ldp32;
    if (!P) {
        set_error("lu16: an outer block above 128 needs the single-precision shadow workspace");
        return NL_EINVAL;
    }
    int nl = 0;
    NL_CUDA_OK(cudaMemsetAsync(w.info, 0, 10 * sizeof(int), st));  // info, flag, ..., the panel's role ticket
    NL_CUDA_OK(cudaMemsetAsync(w.pub, 0, kPubWords * 8, st));
    static bool smem_set = false;
    if (!smem_set) {
        if (set_max_dynamic_smem((const void*)k_offdiag16<float>) != NL_OK ||
            set_max_dynamic_smem((const void*)k_offdiag16<float, 256>) != NL_OK ||
            set_max_dynamic_smem((const void*)k_diag_lu16<float>) != NL_OK)
            return NL_ECUDA;
        smem_set = true;
    }
    for (int K0 = 0; K0 < N; K0 += W) {
        const int Wd = std::min(W, N - K0), far = N - K0 - Wd, C1 = K0 + Wd;
        const bool tc = gemm == 2 && tc_gemm_supported() && (Wd % 64 == 0);
        NL_TRY(copy_block<true>(A, ld, P, ldp, K0, K0, N - K0, Wd, st));
        NL_TRY(copy_block<true>(A, ld, P, ldp, K0, C1, Wd, far, st));
        nl += 2;
        for (int p0 = 0; p0 < Wd; p0 += 128) {
            const int K = K0 + p0, wd = std::min(128, Wd - p0), rest = N - K - wd;
            __half* ut = (tc && far > 0) ? w.ut : nullptr;
            if (rest > 0 && w.stream >= 0) {
                NL_TRY(launch_panel16<float>(P, ldp, K, wd, N, ipiv, w, ut, W, st, (K / 128) & 1, C1, p0));
                ++nl;
            } else {
                prof_begin("k_diag_lu16", st);
                k_diag_lu16<float><<<1, kD16Threads, kDiag16Smem, st>>>(P, ldp, K, wd, ipiv, w.flag,
                                                                     rest > 0 ? (float*)w.stage : nullptr);
                prof_end("k_diag_lu16", st);
                ++nl;
                if (rest > 0) {
                    NL_TRY(launch_offdiag16<float>(P, ldp, K, wd, N, ut, W, w.flag, (const float*)w.stage, C1, p0, st));
                    ++nl;
                }
            }
            // this inner panel's update on the rest of the two strips, unrounded (single
            // precision): SIMT fused multiply-adds in order k (the oracle's arithmetic), or
            // with the tensor-core update the tcgen05 kernel for binary32 C
            const bool tci = gemm == 2 && tc_gemm_supported();
            const int right = C1 - K - wd;  // strip columns right of the inner panel
            if (rest > 0 && right > 0) {
                const float* L21 = P + (K + wd) * ldp + K;
                const float* U12 = P + K * ldp + K + wd;
                float* C22 = P + (K + wd) * ldp + K + wd;
                if (tci) NL_TRY(tc_update_f32(rest, right, wd, L21, ldp, U12, ldp, C22, ldp, st, w.flag));
                else NL_TRY((launch_gemm_simt<float, float>(rest, right, wd, L21, ldp, U12, ldp, C22, ldp, st, w.flag)));
                ++nl;
            }
            const int below = C1 - K - wd;  // rows of the outer block below the inner panel
            if (far > 0 && below > 0) {
                const float* L21 = P + (K + wd) * ldp + K;
                const float* U12 = P + K * ldp + C1;
                float* C22 = P + (K + wd) * ldp + C1;
                if (tci) NL_TRY(tc_update_f32(below, far, wd, L21, ldp, U12, ldp, C22, ldp, st, w.flag));
                else NL_TRY((launch_gemm_simt<float, float>(below, far, wd, L21, ldp, U12, ldp, C22, ldp, st, w.flag)));
                ++nl;
            }
        }
        NL_TRY(copy_block<false>(A, ld, P, ldp, K0, K0, N - K0, Wd, st));
        NL_TRY(copy_block<false>(A, ld, P, ldp, K0, C1, Wd, far, st));
        nl += 2;
        if (far > 0) {
            __half* L21 = A + (int64_t)C1 * ld + K0;
            __half* A22 = A + (int64_t)C1 * ld + C1;
            if (tc) NL_TRY(tc_gemm16_update(far, far, Wd, L21, ld, w.ut, W, A22, ld, st, w.flag));
            else NL_TRY((launch_gemm_simt<__half, float>(far, far, Wd, L21, ld, A + (int64_t)K0 * ld + C1, ld, A22,
                                                        ld, st, w.flag)));
            ++nl;
        }
        NL_CUDA_OK(cudaGetLastError());
    }
    if (launches) *launches += nl;
    return NL_OK;
}

// Outer block nb: a multiple of 16 up to 128 (one level), or 256, 384, 512
// (two levels, fast path only; the interchanging path factors with 128).
bool lu16_nb_valid(int nb) { return (nb >= 16 && nb <= 128 && nb % 16 == 0) || nb == 256 || nb == 384 || nb == 512; }

nl_status lu16_factor(int N, __half* A, int64_t ld, int* ipiv, int nb, int gemm, bool fast, const LuWork& w,
                      cudaStream_t st, int* launches)
{
    if (!lu16_nb_valid(nb)) {
        set_error("lu16: nb must be a multiple of 16 in [16, 128], or 256, 384 or 512");
        return NL_EINVAL;
    }
    if (gemm == 2 && !tc_gemm_supported()) gemm = 1;
    if (nb > 128) {
        if (fast) return lu16_factor_2lvl(N, A, ld, ipiv, nb, gemm, w, st, launches);
        nb = 128;  // the interchanging path (partial pivoting needs row swaps): one level
    }
    return lu_factor_impl<float, __half, 16, true>(N, A, ld, ipiv, nb, gemm, fast, w, st, launches);
}

nl_status lu64_factor(int N, double* A, int64_t ld, int* ipiv, int nb, bool fast, const LuWork& w, cudaStream_t st,
                      int* launches)
{
    if (nb < 16 || nb > 128 || nb % 16) {
        set_error("lu64: nb must be a multiple of 16 in [16, 128]");
        return NL_EINVAL;
    }
    return lu_factor_impl<double, double, 8, false>(N, A, ld, ipiv, nb, 1, fast, w, st, launches);
}

// The single-precision factorisation of the two-precision F32 Newton method
// (Section 1.3): binary32 storage and arithmetic, always the interchanging
// path (leaf panels with pivot search, row swaps, U12 solve, SIMT update).
nl_status lu32_factor(int N, float* A, int64_t ld, int* ipiv, int nb, const LuWork& w, cudaStream_t st, int* launches)
{
    if (nb < 16 || nb > 128 || nb % 16) {
        set_error("lu32: nb must be a multiple of 16 in [16, 128]");
        return NL_EINVAL;
    }
    return lu_factor_impl<float, float, 16, false>(N, A, ld, ipiv, nb, 1, false, w, st, launches);
}

// ------------------------------------------------ binary16 arithmetic LU --
// Partial-pivot LU with every operation rounded to binary16, the arithmetic
// of the paper's F16 column (Section 1.3): at step k the pivot is the first
// row of largest |a_ik| (i >= k), rows k and p are swapped whole,
// l_ik = fl16(a_ik / a_kk) and a_ij <- fl16(a_ij - fl16(l_ik a_kj)) for
// i, j > k, so every entry takes its updates in increasing k.  One
// cooperative launch, one CTA per SM: a warp updates one row at a time, the
// next column's pivot candidates are formed during the update, and each step
// ends at a bounded grid barrier (one more after a row swap).  The product of
// two binary16 numbers is exact in binary32; the difference and the quotient
// are formed in binary32 and rounded once more, to binary16, which is the
// correctly rounded result (24 >= 2 * 11 + 2).  Matrix reads bypass L1
// (other SMs write the rows between barriers).
constexpr int kHaThreads = 512;
constexpr int kHaWarps = kHaThreads / 32;
constexpr int kHaU = 8;  // row entries per lane per batch of loads

__device__ __forceinline__ float h16r(float v) { return __half2float(__float2half_rn(v)); }

// {|a| bits, ~i}: the largest packed value is the first row of largest |a|.
__device__ __forceinline__ unsigned long long ha_pack(float a, int i)
{
    return ((unsigned long long)__float_as_uint(fabsf(a)) << 32) | (unsigned long long)(~(unsigned)i);
}

__device__ __forceinline__ unsigned long long ha_block_max(unsigned long long v, unsigned long long* red)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
        v = w > v ? w : v;
    }
    __syncthreads();  // red is reused across calls
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    v = 0;
#pragma unroll
    for (int q = 0; q < kHaWarps; ++q) v = red[q] > v ? red[q] : v;
    return v;
}

// Grid barrier over co-resident CTAs: bar[0] counts arrivals, bar[1] is the
// generation (both zero at launch).  Bounded: false after recording a timeout,
// or when another CTA recorded an error.
__device__ bool ha_grid_sync(unsigned* bar, unsigned& gen, unsigned* err)
{
    __shared__ int ok_s;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        __threadfence();
        if (atomicAdd(&bar[0], 1u) == gridDim.x - 1) {
            atomicExch(&bar[0], 0u);
            __threadfence();
            atomicAdd(&bar[1], 1u);
        } else {
            long long spins = 0;
            while ((unsigned)ld_acquire_gpu((const int*)&bar[1]) == gen) {
                if (*(volatile unsigned*)err) {
                    ok = 0;
                    break;
                }
                if (++spins > kSpinLimit) {
                    atomicOr(err, (unsigned)ERR_TIMEOUT_OTHER);
                    ok = 0;
                    break;
                }
                __nanosleep(32);
            }
        }
        ++gen;
        __threadfence();
        ok_s = ok;
    }
    __syncthreads();
    return ok_s != 0;
}

__global__ void __launch_bounds__(kHaThreads, 1) k_lu16_arith(__half* __restrict__ A, int64_t lda, int N,
                                                              int* __restrict__ ipiv, int* __restrict__ info,
                                                              unsigned* __restrict__ bar,
                                                              unsigned long long* __restrict__ cand,
                                                              unsigned* __restrict__ err)
{
    __shared__ unsigned long long red[kHaWarps];
    const int tid = threadIdx.x, lane = tid & 31;
    const int G = gridDim.x;
    const int gw = blockIdx.x * kHaWarps + (tid >> 5), nw = G * kHaWarps;  // this warp, all warps
    unsigned gen = 0;
    // pivot candidates of column 0
    unsigned long long nb = 0;
    if (lane == 0)
        for (int i = gw; i < N; i += nw) {
            const unsigned long long c = ha_pack(__half2float(__ldcg(A + (int64_t)i * lda)), i);
            nb = c > nb ? c : nb;
        }
    nb = ha_block_max(nb, red);
    if (tid == 0) cand[blockIdx.x] = nb;
    if (!ha_grid_sync(bar, gen, err)) return;
    for (int k = 0; k < N; ++k) {
        unsigned long long b = 0;
        for (int g = tid; g < G; g += kHaThreads) {
            const unsigned long long c = __ldcg(cand + (k & 1) * G + g);
            b = c > b ? c : b;
        }
        b = ha_block_max(b, red);
        const int p = (int)(~(unsigned)(b & 0xffffffffull));
        if (blockIdx.x == 0 && tid == 0) ipiv[k] = p;
        if (p != k && p > k && p < N) {  // swap rows k and p whole
            __half* Rk = A + (int64_t)k * lda;
            __half* Rp = A + (int64_t)p * lda;
            for (int j = blockIdx.x * kHaThreads + tid; j < N; j += G * kHaThreads) {
                const __half t = __ldcg(Rk + j);
                Rk[j] = __ldcg(Rp + j);
                Rp[j] = t;
            }
            if (!ha_grid_sync(bar, gen, err)) return;
        }
        const __half* Rk = A + (int64_t)k * lda;
        const float akk = __half2float(__ldcg(Rk + k));
        if (akk == 0.0f && blockIdx.x == 0 && tid == 0) atomicCAS(info, 0, k + 1);
        if (k == N - 1) break;
        nb = 0;
        if (akk == 0.0f) {  // no elimination at this step; the next column's candidates as they stand
            if (lane == 0)
                for (int i = k + 1 + gw; i < N; i += nw) {
                    const unsigned long long c = ha_pack(__half2float(__ldcg(A + (int64_t)i * lda + k + 1)), i);
                    nb = c > nb ? c : nb;
                }
        } else {
            bool inf = false;
            for (int i = k + 1 + gw; i < N; i += nw) {
                __half* Ri = A + (int64_t)i * lda;
                const float l = h16r(__fdiv_rn(__half2float(__ldcg(Ri + k)), akk));
                __syncwarp();  // every lane has read a_ik before lane 0 overwrites it
                if (lane == 0) Ri[k] = __float2half_rn(l);
                // kHaU entries per lane: all loads issued before the stores (the rows may alias
                // as far as the compiler knows), the same operations per entry
                for (int j0 = k + 1; j0 < N; j0 += 32 * kHaU) {
                    __half rk[kHaU], ri[kHaU];
#pragma unroll
                    for (int u = 0; u < kHaU; ++u) {
                        const int j = j0 + u * 32 + lane;
                        rk[u] = j < N ? __ldcg(Rk + j) : __ushort_as_half((unsigned short)0);
                        ri[u] = j < N ? __ldcg(Ri + j) : __ushort_as_half((unsigned short)0);
                    }
#pragma unroll
                    for (int u = 0; u < kHaU; ++u) {
                        const int j = j0 + u * 32 + lane;
                        if (j < N) {
                            const float pr = h16r(l * __half2float(rk[u]));
                            const float v = h16r(__half2float(ri[u]) - pr);
                            Ri[j] = __float2half_rn(v);
                            inf |= isinf(v);
                            if (j == k + 1) {
                                const unsigned long long c = ha_pack(v, i);
                                nb = c > nb ? c : nb;
                            }
                        }
                    }
                }
            }
            if (inf) atomicOr(info + 1, 1);
        }
        nb = ha_block_max(nb, red);
        if (tid == 0) cand[((k + 1) & 1) * G + blockIdx.x] = nb;
        if (!ha_grid_sync(bar, gen, err)) return;
    }
}

nl_status lu16_factor_arith(int N, __half* A, int64_t ld, int* ipiv, const LuWork& w, cudaStream_t st)
{
    static std::atomic<int> grid_cache{0};
    int grid = grid_cache.load();
    if (grid == 0) {
        int per_sm = 0;
        NL_CUDA_OK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_lu16_arith, kHaThreads, 0));
        if (per_sm < 1) {
            set_error("binary16-arithmetic LU: the kernel does not fit on an SM");
            return NL_ECUDA;
        }
        grid = std::min(num_sms(), 128 * 128 / 2);  // one CTA per SM; two candidate rows per CTA fit in pub
        grid_cache.store(grid);
    }
    NL_CUDA_OK(cudaMemsetAsync(w.info, 0, 6 * sizeof(int), st));  // info, overflow, (err), barrier count and generation
    unsigned* err = tc_error_word();
    if (!err) err = (unsigned*)(w.info + 2);
    unsigned* bar = (unsigned*)(w.info + 4);
    int* info = w.info;
    unsigned long long* cand = w.pub;
    int Nv = N;
    int64_t ldv = ld;
    void* args[] = {(void*)&A, (void*)&ldv, (void*)&Nv, (void*)&ipiv, (void*)&info, (void*)&bar, (void*)&cand,
                    (void*)&err};
    NL_CUDA_OK(cudaLaunchCooperativeKernel((const void*)k_lu16_arith, dim3(grid), dim3(kHaThreads), args, 0, st));
    return NL_OK;
}

}  // namespace nl

// ================================================================ grouped ==
// Many independent matrices of different N factored in lock step: outer step
// k launches the diagonal-block kernel for every matrix with N > k nb, the
// off-diagonal solves of all of them, and their trailing updates, each as one
// launch over a precomputed task list (largest matrices first).  The kernels
// are the single-matrix fast-path bodies; a matrix whose flag word is non-zero
// (fast path failed, or marked to be skipped) does no work.  No interchanges:
// a matrix that needs them is left with bit 0 of its flag set.
namespace nl {

size_t lu_stage_bytes() { return (size_t)2 * 128 * 128 * 8 + 128 * 8; }

template <typename T, typename S, bool RND>
__global__ void __launch_bounds__(kDiagThreads, 1) k_diag_lu_g(const GInst* __restrict__ inst,
                                                               const GTask* __restrict__ tasks, int K, int nb)
{
    const GInst I = inst[tasks[blockIdx.x].inst];
    diag_lu_body<T, S, RND>(reinterpret_cast<S*>(I.A), I.ld, K, min(nb, I.N - K), I.ipiv, I.flag, I.stage);
}

// WMAX = 64 (panels of at most 64 columns): half the threads, so two blocks share an SM
template <int WMAX>
__global__ void __launch_bounds__(4 * WMAX, 128 / WMAX) k_diag_lu16_g(const GInst* __restrict__ inst,
                                                                      const GTask* __restrict__ tasks, int K, int nb)
{
    const GInst I = inst[tasks[blockIdx.x].inst];
    diag_lu16_body<false, __half, WMAX, 4 * WMAX>(reinterpret_cast<__half*>(I.A), I.ld, K, min(nb, I.N - K), I.ipiv,
                                                  I.flag, reinterpret_cast<float*>(I.stage));
}

template <typename T, typename S>
__global__ void __launch_bounds__(kOffThreads) k_offdiag_g(const GInst* __restrict__ inst,
                                                           const GTask* __restrict__ tasks, int K, int nb)
{
    const GTask t = tasks[blockIdx.x];
    const GInst I = inst[t.inst];
    offdiag_body<T, S>(reinterpret_cast<S*>(I.A), I.ld, K, nb, I.N, t.b, I.flag, I.stage, t.a);
}

__global__ void __launch_bounds__(kO16Threads) k_offdiag16_g(const GInst* __restrict__ inst,
                                                             const GTask* __restrict__ tasks, int K, int nb, int tc)
{
    const GTask t = tasks[blockIdx.x];
    const GInst I = inst[t.inst];
    offdiag16_body(reinterpret_cast<__half*>(I.A), I.ld, K, nb, I.N, t.b, tc ? I.ut : nullptr, nb, I.flag,
                   reinterpret_cast<const float*>(I.stage), t.a);
}

template <typename S, typename T>
__global__ void __launch_bounds__(256) k_gemm_simt_g(const GInst* __restrict__ inst, const GTask* __restrict__ tasks,
                                                     int K, int w)
{
    const GTask t = tasks[blockIdx.x];
    const GInst I = inst[t.inst];
    const int rest = I.N - K - w;
    S* A = reinterpret_cast<S*>(I.A);
    const int64_t ld = I.ld;
    gemm_simt_body<S, T>(rest, rest, w, A + (int64_t)(K + w) * ld + K, ld, A + (int64_t)K * ld + K + w, ld,
                         A + (int64_t)(K + w) * ld + K + w, ld, I.flag, t.a, t.b);
}

// ------------------------------------------- persistent grouped LU --
// The whole grouped factorisation in one launch: CTAs (one per SM) take tasks
// from a device queue in order (an atomic counter) and each task waits, with
// a bounded poll, for the progress word of its matrix:
//   diag(i, k)      needs phase 3k   (matrix i's update of step k-1 done),
//   offdiag(i, k)   needs phase 3k+1 (its diagonal block factored),
//   update(i, k)    needs phase 3k+2 (all its off-diagonal solves done);
// the last task of each phase advances the word (release).  The queue lists
// step k's diagonal tasks, then its off-diagonal tasks, then its update
// tiles, step by step, so every task's dependencies come earlier in the queue
// and were taken by CTAs that are running: no co-residency is needed and the
// launch can be captured in a graph.  A CTA of 512 threads runs a diagonal
// block (diag_lu16_body), four off-diagonal blocks of one role side by side
// (four groups of 128 threads, each with its own shared region; padding
// groups get blocks past the matrix and store nothing), or one update tile of
// TM x 64 with sequential single-precision fused multiply-adds over k and one
// rounding to binary16: the arithmetic of the three-launch SIMT path, so the
// factors are bitwise those of the single-matrix LU with the SIMT update.
// A matrix whose fast path failed (flag set) skips its work but its tasks
// still advance its progress word; a wait that gives up records the error
// and its CTA skips the work the same way, so nothing waits forever.
constexpr int kPgThreads = 512;
constexpr long long kPgSpin = 1LL << 24;

// A queue entry carries its matrix's pointers (one 80-byte record, fetched
// ahead with cp.async while the previous task runs).
struct alignas(16) PTask {
    void* A;
    int* ipiv;
    int* flag;
    void* stage;
    __half* ut;
    int ld, N;
    int inst, kind, step, a, b, n;  // kind 0 diag; 1 off-diagonal quad (a first block, b blocks in it,
                                    // n = 1 row role / 0 column role); 2 update tile (a = m0, b = n0)
};
static_assert(sizeof(PTask) == 80, "queue entries are five 16-byte chunks");

// progress word: the phase reached, with kPgFail once the matrix's flag is set
// (folded in by the task that completes each phase, so a waiting task learns
// both from its one acquire load)
constexpr int kPgFail = 1 << 30;

// Polls before a wait gives up: 0 = kPgSpin; negative = give up at the first
// unmet poll (a test of the timeout path that needs no fault: a wait that runs
// out whatever the producers do).
__device__ long long g_pg_spin_limit = 0;

__device__ __forceinline__ bool pg_wait(const int* p, int need, unsigned* err, int* val)
{
    long long it = 0;
    int v;
    const long long lim = g_pg_spin_limit;
    const long long limit = lim == 0 ? kPgSpin : (lim < 0 ? 0 : lim);
    while (((v = ld_acquire_gpu(p)) & ~kPgFail) < need) {
        if (*(volatile unsigned*)err) return false;
        if (++it > limit) {
            atomicOr(err, (unsigned)ERR_TIMEOUT_OTHER);
            return false;
        }
        __nanosleep(64);
    }
    *val = v;
    return true;
}

__device__ __forceinline__ int atom_add_acq_rel_gpu(int* p, int v)
{
    int old;
    asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}

// thread 0: queue entry t (if any) into a shared slot, asynchronously
__device__ __forceinline__ void pg_fetch(const PTask* tasks, int t, int ntasks, PTask* slot)
{
    if (t < ntasks) {
        const char* src = reinterpret_cast<const char*>(tasks + t);
        const uint32_t dst = smem_u32(slot);
#pragma unroll
        for (int q = 0; q < 5; ++q)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16 * q), "l"(src + 16 * q) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// C[m0.., n0..] (TM x 64) <- fl16(C - A B) over K, 512 threads: thread (ty, tx) =
// (tid / 16, tid % 16) owns rows ty + 32 a and columns tx + 16 b; every entry takes
// its K products in increasing k, one fused multiply-add each.  The operands are
// written by other CTAs of the same launch, so they are read through plain
// (coherent) loads, never the read-only path.
template <int TM>
__device__ __forceinline__ void pg_gemm_tile(int M, int Nc, int K, const __half* A, int64_t lda, const __half* B,
                                             int64_t ldb, __half* C, int64_t ldc, int m0, int n0, float* sm)
{
    constexpr int BK = 16, RA = TM / 32;
    float* As = sm;                    // [BK][TM + 1]
    float* Bs = sm + BK * (TM + 1);    // [BK][64]
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    float acc[RA][4];
#pragma unroll
    for (int a = 0; a < RA; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int i = m0 + ty + 32 * a, j = n0 + tx + 16 * b;
            acc[a][b] = (i < M && j < Nc) ? __half2float(C[(int64_t)i * ldc + j]) : 0.0f;
        }
    for (int k0 = 0; k0 < K; k0 += BK) {
        __syncthreads();
        for (int q = tid; q < TM * BK; q += kPgThreads) {
            const int r = q / BK, kk = q % BK, i = m0 + r, k = k0 + kk;
            As[kk * (TM + 1) + r] = (i < M && k < K) ? __half2float(A[(int64_t)i * lda + k]) : 0.0f;
        }
        for (int q = tid; q < BK * 64; q += kPgThreads) {
            const int kk = q / 64, x = q % 64, k = k0 + kk, j = n0 + x;
            Bs[kk * 64 + x] = (k < K && j < Nc) ? __half2float(B[(int64_t)k * ldb + j]) : 0.0f;
        }
        __syncthreads();
        const int kmax = min(BK, K - k0);
        for (int kk = 0; kk < kmax; ++kk) {
            float av[RA], bv[4];
#pragma unroll
            for (int a = 0; a < RA; ++a) av[a] = As[kk * (TM + 1) + ty + 32 * a];
#pragma unroll
            for (int b = 0; b < 4; ++b) bv[b] = Bs[kk * 64 + tx + 16 * b];
#pragma unroll
            for (int a = 0; a < RA; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[a][b] = fmaf(-av[a], bv[b], acc[a][b]);
        }
    }
#pragma unroll
    for (int a = 0; a < RA; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int i = m0 + ty + 32 * a, j = n0 + tx + 16 * b;
            if (i < M && j < Nc) C[(int64_t)i * ldc + j] = __float2half_rn(acc[a][b]);
        }
}

constexpr long long kPgTcWait = 2000000000LL;  // cycles: bounded mbarrier waits of the tcgen05 tiles

// One 128 x 128 update tile on the tensor cores (TC kernels): thread 0 loads the
// 64-wide A slab (L21 rows, through the matrix's tensor map) and B slab (U12^T
// rows, through its U12^T map) with TMA, issues the four K = 16 tcgen05.mma of
// the slab into the CTA's 128-column TMEM accumulator and commits them; each of
// the 16 warps then reads its 32 lanes x 32 columns (warp w: lanes 32 (w % 4),
// columns 32 (w / 4)) and writes C = fl16(C - acc).  The per-element arithmetic
// is the trailing-update kernels' (same MMAs in the same order, one
// subtraction, one rounding).  `uses` counts the tiles issued by this CTA (the
// mbarrier phases); a wait that gives up marks the CTA dead: its later tiles
// store nothing and it never touches its barriers again.
__device__ __forceinline__ void pg_tc_tile(__half* A, int64_t ld, const TmapBytes* __restrict__ maps, int inst, int K, int w,
                                           int rest, int m0, int n0, bool run, uint32_t tmem, uint32_t& uses,
                                           uint64_t* tbar, int* dead, float* pgsm, unsigned* err)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t raw = smem_u32(pgsm), base = (raw + 1023u) & ~1023u;
    const uint32_t sA = base, sB = base + 128 * 128;
    const uint32_t bl = smem_u32(&tbar[0]), bm = smem_u32(&tbar[1]);
    const uint32_t ph = uses & 1u;
    // this CTA's earlier generic writes to the shared region, before the TMA writes into it
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    run = run && !*(volatile int*)dead;  // CTA-uniform: written by thread 0 only, read after a barrier
    if (run && threadIdx.x == 0) {
        const CUtensorMap* ma = reinterpret_cast<const CUtensorMap*>(&maps[2 * inst]);
        const CUtensorMap* mb = reinterpret_cast<const CUtensorMap*>(&maps[2 * inst + 1]);
        asm volatile("fence.proxy.async.global;" ::: "memory");  // the acquired operands, for the async proxy
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bl), "r"(2u * 128 * 128)
                     : "memory");
        tma_load_2d(sA, ma, K, K + w + m0, bl);
        tma_load_2d(sB, mb, 0, n0, bl);
        if (!mbar_wait(bl, ph, kPgTcWait)) {
            atomicOr(err, (unsigned)ERR_TIMEOUT_OTHER);
            *(volatile int*)dead = 1;
            mbar_wait(bl, ph, kPgTcWait);  // let copies in flight land
        } else {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            constexpr uint32_t idesc = tc_idesc_mn(128, 128);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                const uint64_t ad = sw128_desc(sA + kk * 32), bd = sw128_desc(sB + kk * 32);
                const uint32_t acc = kk ? 1u : 0u;
                asm volatile(
                    "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                    " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
                    "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bm)
                         : "memory");
        }
    }
    // the epilogue's C segment does not depend on the MMAs: load it while they run
    const int q = warp & 3, cg = warp >> 2;
    const int row = m0 + q * 32 + lane, col0 = n0 + cg * 32;
    __half* Crow = A + (int64_t)(K + w + min(row, rest - 1)) * ld + K + w;
    const bool full = run && row < rest && col0 + 32 <= rest;
    uint4 cpre[4];
    if (full) {
        const uint4* p = reinterpret_cast<const uint4*>(Crow + col0);
#pragma unroll
        for (int v = 0; v < 4; ++v) cpre[v] = p[v];
    }
    __syncthreads();
    bool good = run && !*(volatile int*)dead;  // CTA-uniform (a failed load wait set it)
    const bool waited = good ? mbar_wait(bm, ph, kPgTcWait) : true;
    if (__syncthreads_or(!waited)) {
        if (threadIdx.x == 0) {
            atomicOr(err, (unsigned)ERR_TIMEOUT_OTHER);
            *(volatile int*)dead = 1;
            mbar_wait(bm, ph, kPgTcWait);  // let the MMAs in flight finish
        }
        good = false;
    }
    if (run) uses += 1;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (good) {
        uint32_t r[32];
        const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(cg * 32);
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
            "%14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
              "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
              "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]),
              "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]),
              "=r"(r[30]), "=r"(r[31])
            : "r"(taddr));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (full) {
            uint4* p = reinterpret_cast<uint4*>(Crow + col0);
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                uint32_t wds[4] = {cpre[v].x, cpre[v].y, cpre[v].z, cpre[v].w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    __half2 h2;
                    memcpy(&h2, &wds[e], 4);
                    float2 f = __half22float2(h2);
                    f.x -= __uint_as_float(r[v * 8 + 2 * e]);
                    f.y -= __uint_as_float(r[v * 8 + 2 * e + 1]);
                    h2 = __floats2half2_rn(f.x, f.y);
                    memcpy(&wds[e], &h2, 4);
                }
                p[v] = make_uint4(wds[0], wds[1], wds[2], wds[3]);
            }
        } else if (run && row < rest) {
#pragma unroll
            for (int e = 0; e < 32; ++e)
                if (col0 + e < rest)
                    Crow[col0 + e] = __float2half_rn(__half2float(Crow[col0 + e]) - __uint_as_float(r[e]));
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}

// ctl: [0] the queue's next task, [1 .. count] progress words, [1 + count .. 1 + 2 count)
// per-matrix task counters (set by k_pg_init before each launch).  TC: update tiles of
// 128 x 128 on the tensor cores (nb = 64, U12^T written by the column-role solves,
// tensor maps in `maps`); otherwise tm x 64 SIMT tiles.  Thread 0 takes the next queue
// index while it waits for the current task's dependencies and fetches that entry with
// cp.async while the task runs; a phase is handed on with an acquire-release count and
// a release store of the progress word.
template <bool TC>
__global__ void __launch_bounds__(kPgThreads, 1) k_lu_grouped_p(const PTask* __restrict__ tasks, int ntasks, int nb,
                                                                int tm, int tn, const TmapBytes* __restrict__ maps,
                                                                int* __restrict__ ctl, int count,
                                                                unsigned* __restrict__ err,
                                                                unsigned long long* __restrict__ tstat)
{
    extern __shared__ __align__(16) float pgsm[];
    __shared__ PTask qbuf[2];
    __shared__ int qidx[2], go, dead;
    __shared__ __align__(8) uint64_t tbar[2];  // TC: operands landed, MMAs done
    __shared__ uint32_t tslot;
    int* next = ctl;
    int* prog = ctl + 1;
    int* cnt = ctl + 1 + count;
    uint32_t tmem = 0, uses = 0;
    if constexpr (TC) {
        if ((threadIdx.x >> 5) == 0) {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tslot)),
                         "r"(128u));
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
        }
        if (threadIdx.x == 32) {
            dead = 0;
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&tbar[0])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&tbar[1])));
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        tmem = tslot;
    }
    if (threadIdx.x == 0) {
        const int t0 = atomicAdd(next, 1);
        qidx[0] = t0;
        pg_fetch(tasks, t0, ntasks, &qbuf[0]);
        asm volatile("cp.async.wait_all;" ::: "memory");
    }
    int slot = 0;
    for (;;) {
        __syncthreads();
        const int t = qidx[slot];
        if (t >= ntasks) break;
        const PTask& T = qbuf[slot];  // stays put while the task runs (the prefetch fills the other slot)
        const int K = T.step * nb, w = min(nb, T.N - K), rest = T.N - K - w;
        __half* A = reinterpret_cast<__half*>(T.A);
        long long c0 = 0, c1 = 0;  // task timing (tstat): start, dependencies met
        if (threadIdx.x == 0) {
            c0 = clock64();
            const int tnext = atomicAdd(next, 1);  // its latency overlaps the wait below
            int v = 0;
            const bool ok = pg_wait(&prog[T.inst], 3 * T.step + T.kind, err, &v);
            c1 = clock64();
            go = (ok && !(v & kPgFail)) ? 1 : 0;
            qidx[slot ^ 1] = tnext;
            pg_fetch(tasks, tnext, ntasks, &qbuf[slot ^ 1]);  // lands while this task runs
        }
        __syncthreads();
        int* done_word = nullptr;  // thread 0: the counter this task adds to, and by how much
        int add = 0, total = 0, phase = 0;
        if (T.kind == 0) {
            if (go) diag_lu16_body<false, __half>(A, T.ld, K, w, T.ipiv, T.flag, reinterpret_cast<float*>(T.stage));
            phase = rest > 0 ? 3 * T.step + 1 : 3 * T.step + 3;
        } else if (T.kind == 1) {
            const int wp = (w + 31) & ~31;
            const int q = threadIdx.x >> 7, b = T.a + q;
            const int fl = (int)(offdiag16_smem(wp) / sizeof(float));
            if (go)
                offdiag16_body<__half>(A, T.ld, K, w, T.N, T.n ? (1 << 20) : 0, TC ? T.ut : nullptr, nb, T.flag,
                                       reinterpret_cast<const float*>(T.stage), b, -1, 0, threadIdx.x & 127,
                                       pgsm + q * fl);
            done_word = &cnt[T.inst];
            add = T.b;
            total = 2 * ((rest + kO16Rows - 1) / kO16Rows);
            phase = 3 * T.step + 2;
        } else {
            if constexpr (TC) {
                pg_tc_tile(A, T.ld, maps, T.inst, K, w, rest, T.a, T.b, go != 0, tmem, uses, tbar, &dead, pgsm, err);
            } else if (go) {
                const __half* L21 = A + (int64_t)(K + w) * T.ld + K;
                const __half* U12 = A + (int64_t)K * T.ld + K + w;
                __half* C = A + (int64_t)(K + w) * T.ld + K + w;
                if (tm == 128) pg_gemm_tile<128>(rest, rest, w, L21, T.ld, U12, T.ld, C, T.ld, T.a, T.b, pgsm);
                else pg_gemm_tile<64>(rest, rest, w, L21, T.ld, U12, T.ld, C, T.ld, T.a, T.b, pgsm);
            }
            done_word = &cnt[T.inst];
            add = 1;
            total = ((rest + tm - 1) / tm) * ((rest + tn - 1) / tn);
            phase = 3 * T.step + 3;
        }
        // TC: the off-diagonal solves' generic writes (L21 rows and U12^T, the tiles' TMA
        // operands) ordered before the TMA reads of them; the diagonal blocks and the
        // tiles' C are read by generic loads only
        if constexpr (TC)
            if (T.kind == 1) asm volatile("fence.proxy.async.global;" ::: "memory");
        if (threadIdx.x == 0) asm volatile("cp.async.wait_all;" ::: "memory");  // the next entry has landed
        __syncthreads();
        if (threadIdx.x == 0) {
            // the CTA's writes are ordered before thread 0's release by the barrier
            bool last = true;
            if (done_word) {
                last = atom_add_acq_rel_gpu(done_word, add) + add == total;
                if (last) *done_word = 0;
            }
            if (last) st_release_gpu(&prog[T.inst], phase | (*(volatile const int*)T.flag ? kPgFail : 0));
            if (tstat) {  // per kind: tasks, cycles waiting for dependencies, cycles working
                const long long c2 = clock64();
                atomicAdd(&tstat[3 * T.kind], 1ull);
                atomicAdd(&tstat[3 * T.kind + 1], (unsigned long long)(c1 - c0));
                atomicAdd(&tstat[3 * T.kind + 2], (unsigned long long)(c2 - c1));
            }
        }
        slot ^= 1;
    }
    if constexpr (TC) {
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        if ((threadIdx.x >> 5) == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(128u));
        }
    }
}

// Per-task timing of the persistent launch (off unless switched on): per task
// kind, the tasks run, the cycles spent waiting for their dependencies and the
// cycles spent on them (thread 0's clock64 from dependencies met to hand-off).
__device__ unsigned long long g_pg_tstat[9];
static std::atomic<bool> g_pg_tstat_on{false};

static unsigned long long* pg_task_stats_ptr()
{
    if (!g_pg_tstat_on.load()) return nullptr;
    void* p = nullptr;
    return cudaGetSymbolAddress(&p, g_pg_tstat) == cudaSuccess ? static_cast<unsigned long long*>(p) : nullptr;
}

// Before each launch: the queue counter and task counters zeroed, each progress
// word 0 with kPgFail for a matrix whose flag is already set (skipped).
__global__ void k_pg_init(int* __restrict__ ctl, int count, const GInst* __restrict__ inst)
{
    for (int i = threadIdx.x; i < 1 + 2 * count; i += blockDim.x) {
        int v = 0;
        if (i >= 1 && i <= count && *(volatile const int*)inst[i - 1].flag) v = kPgFail;
        ctl[i] = v;
    }
}

static size_t pg_smem_bytes(int nb)
{
    const int wp = (int)round_up(nb, 32);
    size_t b = std::max<size_t>(kDiag16Smem, 4 * offdiag16_smem(wp));
    b = std::max<size_t>(b, (size_t)(16 * (128 + 1) + 16 * 64) * sizeof(float));
    b = std::max<size_t>(b, 1024 + 2 * 128 * 128);  // the tcgen05 tile's A and B slabs, 1024-byte aligned
    return b;
}

// The persistent launch's queue order: a list schedule simulated on the host
// with a cost model (microseconds per task on one CTA).  `workers` CTAs; the
// tasks of a matrix's next phase become ready when its current phase is done
// (diagonal block -> off-diagonal quads -> update tiles -> next diagonal
// block); a free CTA takes the ready task whose matrix has the most outer
// steps left (the longest remaining chain), a diagonal block before quads
// before tiles, then in generation order.  The queue lists the tasks by
// simulated start, so every task's dependencies come earlier in it, and the
// long chains of the largest matrices advance while the others fill the gaps.
static std::vector<PTask> lu_grouped_schedule(int count, const GInst* host_inst, int nb, int tm, int tn, bool tc,
                                              int workers)
{
    struct Ready {
        int rem, kind;
        long long seq;
        PTask t;
        bool operator<(const Ready& o) const  // max-heap: most steps left, then kind, then earliest
        {
            if (rem != o.rem) return rem < o.rem;
            if (kind != o.kind) return kind > o.kind;
            return seq > o.seq;
        }
    };
    struct Busy {
        double end;
        int inst;
        bool operator<(const Busy& o) const { return end > o.end; }  // min-heap on finish time
    };
    std::vector<int> steps(count), step(count, 0), left(count, 0);
    std::priority_queue<Ready> ready;
    std::priority_queue<Busy> busy;
    long long seq = 0;
    size_t total = 0;
    for (int i = 0; i < count; ++i) steps[i] = (int)cdiv(host_inst[i].N, nb);
    // per-task times measured on a GB300 for w = 64 (clock64 around each task of the
    // 512-instance workload): diagonal block ~30 us, off-diagonal quad ~25 us, tile
    // ~6 us (tcgen05 128 x 128), ~15 us (SIMT 128 x 64), ~8 us (SIMT 64 x 64)
    auto dur = [&](int kind, int w) {
        const double f = (double)w / 64.0;
        if (kind == 0) return 0.47 * w;
        if (kind == 1) return 3.0 + 22.0 * f * f;
        return tc ? 6.0 : (tm == 128 ? 15.0 : 8.0) * f;
    };
    std::vector<double> tdur;  // per generated task, indexed by its seq
    auto mk = [&](int i, int kind, int k, int a, int b, int n) {
        const GInst& G = host_inst[i];
        PTask t;
        t.A = G.A;
        t.ipiv = G.ipiv;
        t.flag = G.flag;
        t.stage = G.stage;
        t.ut = G.ut;
        t.ld = (int)G.ld;
        t.N = G.N;
        t.inst = i;
        t.kind = kind;
        t.step = k;
        t.a = a;
        t.b = b;
        t.n = n;
        return t;
    };
    // phase `kind` of matrix i's current step becomes ready
    auto release = [&](int i, int kind) {
        const int k = step[i], K = k * nb, w = std::min(nb, host_inst[i].N - K), rest = host_inst[i].N - K - w;
        const int rem = steps[i] - k;
        auto push = [&](PTask t) {
            ready.push({rem, kind, seq++, t});
            tdur.push_back(dur(kind, w));
            left[i] += 1;
            total += 1;
        };
        if (kind == 0) {
            push(mk(i, 0, k, 0, 0, 0));
        } else if (kind == 1) {
            const int nblk = (int)cdiv(rest, kO16Rows);
            for (int role = 1; role >= 0; --role)
                for (int a = 0; a < nblk; a += 4) push(mk(i, 1, k, a, std::min(4, nblk - a), role));
        } else {
            for (int m0 = 0; m0 < rest; m0 += tm)
                for (int n0 = 0; n0 < rest; n0 += tn) push(mk(i, 2, k, m0, n0, 0));
        }
    };
    for (int i = 0; i < count; ++i) release(i, 0);
    std::vector<PTask> q;
    double t = 0.0;
    int idle = std::max(1, workers);
    while (!ready.empty() || !busy.empty()) {
        while (idle > 0 && !ready.empty()) {
            const Ready r = ready.top();
            ready.pop();
            q.push_back(r.t);
            busy.push({t + tdur[(size_t)r.seq], r.t.inst + count * r.t.kind});
            idle -= 1;
        }
        if (busy.empty()) break;
        const Busy b = busy.top();
        busy.pop();
        t = b.end;
        idle += 1;
        const int i = b.inst % count, kind = b.inst / count;
        if (--left[i] > 0) continue;
        // matrix i's phase `kind` is done
        const int K = step[i] * nb, rest = host_inst[i].N - K - std::min(nb, host_inst[i].N - K);
        if (kind == 0) {
            if (rest > 0) release(i, 1);
        } else if (kind == 1) {
            release(i, 2);
        } else {
            step[i] += 1;
            release(i, 0);
        }
    }
    return q;
}

// The persistent launch's queue (see lu_grouped_schedule).
static nl_status lu_grouped_plan_p(int count, const GInst* host_inst, int nb, int gemm, int tm, GroupPlan* plan)
{
    const int tn = gemm == 2 ? 128 : 64;
    if (gemm == 2) tm = 128;
    int nmax = 0;
    for (int i = 0; i < count; ++i) nmax = std::max(nmax, host_inst[i].N);
    const int steps = (int)cdiv(nmax, nb);
    const int workers = num_sms();
    std::vector<PTask> q = lu_grouped_schedule(count, host_inst, nb, tm, tn, gemm == 2, workers);
    lu_grouped_free(plan);
    plan->count = count;
    plan->nb = nb;
    plan->gemm = gemm;
    plan->steps = steps;
    plan->fp64 = false;
    plan->kind = 1;
    plan->tm = tm;
    plan->tn = tn;
    plan->off.clear();
    plan->n.clear();
    plan->nptasks = (int)q.size();
    plan->grid = std::max(1, std::min(plan->nptasks, num_sms()));
    std::vector<TmapBytes> maps;
    if (gemm == 2) {
        maps.resize(2 * (size_t)count);
        for (int i = 0; i < count; ++i)
            if (host_inst[i].N > nb && !tc_encode_instance_maps(reinterpret_cast<const __half*>(host_inst[i].A),
                                                                host_inst[i].N, host_inst[i].ld, host_inst[i].ut, nb,
                                                                &maps[2 * (size_t)i])) {
                set_error("grouped LU: tensor-map encoding failed for matrix %d", i);
                return NL_ECUDA;
            }
    }
    const size_t qb = q.size() * sizeof(PTask), cb = (size_t)(1 + 2 * count) * sizeof(int);
    const size_t mb = maps.size() * sizeof(TmapBytes);
    plan->bytes = round_up(qb, 256) + round_up(cb, 256) + mb;
    void* p = nullptr;
    NL_CUDA_OK(trim_malloc(&p, plan->bytes));
    plan->tasks = reinterpret_cast<GTask*>(p);  // the allocation's base (freed through it)
    plan->ptasks = reinterpret_cast<PTask*>(p);
    plan->ctl = reinterpret_cast<int*>((char*)p + round_up(qb, 256));
    plan->maps = mb ? reinterpret_cast<TmapBytes*>((char*)p + round_up(qb, 256) + round_up(cb, 256)) : nullptr;
    if (qb) NL_CUDA_OK(cudaMemcpy(plan->ptasks, q.data(), qb, cudaMemcpyHostToDevice));
    if (mb) NL_CUDA_OK(cudaMemcpy(plan->maps, maps.data(), mb, cudaMemcpyHostToDevice));
    return NL_OK;
}

nl_status lu_grouped_plan(int count, const GInst* host_inst, int nb, int gemm, bool fp64, GroupPlan* plan, int kind,
                          int tm)
{
    if (count < 1 || nb < 16 || nb > 128 || nb % 16) {
        set_error("grouped LU: need count >= 1 and nb a multiple of 16 in [16, 128]");
        return NL_EINVAL;
    }
    if (kind == 1) {
        if (fp64 || !(gemm == 1 || gemm == 2) || nb > 64 || (gemm == 2 && nb != 64) || !(tm == 64 || tm == 128) ||
            !tc_gemm_supported() || !tc_error_word()) {
            set_error("grouped LU: the persistent launch needs the binary16 LU, nb <= 64 (nb = 64 with the "
                      "tensor-core update), SIMT tile height 64 or 128");
            return NL_EINVAL;
        }
        return lu_grouped_plan_p(count, host_inst, nb, gemm, tm, plan);
    }
    if (kind != 0) {
        set_error("grouped LU: unknown kind %d", kind);
        return NL_EINVAL;
    }
    if (fp64) gemm = 1;
    if (gemm == 2 && (nb % 64 || !tc_gemm_supported())) gemm = 1;
    int nmax = 0;
    for (int i = 0; i < count; ++i) nmax = std::max(nmax, host_inst[i].N);
    // largest matrices first in every task list
    std::vector<int> order(count);
    for (int i = 0; i < count; ++i) order[i] = i;
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return host_inst[a].N > host_inst[b].N; });
    const int steps = (int)cdiv(nmax, nb);
    const int rows_per_cta = fp64 ? kOffLines : kO16Rows;
    const int tile = (gemm == 2) ? 128 : 64;
    std::vector<GTask> tasks;
    plan->off.assign(3 * steps, 0);
    plan->n.assign(3 * steps, 0);
    for (int k = 0; k < steps; ++k) {
        const int K = k * nb;
        plan->off[3 * k] = (int)tasks.size();
        for (int i : order)
            if (host_inst[i].N > K) tasks.push_back({i, 0, 0, 0});
        plan->n[3 * k] = (int)tasks.size() - plan->off[3 * k];
        plan->off[3 * k + 1] = (int)tasks.size();
        for (int i : order) {
            const int rest = host_inst[i].N - K - nb;
            if (rest <= 0) continue;
            const int nrb = (int)cdiv(rest, rows_per_cta);
            for (int b = 0; b < 2 * nrb; ++b) tasks.push_back({i, b, nrb, 0});
        }
        plan->n[3 * k + 1] = (int)tasks.size() - plan->off[3 * k + 1];
        plan->off[3 * k + 2] = (int)tasks.size();
        for (int i : order) {
            const int rest = host_inst[i].N - K - nb;
            if (rest <= 0) continue;
            const int nt = (int)cdiv(rest, tile);
            for (int a = 0; a < nt; ++a)
                for (int b = 0; b < nt; ++b) tasks.push_back({i, a * tile, b * tile, 0});
        }
        plan->n[3 * k + 2] = (int)tasks.size() - plan->off[3 * k + 2];
    }
    lu_grouped_free(plan);
    plan->count = count;
    plan->nb = nb;
    plan->gemm = gemm;
    plan->steps = steps;
    plan->fp64 = fp64;
    std::vector<TmapBytes> maps;
    if (gemm == 2) {
        maps.resize(2 * (size_t)count);
        for (int i = 0; i < count; ++i)
            if (host_inst[i].N > nb && !tc_encode_instance_maps(reinterpret_cast<const __half*>(host_inst[i].A), host_inst[i].N,
                                         host_inst[i].ld, host_inst[i].ut, nb, &maps[2 * (size_t)i])) {
                set_error("grouped LU: tensor-map encoding failed for matrix %d", i);
                return NL_ECUDA;
            }
    }
    const size_t tb = tasks.size() * sizeof(GTask), mb = maps.size() * sizeof(TmapBytes);
    plan->bytes = round_up(tb, 256) + mb + 256;
    void* p = nullptr;
    NL_CUDA_OK(trim_malloc(&p, plan->bytes));
    plan->tasks = reinterpret_cast<GTask*>(p);
    plan->maps = mb ? reinterpret_cast<TmapBytes*>((char*)p + round_up(tb, 256)) : nullptr;
    if (tb) NL_CUDA_OK(cudaMemcpy(plan->tasks, tasks.data(), tb, cudaMemcpyHostToDevice));
    if (mb) NL_CUDA_OK(cudaMemcpy(plan->maps, maps.data(), mb, cudaMemcpyHostToDevice));
    return NL_OK;
}

void lu_grouped_free(GroupPlan* plan)
{
    if (plan->tasks) cudaFree(plan->tasks);
    plan->tasks = nullptr;
    plan->maps = nullptr;
    plan->ptasks = nullptr;
    plan->ctl = nullptr;
    plan->nptasks = 0;
    plan->kind = 0;
}

nl_status lu_grouped_setup()
{
    static bool smem_set = false;
    if (!smem_set) {
        if (set_max_dynamic_smem((const void*)k_diag_lu16_g<64>) != NL_OK ||
            set_max_dynamic_smem((const void*)k_diag_lu16_g<128>) != NL_OK ||
            set_max_dynamic_smem((const void*)k_offdiag16_g) != NL_OK ||
            set_max_dynamic_smem((const void*)k_diag_lu_g<double, double, false>) != NL_OK ||
            set_max_dynamic_smem((const void*)k_offdiag_g<double, double>) != NL_OK ||
            set_max_dynamic_smem((const void*)k_lu_grouped_p<false>) != NL_OK ||
            set_max_dynamic_smem((const void*)k_lu_grouped_p<true>) != NL_OK)
            return NL_ECUDA;
        smem_set = true;
    }
    return NL_OK;
}

nl_status lu_grouped_factor(const GroupPlan& plan, const GInst* dev_inst, cudaStream_t st, int* launches)
{
    NL_TRY(lu_grouped_setup());
    const int nb = plan.nb, wp = (int)round_up(nb, 32);
    if (plan.kind == 1) {
        k_pg_init<<<1, 256, 0, st>>>(plan.ctl, plan.count, dev_inst);  // a kernel node: legal in conditional bodies
        prof_begin("k_lu_grouped_p", st);
        unsigned long long* ts = pg_task_stats_ptr();
        if (plan.gemm == 2)
            k_lu_grouped_p<true><<<plan.grid, kPgThreads, pg_smem_bytes(nb), st>>>(
                plan.ptasks, plan.nptasks, nb, plan.tm, plan.tn, plan.maps, plan.ctl, plan.count, tc_error_word(),
                ts);
        else
            k_lu_grouped_p<false><<<plan.grid, kPgThreads, pg_smem_bytes(nb), st>>>(
                plan.ptasks, plan.nptasks, nb, plan.tm, plan.tn, nullptr, plan.ctl, plan.count, tc_error_word(),
                ts);
        prof_end("k_lu_grouped_p", st);
        NL_CUDA_OK(cudaGetLastError());
        if (launches) *launches += 2;
        return NL_OK;
    }
    int nl = 0;
    for (int k = 0; k < plan.steps; ++k) {
        const int K = k * nb;
        const GTask* td = plan.tasks + plan.off[3 * k];
        const GTask* to = plan.tasks + plan.off[3 * k + 1];
        const GTask* tg = plan.tasks + plan.off[3 * k + 2];
        const int nd = plan.n[3 * k], no = plan.n[3 * k + 1], ng = plan.n[3 * k + 2];
        if (plan.fp64) {
            if (nd) {
                prof_begin("k_diag_lu", st);
                k_diag_lu_g<double, double, false><<<nd, kDiagThreads, (size_t)wp * (wp + 1) * 8, st>>>(dev_inst, td,
                                                                                                      K, nb);
                prof_end("k_diag_lu", st);
            }
            if (no) {
                prof_begin("k_offdiag", st);
                k_offdiag_g<double, double><<<no, kOffThreads, offdiag_smem(wp, 8), st>>>(dev_inst, to, K, nb);
                prof_end("k_offdiag", st);
            }
            if (ng) k_gemm_simt_g<double, double><<<ng, 256, 0, st>>>(dev_inst, tg, K, nb);
        } else {
            if (nd) {
                prof_begin("k_diag_lu16", st);
                if (nb <= 64) k_diag_lu16_g<64><<<nd, 256, Diag16<64>::smem, st>>>(dev_inst, td, K, nb);
                else k_diag_lu16_g<128><<<nd, 512, Diag16<128>::smem, st>>>(dev_inst, td, K, nb);
                prof_end("k_diag_lu16", st);
            }
            if (no) {
                prof_begin("k_offdiag16", st);
                k_offdiag16_g<<<no, kO16Threads, offdiag16_smem(wp), st>>>(dev_inst, to, K, nb, plan.gemm == 2);
                prof_end("k_offdiag16", st);
            }
            if (ng) {
                if (plan.gemm == 2) {
                    nl_status s = tc_gemm16_grouped(dev_inst, plan.maps, tg, ng, K, nb, st);
                    if (s != NL_OK) return s;
                } else {
                    k_gemm_simt_g<__half, float><<<ng, 256, 0, st>>>(dev_inst, tg, K, nb);
                }
            }
        }
        nl += (nd > 0) + (no > 0) + (ng > 0);
        NL_CUDA_OK(cudaGetLastError());
    }
    if (launches) *launches += nl;
    return NL_OK;
}

// The multiplier rounding of the binary16 LU, elementwise (for tests).
__global__ void k_div_round16(int64_t n, const float* __restrict__ a, const float* __restrict__ b,
                              float* __restrict__ out)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = div_round_h(a[i], b[i]);
}

// The quotients of the double-precision off-diagonal solves and inverses, elementwise (for tests).
__global__ void k_div64(int64_t n, const double* __restrict__ a, const double* __restrict__ b, double* __restrict__ out)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = div_by(a[i], b[i], rcp_in_range(b[i]));
}

}  // namespace nl

extern "C" nl_status nl_k_div_round16(int64_t n, const float* a, const float* b, float* out, void* stream)
{
    using namespace nl;
    if (n < 0 || (n > 0 && (!a || !b || !out))) {
        set_error("nl_k_div_round16: bad argument");
        return NL_EINVAL;
    }
    if (n == 0) return NL_OK;
    k_div_round16<<<(unsigned)cdiv(n, 256), 256, 0, (cudaStream_t)stream>>>(n, a, b, out);
    NL_CUDA_OK(cudaGetLastError());
    return NL_OK;
}

extern "C" nl_status nl_k_div64(int64_t n, const double* a, const double* b, double* out, void* stream)
{
    using namespace nl;
    if (n < 0 || (n > 0 && (!a || !b || !out))) {
        set_error("nl_k_div64: bad argument");
        return NL_EINVAL;
    }
    if (n == 0) return NL_OK;
    k_div64<<<(unsigned)cdiv(n, 256), 256, 0, (cudaStream_t)stream>>>(n, a, b, out);
    NL_CUDA_OK(cudaGetLastError());
    return NL_OK;
}

extern "C" nl_status nl_debug_grouped_task_times(int enable, double* out9)
{
    using namespace nl;
    unsigned long long v[9] = {};
    NL_CUDA_OK(cudaDeviceSynchronize());
    NL_CUDA_OK(cudaMemcpyFromSymbol(v, g_pg_tstat, sizeof(v)));
    const unsigned long long z[9] = {};
    NL_CUDA_OK(cudaMemcpyToSymbol(g_pg_tstat, z, sizeof(z)));
    int dev = 0, khz = 0;
    NL_CUDA_OK(cudaGetDevice(&dev));
    NL_CUDA_OK(cudaDeviceGetAttribute(&khz, cudaDevAttrClockRate, dev));
    if (out9)
        for (int k = 0; k < 3; ++k) {
            out9[3 * k] = (double)v[3 * k];
            out9[3 * k + 1] = khz > 0 ? (double)v[3 * k + 1] / (khz * 1e-3) : 0.0;  // cycles -> microseconds
            out9[3 * k + 2] = khz > 0 ? (double)v[3 * k + 2] / (khz * 1e-3) : 0.0;
        }
    g_pg_tstat_on.store(enable != 0);
    return NL_OK;
}

extern "C" nl_status nl_debug_grouped_wait_limit(long long polls)
{
    using namespace nl;
    NL_CUDA_OK(cudaMemcpyToSymbol(g_pg_spin_limit, &polls, sizeof(polls)));
    return NL_OK;
}
