// fft.cu — the residual of eq. (3.2) in O(N log N) with a fast Fourier
// transform (Section 3: F can be evaluated with an FFT; the Jacobian stays
// analytic).
//
// With 0-based indices the sum of eq. (3.2) is a Hankel product,
//   y_i = sum_j x_j h[i+j],  h[k] = 1/(k+1),  t_i = c/(2N) (i + 1/2) y_i.
// Reversing x (z_m = x_{N-1-m}) turns it into the convolution
//   y_i = (h * z)[i + N - 1],
// and a circular convolution of length L >= 2N gives the same values at the
// indices N-1 .. 2N-2 (a wrapped term would need an index sum of at least
// L + N - 1 > 3N - 3, the largest that occurs).  So one forward transform of z,
// a product with the transform of h (computed once per N), and one inverse
// transform give every y_i, in double precision.
//
// The transforms are hand-written: a four-step split L = L1 L2 (L a power of
// two, L1 <= L2 <= 256) into two launches, each CTA doing one or two radix-2
// Stockham transforms of length L1 or L2 in shared memory,
//   pass A: for each n2, Y[n2][k1] = w_L^(n2 k1) sum_n1 x[L2 n1 + n2] w_L1^(n1 k1),
//   pass B: for each k1, X[k1 + L1 k2] = sum_n2 Y[n2][k1] w_L2^(n2 k2),
// with twiddles w_L^k = exp(-2 pi i k / L) from a table made once with
// sincospi.  The inverse transform is the forward one applied to the
// conjugate (only its real part is needed).  The Newton update x + ||F|| u
// is fused into the first pass, the residual, r and the deterministic norm
// into the last, so one evaluation is four launches.
#include "common.cuh"
#include "internal.h"

namespace nl {

__device__ __forceinline__ double2 cmul(double2 a, double2 b)
{
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// tw[k] = exp(-2 pi i k / L): a thread per entry of the first quadrant.
__global__ void k_fft_twiddles(int L, double2* __restrict__ tw)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x, q = L >> 2;
    if (k < q) {
        double s, c;
        sincospi(2.0 * (double)k / (double)L, &s, &c);
        tw[k] = make_double2(c, -s);
        tw[k + q] = make_double2(-s, -c);
        tw[k + 2 * q] = make_double2(-c, s);
        tw[k + 3 * q] = make_double2(s, c);
    }
}

// Radix-2 Stockham transform of length n (a power of two) held in A, with B
// as the ping-pong buffer, by n / 2 threads (this one: j; act: it takes part;
// every thread of the CTA comes to the barriers); returns the buffer that
// holds the result.  Stage with half-size Ls: thread j combines entries j and
// j + n/2 into positions 2 Ls (j / Ls) + j % Ls and that + Ls, with the twiddle
// w_(2 Ls)^(j % Ls): 1 in the first stage, 1 or -i in the second, else loaded one
// stage ahead.
//
// A double-precision instruction occupies its warp for about 65 cycles,
// dependent on the last one or not and however few lanes are active, until
// four warps keep an SM's few units busy (then 19 cycles per warp
// instruction), so what counts is the number of instructions per warp: 40 in a
// transform of 64, 56 in one of 256.  An evaluation takes 31 us at N = 4096 and
// 48 at 32768 (45 and 70 with the twiddles loaded where they are used, one
// transform per CTA of up to 128 threads and the divisions by L and N in every
// thread).  Not kept, for larger rounding errors: transforms of half the length
// on weighted data (39 us at N = 32768) and a thread per result (30 us at 4096).
// Radix-4 butterflies in n / 4 threads have fewer instructions, but in too few
// warps (at half the length 42 and 46 us).
__device__ __forceinline__ double2* dft_smem(double2* A, double2* B, int n, int j, bool act, int L,
                                             const double2* __restrict__ tw)
{
    const int half = n >> 1;
    double2 w = make_double2(1.0, 0.0);
    for (int Ls = 1; Ls < n; Ls <<= 1) {
        double2 v = w;
        if (Ls > 1 && 4 * Ls <= n) v = __ldg(tw + (j & (2 * Ls - 1)) * (L / (4 * Ls)));
        if (act) {
            const int k = j & (Ls - 1), o = 2 * (j - k) + k;
            const double2 a = A[j];
            double2 b = A[j + half];
            if (Ls > 2) b = cmul(b, w);
            else if (Ls == 2 && k) b = make_double2(b.y, -b.x);
            B[o] = make_double2(a.x + b.x, a.y + b.y);
            B[o + Ls] = make_double2(a.x - b.x, a.y - b.y);
        }
        __syncthreads();
        double2* t = A;
        A = B;
        B = t;
        w = v;
    }
    return A;
}

// A CTA does G = 2^lgG transforms (consecutive n2 or k1, so that 32-byte sectors
// are whole when G = 2), each by n / 2 threads (one for n = 1) with two entries
// each to load and to store.

// Pass A.  MODE 0: the input is `in` (length L, natural order).  MODE 1: the
// input is z_m = v_(N-1-m) for m < N (0 beyond), v = x + scale u (the Newton
// update, rounded as in the direct residual), u may be NULL.  MODE 2: the input
// is h_m = 1/(m+1) for m < 2N - 1 (0 beyond).
template <int MODE, typename TU>
__global__ void __launch_bounds__(256) k_fft_pass_a(int N, int L, int L1, int L2, int lgG, const double2* __restrict__ tw,
                                                    const double2* __restrict__ in, const double* __restrict__ x,
                                                    const TU* __restrict__ u, double scale, double2* __restrict__ Y)
{
    extern __shared__ double2 fsm[];
    const int tpt = max(1, L1 >> 1), nt = tpt << lgG, tid = threadIdx.x, base = blockIdx.x << lgG, G = 1 << lgG;
    const bool act = tid < nt;
    const int lgn = 31 - __clz(L1);
    double2 f[2];  // the four-step twiddles of this thread's results
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int e = tid + q * nt;
        f[q] = make_double2(0.0, 0.0);
        if (act && e < (L1 << lgG)) f[q] = __ldg(tw + (base + (e >> lgn)) * (e & (L1 - 1)));
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int e = tid + q * nt, g = e & (G - 1), n1 = e >> lgG, m = L2 * n1 + base + g;
        if (!act || n1 >= L1) continue;
        double2 v;
        if constexpr (MODE == 0) {
            v = in[m];
        } else if constexpr (MODE == 1) {
            double val = 0.0;
            if (m < N) {
                const int j = N - 1 - m;
                val = x[j];
                if (u) val = __dadd_rn(val, __dmul_rn(scale, (double)u[j]));
            }
            v = make_double2(val, 0.0);
        } else {
            v = make_double2(m < 2 * N - 1 ? 1.0 / (double)(m + 1) : 0.0, 0.0);
        }
        fsm[(g << (lgn + 1)) + n1] = v;
    }
    __syncthreads();
    const int g0 = act ? tid / tpt : 0, j = tid - (tid / tpt) * tpt;
    double2* A = fsm + (g0 << (lgn + 1));
    const int r = (int)(dft_smem(A, A + L1, L1, j, act, L, tw) - A);  // 0 or L1, the same for all groups
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int e = tid + q * nt, g = e >> lgn, k1 = e & (L1 - 1);
        if (act && g < G) Y[(base + g) * L1 + k1] = cmul(fsm[(g << (lgn + 1)) + r + k1], f[q]);
    }
}

// Pass B.  MODE 0: out = X.  MODE 1: out = conj(X * Hh) (the input of the
// inverse transform).  MODE 2: the inverse transform's real part / L at the
// indices N-1 .. 2N-2 gives y_i; then t_i (ct = c / (2N) / L: the division by a
// power of two is exact), r_i = 1/(1 - t_i), F_i = v_i - r_i (v = x + scale u, also
// written to xout when given), and ||F||_2 with a deterministic reduction
// (per-block partials, the last block sums them).
template <int MODE, typename TU>
__global__ void __launch_bounds__(256) k_fft_pass_b(int N, int L, int L1, int L2, int lgG, const double2* __restrict__ tw,
                                                    const double2* __restrict__ Y, const double2* Hh, double2* out,
                                                    double ct, const double* __restrict__ x, const TU* __restrict__ u,
                                                    double scale, double* __restrict__ xout, double* __restrict__ F,
                                                    double* __restrict__ rr, double* __restrict__ part,
                                                    unsigned* __restrict__ cnt, double* __restrict__ fnorm)
{
    extern __shared__ double2 fsm[];
    __shared__ double red[8];
    __shared__ bool last;
    const int tpt = max(1, L2 >> 1), nt = tpt << lgG, tid = threadIdx.x, base = blockIdx.x << lgG, G = 1 << lgG;
    const bool act = tid < nt;
    const int lgn = 31 - __clz(L2);
    double2 f[2];  // MODE 1: Hh, MODE 2: {v, -}, at this thread's results
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int e = tid + q * nt, g = e & (G - 1), n2 = e >> lgG, m = base + g + L1 * n2, i = m - (N - 1);
        f[q] = make_double2(0.0, 0.0);
        if (!act || n2 >= L2) continue;
        fsm[(g << (lgn + 1)) + n2] = Y[n2 * L1 + base + g];
        if constexpr (MODE == 1) f[q] = __ldcg(Hh + m);
        if constexpr (MODE == 2) {
            if (i >= 0 && i < N) {
                f[q].x = x[i];
                if (u) f[q].x = __dadd_rn(f[q].x, __dmul_rn(scale, (double)u[i]));
            }
        }
    }
    __syncthreads();
    const int g0 = act ? tid / tpt : 0, j = tid - (tid / tpt) * tpt;
    double2* A = fsm + (g0 << (lgn + 1));
    const int r = (int)(dft_smem(A, A + L2, L2, j, act, L, tw) - A);
    double acc = 0.0;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int e = tid + q * nt, g = e & (G - 1), k2 = e >> lgG, m = base + g + L1 * k2;
        if (!act || k2 >= L2) continue;
        const double2 R = fsm[(g << (lgn + 1)) + r + k2];
        if constexpr (MODE == 0) {
            out[m] = R;
        } else if constexpr (MODE == 1) {
            const double2 p = cmul(R, f[q]);
            out[m] = make_double2(p.x, -p.y);
        } else {
            const int i = m - (N - 1);
            if (i >= 0 && i < N) {
                const double t = ct * ((double)i + 0.5) * R.x;
                const double ri = 1.0 / (1.0 - t);
                const double fi = f[q].x - ri;
                if (xout) xout[i] = f[q].x;
                F[i] = fi;
                rr[i] = ri;
                acc += fi * fi;
            }
        }
    }
    if constexpr (MODE == 2) {
        // deterministic block sum (up to eight warps)
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if ((tid & 31) == 0) red[tid >> 5] = acc;
        __syncthreads();
        if (tid == 0) {
            double b = 0.0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) b += red[w];
            part[blockIdx.x] = b;
            __threadfence();
            last = (atomicAdd(cnt, 1u) == gridDim.x - 1);
        }
        __syncthreads();
        if (last) {
            __threadfence();
            const double sum = partials_sum(part, (int)gridDim.x, red);
            if (tid == 0) {
                *fnorm = sqrt(sum);
                *cnt = 0u;
            }
        }
    }
}

static void fft_sizes(int N, int* L, int* L1, int* L2)
{
    int l = 4;
    while (l < 2 * N) l <<= 1;
    int lg = 0;
    while ((1 << lg) < l) ++lg;
    *L = l;
    *L1 = 1 << (lg / 2);
    *L2 = l / *L1;
}

size_t fft_work_bytes(int N)
{
    int L, L1, L2;
    fft_sizes(N, &L, &L1, &L2);
    return 4 * round_up((size_t)L * sizeof(double2), 256) + round_up((size_t)L1 * sizeof(double), 256) + 256;
}

void fft_work_carve(void* base, int N, FftPlan* p)
{
    fft_sizes(N, &p->L, &p->L1, &p->L2);
    p->N = N;
    char* q = (char*)base;
    const size_t cb = round_up((size_t)p->L * sizeof(double2), 256);
    p->tw = (double2*)q;
    q += cb;
    p->Hh = (double2*)q;
    q += cb;
    p->Y = (double2*)q;
    q += cb;
    p->V = (double2*)q;
    q += cb;
    p->part = (double*)q;
    q += round_up((size_t)p->L1 * sizeof(double), 256);
    p->cnt = (unsigned*)q;
}

// A pass of `count` transforms of length n: two per CTA once there are more of
// them than SMs (one wave, whole 32-byte sectors), else one.
struct FftLaunch {
    unsigned grid, threads;
    size_t smem;
    int lgG;
};
static FftLaunch fft_launch(int count, int n)
{
    const int lgG = count > num_sms() ? 1 : 0;
    return {(unsigned)(count >> lgG), (unsigned)round_up((int64_t)std::max(1, n / 2) << lgG, 32),
            ((size_t)2 * n << lgG) * sizeof(double2), lgG};
}

template <int MODE, typename TU>
static void fft_pass_a(const FftPlan& p, const double2* in, const double* x, const TU* u, double scale, cudaStream_t st)
{
    const FftLaunch a = fft_launch(p.L2, p.L1);
    k_fft_pass_a<MODE, TU><<<a.grid, a.threads, a.smem, st>>>(p.N, p.L, p.L1, p.L2, a.lgG, p.tw, in, x, u, scale, p.Y);
}

template <int MODE, typename TU>
static void fft_pass_b(const FftPlan& p, double2* out, double ct, const double* x, const TU* u, double scale, double* xout,
                       double* F, double* rr, double* fnorm, cudaStream_t st)
{
    const FftLaunch b = fft_launch(p.L1, p.L2);
    k_fft_pass_b<MODE, TU><<<b.grid, b.threads, b.smem, st>>>(p.N, p.L, p.L1, p.L2, b.lgG, p.tw, p.Y, p.Hh, out, ct, x, u,
                                                              scale, xout, F, rr, p.part, p.cnt, fnorm);
}

nl_status fft_prepare(const FftPlan& p, cudaStream_t st)
{
    NL_CUDA_OK(cudaMemsetAsync(p.cnt, 0, sizeof(unsigned), st));
    k_fft_twiddles<<<(unsigned)cdiv(p.L / 4, 64), 64, 0, st>>>(p.L, p.tw);
    fft_pass_a<2, double>(p, nullptr, nullptr, nullptr, 0.0, st);
    fft_pass_b<0, double>(p, p.Hh, 0.0, nullptr, nullptr, 0.0, nullptr, nullptr, nullptr, nullptr, st);
    NL_CUDA_OK(cudaGetLastError());
    return NL_OK;
}

template <typename TU>
static nl_status residual_fft_t(const FftPlan& p, double c, const double* x, const TU* u, double scale, double* xout,
                                double* F, double* rr, double* fnorm, cudaStream_t st)
{
    const double ct = c / (2.0 * (double)p.N) / (double)p.L;  // (L: a power of two)
    prof_begin("k_fft", st);
    fft_pass_a<1, TU>(p, nullptr, x, u, scale, st);
    fft_pass_b<1, TU>(p, p.V, 0.0, nullptr, nullptr, 0.0, nullptr, nullptr, nullptr, nullptr, st);
    fft_pass_a<0, TU>(p, p.V, nullptr, nullptr, 0.0, st);
    fft_pass_b<2, TU>(p, nullptr, ct, x, u, scale, xout, F, rr, fnorm, st);
    prof_end("k_fft", st);
    NL_CUDA_OK(cudaGetLastError());
    return NL_OK;
}

nl_status launch_residual_fft(const FftPlan& p, double c, const double* x, const void* u, int u_is_double,
                              double scale, double* xout, double* F, double* rr, double* fnorm, cudaStream_t st)
{
    if (u_is_double) return residual_fft_t<double>(p, c, x, (const double*)u, scale, xout, F, rr, fnorm, st);
    return residual_fft_t<float>(p, c, x, (const float*)u, scale, xout, F, rr, fnorm, st);
}

}  // namespace nl
