// Elliptic solve of Section 4.3 on small grids as sine sums (engine 42).
//
// A grid of at most 128 x 256 unknowns gives an FFT a few hundred threads, each
// with a long chain of dependent operations; in FP64, where a sub-partition
// of an SM issues one warp instruction in about 64 clocks, that chain is the
// solve's time (32 x 64: 32 us with the radix-4 engine, 14 us here; FP32 14
// against 10 us).  Here every output is a sum of its own, F_k = sum_n f_n
// sin(pi n k / N), one thread each, spread over the whole GPU: more operations
// (N/2 per output instead of O(log N)) in a chain a tenth as long.  Folding
// halves the sums: sin(pi (N - n) k / N) = -(-1)^k sin(pi n k / N), so odd k
// take f_n + f_{N-n} and even k f_n - f_{N-n}, n <= N/2.  Four partial sums per
// output keep the additions independent and their rounding error small.
//
// Three launches chained by programmatic dependent launch: x pass of one row
// per CTA -> tr[k][row]; y pass, the mode-space solve (Eq. ialpha, or Eqs.
// isub-1/2 for two layers) and the inverse y pass of one x-mode per CTA ->
// work[l][k]; inverse x pass of one row per CTA.  The FP64-evaluated sine
// tables are staged in shared memory before the programmatic wait where they
// fit in 16 KB.
#include <cuda_runtime.h>

#include <cmath>
#include <vector>

#include "bounds.cuh"
#include "dst_engine.cuh"
#include "qg_internal.cuh"

namespace qg {
namespace {

using namespace eng;

constexpr int kMaxN = 256;
constexpr int kStageBytes = 16 * 1024;

// u[n] = f_n + f_{N-n} and v[n] = f_n - f_{N-n}, n < N/2; u = f, v = 0 at N/2
template <typename T>
__device__ __forceinline__ void fold(const T* f, T* u, T* v, int N) {
    const int n = threadIdx.x;
    if (n >= 1 && n <= N / 2) {
        const T a = f[n], b = n < N / 2 ? f[N - n] : T(0);
        u[n] = a + b;
        v[n] = n < N / 2 ? a - b : T(0);
    }
}

// F_k from the folded values: S[(n - 1) N + k] = sin(pi n k / N)
template <typename T>
__device__ __forceinline__ T sine_sum(const T* S, const T* u, const T* v, int N, int k) {
    const T* x = (k & 1) ? u : v;
    T a[4] = {T(0), T(0), T(0), T(0)};
    const int h = N / 2;                       // a multiple of 4
#pragma unroll 4
    for (int n = 0; n < h; n += 4) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (QG_IN((n + q) * N + k, h * N, 121)) a[q] = fma(S[(n + q) * N + k], x[n + q + 1], a[q]);
    }
    return (a[0] + a[2]) + (a[1] + a[3]);
}

// The table in shared memory when it fits.
template <typename T>
__device__ __forceinline__ const T* stage_table(const T* S, T* buf, int N, bool fits) {
    if (!fits) return S;
    // (16 bytes a thread and load, eight loads in flight)
    const int4* src = reinterpret_cast<const int4*>(S);
    int4* dst = reinterpret_cast<int4*>(buf);
    const int n = N / 2 * N * (int)sizeof(T) / 16;
    for (int e = threadIdx.x; e < n; e += 8 * blockDim.x) {
        int4 v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (e + q * (int)blockDim.x < n) v[q] = __ldg(src + e + q * blockDim.x);
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (e + q * (int)blockDim.x < n) dst[e + q * blockDim.x] = v[q];
    }
    return buf;
}

// X pass of row 1 + blockIdx.x of layer blockIdx.y: forward (the sum of the
// right-hand side's planes -> tr) or inverse (work -> out).
template <typename T, bool FWD>
__global__ void __launch_bounds__(kMaxN) dense_x_kernel(SolveParams<T> P, const T* S, int fits) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ T f[kMaxN], u[kMaxN / 2 + 1], v[kMaxN / 2 + 1];
    const int N = P.mx, k = threadIdx.x, r = 1 + blockIdx.x, L = blockIdx.y;
    const T* tab = stage_table(S, reinterpret_cast<T*>(smem), N, fits != 0);
    pdl_wait();
    pdl_trigger();
    const long long n = (long long)(P.my + 1) * P.ld;
    (void)n;
    if (k >= 1 && k < N && QG_IN((long long)r * P.ld + k, n, 122)) {
        const size_t o = (size_t)r * P.ld + k;
        T x;
        if (FWD) {
            const T* const in[4] = {L ? P.in[1][0] : P.in[0][0], L ? P.in[1][1] : P.in[0][1],
                                    L ? P.in[1][2] : P.in[0][2], L ? P.in[1][3] : P.in[0][3]};
            x = in[0][o];
            if (P.nin > 1) {
                const bool cx = (k & (P.part_px - 1)) == 0, cy = (r & (P.part_py - 1)) == 0;
                const T b = cx ? in[1][o] : T(0), c = cy ? in[2][o] : T(0);
                const T d = cx && cy ? in[3][o] : T(0);
                x += b;
                x += c;
                x += d;
            }
        } else {
            x = (L ? P.work[1] : P.work[0])[o];
        }
        f[k] = x;
    }
    __syncthreads();
    fold(f, u, v, N);
    __syncthreads();
    if (k >= 1 && k < N) {
        const T F = sine_sum(tab, u, v, N, k);
        const long long nt = (long long)(P.mx + 1) * P.ld_tr;
        (void)nt;
        if (FWD) {
            if (QG_IN((long long)k * P.ld_tr + r, nt, 123))
                (L ? P.tr[1] : P.tr[0])[(size_t)k * P.ld_tr + r] = F;
        } else if (QG_IN((long long)r * P.ld + k, n, 124)) {
            (L ? P.out[1] : P.out[0])[(size_t)r * P.ld + k] = F;
        }
    }
}

// Y pass of x-mode 1 + blockIdx.x: forward sums, mode-space solve, inverse.
template <typename T, int NL>
__global__ void __launch_bounds__(kMaxN) dense_y_kernel(SolveParams<T> P, const T* S, int fits) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ T f[NL][kMaxN], u[NL][kMaxN / 2 + 1], v[NL][kMaxN / 2 + 1];
    const int N = P.my, l = threadIdx.x, k = 1 + blockIdx.x;
    const bool in = l >= 1 && l < N;
    const T* tab = stage_table(S, reinterpret_cast<T*>(smem), N, fits != 0);
    const T lam = in ? P.lamx[k] + P.lamy[l] : T(1);
    pdl_wait();
    pdl_trigger();
    const long long nt = (long long)(P.mx + 1) * P.ld_tr;
    (void)nt;
    if (in && QG_IN((long long)k * P.ld_tr + l, nt, 125)) {
#pragma unroll
        for (int L = 0; L < NL; ++L) f[L][l] = P.tr[L][(size_t)k * P.ld_tr + l];
    }
    __syncthreads();
#pragma unroll
    for (int L = 0; L < NL; ++L) fold(f[L], u[L], v[L], N);
    __syncthreads();
    if (in) {
        T F[NL];
#pragma unroll
        for (int L = 0; L < NL; ++L) F[L] = sine_sum(tab, u[L], v[L], N, l);
        if (NL == 1) {
            f[0][l] = F[0] * (P.scale / lam);
        } else {
            const T q1 = P.scale * F[0], q2 = P.scale * F[NL - 1];
            const T al = P.Ro * lam;
            const T den = al * (al - P.f1 - P.f2);
            f[0][l] = (al * q1 - P.f2 * q1 - P.f1 * q2) / den;
            f[NL - 1][l] = (al * q2 - P.f2 * q1 - P.f1 * q2) / den;
        }
    }
    __syncthreads();
#pragma unroll
    for (int L = 0; L < NL; ++L) fold(f[L], u[L], v[L], N);
    __syncthreads();
    const long long n = (long long)(P.my + 1) * P.ld;
    (void)n;
    if (in && QG_IN((long long)l * P.ld + k, n, 126)) {
#pragma unroll
        for (int L = 0; L < NL; ++L)
            P.work[L][(size_t)l * P.ld + k] = sine_sum(tab, u[L], v[L], N, l);
    }
}

template <typename T>
cudaError_t launch(void (*k)(SolveParams<T>, const T*, int), const SolveParams<T>& P, const T* S,
                   int N, dim3 grid, cudaStream_t s) {
    const size_t bytes = (size_t)N / 2 * N * sizeof(T);
    const int fits = bytes <= (size_t)kStageBytes;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(N < 32 ? 32 : N);
    cfg.dynamicSmemBytes = fits ? bytes : 0;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = P.no_pdl ? nullptr : at;
    cfg.numAttrs = P.no_pdl ? 0 : 1;
    return cudaLaunchKernelEx(&cfg, k, P, S, fits);
}

}  // namespace

bool dense_supports(int mx, int my) {
    return is_pow2(mx) && is_pow2(my) && mx >= 8 && my >= 8 && mx <= kMaxN && my <= kMaxN;
}

void dense_table(int N, double* out) {
    const double pi = 3.14159265358979323846;
    // 2N sines, then copies: the table's N^2/2 sines were 0.4 ms of a 256-wide
    // handle's creation
    std::vector<double> sn(2 * N);
    for (int m = 0; m < 2 * N; ++m) sn[m] = std::sin(pi * (long long)m / N);
    for (int n = 1; n <= N / 2; ++n)
        for (int k = 0; k < N; ++k)
            out[(size_t)(n - 1) * N + k] = sn[(long long)n * k % (2 * N)];
}

template <typename T>
cudaError_t launch_solve_dense(const SolveParams<T>& P, cudaStream_t s) {
    if (!dense_supports(P.mx, P.my) || !P.dsx || !P.dsy || P.batch) return cudaErrorInvalidValue;
    const dim3 gx(P.my - 1, P.layers), gy(P.mx - 1);
    cudaError_t e = launch<T>(dense_x_kernel<T, true>, P, P.dsx, P.mx, gx, s);
    if (e == cudaSuccess)
        e = P.layers == 2 ? launch<T>(dense_y_kernel<T, 2>, P, P.dsy, P.my, gy, s)
                          : launch<T>(dense_y_kernel<T, 1>, P, P.dsy, P.my, gy, s);
    if (e == cudaSuccess) e = launch<T>(dense_x_kernel<T, false>, P, P.dsx, P.mx, gx, s);
    return e;
}

template cudaError_t launch_solve_dense<float>(const SolveParams<float>&, cudaStream_t);
template cudaError_t launch_solve_dense<double>(const SolveParams<double>&, cudaStream_t);

QG_BOUNDS_QUERY(bounds_site_dense)

}  // namespace qg
