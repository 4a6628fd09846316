// FP64 diagnostics of a basin state: the basin-integrated kinetic energy
// (Section 5.2, E = 1/2 iint |grad psi|^2, one-sided differences on grid
// edges), the enstrophy 1/2 iint w^2, and max(|psi_x|, |psi_y|) (the
// denominator of the CFL time step, Eq. dt).
//
// Differences are formed in the working precision and squared and summed in
// FP64.  An FP32 basin's psi is refined once before (residual_kernel, one more
// solve, prolong_pair_kernel): the steepest difference is a few per cent of
// psi itself, so the rounding of an FP32 solve (1.5e-7 of psi) stands in
// max |grad psi| at 2e-6; refined, 1e-7 is left.  Each CTA covers a fixed strided set of nodes and reduces through a
// fixed shared-memory tree; one CTA then folds the per-CTA results in index
// order, so the result is bitwise reproducible run to run.
#include <cuda_runtime.h>

#include "bounds.cuh"
#include "qg_internal.cuh"

namespace qg {
namespace {

constexpr int kDiagThreads = 256;
constexpr int kDiagBlocks = 304;  // 2 per SM on a 152-SM GB300

// psi is `psi`, plus `lo` (the part below its rounding) when that is given.
// nx is a power of two (2^lgx): no division per node.
template <typename T>
__global__ void __launch_bounds__(kDiagThreads)
diag_partial_kernel(const T* __restrict__ psi, const T* __restrict__ lo, const T* __restrict__ w,
                    int nx, int lgx, int ny, int ld, double* __restrict__ partial) {
    __shared__ double sh[5][kDiagThreads];
    double sx = 0.0, sy = 0.0, sw = 0.0;
    T ux = T(0), uy = T(0);
    const int total = nx * ny;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += gridDim.x * blockDim.x) {
        const int i = idx & (nx - 1), j = idx >> lgx;
        const size_t c = (size_t)j * ld + i;
        const long long n = (long long)(ny + 1) * ld;
        (void)n;
        if (!(QG_IN((long long)c + ld, n, 101) && QG_IN((long long)c + 1, n, 101) &&
              (i < 1 || j < 1 || (QG_IN((long long)c - ld, n, 102) && QG_IN((long long)c - 1, n, 102)))))
            continue;
        auto diff = [&](size_t p, size_t q) {
            const T d = psi[p] - psi[q];
            return lo ? d + (lo[p] - lo[q]) : d;
        };
        if (j >= 1) {
            const double d = (double)diff(c + 1, c);
            sx += d * d;
        }
        if (i >= 1) {
            const double d = (double)diff(c + ld, c);
            sy += d * d;
        }
        if (i >= 1 && j >= 1) {
            const double v = (double)w[c];
            sw += v * v;
            const T a = fabs(diff(c + 1, c - 1)), b = fabs(diff(c + ld, c - ld));
            ux = a > ux ? a : ux;   // (as fmax: a NaN shows in the sums)
            uy = b > uy ? b : uy;
        }
    }
    sh[0][threadIdx.x] = sx;
    sh[1][threadIdx.x] = sy;
    sh[2][threadIdx.x] = sw;
    sh[3][threadIdx.x] = (double)ux;
    sh[4][threadIdx.x] = (double)uy;
    __syncthreads();
    for (int s = kDiagThreads / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            sh[0][threadIdx.x] += sh[0][threadIdx.x + s];
            sh[1][threadIdx.x] += sh[1][threadIdx.x + s];
            sh[2][threadIdx.x] += sh[2][threadIdx.x + s];
            sh[3][threadIdx.x] = fmax(sh[3][threadIdx.x], sh[3][threadIdx.x + s]);
            sh[4][threadIdx.x] = fmax(sh[4][threadIdx.x], sh[4][threadIdx.x + s]);
        }
        __syncthreads();
    }
    if (threadIdx.x < 5) partial[blockIdx.x * 5 + threadIdx.x] = sh[threadIdx.x][0];
}

__global__ void __launch_bounds__(kDiagThreads)
diag_final_kernel(const double* __restrict__ partial, int nblocks,
                  double* __restrict__ out) {
    __shared__ double sh[5][kDiagThreads];
    double a[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    for (int b = threadIdx.x; b < nblocks; b += blockDim.x) {
        a[0] += partial[b * 5 + 0];
        a[1] += partial[b * 5 + 1];
        a[2] += partial[b * 5 + 2];
        a[3] = fmax(a[3], partial[b * 5 + 3]);
        a[4] = fmax(a[4], partial[b * 5 + 4]);
    }
    for (int k = 0; k < 5; ++k) sh[k][threadIdx.x] = a[k];
    __syncthreads();
    for (int s = kDiagThreads / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            sh[0][threadIdx.x] += sh[0][threadIdx.x + s];
            sh[1][threadIdx.x] += sh[1][threadIdx.x + s];
            sh[2][threadIdx.x] += sh[2][threadIdx.x + s];
            sh[3][threadIdx.x] = fmax(sh[3][threadIdx.x], sh[3][threadIdx.x + s]);
            sh[4][threadIdx.x] = fmax(sh[4][threadIdx.x], sh[4][threadIdx.x + s]);
        }
        __syncthreads();
    }
    if (threadIdx.x < 5) out[threadIdx.x] = sh[threadIdx.x][0];
}

// r = R^l w - lap_h psi at the interior nodes of the elliptic grid: the
// restriction's sums in FP32 (restrict_kernel's), the cancelling differences
// in FP64.  cx, cy = 1/dx^2, 1/dy^2 of the elliptic grid.
__global__ void residual_kernel(const float* __restrict__ w, int ldf, const float* __restrict__ psi,
                                float* __restrict__ r, int ld, int mx, int my, int levels,
                                double cx, double cy) {
    const int I = blockIdx.x * blockDim.x + threadIdx.x + 1;
    const int J = blockIdx.y * blockDim.y + threadIdx.y + 1;
    if (I >= mx || J >= my) return;
    const int f = 1 << levels;
    const float* base = w + (size_t)(f * J) * ldf + f * I;
    const long long fn = (long long)(f * my + 1) * ldf, cn = (long long)(my + 1) * ld;
    (void)fn;
    (void)cn;
    float acc = 0.0f;
    for (int dj = -(f - 1); dj <= f - 1; ++dj) {
        float racc = 0.0f;
        for (int di = -(f - 1); di <= f - 1; ++di)
            if (QG_IN((long long)(f * J + dj) * ldf + f * I + di, fn, 103))
                racc += (float)(f - (di < 0 ? -di : di)) * base[(ptrdiff_t)dj * ldf + di];
        acc += (float)(f - (dj < 0 ? -dj : dj)) * racc;
    }
    acc *= 1.0f / ((float)f * f * f * f);
    const size_t c = (size_t)J * ld + I;
    if (!(QG_IN((long long)c + ld, cn, 104) && QG_IN((long long)c - ld, cn, 104))) return;
    const double p0 = psi[c];
    const double lap = (((double)psi[c + 1] - p0) + ((double)psi[c - 1] - p0)) * cx +
                       (((double)psi[c + ld] - p0) + ((double)psi[c - ld] - p0)) * cy;
    r[c] = (float)((double)acc - lap);
}

// hi + lo = P^l (c + d) at every fine node, lo the part below hi's rounding:
// error-free products and sums (Dekker, Knuth) of the bilinear terms of c, d
// being the small correction.  c and hi may be one array at levels = 0.
__global__ void prolong_pair_kernel(const float* c, const float* __restrict__ d, int ldc, float* hi,
                                    float* __restrict__ lo, int ldf, int nx, int ny, int levels) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    if (i > nx || j > ny) return;
    const int f = 1 << levels, I = i >> levels, J = j >> levels;
    const float a = (float)(i & (f - 1)) / (float)f, b = (float)(j & (f - 1)) / (float)f;
    const float wt[4] = {(1.0f - a) * (1.0f - b), a * (1.0f - b), (1.0f - a) * b, a * b};   // exact
    const size_t o = (size_t)J * ldc + I;
    const int mx = nx >> levels, my = ny >> levels;
    const long long cn = (long long)(my + 1) * ldc;
    (void)cn;
    float s = 0.0f, e = 0.0f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const size_t q = o + (k & 1) + (size_t)(k >> 1) * ldc;
        // (past the grid, or a wall: zero, whatever a solve left there)
        const int In = I + (k & 1), Jn = J + (k >> 1);
        if (wt[k] == 0.0f || In == 0 || Jn == 0 || In >= mx || Jn >= my || !QG_IN((long long)q, cn, 105))
            continue;
        const float x = c[q], p = __fmul_rn(wt[k], x);
        const float t = __fadd_rn(s, p), z = __fsub_rn(t, s);
        e = __fadd_rn(e, __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(p, z)));
        e = __fadd_rn(e, __fmaf_rn(wt[k], x, -p));
        e = __fmaf_rn(wt[k], d[q], e);
        s = t;
    }
    const size_t n = (size_t)j * ldf + i;
    if (!QG_IN((long long)n, (long long)(ny + 1) * ldf, 106)) return;
    const float h = __fadd_rn(s, e);
    hi[n] = h;
    lo[n] = __fadd_rn(__fsub_rn(s, h), e);
}

// acc += c0 out[0] + c1 out[1]: the kinetic energy of Section 5.2 from the
// two edge sums of diag_final_kernel, scaled, added in FP64 by one thread.
__global__ void energy_add_kernel(const double* __restrict__ out, double c0, double c1,
                                  double* __restrict__ acc) {
    if (threadIdx.x == 0 && blockIdx.x == 0) acc[0] += c0 * out[0] + c1 * out[1];
}

}  // namespace

int diag_blocks() { return kDiagBlocks; }

QG_BOUNDS_QUERY(bounds_site_diag)

cudaError_t launch_energy_add(const double* out, double c0, double c1, double* acc,
                              cudaStream_t s) {
    energy_add_kernel<<<1, 32, 0, s>>>(out, c0, c1, acc);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_diagnostics(const T* psi, const T* lo, const T* w, int nx, int ny, int ld,
                               double* partial, int nblocks, double* out, cudaStream_t s) {
    diag_partial_kernel<T><<<nblocks, kDiagThreads, 0, s>>>(psi, lo, w, nx, ilog2(nx), ny, ld,
                                                           partial);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    diag_final_kernel<<<1, kDiagThreads, 0, s>>>(partial, nblocks, out);
    return cudaGetLastError();
}

template cudaError_t launch_diagnostics<float>(const float*, const float*, const float*, int, int,
                                               int, double*, int, double*, cudaStream_t);
template cudaError_t launch_diagnostics<double>(const double*, const double*, const double*, int,
                                                int, int, double*, int, double*, cudaStream_t);

cudaError_t launch_residual(const float* w, int ldf, const float* psi, float* r, int ld, int mx,
                            int my, int levels, double cx, double cy, cudaStream_t s) {
    const dim3 block(32, 8), grid((mx - 1 + 31) / 32, (my - 1 + 7) / 8);
    residual_kernel<<<grid, block, 0, s>>>(w, ldf, psi, r, ld, mx, my, levels, cx, cy);
    return cudaGetLastError();
}

cudaError_t launch_prolong_pair(const float* c, const float* d, int ldc, float* hi, float* lo,
                                int ldf, int nx, int ny, int levels, cudaStream_t s) {
    const dim3 block(32, 8), grid((nx + 1 + 31) / 32, (ny + 1 + 7) / 8);
    prolong_pair_kernel<<<grid, block, 0, s>>>(c, d, ldc, hi, lo, ldf, nx, ny, levels);
    return cudaGetLastError();
}

}  // namespace qg
