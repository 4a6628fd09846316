// Tiles of 16 x 8 fine nodes (16 x 16 at l = 4), one thread per node: the
// staging, prolongation and restriction that the kernels of fused_node.cu and
// adjoint.cu share.
#pragma once

#include <cuda_runtime.h>

#include "bounds.cuh"
#include "qg_internal.cuh"

namespace qg {
namespace node {

constexpr int NX = 16;                                   // tile columns

template <int LV>
struct Tile {
    static constexpr int F = 1 << LV, NY = LV == 4 ? 16 : 8, THREADS = NX * NY;
    static constexpr int WX = NX + 2, WY = NY + 2;              // halo tile
    static constexpr int CX = NX / F + 3, CY = NY / F + 3;      // elliptic-grid patch
    static constexpr int SX = NX / F + 1, SY = NY / F + 1;      // elliptic nodes the tile touches
};

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// The halo tile of a fine field with corner node (x0, y0) (zero outside the
// grid).
template <typename T, int LV>
__device__ __forceinline__ void load_halo(const T* src, T* dst, int x0, int y0, int nx, int ny, int ld) {
    using Q = Tile<LV>;
    for (int e = threadIdx.x; e < Q::WY * Q::WX; e += Q::THREADS) {
        const int hx = x0 - 1 + e % Q::WX, hy = y0 - 1 + e / Q::WX;
        const bool ok = hx >= 0 && hx <= nx && hy >= 0 && hy <= ny &&
                        QG_IN((long long)hy * ld + hx, (long long)(ny + 1) * ld, 131);
        dst[e] = ok ? src[(size_t)hy * ld + hx] : T(0);
    }
}

// The elliptic-grid patch of the tile: node (a, b) is elliptic node
// ((x0 >> LV) - 1 + a, (y0 >> LV) - 1 + b).
template <typename T, int LV>
__device__ __forceinline__ void load_patch(const T* src, T* cp, int x0, int y0, int nx, int ny, int ldp) {
    using Q = Tile<LV>;
    const int mx = nx >> LV, my = ny >> LV, I0 = (x0 >> LV) - 1, J0 = (y0 >> LV) - 1;
    for (int e = threadIdx.x; e < Q::CX * Q::CY; e += Q::THREADS) {
        const int I = I0 + e % Q::CX, J = J0 + e / Q::CX;
        const bool ok = I >= 0 && I <= mx && J >= 0 && J <= my &&
                        QG_IN((long long)J * ldp + I, (long long)(my + 1) * ldp, 133);
        cp[e] = ok ? src[(size_t)J * ldp + I] : T(0);
    }
}

// The patch prolonged to the halo tile (Eq. pro applied l times: bilinear):
// rows of the patch at the fine rows, then columns; halo row r is fine row
// y0 - 1 + r, patch row (F - 1 + r) / F.  A row or column past a wall is not
// read by an interior node.  Barriers before, between and after.
template <typename T, int LV>
__device__ __forceinline__ void prolong_halo(const T* cp, T* cr, T* sp) {
    using Q = Tile<LV>;
    constexpr int F = Q::F;
    __syncthreads();
    for (int e = threadIdx.x; e < Q::WY * Q::CX; e += Q::THREADS) {
        const int r = e / Q::CX, c = e % Q::CX;
        const int b = (F - 1 + r) / F, ph = (F - 1 + r) % F;
        const bool ok = QG_IN((b + 1) * Q::CX + c, Q::CX * Q::CY, 134);
        const T lo = ok ? cp[b * Q::CX + c] : T(0), hi = ok ? cp[(b + 1) * Q::CX + c] : T(0);
        const T wt = T(ph) * (T(1) / T(F));
        cr[e] = ph == 0 ? lo : fma(wt, hi, (T(1) - wt) * lo);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < Q::WY * Q::WX; e += Q::THREADS) {
        const int r = e / Q::WX, c = e % Q::WX;
        const int a = (F - 1 + c) / F, ph = (F - 1 + c) % F;
        const bool ok = QG_IN(r * Q::CX + a + 1, Q::WY * Q::CX, 135);
        const T lo = ok ? cr[r * Q::CX + a] : T(0), hi = ok ? cr[r * Q::CX + a + 1] : T(0);
        const T wt = T(ph) * (T(1) / T(F));
        sp[e] = ph == 0 ? lo : fma(wt, hi, (T(1) - wt) * lo);
    }
    __syncthreads();
}

// The patch prolonged to the thread's own node (i, j) of the tile.
template <typename T, int LV>
__device__ __forceinline__ T prolong_own(const T* cp, int i, int j) {
    using Q = Tile<LV>;
    constexpr int F = Q::F;
    const T* c = cp + (1 + j / F) * Q::CX + 1 + i / F;
    const T a = T(i % F) * (T(1) / T(F)), b = T(j % F) * (T(1) / T(F));
    if (!QG_IN((2 + j / F) * Q::CX + 2 + i / F, Q::CX * Q::CY, 134)) return T(0);
    const T lo = fma(a, c[1], (T(1) - a) * c[0]);
    const T hi = fma(a, c[Q::CX + 1], (T(1) - a) * c[Q::CX]);
    return fma(b, hi, (T(1) - b) * lo);
}

// The hat weights (f - |d|)/f^2 of the restriction over the tile's nodes
// `so` (zero at walls and outside), x shares then y shares, into the four
// partial planes of fused.cu (plane 0, bit 0: the tile's right edge line,
// bit 1: the line above its last row; one writer per plane and node).
template <typename T, int LV>
__device__ __forceinline__ void restrict_tile(const T* so, T* sx, T* const (&part)[4], int ldc, int x0,
                                              int y0, int nx, int ny) {
    using Q = Tile<LV>;
    constexpr int F = Q::F, NY = Q::NY;
    const int mx = nx >> LV, my = ny >> LV;
    __syncthreads();
    for (int e = threadIdx.x; e < NY * Q::SX; e += Q::THREADS) {
        const int r = e / Q::SX, c = e % Q::SX;
        T v = T(0);
#pragma unroll
        for (int d = -(F - 1); d < F; ++d) {
            const int k = c * F + d;
            if (k >= 0 && k < NX && QG_IN(r * NX + k, NY * NX, 137))
                v = fma(T(F - (d < 0 ? -d : d)) * (T(1) / T(F * F)), so[r * NX + k], v);
        }
        sx[e] = v;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < Q::SY * Q::SX; e += Q::THREADS) {
        const int m = e / Q::SX, c = e % Q::SX;
        T v = T(0);
#pragma unroll
        for (int d = -(F - 1); d < F; ++d) {
            const int r = m * F + d;
            if (r >= 0 && r < NY && QG_IN(r * Q::SX + c, NY * Q::SX, 138))
                v = fma(T(F - (d < 0 ? -d : d)) * (T(1) / T(F * F)), sx[r * Q::SX + c], v);
        }
        const int I = (x0 >> LV) + c, J = (y0 >> LV) + m;
        const int pl = (c == Q::SX - 1 ? 1 : 0) + (m == Q::SY - 1 ? 2 : 0);
        if (I >= 1 && I <= mx - 1 && J >= 1 && J <= my - 1 &&
            QG_IN((long long)J * ldc + I, (long long)(my + 1) * ldc, 139))
            part[pl][(size_t)J * ldc + I] = v;
    }
}

// Launch of a tile kernel, dependent programmatically on the launch before.
template <typename... P, typename... A>
cudaError_t launch(void (*k)(P...), int nx, int ny, int rows, cudaStream_t s, const A&... a) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((nx + NX - 1) / NX, (ny + rows - 1) / rows);
    cfg.blockDim = dim3(NX * rows);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, a...);
}

}  // namespace node
}  // namespace qg
