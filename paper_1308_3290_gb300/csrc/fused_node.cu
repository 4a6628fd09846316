// Fused fine-grid stage of the one-layer model with one node per thread: the
// same stage as the sweep of fused.cu (prolongation on load, Arakawa / beta /
// dissipation / forcing, the TVDRK3 combination, restriction on store) for
// grids whose sweep tiles leave most of the GPU idle.
//
// The bound is FP64: an SM sub-partition issues one FP64 warp instruction per
// ~64 clocks, so a thread that sweeps 8 rows of 4 columns (about 1600 FP64
// instructions) holds its sub-partition for 50 us, however few tiles there
// are.  One node per thread and tiles of 16 x 8 nodes spread the same number
// of instructions (about 40 a node: the sweep's shared differences save
// little more than its halo rows cost) over every sub-partition.
//
// A CTA stages w^(s) with its halo and the elliptic-grid patch (or the fine
// psi, l = 0) in shared memory; prolongs in two steps, rows of the patch at
// the fine rows, then columns (Eq. pro applied l times is bilinear); updates
// its nodes; and sums the hat weights (f - |d|)/f^2 of the restriction the
// same way, into the four planes of fused.cu (plane 0, bit 0: the tile's right
// edge line, bit 1: the line above its last row; one writer per plane and
// node).
#include <cuda_runtime.h>

#include "bounds.cuh"
#include "qg_internal.cuh"

namespace qg {
namespace {

constexpr int NX = 16;                                   // tile columns
template <int LV> struct NodeRows { static constexpr int value = LV == 4 ? 16 : 8; };

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename T, int LV>
__global__ void __launch_bounds__(NX * NodeRows<LV>::value)
node_stage_kernel(const FusedParams<T> p) {
    constexpr int NY = NodeRows<LV>::value, F = 1 << LV, THREADS = NX * NY;
    constexpr int WX = NX + 2, WY = NY + 2;              // halo tile
    constexpr int CX = NX / F + 3, CY = NY / F + 3;      // elliptic-grid patch
    constexpr int SX = NX / F + 1, SY = NY / F + 1;      // elliptic nodes the tile touches
    __shared__ T sw[WY * WX], sp[WY * WX];
    __shared__ T so[LV > 0 ? NY * NX : 1], sx[LV > 0 ? NY * SX : 1];
    __shared__ T cp[LV > 0 ? CY * CX : 1], cr[LV > 0 ? WY * CX : 1];
    __shared__ T s_dt;
    const int nx = p.nx, ny = p.ny, ld = p.ld;
    const int x0 = blockIdx.x * NX, y0 = blockIdx.y * NY;
    const int i = threadIdx.x % NX, j = threadIdx.x / NX;
    const int x = x0 + i, y = y0 + j;
    const bool in = x >= 1 && x <= nx - 1 && y >= 1 && y <= ny - 1;
    const long long fine_n = (long long)(ny + 1) * ld;
    (void)fine_n;
    // a halo tile of a fine field (zero outside the grid)
    auto halo = [&](const T* src, T* dst) {
        for (int e = threadIdx.x; e < WY * WX; e += THREADS) {
            const int hx = x0 - 1 + e % WX, hy = y0 - 1 + e / WX;
            const bool ok = hx >= 0 && hx <= nx && hy >= 0 && hy <= ny &&
                            QG_IN((long long)hy * ld + hx, fine_n, 81);
            dst[e] = ok ? src[(size_t)hy * ld + hx] : T(0);
        }
    };
    // w^(s), w^n and the forcing were complete before the solve began
    halo(p.w, sw);
    T wn = T(0), f = T(0);
    const size_t o = (size_t)y * ld + x;
    if (in && QG_IN(o, fine_n, 82)) {
        if (p.a != T(0)) wn = p.wn[o];
        f = p.f2d ? p.f2d[o] : p.frow[y];
    }
    pdl_wait();
    pdl_trigger();
    if (threadIdx.x == 0) {
        // the step size: fixed, or Eq. dt from this step's first psi
        double dtd = (double)p.dt;
        if (p.umax) {
            const double u = __longlong_as_double((long long)*p.umax);
            dtd = u > 0.0 ? fmin(p.dt_cap, p.cfl_h / u) : p.dt_cap;
        }
        s_dt = (T)dtd;
        if (p.last_stage && blockIdx.x == 0 && blockIdx.y == 0) {
            p.clock[0] += dtd;
            p.clock[1] = dtd;
        }
    }
    const int mx = nx >> LV, my = ny >> LV;
    if constexpr (LV == 0) {
        halo(p.psi, sp);
        __syncthreads();
    } else {
        // patch node (a, b) is elliptic node (I0 + a, J0 + b)
        const int I0 = (x0 >> LV) - 1, J0 = (y0 >> LV) - 1;
        for (int e = threadIdx.x; e < CX * CY; e += THREADS) {
            const int I = I0 + e % CX, J = J0 + e / CX;
            const bool ok = I >= 0 && I <= mx && J >= 0 && J <= my &&
                            QG_IN((long long)J * p.ldp + I, (long long)(my + 1) * p.ldp, 83);
            cp[e] = ok ? p.psi[(size_t)J * p.ldp + I] : T(0);
        }
        __syncthreads();
        // halo row r is fine row y0 - 1 + r: patch row (F - 1 + r) / F
        for (int e = threadIdx.x; e < WY * CX; e += THREADS) {
            const int r = e / CX, c = e % CX;
            const int b = (F - 1 + r) / F, ph = (F - 1 + r) % F;
            const bool ok = QG_IN((b + 1) * CX + c, CX * CY, 84);
            const T lo = ok ? cp[b * CX + c] : T(0), hi = ok ? cp[(b + 1) * CX + c] : T(0);
            const T wt = T(ph) * (T(1) / T(F));
            cr[e] = ph == 0 ? lo : fma(wt, hi, (T(1) - wt) * lo);
        }
        __syncthreads();
        for (int e = threadIdx.x; e < WY * WX; e += THREADS) {
            const int r = e / WX, c = e % WX;
            const int a = (F - 1 + c) / F, ph = (F - 1 + c) % F;
            const bool ok = QG_IN(r * CX + a + 1, WY * CX, 85);
            const T lo = ok ? cr[r * CX + a] : T(0), hi = ok ? cr[r * CX + a + 1] : T(0);
            const T wt = T(ph) * (T(1) / T(F));
            // (a row or column past a wall is not read by an interior node)
            sp[e] = ph == 0 ? lo : fma(wt, hi, (T(1) - wt) * lo);
        }
        __syncthreads();
    }
    const T dt = s_dt;
    T out = T(0);
    if (in) {
        const T* q = sw + (j + 1) * WX + i + 1;
        const T* s = sp + (j + 1) * WX + i + 1;
        const T p10 = s[1], pm0 = s[-1], p01 = s[WX], p0m = s[-WX];
        const T p11 = s[WX + 1], pm1 = s[WX - 1], p1m = s[1 - WX], pmm = s[-1 - WX];
        const T q00 = q[0], q10 = q[1], qm0 = q[-1], q01 = q[WX], q0m = q[-WX];
        // vertical differences of psi at columns x - 1, x, x + 1, horizontal
        // ones at rows y - 1, y, y + 1
        const T vm = pm1 - pmm, v0 = p01 - p0m, vp = p11 - p1m;
        const T hm = p1m - pmm, h0 = p10 - pm0, hp = p11 - pm1;
        // Arakawa J1 + J2 + J3 by neighbour of q (Eqs. j1-j3), as in fused.cu
        T jac = -q10 * (v0 + vp);
        jac = fma(qm0, vm + v0, jac);
        jac = fma(q01, h0 + hp, jac);
        jac = fma(-q0m, h0 + hm, jac);
        jac = fma(-q[WX + 1], p01 - p10, jac);
        jac = fma(q[-1 - WX], pm0 - p0m, jac);
        jac = fma(q[WX - 1], p01 - pm0, jac);
        jac = fma(-q[1 - WX], p10 - p0m, jac);
        const T beta = fma(T(4), h0, hp + hm);
        // w^(s+1) = a w^n + b w^(s) + b dt G
        const T bdt = p.b * dt;
        const T k_0 = fma(T(-2) * (p.c_lapx + p.c_lapy), bdt, p.b);
        T g = fma(-p.c_beta * bdt, beta, bdt * f);
        g = fma(-p.c_jac * bdt, jac, g);
        g = fma(k_0, q00, g);
        g = fma(p.c_lapy * bdt, q01 + q0m, g);
        g = fma(p.c_lapx * bdt, q10 + qm0, g);
        out = fma(p.a, wn, g);
        if (QG_IN(o, fine_n, 86)) p.wout[o] = out;
    }
    if constexpr (LV > 0) {
        so[threadIdx.x] = out;
        __syncthreads();
        // x shares of each row at the tile's elliptic columns
        for (int e = threadIdx.x; e < NY * SX; e += THREADS) {
            const int r = e / SX, c = e % SX;
            T v = T(0);
#pragma unroll
            for (int d = -(F - 1); d < F; ++d) {
                const int k = c * F + d;
                if (k >= 0 && k < NX && QG_IN(r * NX + k, NY * NX, 87))
                    v = fma(T(F - (d < 0 ? -d : d)) * (T(1) / T(F * F)), so[r * NX + k], v);
            }
            sx[e] = v;
        }
        __syncthreads();
        for (int e = threadIdx.x; e < SY * SX; e += THREADS) {
            const int m = e / SX, c = e % SX;
            T v = T(0);
#pragma unroll
            for (int d = -(F - 1); d < F; ++d) {
                const int r = m * F + d;
                if (r >= 0 && r < NY && QG_IN(r * SX + c, NY * SX, 88))
                    v = fma(T(F - (d < 0 ? -d : d)) * (T(1) / T(F * F)), sx[r * SX + c], v);
            }
            const int I = (x0 >> LV) + c, J = (y0 >> LV) + m;
            const int pl = (c == SX - 1 ? 1 : 0) + (m == SY - 1 ? 2 : 0);
            const long long pn = (long long)(my + 1) * p.ldc;
            (void)pn;
            if (I >= 1 && I <= mx - 1 && J >= 1 && J <= my - 1 &&
                QG_IN((long long)J * p.ldc + I, pn, 89))
                p.part[pl][(size_t)J * p.ldc + I] = v;
        }
    }
}

template <typename T, int LV>
cudaError_t launch_lv(const FusedParams<T>& p, cudaStream_t s) {
    constexpr int NY = NodeRows<LV>::value;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((p.nx + NX - 1) / NX, (p.ny + NY - 1) / NY);
    cfg.blockDim = dim3(NX * NY);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, node_stage_kernel<T, LV>, p);
}

}  // namespace

int node_tile_rows(int levels) { return levels == 4 ? 16 : 8; }
int node_tile_cols() { return NX; }

template <typename T>
cudaError_t launch_fine_node(const FusedParams<T>& p, int levels, cudaStream_t s) {
    switch (levels) {
        case 0: return launch_lv<T, 0>(p, s);
        case 1: return launch_lv<T, 1>(p, s);
        case 2: return launch_lv<T, 2>(p, s);
        case 3: return launch_lv<T, 3>(p, s);
        case 4: return launch_lv<T, 4>(p, s);
        default: return cudaErrorInvalidValue;
    }
}

template cudaError_t launch_fine_node<float>(const FusedParams<float>&, int, cudaStream_t);
template cudaError_t launch_fine_node<double>(const FusedParams<double>&, int, cudaStream_t);

QG_BOUNDS_QUERY(bounds_site_node)

}  // namespace qg
