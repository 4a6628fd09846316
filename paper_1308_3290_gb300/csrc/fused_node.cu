// Fused fine-grid stage of the one-layer model with one node per thread: the
// same stage as the sweep of fused.cu (prolongation on load, Arakawa / beta /
// dissipation / forcing, the TVDRK3 combination, restriction on store) for
// grids whose sweep tiles leave most of the GPU idle.
//
// The bound is FP64: an SM sub-partition issues one FP64 warp instruction per
// ~64 clocks, so a thread that sweeps 8 rows of 4 columns (about 1600 FP64
// instructions) holds its sub-partition for some 50 us at that rate, however few tiles there
// are.  One node per thread and tiles of 16 x 8 nodes spread the same number
// of instructions (about 40 a node: the sweep's shared differences save
// little more than its halo rows cost) over every sub-partition.  64 x 128,
// l = 1, FP64: 203 us a step with the sweep and an FFT engine, 43 us with this
// stage and the sine sums of solve_dense.cu; FP32 35 and 23 to 25 us.  Which
// tile a handle takes is timed when it is created.
//
// A CTA stages w^(s) with its halo and the elliptic-grid patch (or the fine
// psi, l = 0) in shared memory, prolongs, updates its nodes and sums the
// restriction into the four planes of fused.cu (node_tile.cuh).
#include <cuda_runtime.h>

#include "node_tile.cuh"

namespace qg {
namespace {

using namespace node;

template <typename T, int LV>
__global__ void __launch_bounds__(Tile<LV>::THREADS)
node_stage_kernel(FusedParams<T> p) {
    using Q = Tile<LV>;
    constexpr int NY = Q::NY, WX = Q::WX, WY = Q::WY;
    __shared__ T sw[WY * WX], sp[WY * WX];
    __shared__ T so[LV > 0 ? NY * NX : 1], sx[LV > 0 ? NY * Q::SX : 1];
    __shared__ T cp[LV > 0 ? Q::CY * Q::CX : 1], cr[LV > 0 ? WY * Q::CX : 1];
    __shared__ T s_dt;
    const int nx = p.nx, ny = p.ny, ld = p.ld;
    const int x0 = blockIdx.x * NX, y0 = blockIdx.y * NY;
    const int i = threadIdx.x % NX, j = threadIdx.x / NX;
    const int x = x0 + i, y = y0 + j;
    const bool in = x >= 1 && x <= nx - 1 && y >= 1 && y <= ny - 1;
    const long long fine_n = (long long)(ny + 1) * ld;
    (void)fine_n;
    // w^(s), w^n and the forcing were complete before the solve began
    load_halo<T, LV>(p.w, sw, x0, y0, nx, ny, ld);
    T wn = T(0), f = T(0);
    const size_t o = (size_t)y * ld + x;
    if (in && QG_IN(o, fine_n, 132)) {
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
    if constexpr (LV == 0) {
        load_halo<T, LV>(p.psi, sp, x0, y0, nx, ny, ld);
        __syncthreads();
    } else {
        load_patch<T, LV>(p.psi, cp, x0, y0, nx, ny, p.ldp);
        prolong_halo<T, LV>(cp, cr, sp);
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
        // w^(s+1) = a w^n + b w^(s) + b dt G, the centre's weights and the order as in fused.cu
        constexpr bool kApart = sizeof(T) == 4;
        const T bdt = p.b * dt;
        const T k_lx = p.c_lapx * bdt, k_ly = p.c_lapy * bdt;
        const T k_0 = kApart ? T(-2) * (k_lx + k_ly) : fma(T(-2) * (p.c_lapx + p.c_lapy), bdt, p.b);
        T g = fma(-p.c_beta * bdt, beta, bdt * f);
        g = fma(-p.c_jac * bdt, jac, g);
        g = fma(k_0, q00, g);
        g = fma(k_ly, q01 + q0m, g);
        g = fma(k_lx, q10 + qm0, g);
        out = fma(p.a, wn, g);
        if constexpr (kApart) out = fma(p.b, q00, out);
        if (QG_IN(o, fine_n, 136)) p.wout[o] = out;
    }
    if constexpr (LV > 0) {
        so[threadIdx.x] = out;
        restrict_tile<T, LV>(so, sx, p.part, p.ldc, x0, y0, nx, ny);
    }
}

}  // namespace

int node_tile_rows(int levels) { return levels == 4 ? 16 : 8; }
int node_tile_cols() { return node::NX; }

template <typename T>
cudaError_t launch_fine_node(const FusedParams<T>& p, int levels, cudaStream_t s) {
    switch (levels) {
        case 0: return node::launch(node_stage_kernel<T, 0>, p.nx, p.ny, node_tile_rows(0), s, p);
        case 1: return node::launch(node_stage_kernel<T, 1>, p.nx, p.ny, node_tile_rows(1), s, p);
        case 2: return node::launch(node_stage_kernel<T, 2>, p.nx, p.ny, node_tile_rows(2), s, p);
        case 3: return node::launch(node_stage_kernel<T, 3>, p.nx, p.ny, node_tile_rows(3), s, p);
        case 4: return node::launch(node_stage_kernel<T, 4>, p.nx, p.ny, node_tile_rows(4), s, p);
        default: return cudaErrorInvalidValue;
    }
}

template cudaError_t launch_fine_node<float>(const FusedParams<float>&, int, cudaStream_t);
template cudaError_t launch_fine_node<double>(const FusedParams<double>&, int, cudaStream_t);

QG_BOUNDS_QUERY(bounds_site_node)

}  // namespace qg
