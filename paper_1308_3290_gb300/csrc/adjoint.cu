// Kernels of the discrete adjoint of the one-layer CGPRK3 step (the paper has
// no adjoint; these transpose the Jacobian of the step of Section 3.2).
//
// With psi = A w (A = P^l S R^l, symmetric) the transposed right-hand side is
//   G_w^T lam = J(psi, lam) + (1/Re) lap lam - A[J(w, lam) - (1/Ro) J(lam, y)],
// because J(p, .) (Arakawa's enstrophy conservation, Section 4.1) and the beta
// operator J(., y) are skew-symmetric on fields that vanish on the walls.
// Per transposed TVDRK3 stage (Eq. TVDRK in stage form w^(s+1) = a w^n +
// b (w^(s) + dt G(w^(s)))) there are two launches around the forward solve:
// adj_source computes the bracket and restricts it on store, adj_stage
// prolongs psi and the solve's result on load and assembles the stage.  The
// fields live on the elliptic grid in between (the unfused form wrote and
// read three more fine fields and took 13 launches a stage).  The grids are
// small (256 x 512: 0.6 MB a field), the launches' latency is the bound: tiles
// of 16 x 8 nodes, one thread each (node_tile.cuh), chained by programmatic
// dependent launch.  256 x 512, l = 1, 40 steps and their gradient: 15.4 ms
// unfused, 9.2 ms with these launches and the reverse steps replayed as graphs.
#include <cuda_runtime.h>

#include "arakawa.cuh"
#include "node_tile.cuh"

namespace qg {
namespace {

using namespace node;

template <typename T>
struct Nine {   // a node's nine neighbours in a halo tile of pitch W
    T m0, p0, z0, z1, mm, pm, mp, pp, c;
    __device__ __forceinline__ Nine(const T* s, int W)
        : m0(s[-1]), p0(s[1]), z0(s[-W]), z1(s[W]), mm(s[-W - 1]), pm(s[-W + 1]), mp(s[W - 1]),
          pp(s[W + 1]), c(s[0]) {}
};
template <typename T>
__device__ __forceinline__ T arakawa9(const Nine<T>& p, const Nine<T>& q) {
    return arakawa_sum(p.m0, p.p0, p.z0, p.z1, p.mm, p.pm, p.mp, p.pp, q.m0, q.p0, q.z0, q.z1,
                       q.mm, q.pm, q.mp, q.pp);
}

// U = J(w, lam) - (1/Ro) J(lam, y), restricted into the partial planes
// (l >= 1) or written to `fine` (l = 0).
template <typename T, int LV>
__global__ void __launch_bounds__(Tile<LV>::THREADS)
adj_source_kernel(const T* w, const T* lam, AdjOut<T> out, AdjParams<T> p) {
    using Q = Tile<LV>;
    __shared__ T sp[Q::WY * Q::WX], sq[Q::WY * Q::WX];
    __shared__ T so[LV > 0 ? Q::THREADS : 1], sx[LV > 0 ? Q::NY * Q::SX : 1];
    const int x0 = blockIdx.x * NX, y0 = blockIdx.y * Q::NY;
    const int i = threadIdx.x % NX, j = threadIdx.x / NX, x = x0 + i, y = y0 + j;
    pdl_wait();
    pdl_trigger();
    load_halo<T, LV>(w, sp, x0, y0, p.nx, p.ny, p.ld);
    load_halo<T, LV>(lam, sq, x0, y0, p.nx, p.ny, p.ld);
    __syncthreads();
    T u = T(0);
    const size_t o = (size_t)y * p.ld + x;
    if (x >= 1 && x <= p.nx - 1 && y >= 1 && y <= p.ny - 1) {
        const Nine<T> P(sp + (j + 1) * Q::WX + i + 1, Q::WX), L(sq + (j + 1) * Q::WX + i + 1, Q::WX);
        // (1/Ro) J(lam, y): the closed form (4 c_j + c_{j+1} + c_{j-1}) / (6 Ro)
        // with c the central x difference of lam
        const T beta = (T(4) * (L.p0 - L.m0) + (L.pp - L.mp) + (L.pm - L.mm)) * p.c_beta;
        u = arakawa9(P, L) * p.c_jac - beta;
        if (LV == 0 && QG_IN(o, (long long)(p.ny + 1) * p.ld, 111)) out.fine[o] = u;
    }
    if constexpr (LV > 0) {
        so[threadIdx.x] = u;
        restrict_tile<T, LV>(so, sx, out.part, out.ldc, x0, y0, p.nx, p.ny);
    }
}

// One transposed TVDRK3 stage: next = b lam + b dt v,
//   v = J(psi, lam) + (1/Re) lap lam - phi      (phi = A of adj_source),
// psi and phi prolonged on load.  The step's first stage (the last to be
// reversed; f.g non-null) adds what the others send to w^n, a_2 lam_2 +
// a_1 lam_1, and the forcing gradient of all three, dt (b_2 lam_2 + b_1 lam_1
// + b lam); lam_2 may be next itself.
template <typename T, int LV>
__global__ void __launch_bounds__(Tile<LV>::THREADS)
adj_stage_kernel(const T* psi, const T* phi, int ldp, const T* lam, T* next, AdjFirst<T> f,
                 AdjParams<T> p) {
    using Q = Tile<LV>;
    __shared__ T sp[Q::WY * Q::WX], sq[Q::WY * Q::WX];
    __shared__ T cp[LV > 0 ? Q::CY * Q::CX : 1], cr[LV > 0 ? Q::WY * Q::CX : 1];
    __shared__ T cf[LV > 0 ? Q::CY * Q::CX : 1];
    const int x0 = blockIdx.x * NX, y0 = blockIdx.y * Q::NY;
    const int i = threadIdx.x % NX, j = threadIdx.x / NX, x = x0 + i, y = y0 + j;
    pdl_wait();
    pdl_trigger();
    load_halo<T, LV>(lam, sq, x0, y0, p.nx, p.ny, p.ld);
    if constexpr (LV == 0) {
        load_halo<T, LV>(psi, sp, x0, y0, p.nx, p.ny, p.ld);
        __syncthreads();
    } else {
        load_patch<T, LV>(psi, cp, x0, y0, p.nx, p.ny, ldp);
        load_patch<T, LV>(phi, cf, x0, y0, p.nx, p.ny, ldp);
        prolong_halo<T, LV>(cp, cr, sp);
    }
    const size_t o = (size_t)y * p.ld + x;
    if (!(x >= 1 && x <= p.nx - 1 && y >= 1 && y <= p.ny - 1) ||
        !QG_IN(o, (long long)(p.ny + 1) * p.ld, 111))
        return;
    const Nine<T> P(sp + (j + 1) * Q::WX + i + 1, Q::WX), L(sq + (j + 1) * Q::WX + i + 1, Q::WX);
    T ph;
    if constexpr (LV == 0) ph = phi[o];
    else ph = prolong_own<T, LV>(cf, i, j);
    const T lap = (L.p0 + L.m0 - T(2) * L.c) * p.c_lapx + (L.z1 + L.z0 - T(2) * L.c) * p.c_lapy;
    const T v = arakawa9(P, L) * p.c_jac + lap - ph;
    T out = p.b * (L.c + p.dt * v);
    if (f.g) {
        const T l2 = f.lam2[o], l1 = f.lam1[o];
        out += f.a2 * l2 + f.a1 * l1;
        f.g[o] += p.dt * (f.b2 * l2 + f.b1 * l1 + p.b * L.c);
    }
    next[o] = out;
}

// -dx dy lap psi (dE/dpsi of E = 1/2 dx dy sum over edges of the squared
// one-sided differences, = -1/2 dx dy sum psi lap psi with zero walls), psi
// prolonged on load, restricted on store as in adj_source.
template <typename T, int LV>
__global__ void __launch_bounds__(Tile<LV>::THREADS)
energy_source_kernel(const T* psi, int ldp, AdjOut<T> out, AdjParams<T> p) {
    using Q = Tile<LV>;
    __shared__ T sp[Q::WY * Q::WX];
    __shared__ T cp[LV > 0 ? Q::CY * Q::CX : 1], cr[LV > 0 ? Q::WY * Q::CX : 1];
    __shared__ T so[LV > 0 ? Q::THREADS : 1], sx[LV > 0 ? Q::NY * Q::SX : 1];
    const int x0 = blockIdx.x * NX, y0 = blockIdx.y * Q::NY;
    const int i = threadIdx.x % NX, j = threadIdx.x / NX, x = x0 + i, y = y0 + j;
    pdl_wait();
    pdl_trigger();
    if constexpr (LV == 0) {
        load_halo<T, LV>(psi, sp, x0, y0, p.nx, p.ny, p.ld);
        __syncthreads();
    } else {
        load_patch<T, LV>(psi, cp, x0, y0, p.nx, p.ny, ldp);
        prolong_halo<T, LV>(cp, cr, sp);
    }
    T u = T(0);
    const size_t o = (size_t)y * p.ld + x;
    if (x >= 1 && x <= p.nx - 1 && y >= 1 && y <= p.ny - 1) {
        const T* s = sp + (j + 1) * Q::WX + i + 1;
        const T lap = (s[1] + s[-1] - T(2) * s[0]) * p.inv_dx2 +
                      (s[Q::WX] + s[-Q::WX] - T(2) * s[0]) * p.inv_dy2;
        u = -p.dxdy * lap;
        if (LV == 0 && QG_IN(o, (long long)(p.ny + 1) * p.ld, 111)) out.fine[o] = u;
    }
    if constexpr (LV > 0) {
        so[threadIdx.x] = u;
        restrict_tile<T, LV>(so, sx, out.part, out.ldc, x0, y0, p.nx, p.ny);
    }
}

// dense[(j-1)(nx-1) + i-1] += scale * (c prolonged `levels` times)(i, j)
template <typename T>
__global__ void add_prolonged_kernel(T* dense, const T* __restrict__ c, int ldc, T scale, int nx,
                                     int ny, int levels) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x + 1;
    const int j = blockIdx.y * blockDim.y + threadIdx.y + 1;
    if (i >= nx || j >= ny) return;
    const int f = 1 << levels, I = i >> levels, J = j >> levels;
    const size_t q = (size_t)J * ldc + I;
    const long long cn = (long long)((ny >> levels) + 1) * ldc;
    (void)cn;
    if (!QG_IN((long long)q + (levels ? ldc + 1 : 0), cn, 112) ||
        !QG_IN((long long)(j - 1) * (nx - 1) + (i - 1), (long long)(nx - 1) * (ny - 1), 112))
        return;
    T v = c[q];
    if (levels) {
        const T a = T(i & (f - 1)) / T(f), b = T(j & (f - 1)) / T(f);
        const T lo = fma(a, c[q + 1], (T(1) - a) * v);
        const T hi = fma(a, c[q + ldc + 1], (T(1) - a) * c[q + ldc]);
        v = fma(b, hi, (T(1) - b) * lo);
    }
    dense[(size_t)(j - 1) * (nx - 1) + (i - 1)] += scale * v;
}

}  // namespace

#define QG_BY_LEVEL(CALL)            \
    switch (levels) {                \
        case 0: return CALL(0);      \
        case 1: return CALL(1);      \
        case 2: return CALL(2);      \
        case 3: return CALL(3);      \
        case 4: return CALL(4);      \
        default: return cudaErrorInvalidValue; \
    }

template <typename T>
cudaError_t launch_adj_source(const T* w, const T* lam, const AdjOut<T>& out,
                              const AdjParams<T>& p, int levels, cudaStream_t s) {
#define CALL(L) node::launch(adj_source_kernel<T, L>, p.nx, p.ny, Tile<L>::NY, s, w, lam, out, p)
    QG_BY_LEVEL(CALL)
#undef CALL
}

template <typename T>
cudaError_t launch_adj_stage(const T* psi, const T* phi, int ldp, const T* lam, T* next,
                             const AdjFirst<T>& f, const AdjParams<T>& p, int levels,
                             cudaStream_t s) {
#define CALL(L) \
    node::launch(adj_stage_kernel<T, L>, p.nx, p.ny, Tile<L>::NY, s, psi, phi, ldp, lam, next, f, p)
    QG_BY_LEVEL(CALL)
#undef CALL
}

template <typename T>
cudaError_t launch_energy_source(const T* psi, int ldp, const AdjOut<T>& out,
                                 const AdjParams<T>& p, int levels, cudaStream_t s) {
#define CALL(L) node::launch(energy_source_kernel<T, L>, p.nx, p.ny, Tile<L>::NY, s, psi, ldp, out, p)
    QG_BY_LEVEL(CALL)
#undef CALL
}

template <typename T>
cudaError_t launch_add_prolonged(T* dense, const T* c, int ldc, double scale, int nx, int ny,
                                 int levels, cudaStream_t s) {
    const dim3 b(32, 8), g((nx - 1 + 31) / 32, (ny - 1 + 7) / 8);
    add_prolonged_kernel<T><<<g, b, 0, s>>>(dense, c, ldc, (T)scale, nx, ny, levels);
    return cudaGetLastError();
}

#define QG_INST(T)                                                                          \
    template cudaError_t launch_adj_source<T>(const T*, const T*, const AdjOut<T>&,         \
                                              const AdjParams<T>&, int, cudaStream_t);      \
    template cudaError_t launch_adj_stage<T>(const T*, const T*, int, const T*, T*,         \
                                             const AdjFirst<T>&, const AdjParams<T>&, int,  \
                                             cudaStream_t);                                 \
    template cudaError_t launch_energy_source<T>(const T*, int, const AdjOut<T>&,           \
                                                 const AdjParams<T>&, int, cudaStream_t);   \
    template cudaError_t launch_add_prolonged<T>(T*, const T*, int, double, int, int, int,  \
                                                 cudaStream_t);
QG_INST(float)
QG_INST(double)
#undef QG_INST

QG_BOUNDS_QUERY(bounds_site_adjoint)

}  // namespace qg
