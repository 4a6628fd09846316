// Geometric multigrid for the elliptic sub-problem (Section 3: the CGP step
// does not depend on which Poisson solver runs on the coarse grid; the paper
// names the V-cycle multigrid as the solver of choice where sine transforms
// do not apply).
//
// lap_h psi = f on an mx x my grid of intervals with psi = 0 on the walls
// (the 5-point operator whose eigenvalues Eq. ialpha gives, Section 4.3,
// with the grid's own spacings).  One V(2,2)
// cycle:
//   - two red-black Gauss-Seidel sweeps (each point solves its own 5-point
//     equation for the current neighbours);
//   - the residual r = f - lap_h psi restricted to the next grid by full
//     weighting, the operator of Eq. res (fine wall residuals are zero);
//   - the coarse-grid correction (recursively, from a zero guess);
//   - the correction prolonged by bilinear interpolation, the operator of
//     Eq. pro, and added;
//   - two more sweeps.
// Grids are halved until the shorter side has 2 intervals; there the
// unknowns form one line and the 5-point equations a tridiagonal system,
// solved exactly (Thomas algorithm).
//
// The grids are small (512 x 1024: 2 MB a field) and every half sweep depends
// on the one before, so launches are the bound: one per operation, ten a
// level, took 146 us a cycle on 512 x 1024 (in a step of 1024 x 2048, l = 1,
// with the cycle's share of the fine stage).  A level takes two launches
// instead: 70 us.  A CTA loads a tile of 32 x 32 nodes with a halo as wide as the half
// sweeps (and the residual's restriction) reach, and does them all in shared
// memory; the halo's nodes are updated by every CTA that holds them, from the
// same values in the same order, so the result is that of the whole-grid
// sweeps.  The tiles of a launch read one array and write another.  The
// halo costs 1.9 times the arithmetic on the way down and 1.6 on the way up,
// which the saved passes over the grid repay on large grids too.  The levels
// from `tail` down run in one CTA out of shared memory.
#include <cuda_runtime.h>

#include <mutex>

#include "bounds.cuh"
#include "qg_internal.cuh"

namespace qg {
namespace {

constexpr int kPre = 2, kPost = 2;

template <typename T>
struct Grid {
    T* psi;
    const T* rhs;
    int mx, my, ld, ldr;   // intervals, pitch of psi, pitch of rhs
    T cx, cy;              // 1/dx^2, 1/dy^2
};

// ---- one operation on one grid, for a range of threads ---------------
// (the tail kernel's)

template <typename T>
__device__ __forceinline__ void rb_half(const Grid<T>& g, int color, int tid, int nthr) {
    const int hw = g.mx / 2;                   // points of one colour per row (upper bound)
    const int lh = 31 - __clz(hw);             // (sides are powers of two)
    const int n = hw * (g.my - 1);
    const T inv = T(1) / (T(2) * (g.cx + g.cy));
    for (int e = tid; e < n; e += nthr) {
        const int j = 1 + (e >> lh);
        const int i = 2 * (e & (hw - 1)) + (((1 + j) & 1) == color ? 1 : 2);
        if (i > g.mx - 1) continue;
        const long long o = (long long)j * g.ld + i, n = (long long)(g.my + 1) * g.ld;
        if (!(QG_IN(o - g.ld, n, 91) && QG_IN(o + g.ld, n, 91) &&
              QG_IN((long long)j * g.ldr + i, (long long)(g.my + 1) * g.ldr, 92)))
            continue;
        T* p = g.psi + (size_t)j * g.ld + i;
        const T f = g.rhs[(size_t)j * g.ldr + i];
        p[0] = (g.cx * (p[-1] + p[1]) + g.cy * (p[-g.ld] + p[g.ld]) - f) * inv;
    }
}

// lap_h psi at p, from the differences to the neighbours: where psi is smooth
// they are exact, while (p[-1] + p[1]) - 2 p[0] rounds a sum of the size of
// 2 psi that 1/dx^2 then multiplies.  On 512 x 1024 in FP32 that rounding held
// psi's error between 2e-6 and 1e-5 however many cycles ran; with the
// differences it is 5.5e-8 from the sixth cycle on.  (One operation more a
// direction, in a phase that waits for shared memory.)
template <typename T>
__device__ __forceinline__ T lap_at(const Grid<T>& g, const T* p, int ld) {
    const T c = p[0];
    return g.cx * ((p[-1] - c) + (p[1] - c)) + g.cy * ((p[-ld] - c) + (p[ld] - c));
}

template <typename T>
__device__ __forceinline__ T residual_at(const Grid<T>& g, int i, int j) {
    if (i < 1 || j < 1 || i > g.mx - 1 || j > g.my - 1) return T(0);
    const long long o = (long long)j * g.ld + i, n = (long long)(g.my + 1) * g.ld;
    if (!(QG_IN(o - g.ld, n, 93) && QG_IN(o + g.ld, n, 93) &&
          QG_IN((long long)j * g.ldr + i, (long long)(g.my + 1) * g.ldr, 93)))
        return T(0);
    const T* p = g.psi + (size_t)j * g.ld + i;
    return g.rhs[(size_t)j * g.ldr + i] - lap_at(g, p, g.ld);
}

// coarse f = R(f - lap_h psi) (Eq. res on the residual), coarse psi = 0
template <typename T>
__device__ __forceinline__ void restrict_residual(const Grid<T>& g, T* cf, T* cpsi, int cmx,
                                                  int cmy, int cld, int tid, int nthr) {
    const int n = cmx * cmy, lc = 31 - __clz(cmx);   // (sides are powers of two)
    for (int e = tid; e < n; e += nthr) {
        const int I = e & (cmx - 1), J = e >> lc;
        const int i = 2 * I, j = 2 * J;
        if (I < 1 || J < 1 || !QG_IN((long long)J * cld + I, (long long)(cmy + 1) * cld, 94)) continue;
        const T c = residual_at(g, i, j);
        const T ed = residual_at(g, i - 1, j) + residual_at(g, i + 1, j) +
                     residual_at(g, i, j - 1) + residual_at(g, i, j + 1);
        const T co = residual_at(g, i - 1, j - 1) + residual_at(g, i + 1, j - 1) +
                     residual_at(g, i - 1, j + 1) + residual_at(g, i + 1, j + 1);
        cf[(size_t)J * cld + I] = (T(4) * c + T(2) * ed + co) * T(0.0625);
        cpsi[(size_t)J * cld + I] = T(0);
    }
}

// fine psi += P(coarse psi) (Eq. pro; coarse wall values are zero)
template <typename T>
__device__ __forceinline__ void prolong_add(const Grid<T>& g, const T* cpsi, int cld, int tid,
                                            int nthr) {
    const int n = g.mx * g.my, lx = 31 - __clz(g.mx);
    for (int e = tid; e < n; e += nthr) {
        const int i = e & (g.mx - 1), j = e >> lx;
        const int I = i >> 1, J = j >> 1;
        const long long cn = (long long)((g.my >> 1) + 1) * cld;
        (void)cn;
        if (i < 1 || j < 1 || !(QG_IN((long long)J * cld + I, cn, 95) && QG_IN((long long)(J + 1) * cld + I + 1, cn, 95) &&
              QG_IN((long long)j * g.ld + i, (long long)(g.my + 1) * g.ld, 96)))
            continue;
        const T* c = cpsi + (size_t)J * cld + I;
        T v;
        if (!(i & 1) && !(j & 1)) v = c[0];
        else if (!(j & 1)) v = T(0.5) * (c[0] + c[1]);
        else if (!(i & 1)) v = T(0.5) * (c[0] + c[cld]);
        else v = T(0.25) * (c[0] + c[1] + c[cld] + c[cld + 1]);
        g.psi[(size_t)j * g.ld + i] += v;
    }
}

// The coarsest grid: a shorter side of 2 intervals leaves one line of n <= 7
// unknowns u_k (the sides are within a factor 4); the walls beside it are
// zero, so its 5-point equations read  c u_{k-1} + d u_k + c u_{k+1} = f_k,
// d = -2 (cx + cy), c the coefficient along the line.  Forward elimination
// and back substitution (one thread; |d| > 2c keeps it stable).
template <typename T>
__device__ void line_solve(const Grid<T>& g) {
    const bool along_y = g.mx == 2;
    const int n = along_y ? g.my - 1 : g.mx - 1;
    if (n > 8) return;
    const T c = along_y ? g.cy : g.cx;
    const T d = -T(2) * (g.cx + g.cy);
    auto u = [&](int k) -> T& {
        return along_y ? g.psi[(size_t)(k + 1) * g.ld + 1] : g.psi[(size_t)g.ld + k + 1];
    };
    auto f = [&](int k) -> T {
        return along_y ? g.rhs[(size_t)(k + 1) * g.ldr + 1] : g.rhs[(size_t)g.ldr + k + 1];
    };
    T cs[8];
    T cprev = T(0), uprev = T(0);
    for (int k = 0; k < n; ++k) {
        const T den = d - c * cprev;
        cs[k] = c / den;
        uprev = (f(k) - c * uprev) / den;
        u(k) = uprev;
        cprev = cs[k];
    }
    for (int k = n - 2; k >= 0; --k) u(k) -= cs[k] * u(k + 1);
}

// ---- per-level kernels ---------------------------------------------------

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

constexpr int TW = 32;                        // tile sides
constexpr int kThreads = 256;

// A tile and its halo of HALO nodes in shared memory: local node (c, r) is
// node (x0 - HALO + c, y0 - HALO + r).
template <typename T, int HALO>
struct Patch {
    static constexpr int W = TW + 2 * HALO, P = W + 1;   // side, pitch
    T psi[W * P], rhs[W * P];
};

// SWEEPS red-black sweeps of the patch: each half sweep updates the nodes one
// node further in than the last, so that the tile (and what the caller needs
// around it) sees none of the stale border.
template <typename T, int HALO, int SWEEPS>
__device__ __forceinline__ void patch_sweeps(Patch<T, HALO>& s, const Grid<T>& g, int x0, int y0) {
    using Q = Patch<T, HALO>;
    constexpr int W = Q::W, HW = W / 2, P = Q::P;
    const T inv = T(1) / (T(2) * (g.cx + g.cy));
    constexpr int ITER = (W * HW + kThreads - 1) / kThreads;
#pragma unroll
    for (int h = 1; h <= 2 * SWEEPS; ++h) {
        const int color = (h - 1) & 1;
        // (the nodes of a colour do not depend on one another: all loads first)
        T v[ITER];
        bool ok[ITER];
        int at[ITER];
#pragma unroll
        for (int k = 0; k < ITER; ++k) {
            const int e = threadIdx.x + k * kThreads;
            const int r = e / HW, j = y0 - HALO + r;
            // nodes with (i + j) mod 2 == color (x0, y0 and HALO are even)
            const int c = 2 * (e - r * HW) + ((r + color) & 1), i = x0 - HALO + c;
            ok[k] = r >= h && r < W - h && c >= h && c < W - h && i >= 1 && j >= 1 &&
                    i <= g.mx - 1 && j <= g.my - 1 && QG_IN(r * P + c - P, W * P, 91) &&
                    QG_IN(r * P + c + P, W * P, 91);
            at[k] = r * P + c;
            if (ok[k]) {
                const T* p = s.psi + at[k];
                v[k] = (g.cx * (p[-1] + p[1]) + g.cy * (p[-P] + p[P]) - s.rhs[at[k]]) * inv;
            }
        }
#pragma unroll
        for (int k = 0; k < ITER; ++k)
            if (ok[k]) s.psi[at[k]] = v[k];
        __syncthreads();
    }
}

template <typename T, int HALO>
__device__ __forceinline__ T patch_residual(const Patch<T, HALO>& s, const Grid<T>& g, int x0,
                                            int y0, int c, int r) {
    constexpr int P = Patch<T, HALO>::P, W = Patch<T, HALO>::W;
    const int i = x0 - HALO + c, j = y0 - HALO + r;
    if (i < 1 || j < 1 || i > g.mx - 1 || j > g.my - 1) return T(0);
    if (!(QG_IN(r * P + c - P, W * P, 93) && QG_IN(r * P + c + P, W * P, 93)))
        return T(0);
    return s.rhs[r * P + c] - lap_at(g, s.psi + r * P + c, P);
}

// Down: the pre-smoothing sweeps of g (from zero when `zero`, else from
// g.psi) -> out, and the residual's restriction -> cf.
template <typename T>
__global__ void __launch_bounds__(kThreads)
mg_down_kernel(Grid<T> g, int zero, T* out, T* cf, int cmx, int cmy, int cld) {
    // 2 kPre half sweeps, the residual beside the tile, its stencil
    constexpr int HALO = 2 * kPre + 2;
    using Q = Patch<T, HALO>;
    __shared__ Q s;
    const int x0 = blockIdx.x * TW, y0 = blockIdx.y * TW;
    pdl_wait();
    pdl_trigger();
    constexpr int ITER = (Q::W * Q::W + kThreads - 1) / kThreads;
    T pv[ITER], fv[ITER];
#pragma unroll
    for (int k = 0; k < ITER; ++k) {
        const int e = threadIdx.x + k * kThreads;
        const int r = e / Q::W, c = e - r * Q::W, i = x0 - HALO + c, j = y0 - HALO + r;
        const bool in = r < Q::W && i >= 1 && j >= 1 && i <= g.mx - 1 && j <= g.my - 1 &&
                        QG_IN((long long)j * g.ld + i, (long long)(g.my + 1) * g.ld, 92) &&
                        QG_IN((long long)j * g.ldr + i, (long long)(g.my + 1) * g.ldr, 92);
        pv[k] = in && !zero ? g.psi[(size_t)j * g.ld + i] : T(0);
        fv[k] = in ? g.rhs[(size_t)j * g.ldr + i] : T(0);
    }
#pragma unroll
    for (int k = 0; k < ITER; ++k) {
        const int e = threadIdx.x + k * kThreads;
        const int r = e / Q::W, c = e - r * Q::W;
        if (r < Q::W) {
            s.psi[r * Q::P + c] = pv[k];
            s.rhs[r * Q::P + c] = fv[k];
        }
    }
    __syncthreads();
    patch_sweeps<T, HALO, kPre>(s, g, x0, y0);
    for (int e = threadIdx.x; e < TW * TW; e += kThreads) {
        const int c = e % TW, r = e / TW, i = x0 + c, j = y0 + r;
        if (i >= 1 && j >= 1 && i <= g.mx - 1 && j <= g.my - 1 &&
            QG_IN((long long)j * g.ld + i, (long long)(g.my + 1) * g.ld, 96))
            out[(size_t)j * g.ld + i] = s.psi[(r + HALO) * Q::P + c + HALO];
    }
    for (int e = threadIdx.x; e < TW * TW / 4; e += kThreads) {
        const int I = x0 / 2 + e % (TW / 2), J = y0 / 2 + e / (TW / 2);
        if (I < 1 || J < 1 || I > cmx - 1 || J > cmy - 1 ||
            !QG_IN((long long)J * cld + I, (long long)(cmy + 1) * cld, 94))
            continue;
        const int c = 2 * I - x0 + HALO, r = 2 * J - y0 + HALO;
        auto res = [&](int dc, int dr) { return patch_residual<T, HALO>(s, g, x0, y0, c + dc, r + dr); };
        const T ed = res(-1, 0) + res(1, 0) + res(0, -1) + res(0, 1);
        const T co = res(-1, -1) + res(1, -1) + res(-1, 1) + res(1, 1);
        cf[(size_t)J * cld + I] = (T(4) * res(0, 0) + T(2) * ed + co) * T(0.0625);
    }
}

// Up: g.psi + P(coarse psi), the post-smoothing sweeps -> out.
template <typename T>
__global__ void __launch_bounds__(kThreads)
mg_up_kernel(Grid<T> g, T* out, const T* cpsi, int cld) {
    constexpr int HALO = 2 * kPost;
    using Q = Patch<T, HALO>;
    __shared__ Q s;
    const int x0 = blockIdx.x * TW, y0 = blockIdx.y * TW;
    pdl_wait();
    pdl_trigger();
    constexpr int ITER = (Q::W * Q::W + kThreads - 1) / kThreads;
    T q[ITER][4], pv[ITER], fv[ITER];
#pragma unroll
    for (int k = 0; k < ITER; ++k) {
        const int e = threadIdx.x + k * kThreads;
        const int r = e / Q::W, c = e - r * Q::W, i = x0 - HALO + c, j = y0 - HALO + r;
        const long long cn = (long long)((g.my >> 1) + 1) * cld;
        (void)cn;
        const int I = i >> 1, J = j >> 1;
        const bool in = r < Q::W && i >= 1 && j >= 1 && i <= g.mx - 1 && j <= g.my - 1 &&
                        QG_IN((long long)(J + 1) * cld + I + 1, cn, 95) &&
                        QG_IN((long long)j * g.ld + i, (long long)(g.my + 1) * g.ld, 92);
        // the four elliptic nodes around (zero walls)
        const T* cq = cpsi + (in ? (size_t)J * cld + I : 0);
        q[k][0] = in ? cq[0] : T(0);
        q[k][1] = in ? cq[1] : T(0);
        q[k][2] = in ? cq[cld] : T(0);
        q[k][3] = in ? cq[cld + 1] : T(0);
        pv[k] = in ? g.psi[(size_t)j * g.ld + i] : T(0);
        fv[k] = in ? g.rhs[(size_t)j * g.ldr + i] : T(0);
    }
#pragma unroll
    for (int k = 0; k < ITER; ++k) {
        const int e = threadIdx.x + k * kThreads;
        const int r = e / Q::W, c = e - r * Q::W;   // (x0, y0 and HALO are even)
        const T lo = (c & 1) ? T(0.5) * (q[k][0] + q[k][1]) : q[k][0];
        const T hi = (c & 1) ? T(0.5) * (q[k][2] + q[k][3]) : q[k][2];
        pv[k] += (r & 1) ? T(0.5) * (lo + hi) : lo;
    }
#pragma unroll
    for (int k = 0; k < ITER; ++k) {
        const int e = threadIdx.x + k * kThreads;
        const int r = e / Q::W, c = e - r * Q::W;
        if (r < Q::W) {
            s.psi[r * Q::P + c] = pv[k];
            s.rhs[r * Q::P + c] = fv[k];
        }
    }
    __syncthreads();
    patch_sweeps<T, HALO, kPost>(s, g, x0, y0);
    for (int e = threadIdx.x; e < TW * TW; e += kThreads) {
        const int c = e % TW, r = e / TW, i = x0 + c, j = y0 + r;
        if (i >= 1 && j >= 1 && i <= g.mx - 1 && j <= g.my - 1 &&
            QG_IN((long long)j * g.ld + i, (long long)(g.my + 1) * g.ld, 96))
            out[(size_t)j * g.ld + i] = s.psi[(r + HALO) * Q::P + c + HALO];
    }
}

// rhs0 = P0 + P1 + ... (the restriction's partial planes, in that order),
// psi0 = 0 when `zero`
template <typename T>
__global__ void __launch_bounds__(256) mg_sum_kernel(MGSumParams<T> q) {
    const int n = q.mx * q.my, lx = 31 - __clz(q.mx);
    pdl_wait();
    pdl_trigger();
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
        const int i = e & (q.mx - 1), j = e >> lx;
        if (i < 1 || j < 1) continue;
        const size_t o = (size_t)j * q.ld_in + i;
        if (!(QG_IN((long long)o, (long long)(q.my + 1) * q.ld_in, 90) &&
              QG_IN((long long)j * q.ld + i, (long long)(q.my + 1) * q.ld, 90)))
            continue;
        T v = q.in[0][o];
        for (int k = 1; k < q.nin; ++k) v = v + q.in[k][o];
        q.rhs[(size_t)j * q.ld + i] = v;
        if (q.zero) q.psi[(size_t)j * q.ld + i] = T(0);
    }
}

constexpr int kTailThreads = 512;

// ---- the tail: levels t..C in one CTA, out of shared memory -------------
// On entry psi_t (global) holds the initial guess (zero: a.zero) and rhs_t (global) the
// right-hand side; one V-cycle over levels t..C; psi_t is written back.
template <typename T>
__global__ void __launch_bounds__(kTailThreads) mg_tail_kernel(MGTail<T> a) {
    extern __shared__ __align__(16) unsigned char smem[];
    T* base = reinterpret_cast<T*>(smem);
    const int tid = threadIdx.x, nthr = blockDim.x;
    // smem layout: for each level k: psi[(my+1)(mx+1)], rhs[(my+1)(mx+1)]
    Grid<T> g[kMaxTail];
    size_t off = 0;
    for (int k = 0; k < a.n; ++k) {
        const int ld = a.mx[k] + 1;
        const size_t sz = (size_t)(a.my[k] + 1) * ld;
        g[k].psi = base + off;
        g[k].rhs = base + off + sz;
        g[k].mx = a.mx[k];
        g[k].my = a.my[k];
        g[k].ld = g[k].ldr = ld;
        g[k].cx = a.cx[k];
        g[k].cy = a.cy[k];
        off += 2 * sz;
    }
#ifdef QG_BOUNDS_CHECK
    {
        // the levels' arrays inside the launch's dynamic shared memory (the
        // same test in every thread)
        unsigned dyn;
        asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn));
        if (!QG_IN((long long)(off * sizeof(T)) - 1, (long long)dyn, 97)) return;
    }
#endif
    for (size_t e = tid; e < off; e += nthr) base[e] = T(0);
    __syncthreads();
    pdl_wait();
    pdl_trigger();
    {
        const int n = a.mx[0] * a.my[0], lx = 31 - __clz(a.mx[0]), ld0 = g[0].ld;
        T* rhs0 = const_cast<T*>(g[0].rhs);
        constexpr int U = 4;                      // loads in flight
        for (int e0 = tid; e0 < n; e0 += U * nthr) {
            T pv[U], fv[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int e = e0 + u * nthr, i = e & (a.mx[0] - 1), j = e >> lx;
                const bool in = e < n && i >= 1 && j >= 1 &&
                                QG_IN((long long)j * a.ld + i, (long long)(a.my[0] + 1) * a.ld, 98) &&
                                QG_IN((long long)j * a.ldr + i, (long long)(a.my[0] + 1) * a.ldr, 98);
                pv[u] = in && !a.zero ? a.psi[(size_t)j * a.ld + i] : T(0);
                fv[u] = in ? a.rhs[(size_t)j * a.ldr + i] : T(0);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int e = e0 + u * nthr, i = e & (a.mx[0] - 1), j = e >> lx;
                if (e < n) {
                    g[0].psi[j * ld0 + i] = pv[u];
                    rhs0[j * ld0 + i] = fv[u];
                }
            }
        }
    }
    __syncthreads();
    for (int k = 0; k + 1 < a.n; ++k) {
        for (int s = 0; s < kPre; ++s)
            for (int c = 0; c < 2; ++c) {
                rb_half(g[k], c, tid, nthr);
                __syncthreads();
            }
        restrict_residual(g[k], const_cast<T*>(g[k + 1].rhs), g[k + 1].psi, g[k + 1].mx,
                          g[k + 1].my, g[k + 1].ld, tid, nthr);
        __syncthreads();
    }
    if (tid == 0) line_solve(g[a.n - 1]);
    __syncthreads();
    for (int k = a.n - 2; k >= 0; --k) {
        prolong_add(g[k], g[k + 1].psi, g[k + 1].ld, tid, nthr);
        __syncthreads();
        for (int s = 0; s < kPost; ++s)
            for (int c = 0; c < 2; ++c) {
                rb_half(g[k], c, tid, nthr);
                __syncthreads();
            }
    }
    const int n = a.mx[0] * a.my[0], lx = 31 - __clz(a.mx[0]);
    for (int e = tid; e < n; e += nthr) {
        const int i = e & (a.mx[0] - 1), j = e >> lx;
        if (i < 1 || j < 1) continue;
        if (!QG_IN((long long)j * a.ld + i, (long long)(a.my[0] + 1) * a.ld, 99)) continue;
        a.psi[(size_t)j * a.ld + i] = g[0].psi[(size_t)j * g[0].ld + i];
    }
}

int blocks_for(long n) {
    long b = (n + 255) / 256;
    if (b < 1) b = 1;
    if (b > 4096) b = 4096;
    return (int)b;
}

}  // namespace

// The tail kernel's shared-memory limit, raised once per process to the
// most any hierarchy uses (called when a hierarchy is built, outside any
// stream capture).
cudaError_t mg_reserve_tail_smem(size_t bytes, size_t esz) {
    static std::mutex mu;             // handles on other host threads share it
    static size_t have[2] = {0, 0};
    std::lock_guard<std::mutex> lock(mu);
    const int k = esz == 8 ? 1 : 0;
    if (bytes <= have[k]) return cudaSuccess;
    const cudaError_t e =
        esz == 8 ? cudaFuncSetAttribute(mg_tail_kernel<double>,
                                        cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes)
                 : cudaFuncSetAttribute(mg_tail_kernel<float>,
                                        cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) have[k] = bytes;
    return e;
}

int mg_cycle_launches(int tail) { return 2 * tail + 1; }

size_t mg_tail_smem(const int* mx, const int* my, int n, size_t esz) {
    size_t s = 0;
    for (int k = 0; k < n; ++k) s += 2 * (size_t)(mx[k] + 1) * (my[k] + 1) * esz;
    return s;
}

// A launch that depends programmatically on the one before it.
template <typename... P, typename... A>
static cudaError_t launch(void (*k)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s,
                          const A&... a) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, P(a)...);
}

template <typename T>
cudaError_t launch_mg_sum(const MGSumParams<T>& q, cudaStream_t s) {
    return launch(mg_sum_kernel<T>, dim3(blocks_for((long)q.mx * q.my)), 256, 0, s, q);
}

// One V-cycle.  lv[0..nl): the grids (psi, psi2, rhs, sizes, pitches, 1/dx^2,
// 1/dy^2); the levels from `tail` on are the tail's.  Level 0 starts from its
// psi, the others from zero; every level's result is in psi (its smoothed
// state on the way down in psi2).
template <typename T>
cudaError_t launch_mg_cycle(const MGLevelDesc<T>* lv, int nl, int tail, cudaStream_t s) {
    auto grid = [&](int k, T* psi) {
        Grid<T> g;
        g.psi = psi;
        g.rhs = lv[k].rhs;
        g.mx = lv[k].mx;
        g.my = lv[k].my;
        g.ld = lv[k].ld;
        g.ldr = lv[k].ldr;
        g.cx = lv[k].cx;
        g.cy = lv[k].cy;
        return g;
    };
    auto tiles = [&](int k) { return dim3((lv[k].mx + TW - 1) / TW, (lv[k].my + TW - 1) / TW); };
    cudaError_t e = cudaSuccess;
    for (int k = 0; k < tail && e == cudaSuccess; ++k)
        e = launch(mg_down_kernel<T>, tiles(k), kThreads, 0, s, grid(k, lv[k].psi), k > 0 ? 1 : 0,
                   lv[k].psi2, lv[k + 1].rhs_w, lv[k + 1].mx, lv[k + 1].my, lv[k + 1].ld);
    if (e != cudaSuccess) return e;
    MGTail<T> a = {};
    a.n = nl - tail;
    if (a.n > kMaxTail) return cudaErrorInvalidValue;
    for (int k = 0; k < a.n; ++k) {
        a.mx[k] = lv[tail + k].mx;
        a.my[k] = lv[tail + k].my;
        a.cx[k] = lv[tail + k].cx;
        a.cy[k] = lv[tail + k].cy;
    }
    a.psi = lv[tail].psi;
    a.rhs = lv[tail].rhs;
    a.ld = lv[tail].ld;
    a.ldr = lv[tail].ldr;
    a.zero = tail > 0 ? 1 : 0;
    e = launch(mg_tail_kernel<T>, dim3(1), kTailThreads, mg_tail_smem(a.mx, a.my, a.n, sizeof(T)), s, a);
    for (int k = tail - 1; k >= 0 && e == cudaSuccess; --k)
        e = launch(mg_up_kernel<T>, tiles(k), kThreads, 0, s, grid(k, lv[k].psi2), lv[k].psi,
                   lv[k + 1].psi, lv[k + 1].ld);
    return e;
}

QG_BOUNDS_QUERY(bounds_site_mg)

template cudaError_t launch_mg_sum<float>(const MGSumParams<float>&, cudaStream_t);
template cudaError_t launch_mg_sum<double>(const MGSumParams<double>&, cudaStream_t);
template cudaError_t launch_mg_cycle<float>(const MGLevelDesc<float>*, int, int, cudaStream_t);
template cudaError_t launch_mg_cycle<double>(const MGLevelDesc<double>*, int, int, cudaStream_t);

}  // namespace qg
