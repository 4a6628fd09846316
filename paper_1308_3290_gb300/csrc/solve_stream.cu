// Elliptic solve of Section 4.3 with half-length sine transforms (engine 50).
//
// The x pass of the right-hand side, the y pass with the mode-space solve of
// Eq. ialpha (or Eqs. isub-1/2 for two layers), and the inverse x pass.  Each
// is a DST-I of two real sequences a, b at once, z = a + i b, defined through
// the FFT of length L = 2N of the odd extension of z (Z_k = -2i F_k, so
// F(a)_k = -Im Z_k / 2, F(b)_k = Re Z_k / 2), but only the half that the odd
// symmetry leaves is computed:
//
//   * with G = L/16, butterfly t of the first radix-16 pass takes x[t + G r],
//     r < 16, which are z[t + G r], r < 8, and -z[c G - t], c = 16 - r <= 8:
//     no odd extension is ever stored.  Butterfly G - t is that of t with its
//     inputs reversed and negated, Y_{G-t}[s] = -e^{2 pi i s/16} Y_t[-s], so
//     only t = 0 .. G/2 are computed;
//   * the sixteen sub-transforms of length G that follow, over
//     u_s[t] = e^{-2 pi i t s/L} Y_t[s], give X[s + 16 k]; by u_s[G - t] =
//     -u_{-s}[t] and X[L - m] = -X[m] the rows s = 1..7 also hold the rows
//     16 - s, so only rows s = 0..8 are computed (rows 0 and 8 are their own
//     images and come out twice: 9/16 of the work instead of 1/2).
//
// The sine sum is symmetric, so the same factors in the opposite order
// (rows first, then the radix-16 pass over s) transform from the rows' order
// back to natural order.  Every output is a sum of products with unit-modulus
// factors (no running sum, no division by a sine), so the rounding error
// grows like log N as for the full-length FFT.
//
// Layout of the work: a pair of sequences has 9 G/16 threads.  In the radix-16
// pass thread t <= G/2 does butterfly t; in the rows thread (s, j), j < H =
// G/16, holds 16 values u_s[j + H r], does a 16-point DFT, exchanges with the
// H threads of its row (a warp or less, so no CTA barrier below L = 16384)
// and finishes with H-point DFTs (H = 32, 64: 8 x 4, 16 x 4, one more
// exchange).  One CTA barrier lies between the pass and the rows.
//
//   x forward: pass, rows;        modes in position order -> tr
//   y:         pass, rows, mode-space solve, rows, pass  -> work
//   x inverse: rows, pass                                -> out
//
// An x-mode m = s + 16 k (k < G/2) has position s G/2 + k: the order in
// which the inverse x pass's rows read, so that its loads are contiguous.
// tr and work are scratch arrays and interleave the two sequences of the
// pass that reads them (tr: [pair of positions][row][2]; work: [pair of
// rows][position][2]; two layers: [position][row][layer] and
// [row][position][layer]), so a pass loads z as one vector and the pass
// before writes runs of 4 values a pair: 32-byte sectors from two pairs on.
//
// Three launches chained by programmatic dependent launch; an ensemble group's
// batch runs as one launch, a work queue over the items of the three passes
// of every member (stream_queue_kernel).
//
// All twiddles come from one FP64-generated table per length (half_table):
// every factor is a rounded exact value.
#include <cuda_runtime.h>

#include <cmath>

#include "bounds.cuh"
#include "dst_engine.cuh"
#include "qg_internal.cuh"

namespace qg {
namespace {

using namespace eng;

// Geometry of a length L = 2^LG = 2N.
template <int LG>
struct Half {
    static constexpr int L = 1 << LG, N = L / 2, G = L / 16, H = G / 16;
    static constexpr int HC = H <= 16 ? 1 : 4, HB = H / HC;   // the rows' second DFTs
    static constexpr int TP = 9 * H;                          // threads per pair
    static constexpr int P2 = H + 1;   // pitch of a row's exchange [q][j], q < 16, j < H
    // pitch of a row: 16 P2 = G + 16, and more where several rows share a
    // half warp, so that their lanes fall on different banks
    static constexpr int RP = H == 1 ? 17 : 16 * P2 + (H <= 8 ? H : 0);
    static constexpr int BUF = 9 * RP;                        // complex elements per pair
    // table: T1[s - 1][t] = e^{-2 pi i t s/L}, s = 1..8, t <= G/2 (pitch PT);
    // T2[q - 1][j] = e^{-2 pi i q j/G}, q = 1..15, j < H;
    // T3[p][c] = e^{-2 pi i p c/H}, p < HB, c < HC (HC > 1)
    static constexpr int PT = G / 2 + 2;
    static constexpr int T2 = 8 * PT, T3 = T2 + 15 * H, TABLE = T3 + (HC > 1 ? H : 0);
};

template <typename T>
__device__ __forceinline__ Cplx<T> lds_(const CT<T>* b, int i, int lim) {
    (void)lim;
    if (!QG_IN(i, lim, 61)) return Cplx<T>{T(0), T(0)};
    const CT<T> v = b[i];
    return Cplx<T>{v.x, v.y};
}
template <typename T>
__device__ __forceinline__ void sts_(CT<T>* b, int i, Cplx<T> v, int lim) {
    (void)lim;
    if (!QG_IN(i, lim, 62)) return;
    CT<T> w;
    w.x = v.x;
    w.y = v.y;
    b[i] = w;
}
// a conj(w)
template <typename T>
__device__ __forceinline__ Cplx<T> cmulc(Cplx<T> a, Cplx<T> w) {
    return {a.x * w.x + a.y * w.y, a.y * w.x - a.x * w.y};
}
template <typename T>
__device__ __forceinline__ Cplx<T> ldt(const CT<T>* t, int i, int lim) {
    (void)lim;
    if (!QG_IN(i, lim, 68)) return Cplx<T>{T(1), T(0)};
    const CT<T> v = __ldg(t + i);
    return Cplx<T>{v.x, v.y};
}

// The outputs of dft<R> in natural order.
template <typename T, int R>
__device__ __forceinline__ void dft_nat(Cplx<T>* v) {
    dft<T, R>(v);
    if constexpr (R >= 8) {
        Cplx<T> o[R];
#pragma unroll
        for (int r = 0; r < R; ++r) o[r] = v[out_slot<R>(r)];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = o[r];
    }
}

// Threads of one row: a warp's lanes (H <= 32), else (H = 64) two warps,
// which meet at the CTA barrier (every thread of the CTA runs the same
// stages).
template <int LG>
__device__ __forceinline__ void row_sync() {
    if constexpr (Half<LG>::H > 32) __syncthreads();
    else if constexpr (Half<LG>::H > 1) __syncwarp();
}

// Radix-16 pass: v[r] = x[t + G r] -> u_s[t] and u_s[G - t] of the rows
// s = 0..8 in buf (t <= G/2).
template <typename T, int LG>
__device__ __forceinline__ void pass_fwd(Cplx<T> (&v)[16], CT<T>* buf, int t,
                                         const CT<T>* __restrict__ tab) {
    using Q = Half<LG>;
    dft_nat<T, 16>(v);
    const bool both = t > 0 && t < Q::G / 2;
#pragma unroll
    for (int s = 0; s <= 8; ++s) {
        Cplx<T> a = v[s], b = v[(16 - s) & 15];
        if (s > 0) {
            const Cplx<T> w = ldt<T>(tab, (s - 1) * Q::PT + t, Q::TABLE);
            a = cmul(a, w.x, w.y);
            b = cmulc(b, w);
        }
        sts_<T>(buf, s * Q::RP + t, a, Q::BUF);
        if (both) sts_<T>(buf, s * Q::RP + Q::G - t, Cplx<T>{-b.x, -b.y}, Q::BUF);
    }
}

// The transposed pass: rows V_s[t], V_s[G - t] in buf -> v[r] = z[t + G r]
// (r >= 8: -z[(16 - r) G - t]), t <= G/2.
template <typename T, int LG>
__device__ __forceinline__ void pass_bwd(Cplx<T> (&v)[16], const CT<T>* buf, int t,
                                         const CT<T>* __restrict__ tab) {
    using Q = Half<LG>;
    const int tm = t == 0 ? 0 : Q::G - t;
    v[0] = lds_<T>(buf, t, Q::BUF);
#pragma unroll
    for (int s = 1; s <= 8; ++s) {
        const Cplx<T> w = ldt<T>(tab, (s - 1) * Q::PT + t, Q::TABLE);
        const Cplx<T> a = lds_<T>(buf, s * Q::RP + t, Q::BUF);
        v[s] = cmul(a, w.x, w.y);
        if (s < 8) {
            const Cplx<T> b = cmulc(lds_<T>(buf, s * Q::RP + tm, Q::BUF), w);
            v[16 - s] = Cplx<T>{-b.x, -b.y};
        }
    }
    dft_nat<T, 16>(v);
}

// The index k (of X[s + 16 k]) of register i of thread j of a row.
template <int LG>
__device__ __forceinline__ int row_k(int j, int i) {
    using Q = Half<LG>;
    if constexpr (Q::HC == 1) {
        return j + (i / Q::H) * Q::H + 16 * (i % Q::H);
    } else {
        const int p1 = (j >> 4) + (Q::H / 16) * (i >> 2);
        return (j & 15) + 16 * (p1 + Q::HB * (i & 3));
    }
}

// Its part that does not depend on the thread: k = 0 and k = G/2 (the walls of
// row 0) lie at j = 0 of the registers whose part is 0 and G/2.
template <int LG>
__host__ __device__ constexpr int row_k0(int i) {
    using Q = Half<LG>;
    return Q::HC == 1 ? (i / Q::H) * Q::H + 16 * (i % Q::H)
                      : 16 * ((Q::H / 16) * (i >> 2) + Q::HB * (i & 3));
}

// Whether that index is below G/2, the same for every thread.
template <int LG>
__host__ __device__ constexpr bool row_low(int i) {
    using Q = Half<LG>;
    return Q::H == 1 ? i < 8 : Q::HC == 1 ? i % Q::H < Q::H / 2 : (i & 3) < 2;
}

// Row transform, natural order to row_k order: v[r] = u[j + H r] on entry;
// row: the row's G + 16 elements of shared memory (its values have been
// read).
template <typename T, int LG>
__device__ __forceinline__ void row_fwd(Cplx<T> (&v)[16], CT<T>* row, int j,
                                        const CT<T>* __restrict__ tab) {
    using Q = Half<LG>;
    constexpr int H = Q::H, P2 = Q::P2, LIM = Q::RP;
    dft_nat<T, 16>(v);
    if constexpr (H > 1) {
#pragma unroll
        for (int q = 1; q < 16; ++q) {
            const Cplx<T> w = ldt<T>(tab + Q::T2, (q - 1) * H + j, Q::TABLE - Q::T2);
            v[q] = cmul(v[q], w.x, w.y);
        }
        row_sync<LG>();   // every thread of the row has read its values
#pragma unroll
        for (int q = 0; q < 16; ++q) sts_<T>(row, q * P2 + j, v[q], LIM);
        row_sync<LG>();
        if constexpr (Q::HC == 1) {
#pragma unroll
            for (int b = 0; b < 16 / H; ++b) {
#pragma unroll
                for (int e = 0; e < H; ++e)
                    v[b * H + e] = lds_<T>(row, (j + H * b) * P2 + e, LIM);
                dft_nat<T, H>(v + b * H);
            }
        } else {
            constexpr int HB = Q::HB, NB = 16 / HB;
            const int q = j & 15;
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                const int c = (j >> 4) + (H / 16) * b;   // j0
#pragma unroll
                for (int e = 0; e < HB; ++e)
                    v[b * HB + e] = lds_<T>(row, q * P2 + c + 4 * e, LIM);
                dft_nat<T, HB>(v + b * HB);
#pragma unroll
                for (int e = 0; e < HB; ++e) {
                    if (e > 0) {
                        const Cplx<T> w = ldt<T>(tab + Q::T3, e * 4 + c, Q::TABLE - Q::T3);
                        v[b * HB + e] = cmul(v[b * HB + e], w.x, w.y);
                    }
                    sts_<T>(row, q * P2 + c + 4 * e, v[b * HB + e], LIM);   // in place
                }
            }
            row_sync<LG>();
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int p = (j >> 4) + (H / 16) * b;
#pragma unroll
                for (int e = 0; e < 4; ++e) v[b * 4 + e] = lds_<T>(row, q * P2 + 4 * p + e, LIM);
                dft_nat<T, 4>(v + b * 4);
            }
        }
    }
}

// The same transform from row_k order to natural order: v[r] = V[j + H r]
// on return.
template <typename T, int LG>
__device__ __forceinline__ void row_bwd(Cplx<T> (&v)[16], CT<T>* row, int j,
                                        const CT<T>* __restrict__ tab) {
    using Q = Half<LG>;
    constexpr int H = Q::H, P2 = Q::P2, LIM = Q::RP;
    if constexpr (H > 1) {
        if constexpr (Q::HC == 1) {
            row_sync<LG>();   // row_fwd's reads are done
#pragma unroll
            for (int b = 0; b < 16 / H; ++b) {
                dft_nat<T, H>(v + b * H);
#pragma unroll
                for (int e = 0; e < H; ++e)
                    sts_<T>(row, (j + H * b) * P2 + e, v[b * H + e], LIM);
            }
        } else {
            constexpr int HB = Q::HB, NB = 16 / HB;
            const int q = j & 15;
            row_sync<LG>();
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int p = (j >> 4) + (H / 16) * b;
                dft_nat<T, 4>(v + b * 4);
#pragma unroll
                for (int e = 0; e < 4; ++e) sts_<T>(row, q * P2 + 4 * p + e, v[b * 4 + e], LIM);
            }
            row_sync<LG>();
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                const int c = (j >> 4) + (H / 16) * b;
#pragma unroll
                for (int e = 0; e < HB; ++e) {
                    v[b * HB + e] = lds_<T>(row, q * P2 + c + 4 * e, LIM);
                    if (e > 0) {
                        const Cplx<T> w = ldt<T>(tab + Q::T3, e * 4 + c, Q::TABLE - Q::T3);
                        v[b * HB + e] = cmul(v[b * HB + e], w.x, w.y);
                    }
                }
                dft_nat<T, HB>(v + b * HB);
#pragma unroll
                for (int e = 0; e < HB; ++e)
                    sts_<T>(row, q * P2 + c + 4 * e, v[b * HB + e], LIM);   // in place
            }
        }
        row_sync<LG>();
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            v[q] = lds_<T>(row, q * P2 + j, LIM);
            if (q > 0) {
                const Cplx<T> w = ldt<T>(tab + Q::T2, (q - 1) * H + j, Q::TABLE - Q::T2);
                v[q] = cmul(v[q], w.x, w.y);
            }
        }
    }
    dft_nat<T, 16>(v);
}

// Columns j = t + G r (r < 8) and c G - t (c = 16 - r) of the right-hand side
// rows ra and rb (existing: va, vb; planes ia, ib): plane 0, plus plane 2 on
// rows with row % part_py == 0, plus planes 1 and 3 at columns with column %
// part_px == 0.  One test of t serves every column where the period divides G.
// At 128 intervals G is 16 and the period of a 64-column tile at l = 1 is 32:
// there t = 0 also reads planes 1 and 3 at columns between the seams, where they
// hold zeros (testing each column cost 4 % of a 256 x 512, l = 1 step).  Eight columns at a time: the loads of all their planes are in flight
// together, within the register budget.
template <typename T, int LG>
__device__ __forceinline__ void load_rhs(const SolveParams<T>& P, const T* const (&ia)[4],
                                         const T* const (&ib)[4], int ra, int rb, bool va, bool vb,
                                         int t, Cplx<T> (&v)[16]) {
    using Q = Half<LG>;
    // (a row that does not exist reads row 0, a wall: zeros)
    const int oa = (va ? ra : 0) * P.ld, ob = (vb ? rb : 0) * P.ld;
    const bool cx = P.nin > 1 && (t & (P.part_px - 1)) == 0;
    const bool ya = P.nin > 1 && va && (ra & (P.part_py - 1)) == 0;
    const bool yb = P.nin > 1 && vb && (rb & (P.part_py - 1)) == 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        auto col = [&](int r) { return h == 0 ? t + Q::G * r : (8 - r) * Q::G - t; };
        // not a wall (z_0, z_N)
        auto ok = [&](int r) { return (t > 0 || r != 0) && QG_IN(col(r), P.mx, 63); };
        T a[8], b[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            a[r] = ok(r) ? __ldg(ia[0] + oa + col(r)) : T(0);
            b[r] = ok(r) ? __ldg(ib[0] + ob + col(r)) : T(0);
        }
        if (cx) {
            T c[8], d[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                c[r] = ok(r) ? __ldg(ia[1] + oa + col(r)) : T(0);
                d[r] = ok(r) ? __ldg(ib[1] + ob + col(r)) : T(0);
            }
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                a[r] += c[r];
                b[r] += d[r];
            }
        }
        auto add_seam = [&](const T* const (&in)[4], int o, T (&x)[8]) {
            T c[8], d[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                c[r] = ok(r) ? __ldg(in[2] + o + col(r)) : T(0);
                d[r] = cx && ok(r) ? __ldg(in[3] + o + col(r)) : T(0);
            }
#pragma unroll
            for (int r = 0; r < 8; ++r) x[r] += c[r] + d[r];
        };
        if (ya) add_seam(ia, oa, a);
        if (yb) add_seam(ib, ob, b);
#pragma unroll
        for (int r = 0; r < 8; ++r)
            v[8 * h + r] = h == 0 ? Cplx<T>{a[r], b[r]} : Cplx<T>{-a[r], -b[r]};
    }
}

// 1/x for the normal range (an eigenvalue): the hardware's approximation
// and Newton's iteration r (2 - x r) until the working precision.
__device__ __forceinline__ float recip(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return fmaf(r, fmaf(-x, r, 1.0f), r);
}
__device__ __forceinline__ double recip(double x) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));   // 20 bits
    r = fma(r, fma(-x, r, 1.0), r);
    return fma(r, fma(-x, r, 1.0), r);
}

// Four consecutive values as vector stores (16-byte aligned).
__device__ __forceinline__ void st4(float* p, float a, float b, float c, float d) {
    *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
}
__device__ __forceinline__ void st4(double* p, double a, double b, double c, double d) {
    *reinterpret_cast<double2*>(p) = make_double2(a, b);
    *reinterpret_cast<double2*>(p + 2) = make_double2(c, d);
}

// Staging pitch in complex elements of the outputs of PPC pairs.
__host__ __device__ constexpr int stage_pitch(int ppc) { return ppc == 1 ? 1 : ppc + 1; }
__host__ __device__ constexpr int round32(int v) { return (v + 31) / 32 * 32; }

// Threads of a CTA of PPC pairs, and its shared memory in complex elements:
// the pairs' buffers (and a spare row when the last warp is not full), or
// the staged outputs, never both at once.
template <int LG, int PPC>
__host__ __device__ constexpr int cta_threads() { return round32(Half<LG>::TP * PPC); }
template <int LG, int PPC>
__host__ __device__ constexpr int cta_elems(bool staged) {
    const int buf = PPC * Half<LG>::BUF + (Half<LG>::TP * PPC % 32 ? Half<LG>::RP : 0);
    const int stg = staged ? Half<LG>::N * stage_pitch(PPC) : 0;
    return buf > stg ? buf : stg;
}

// One pass of the solve for PPC sequence pairs (pair blk PPC + group, one
// group of TP threads each; threads past the last group only meet the
// barriers).  Pairs, one layer: two rows of the grid (x passes), two
// positions (y pass); two layers: the two layers of a row or position.
// Every thread of the CTA takes part.
template <typename T, int OPY, int PH, int LG, int PPC>
__device__ __forceinline__ void stream_item(const SolveParams<T>& P, int npairs, int blk,
                                            unsigned char* smem) {
    using Q = Half<LG>;
    constexpr int G = Q::G, H = Q::H, N = Q::N;
    const int grp = PPC == 1 && Q::TP % 32 == 0 ? 0 : (int)threadIdx.x / Q::TP;
    const int tt = (int)threadIdx.x - grp * Q::TP;
    const bool act = grp < PPC;
    const int s = tt / H, j = tt - s * H;      // the thread's row and place in it
    const bool tpass = act && tt <= G / 2;     // takes part in the radix-16 pass
    const int pair0 = blk * PPC, pair = pair0 + grp;
    const bool vp = act && pair < npairs;
    CT<T>* buf = reinterpret_cast<CT<T>*>(smem) + (act ? grp : 0) * Q::BUF;
    // (threads past the last group run the row stages on a spare row)
    CT<T>* row = act ? buf + s * Q::RP : reinterpret_cast<CT<T>*>(smem) + PPC * Q::BUF;
    const CT<T>* tab = PH == 1 ? P.hty : P.htx;
    // scratch arrays, in complex units of two interleaved sequences
    CT<T>* tr = reinterpret_cast<CT<T>*>(P.tr[0]);
    CT<T>* wk = reinterpret_cast<CT<T>*>(P.work[0] + P.ld);   // from row 1 of the array on
    const long long ntr = (long long)(OPY == 2 ? P.mx : P.mx / 2) * P.ld_tr;
    const long long nwk = (long long)(OPY == 2 ? P.my - 1 : P.my / 2) * P.ld;
    (void)ntr;
    (void)nwk;

    Cplx<T> v[16];
    if constexpr (PH == 2) {
        // row s of the inverse x pass: modes s + 16 k, k = j + H r; k >= G/2
        // are the negated modes 16 - s + 16 (G - 1 - k)
        // (a pair or row that does not exist reads one that does)
        const int pe = vp ? pair : 0, se = act ? s : 0;
        const CT<T>* lo = wk + (size_t)pe * P.ld + se * (G / 2) + j;
        const CT<T>* hi = wk + (size_t)pe * P.ld + (se == 0 ? G : (16 - se) * (G / 2) + G - 1) - j;
        const bool wall = se == 0 && j == 0;      // modes 0 and mx: r = 0 and 8
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            CT<T> x;
            x.x = x.y = T(0);
            if (!((r & 7) == 0 && wall) &&
                QG_IN((r < 8 ? lo + H * r : hi - H * r) - wk, nwk, 64))
                x = r < 8 ? lo[H * r] : hi[-H * r];
            v[r] = r < 8 ? Cplx<T>{x.x, x.y} : Cplx<T>{-x.x, -x.y};
        }
        row_fwd<T, LG>(v, row, j, tab);
        row_sync<LG>();
        if (act) {
#pragma unroll
            for (int i = 0; i < 16; ++i) sts_<T>(row, row_k<LG>(j, i), v[i], Q::RP);
        }
    } else {
        if (tpass) {
            if constexpr (PH == 0) {
                const int ra = OPY == 2 ? 1 + pair : 1 + 2 * pair, rb = OPY == 2 ? ra : ra + 1;
                load_rhs<T, LG>(P, P.in[0], P.in[OPY == 2 ? 1 : 0], ra, rb, vp,
                                vp && rb <= P.my - 1, tt, v);
            } else {
                const CT<T>* src = tr + (vp ? (size_t)pair * P.ld_tr : 0) - 1;
#pragma unroll
                for (int r = 0; r < 16; ++r) {
                    const int n = r < 8 ? tt + G * r : (16 - r) * G - tt;
                    CT<T> x;
                    x.x = x.y = T(0);
                    if ((tt > 0 || (r & 7) != 0) &&
                        QG_IN((long long)(vp ? pair : 0) * P.ld_tr + n - 1, ntr, 65))
                        x = src[n];
                    v[r] = r < 8 ? Cplx<T>{x.x, x.y} : Cplx<T>{-x.x, -x.y};
                }
            }
            pass_fwd<T, LG>(v, buf, tt, tab);
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < 16; ++r) v[r] = lds_<T>(row, j + H * r, Q::RP);
        row_fwd<T, LG>(v, row, j, tab);
    }

    if constexpr (PH == 1) {
        // mode-space solve of the modes l = s + 16 k, their images included
        // (the eigenvalues of l and 2 my - l are the same)
        auto mode = [&](int pos) { return pos / (P.mx / 16) + 16 * (pos % (P.mx / 16)); };
        const int ka = OPY == 2 ? mode(pair) : mode(2 * pair);
        const int kb = OPY == 2 ? ka : mode(2 * pair + 1);
        const bool ok = vp && QG_IN(ka, P.mx + 1, 66) && QG_IN(kb, P.mx + 1, 66);
        // lamyr comes divided by P.scale, a power of two: so do lamx and Ro, and
        // the scaling takes no operation per mode
        const T inv = T(1) / P.scale;
        const T lxa = (ok ? __ldg(P.lamx + ka) : T(1)) * inv, lxb = (ok ? __ldg(P.lamx + kb) : T(1)) * inv;
        const T ro = P.Ro * P.scale;
        const T* ly_s = P.lamyr + (act ? s : 0) * G;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int k = row_k<LG>(j, i);
            const T ly = QG_IN((act ? s : 0) * G + k, 9 * G, 67) ? __ldg(ly_s + k) : T(1);
            // the pair's 2 F are -Im Z and Re Z
            const T Fa = -v[i].y, Fb = v[i].x;
            T x, y;
            if (OPY == 1) {
                x = Fa * recip(lxa + ly);
                y = Fb * recip(lxb + ly);
            } else {
                const T q1 = P.scale * Fa, q2 = P.scale * Fb;
                const T al = ro * (lxa + ly);
                // the two quotients without a division, whose rare path splits
                // the chains of the 16 modes (FP32 256 x 256, l = 0: 51.4 us a
                // step with two divisions a mode, 43.1 with one, 36.9 without):
                // a reciprocal factor by factor, both negative, and the residual
                // correction of Markstein (1990), which rounds them as a
                // division would
                const T den = al * (al - P.f1 - P.f2);
                const T r = recip(al) * recip(al - P.f1 - P.f2);
                const T n1 = al * q1 - P.f2 * q1 - P.f1 * q2, n2 = al * q2 - P.f2 * q1 - P.f1 * q2;
                x = n1 * r;
                y = n2 * r;
                x = fma(fma(-den, x, n1), r, x);
                y = fma(fma(-den, y, n2), r, y);
            }
            v[i] = Cplx<T>{x, y};
            // the walls l = 0 and my stay 0
            if ((row_k0<LG>(i) == 0 || row_k0<LG>(i) == G / 2) && s == 0 && j == 0)
                v[i] = Cplx<T>{T(0), T(0)};
        }
        row_bwd<T, LG>(v, row, j, tab);
        row_sync<LG>();
        if (act) {
#pragma unroll
            for (int r = 0; r < 16; ++r) sts_<T>(row, j + H * r, v[r], Q::RP);
        }
    }
    if constexpr (PH >= 1) {
        __syncthreads();
        if (tpass) pass_bwd<T, LG>(v, buf, tt, tab);
    }

    // 2 F(a)_k = -Im Z_k, 2 F(b)_k = Re Z_k (P.scale holds the 2^-4)
    if constexpr (PH == 2) {
        if (tpass) {
            const int ra = OPY == 2 ? 1 + pair : 1 + 2 * pair, rb = OPY == 2 ? ra : ra + 1;
            const bool vb = vp && rb <= P.my - 1;
            const long long nw = (long long)(P.my + 1) * P.ld;
            (void)nw;
            T* oa = P.out[0] + (size_t)ra * P.ld;
            T* ob = P.out[OPY == 2 ? 1 : 0] + (size_t)rb * P.ld;
            // (columns 0 and mx and the wall row my are zero: out may be the
            // array that held the scratch values.  Threads 0 and G/2 hold
            // some columns twice, at r < 8 and r >= 8, and write them twice.)
            if (vp) {
#pragma unroll
                for (int r = 0; r < 16; ++r) {
                    const bool second = r >= 8;
                    const int n = second ? (16 - r) * G - tt : tt + G * r;
                    const T sg = second ? T(-1) : T(1);
                    T fa = -sg * v[r].y, fb = sg * v[r].x;
                    if ((r & 7) == 0 && tt == 0) fa = fb = T(0);
                    if (QG_IN((long long)ra * P.ld + n, nw, 70)) oa[n] = fa;
                    if (QG_IN((long long)rb * P.ld + n, nw, 70)) ob[n] = fb;
                }
                if (!vb) {
#pragma unroll
                    for (int r = 0; r < 16; ++r) {
                        const int n = r >= 8 ? (16 - r) * G - tt : tt + G * r;
                        if (QG_IN((long long)rb * P.ld + n, nw, 70)) ob[n] = T(0);
                    }
                }
            }
        }
    } else {
        constexpr int SP = stage_pitch(PPC);
        CT<T>* stg = reinterpret_cast<CT<T>*>(smem);
        constexpr int SLIM = cta_elems<LG, PPC>(true);
        __syncthreads();   // every group is done with its buffer
        if constexpr (PH == 0) {
            // modes s + 16 k by position
            if (act) {
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const int k = row_k<LG>(j, i);
                    const bool low = row_low<LG>(i);
                    if (!low && (s == 0 || s == 8)) continue;   // images of the low half
                    const int pos = low ? s * (G / 2) + k : (16 - s) * (G / 2) + G - 1 - k;
                    const T sg = low ? T(1) : T(-1);
                    Cplx<T> o{-sg * v[i].y, sg * v[i].x};
                    if (i == 0 && s == 0 && j == 0) o = Cplx<T>{T(0), T(0)};   // the wall mode
                    sts_<T>(stg, pos * SP + grp, o, SLIM);
                }
            }
        } else {
            if (tpass) {
#pragma unroll
                for (int r = 0; r < 16; ++r) {
                    const bool second = r >= 8;
                    const int n = second ? (16 - r) * G - tt : tt + G * r;
                    // (elements 0 and N are walls: N has no place; threads 0 and
                    // G/2 hold some elements twice)
                    if (r == 8 && tt == 0) continue;
                    const T sg = second ? T(-1) : T(1);
                    sts_<T>(stg, n * SP + grp, Cplx<T>{-sg * v[r].y, sg * v[r].x}, SLIM);
                }
            }
        }
        __syncthreads();
        // thread e writes for pair g = e mod PPC the items e / PPC + i STEP
        constexpr int BT = cta_threads<LG, PPC>(), STEP = BT / PPC;
        static_assert(BT % PPC == 0, "");
        const int g = (int)threadIdx.x % PPC, q0 = (int)threadIdx.x / PPC;
        const int ldo = PH == 0 ? P.ld_tr : P.ld;
        if (pair0 + g < npairs) {
            if constexpr (OPY == 1) {
                // 2 x 2 blocks: positions 2 q, 2 q + 1 (x forward) or rows
                // 2 q + 1, 2 q + 2 (y) of a pair, transposed into a run of 4
                // values
                constexpr int ITEMS = N / 2, ITER = (ITEMS + STEP - 1) / STEP;
                const CT<T>* src = stg + (PH == 0 ? 2 * q0 : 2 * q0 + 1) * SP + g;
                long long o = (long long)q0 * ldo + 2 * (pair0 + g);
                CT<T>* dst = PH == 0 ? tr : wk;
#pragma unroll 4
                for (int i = 0; i < ITER; ++i) {
                    const int q = q0 + i * STEP;
                    if (q < ITEMS && QG_IN((2 * q + 1) * SP + g, SLIM, 61) &&
                        QG_IN(o + 1, PH == 0 ? ntr : nwk, PH == 0 ? 69 : 72)) {
                        const CT<T> c0 = src[2 * i * STEP * SP];
                        CT<T> c1;
                        c1.x = c1.y = T(0);      // (row N is the wall)
                        if (PH == 0 || q < ITEMS - 1) c1 = src[(2 * i * STEP + 1) * SP];
                        st4(reinterpret_cast<T*>(dst + o), c0.x, c1.x, c0.y, c1.y);
                    }
                    o += (long long)STEP * ldo;
                }
            } else {
                // [position][row][layer] (x forward), [row][position][layer] (y)
                constexpr int ITER = (N + STEP - 1) / STEP;
                const CT<T>* src = stg + q0 * SP + g;
                long long o = (long long)(PH == 0 ? q0 : q0 - 1) * ldo + pair0 + g;
                CT<T>* dst = PH == 0 ? tr : wk;
#pragma unroll 4
                for (int i = 0; i < ITER; ++i) {
                    const int q = q0 + i * STEP;
                    if (q < N && (PH == 0 || q > 0) && QG_IN(q * SP + g, SLIM, 61) &&
                        QG_IN(o, PH == 0 ? ntr : nwk, PH == 0 ? 69 : 72))
                        dst[o] = src[i * STEP * SP];
                    o += (long long)STEP * ldo;
                }
            }
        }
    }
}

// Registers per thread the CTA shapes are budgeted for: FP32 72 (three CTAs
// of 288 threads per SM; at 96, two, the passes of the 2048 x 4096 grid took
// 29, 59 and 20 us instead of 22, 41 and 20), FP64 as many as it takes.
template <typename T>
__host__ __device__ constexpr int minb_for(int threads, int regs32 = 72) {
    const int regs = sizeof(T) == 8 ? 160 : regs32;
    const int b = 65536 / (round32(threads) * regs);
    return b < 1 ? 1 : (b > 16 ? 16 : b);
}

// One launch per pass.  Batches (ensembles, one layer): member
// blockIdx.x / cpm takes CTAs blockIdx.x mod cpm, with its arrays from
// P.batch.
template <typename T, int OPY, int PH, int LG, int PPC>
__global__ void __launch_bounds__(cta_threads<LG, PPC>(), minb_for<T>(cta_threads<LG, PPC>()))
stream_kernel(SolveParams<T> Pin, int npairs, int cpm) {
    extern __shared__ __align__(16) unsigned char smem[];
    SolveParams<T> P = Pin;
    int blk = blockIdx.x;
    if (Pin.batch) {
        const int m = blk / cpm;
        blk -= m * cpm;
        const SolveMember<T>& M = Pin.batch[m];
#pragma unroll
        for (int q = 0; q < 4; ++q) P.in[0][q] = M.in[q];
        P.nin = M.nin;
        P.part_px = M.part_px;
        P.part_py = M.part_py;
        P.tr[0] = M.tr;
        P.work[0] = M.work;
        P.out[0] = M.out;
    }
    pdl_wait();
    pdl_trigger();
    stream_item<T, OPY, PH, LG, PPC>(P, npairs, blk, smem);
}

// Pairs per y item of the work queue (twice as many per x item, half as
// long) and its CTA size.
__host__ __device__ constexpr int queue_ppc(int lgx) { return lgx <= 10 ? 4 : 2; }
__host__ __device__ constexpr int queue_threads(int lgx) {
    return round32(9 * (1 << (lgx + 1)) / 256 * queue_ppc(lgx));
}

// Batched solve of an ensemble group in one launch (one layer, y length
// twice the x length): a work queue over the items of the three passes of
// every member, claimed in order from the counter q[0] (pass by pass,
// member by member).  An item of pass ph >= 1 of member m first waits
// (bounded) until the q[2 + 3 m + ph - 1] items of the pass before are
// done; those were claimed earlier by CTAs that are running and depend on
// no later item, so the wait ends without any co-residency.  A wait that
// runs out sets the member's error flag and the item is counted done
// unprocessed.  The last CTA to leave resets the counters for the next
// launch.
constexpr int kQueueSpin = 1 << 22;

__device__ __forceinline__ bool wait_done(const unsigned* c, unsigned want, int limit) {
    for (int i = 0; i < limit; ++i) {
        unsigned v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(c) : "memory");
        if (v >= want) return true;
    }
    return false;
}

template <typename T, int LGX>
__global__ void __launch_bounds__(queue_threads(LGX), minb_for<T>(queue_threads(LGX), 96))
stream_queue_kernel(SolveParams<T> P) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_item;
    constexpr int LGY = LGX + 1;
    constexpr int PX = 2 * queue_ppc(LGX), PY = queue_ppc(LGX);
    unsigned* q = P.bar;
    const int nb = P.nbatch;
    const int rows = P.my / 2, cols = P.mx / 2;
    const int n0i = (rows + PX - 1) / PX, n1i = (cols + PY - 1) / PY;
    const int e0 = nb * n0i, e1 = e0 + nb * n1i, total = e1 + nb * n0i;
    pdl_wait();
    pdl_trigger();
    for (;;) {
        if (threadIdx.x == 0) s_item = (int)atomicAdd(q, 1u);
        __syncthreads();
        const int item = s_item;
        __syncthreads();
        if (item >= total) break;
        int ph, m, blk;
        if (item < e0) {
            ph = 0; m = item / n0i; blk = item - m * n0i;
        } else if (item < e1) {
            ph = 1; m = (item - e0) / n1i; blk = item - e0 - m * n1i;
        } else {
            ph = 2; m = (item - e1) / n0i; blk = item - e1 - m * n0i;
        }
        const SolveMember<T>& M = P.batch[m];
        int ok = 1;
        if (ph > 0 && threadIdx.x == 0)
            ok = wait_done(q + 2 + 3 * m + ph - 1, (unsigned)(ph == 1 ? n0i : n1i), kQueueSpin);
        if (__syncthreads_and(ok)) {
            SolveParams<T> Q = P;
#pragma unroll
            for (int k = 0; k < 4; ++k) Q.in[0][k] = M.in[k];
            Q.nin = M.nin;
            Q.part_px = M.part_px;
            Q.part_py = M.part_py;
            Q.tr[0] = M.tr;
            Q.work[0] = M.work;
            Q.out[0] = M.out;
            if (ph == 0) stream_item<T, 1, 0, LGX, PX>(Q, rows, blk, smem);
            else if (ph == 1) stream_item<T, 1, 1, LGY, PY>(Q, cols, blk, smem);
            else stream_item<T, 1, 2, LGX, PX>(Q, rows, blk, smem);
            __syncthreads();
        } else if (threadIdx.x == 0) {
            atomicExch(M.err, 1);
        }
        if (threadIdx.x == 0) {
            // this CTA's stores of the item are ordered before the count by
            // the CTA barrier above and the release
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(q + 2 + 3 * m + ph)
                         : "memory");
        }
    }
    if (threadIdx.x == 0) {
        unsigned old;
        asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(old) : "l"(q + 1)
                     : "memory");
        if (old == gridDim.x - 1) {
            for (int i = 0; i < 2 + 3 * nb; ++i) q[i] = 0u;
        }
    }
}

// Lengths 2^LG of the engine: L = 256 .. 16384 (FP32), .. 8192 (FP64).
constexpr int kMinLg = 8, kMaxLg = 14;

template <typename T, int OPY, int PH, int LG, int PPC>
cudaError_t launch_ppc(const SolveParams<T>& P, int npairs, cudaStream_t s) {
    const int cpm = (npairs + PPC - 1) / PPC;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cpm * (P.batch ? P.nbatch : 1));
    cfg.blockDim = dim3(cta_threads<LG, PPC>());
    cfg.dynamicSmemBytes = (size_t)cta_elems<LG, PPC>(PH != 2) * sizeof(CT<T>);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    // (ensemble branches run side by side: a dependent started early would
    // hold SM resources idle, so their launches may go without)
    cfg.attrs = P.no_pdl ? nullptr : at;
    cfg.numAttrs = P.no_pdl ? 0 : 1;
    auto k = stream_kernel<T, OPY, PH, LG, PPC>;
    int per = 0, nsm = 0;
    cudaError_t e = launch_shape(reinterpret_cast<const void*>(k), (int)cfg.blockDim.x,
                                 cfg.dynamicSmemBytes, &per, &nsm);
    if (e != cudaSuccess) return e;
    return cudaLaunchKernelEx(&cfg, k, P, npairs, cpm);
}

// Pairs per CTA, of 1, 2, .. ppc_max (CTAs of at most 288 threads, FP32 at
// LG = 12 576): the number that leaves the fullest SM the fewest warps.  More
// pairs fill the CTA's last warp and write longer runs, so a tie takes more
// pairs (the inverse x pass writes whole rows either way: fewer, in FP32);
// with few warps on an SM the pass is bound by latency, and fewer pairs are
// taken for up to an eighth more warps.  Measured in whole FP32 steps at
// l = 0 (us; pairs in the three passes): 512 x 1024 51.8 with (4, 2, 2),
// 55.4 with (4, 1, 1); 1024 x 2048 79.9 with (4, 4, 1), 93.1 with (4, 2, 1);
// 512 x 2048 64.4 with (4, 1, 4), 69.8 with (8, 1, 4); 2048 x 4096 291 with
// (2, 1, 2), 298 with (4, 1, 1); FP64 512 x 1024 575 with (4, 2, 4), 661
// with (4, 2, 1).
// Two layers in FP32 store one value of each layer per pair and element, 8
// bytes: the two passes that write the scratch arrays take four pairs at
// least, a 32-byte sector (l = 0, 1024 x 2048: 183 us with (4, 4, 2), 222 with
// (1, 1, 1), 197 with (2, 2, 1); 256 x 256 36.9, 39.0 and 39.0).
template <typename T>
__host__ __device__ constexpr int ppc_max(int lg) {
    return lg <= 10 ? 8 : lg == 11 ? 4 : lg == 12 ? (sizeof(T) == 4 ? 4 : 2) : 1;
}
template <typename T, int OPY, int PH>
__host__ __device__ constexpr int ppc_min(int lg) {
    const int least = OPY == 2 && PH < 2 && sizeof(T) == 4 ? 4 : 1;
    return least < ppc_max<T>(lg) ? least : ppc_max<T>(lg);
}
template <typename T>
int pick_ppc(int ph, int lg, int npairs, int batch, int nsm, int least) {
    const int tp = 9 * (1 << lg) / 256;
    int best = least, cost = 0;
    for (int c = least; c <= ppc_max<T>(lg); c *= 2) {
        const int ctas = (npairs + c - 1) / c * batch;
        const int w = (ctas + nsm - 1) / nsm * (round32(tp * c) / 32);
        const bool keep_tie = ph == 2 && sizeof(T) == 4;
        if (c == least || w < cost || (w == cost && !keep_tie)) {
            if (c > least && cost <= 16 && 8 * cost <= 9 * w) continue;
            best = c;
            cost = w;
        }
    }
    return best;
}
template <typename T, int OPY, int PH, int LG>
cudaError_t launch_pass(const SolveParams<T>& P, int npairs, cudaStream_t s) {
    int dev = 0, nsm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    constexpr int M = ppc_max<T>(LG), LEAST = ppc_min<T, OPY, PH>(LG);
    const int c = pick_ppc<T>(PH, LG, npairs, P.batch ? P.nbatch : 1, nsm, LEAST);
    if constexpr (M >= 8) {
        if (c == 8) return launch_ppc<T, OPY, PH, LG, 8>(P, npairs, s);
    }
    if constexpr (M >= 4) {
        if (c == 4) return launch_ppc<T, OPY, PH, LG, 4>(P, npairs, s);
    }
    if constexpr (M >= 2 && LEAST <= 2) {
        if (c == 2) return launch_ppc<T, OPY, PH, LG, 2>(P, npairs, s);
    }
    if constexpr (LEAST == 1) {
        return launch_ppc<T, OPY, PH, LG, 1>(P, npairs, s);
    }
    return cudaErrorInvalidValue;   // (not reached: c is one of the above)
}

template <typename T, int OPY, int PH>
cudaError_t launch_lg(const SolveParams<T>& P, int lg, int npairs, cudaStream_t s) {
    switch (lg) {
        case 8: return launch_pass<T, OPY, PH, 8>(P, npairs, s);
        case 9: return launch_pass<T, OPY, PH, 9>(P, npairs, s);
        case 10: return launch_pass<T, OPY, PH, 10>(P, npairs, s);
        case 11: return launch_pass<T, OPY, PH, 11>(P, npairs, s);
        case 12: return launch_pass<T, OPY, PH, 12>(P, npairs, s);
        case 13: return launch_pass<T, OPY, PH, 13>(P, npairs, s);
        case 14:
            if constexpr (sizeof(T) == 4) return launch_pass<T, OPY, PH, 14>(P, npairs, s);
            return cudaErrorInvalidValue;
        default: return cudaErrorInvalidValue;
    }
}

template <typename T, int OPY>
cudaError_t launch_all(const SolveParams<T>& P, cudaStream_t s) {
    const int lgx = ilog2(2 * P.mx), lgy = ilog2(2 * P.my);
    const int rows = OPY == 2 ? P.my - 1 : P.my / 2;
    const int cols = OPY == 2 ? P.mx : P.mx / 2;
    cudaError_t e = launch_lg<T, OPY, 0>(P, lgx, rows, s);
    if (e == cudaSuccess) e = launch_lg<T, OPY, 1>(P, lgy, cols, s);
    if (e == cudaSuccess) e = launch_lg<T, OPY, 2>(P, lgx, rows, s);
    return e;
}

template <typename T, int LGX>
cudaError_t launch_queue_lg(const SolveParams<T>& P, cudaStream_t s) {
    constexpr int BT = queue_threads(LGX);
    constexpr int PX = 2 * queue_ppc(LGX), PY = queue_ppc(LGX);
    auto k = stream_queue_kernel<T, LGX>;
    constexpr int ex = cta_elems<LGX, PX>(true), ey = cta_elems<LGX + 1, PY>(true);
    const size_t sm = (size_t)(ex > ey ? ex : ey) * sizeof(CT<T>);
    int nsm = 0, per = 0;
    cudaError_t e = launch_shape(reinterpret_cast<const void*>(k), BT, sm, &per, &nsm);
    if (e != cudaSuccess) return e;
    if (per < 1) return cudaErrorInvalidConfiguration;
    const int rows = P.my / 2, cols = P.mx / 2;
    const int total = P.nbatch * (2 * ((rows + PX - 1) / PX) + (cols + PY - 1) / PY);
    int grid = per * nsm;
    if (total < grid) grid = total;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(BT);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = P.no_pdl ? nullptr : at;
    cfg.numAttrs = P.no_pdl ? 0 : 1;
    return cudaLaunchKernelEx(&cfg, k, P);
}

}  // namespace

// Batches of one-layer grids with my = 2 mx and 2 mx = 2^8 .. 2^11 run as
// one work-queue launch; other batches as three launches.
bool stream_queue_ok(int mx, int my, int layers) {
    if (layers != 1 || my != 2 * mx || !is_pow2(mx)) return false;
    const int lx = ilog2(2 * mx);
    return lx >= 8 && lx <= 11;
}

bool stream_supports(int mx, int my, size_t esz) {
    if (!is_pow2(mx) || !is_pow2(my)) return false;
    const int lx = ilog2(2 * mx), ly = ilog2(2 * my);
    const int hi = esz == 4 ? kMaxLg : kMaxLg - 1;
    // (128 x 128 and less are left to the engines of one launch)
    if (lx == kMinLg && ly == kMinLg) return false;
    return lx >= kMinLg && ly >= kMinLg && lx <= hi && ly <= hi;
}

size_t half_table_size(int L) {
    const int G = L / 16, H = G / 16;
    return (size_t)8 * (G / 2 + 2) + 15 * H + (H > 16 ? H : 0);
}

void half_table(int L, double* re, double* im) {
    const int G = L / 16, H = G / 16, PT = G / 2 + 2;
    const double pi = 3.14159265358979323846;
    auto put = [&](size_t i, long long num, long long den) {   // e^{-2 pi i num/den}
        const double a = -2.0 * pi * (double)(num % den) / (double)den;
        re[i] = std::cos(a);
        im[i] = std::sin(a);
    };
    for (int s = 1; s <= 8; ++s)
        for (int t = 0; t < PT; ++t) put((size_t)(s - 1) * PT + t, (long long)t * s, L);
    const size_t t2 = (size_t)8 * PT, t3 = t2 + 15 * (size_t)H;
    for (int q = 1; q < 16; ++q)
        for (int j = 0; j < H; ++j) put(t2 + (size_t)(q - 1) * H + j, (long long)q * j, G);
    if (H > 16)
        for (int p = 0; p < H / 4; ++p)
            for (int c = 0; c < 4; ++c) put(t3 + 4 * p + c, (long long)p * c, H);
}

void half_lam(int M, const double* lam, double* out) {
    const int G = M / 8;
    for (int s = 0; s <= 8; ++s)
        for (int k = 0; k < G; ++k) {
            const int m = s + 16 * k;
            out[(size_t)s * G + k] = lam[m <= M ? m : 2 * M - m];
        }
}

template <typename T>
cudaError_t launch_solve_stream(const SolveParams<T>& Pin, cudaStream_t s) {
    if (!stream_supports(Pin.mx, Pin.my, sizeof(T)) || !Pin.htx || !Pin.hty || !Pin.lamyr ||
        (Pin.batch && (Pin.layers != 1 || Pin.nbatch < 1)))
        return cudaErrorInvalidValue;
    // two layers: the scratch rows of both layers lie in one run from work[0]
    // (tr[0]), so the output may not share them
    if (Pin.layers == 2 && (Pin.out[0] == Pin.work[0] || Pin.out[1] == Pin.work[1]))
        return cudaErrorInvalidValue;
    SolveParams<T> P = Pin;
    P.scale *= T(1) / T(16);   // the passes leave 2 F (exact)
    if (P.batch && stream_queue_ok(P.mx, P.my, P.layers) && P.bar) {
        switch (ilog2(2 * P.mx)) {
            case 8: return launch_queue_lg<T, 8>(P, s);
            case 9: return launch_queue_lg<T, 9>(P, s);
            case 10: return launch_queue_lg<T, 10>(P, s);
            default: return launch_queue_lg<T, 11>(P, s);
        }
    }
    return P.layers == 2 ? launch_all<T, 2>(P, s) : launch_all<T, 1>(P, s);
}

QG_BOUNDS_QUERY(bounds_site_stream)

template cudaError_t launch_solve_stream<float>(const SolveParams<float>&, cudaStream_t);
template cudaError_t launch_solve_stream<double>(const SolveParams<double>&, cudaStream_t);

}  // namespace qg
