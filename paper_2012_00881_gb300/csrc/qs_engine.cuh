// The slice engine: one persistent cooperative kernel runs the whole xi loop
// of Algorithm 1 (Collect_Source, Solve_Wakefield, Push_Trajectory,
// Step_Size_Refinement) for one 3D step.  Phases are separated by a grid
// barrier whose waits are bounded in time; a timed-out wait records
// QS_ERR_TIMEOUT and every block leaves the kernel at its next barrier.
//
// The solves (qs_solve.cuh) are direct, by sine transforms, and for B_perp
// conjugate gradients preconditioned with them; sources are formed where their
// row transforms read them.  Grid sides without the transforms (odd, below 8 or
// above 2048, clusters on request) and solves that the iterations do not finish
// take red-black Gauss-Seidel V(nu1, nu2) cycles
// with 4-cell-average restriction, bilinear prolongation and rediscretised
// coarse operators (kappa averaged).  Levels of side <= block_level_n are
// solved redundantly by every block in its shared memory, down to a coarsest
// grid of side <= 4 whose dense inverse is cached.  Refined form: float64
// residual, float32 inner cycles whose grid-wide levels are staged tile by
// tile in shared memory, float64 correction.
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

#include "qs_solve.cuh"

namespace {

// ---------------------------------------------------------------------------
// particle and grid phases
// ---------------------------------------------------------------------------

// Plasma macroparticles and the grids they deposit into.  Positions and
// n_* are float64 in both forms (the density source n_* - n_ion and the
// sources built on it are small differences of O(1) numbers); momenta,
// weights and the other six moments are in the particle precision P (float64
// form: double; refined form: float).  In the refined form the gamma moment
// holds n_* <gamma - 1>, which has no cancellation.
template <typename P>
struct PS {
    double *x, *y;
    P *px, *py, *w;
    double *wd;  // float64 weights: n_* must cancel n_ion to rounding
    double *na, *nb;   // n_* of this slice and of the next one
    // the moments j_x, j_y, T_xx, T_xy, T_yy, n_* <gamma> (refined form: <gamma - 1>):
    // six grids (float64), or the interleaved cells of EngineArgs::mom32
    P *m[6];
    static constexpr int stride = sizeof(P) == 8 ? 1 : 8;  // between cells of a moment
    __device__ __forceinline__ P mom(int k, int i) const { return m[k][(size_t)i * stride]; }
};

enum { M_JX = 0, M_JY, M_TXX, M_TXY, M_TYY, M_G };

// n_* <gamma> from the gamma moment of either form
template <typename P>
__device__ __forceinline__ double g_total(P G, double n) {
    if constexpr (sizeof(P) == 8) return G;
    else return n + (double)G;
}

template <typename P>
struct CicP {
    int i00, i01, i10, i11;
    P w00, w01, w10, w11;
};

// CIC weights of a float64 stencil in the particle precision
template <typename P>
__device__ __forceinline__ CicP<P> cic_p(const Cic &c) {
    CicP<P> r;
    r.i00 = c.i00; r.i01 = c.i01; r.i10 = c.i10; r.i11 = c.i11;
    r.w00 = (P)c.w00; r.w01 = (P)c.w01; r.w10 = (P)c.w10; r.w11 = (P)c.w11;
    return r;
}

template <typename P, typename G>
__device__ __forceinline__ P gat(const G *u, const CicP<P> &c) {
    return (P)u[c.i00] * c.w00 + (P)u[c.i01] * c.w01 + (P)u[c.i10] * c.w10 + (P)u[c.i11] * c.w11;
}

template <typename P>
__device__ __forceinline__ void dep(P *g, const CicP<P> &c, P q) {
    atomicAdd(g + c.i00, q * c.w00);
    atomicAdd(g + c.i01, q * c.w01);
    atomicAdd(g + c.i10, q * c.w10);
    atomicAdd(g + c.i11, q * c.w11);
}

// Six float32 moments of a lane's particle, times the weights, to its four
// cells of the interleaved grid (two float4 a cell: six moments and two zeros).
// A pair of lanes does the even lane's particle and then the odd one's, the even
// lane the first float4 of every cell and the odd lane the second: a request
// then covers whole 32-byte sectors, half as many of them, which is what the
// reductions are bound by.  The moments phase at 512^2, nine particles a cell:
// 97 us, with each lane on its own particle 120, with six scalar reductions and
// float64 arithmetic 247; at 256^2, four a cell: 14.0 and 18.6.  All 32 lanes call.
__device__ __forceinline__ void dep6_pairs(float4 *g, const CicP<float> &c, const float q[6]) {
    const bool odd = (threadIdx.x & 1) != 0;
    const float own[4] = {odd ? q[4] : q[0], odd ? q[5] : q[1], odd ? 0.f : q[2],
                          odd ? 0.f : q[3]};
    auto swap = [](auto v) { return __shfl_xor_sync(0xffffffffu, v, 1); };
    const float got[4] = {swap(odd ? q[0] : q[4]), swap(odd ? q[1] : q[5]),
                          swap(odd ? q[2] : 0.f), swap(odd ? q[3] : 0.f)};
    const int i[4] = {c.i00, c.i01, c.i10, c.i11};
    const float w[4] = {c.w00, c.w01, c.w10, c.w11};
    int j[4];
    float v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        j[k] = swap(i[k]);
        v[k] = swap(w[k]);
    }
    g += odd;
#pragma unroll
    for (int turn = 0; turn < 2; ++turn) {
        const bool mine = odd == (turn == 1);
        float d[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) d[k] = mine ? own[k] : got[k];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float wk = mine ? w[k] : v[k];
            asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(
                             g + 2 * (size_t)(mine ? i[k] : j[k])),
                         "f"(d[0] * wk), "f"(d[1] * wk), "f"(d[2] * wk), "f"(d[3] * wk)
                         : "memory");
        }
    }
}

// Whether the refined form sums its moments in float64, in the grids of the float64
// form, and rounds the sums: in steps that a gradient is taken of.  The order in
// which float32 reductions arrive made two losses of one input differ by 3e-10 to
// 2e-9 at 256^2, which a line search or a difference quotient sees; with float64
// sums 2e-13 to 4e-11, nearer to the float64 form's.  The moments phase takes 40 us
// instead of 14 there (a gradient 43.6 -> 44.9 ms).  Privatised deposits keep theirs.
__device__ __forceinline__ bool sums64(const EngineArgs &A) {
    return A.precision == QS_FP32_REFINED && (A.ckpt || A.seg_g) && A.band_rows == 0;
}

__device__ __forceinline__ void dep6_float64(const EngineArgs &A, const CicP<float> &c,
                                             const float q[6]) {
    double *const g[6] = {A.jx, A.jy, A.txx, A.txy, A.tyy, A.G};
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        atomicAdd(g[k] + c.i00, qsff::widen(q[k] * c.w00));
        atomicAdd(g[k] + c.i01, qsff::widen(q[k] * c.w01));
        atomicAdd(g[k] + c.i10, qsff::widen(q[k] * c.w10));
        atomicAdd(g[k] + c.i11, qsff::widen(q[k] * c.w11));
    }
}

// a cell's accumulators before the deposit
__device__ __forceinline__ void clear_moments(const EngineArgs &A, int i) {
    if (sums64(A)) A.jx[i] = A.jy[i] = A.txx[i] = A.txy[i] = A.tyy[i] = A.G[i] = 0.0;
    else
        A.mom32[2 * (size_t)i] = A.mom32[2 * (size_t)i + 1] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// the rounded sums to the refined form's cells
__device__ __noinline__ void round_moments(const EngineArgs &A, Thr T) {
    auto f = [](double v) { return qsff::split(v).h; };
    for (int i = T.t0; i < A.N * A.N; i += T.nt) {
        A.mom32[2 * (size_t)i] = make_float4(f(A.jx[i]), f(A.jy[i]), f(A.txx[i]), f(A.txy[i]));
        A.mom32[2 * (size_t)i + 1] = make_float4(f(A.tyy[i]), f(A.G[i]), 0.f, 0.f);
    }
}

// ---------------------------------------------------------------------------
// Privatised deposits.  With the plasma sorted by cell, a block that takes a
// contiguous chunk of the particle array finds its CIC stencils in a narrow
// band of grid rows (a 262,144-particle chunk of 1/152 covers about two rows
// of a 256^2 grid).  The block accumulates the band in shared memory and
// adds it to the grid once per cell: one global atomic per cell and moment
// instead of four per particle and moment.  A stencil outside the band (a
// particle that moved far since the last sort) is added to the grid directly.
// ---------------------------------------------------------------------------

// the block's contiguous chunk [p0, p1) of np particles
__device__ __forceinline__ void chunk_of(int64_t np, int bid, int nblk, int64_t &p0,
                                         int64_t &p1) {
    const int64_t cs = (np + nblk - 1) / nblk;
    p0 = min(np, (int64_t)bid * cs);
    p1 = min(np, p0 + cs);
}

// Rows [r0, r0 + rows) holding the CIC stencils (rows of y - h/2 and the
// next) of the chunk's particles, widened by `margin` rows on each side and
// clipped to the grid and to max_rows; rows = 0 for an empty chunk.
struct Band {
    int r0, rows;
};

__device__ Band band_of(const EngineArgs &A, const double *y, int64_t p0, int64_t p1, int margin,
                        int max_rows) {
    __shared__ int s_lo, s_hi;
    if (threadIdx.x == 0) {
        s_lo = A.N;
        s_hi = -1;
    }
    __syncthreads();
    int lo = A.N, hi = -1;
    for (int64_t p = p0 + threadIdx.x; p < p1; p += blockDim.x) {
        const int a = (int)floor((y[p] - A.y_min) * A.inv_h - 0.5);
        lo = min(lo, a);
        hi = max(hi, a + 1);
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if ((threadIdx.x & 31) == 0) {
        atomicMin(&s_lo, lo);
        atomicMax(&s_hi, hi);
    }
    __syncthreads();
    Band b{0, 0};
    if (s_hi >= 0) {
        const int r0 = max(0, s_lo - margin);
        const int r1 = min(A.N - 1, s_hi + margin);
        b.r0 = r0;
        b.rows = min(r1 - r0 + 1, max_rows);
    }
    __syncthreads();  // s_lo, s_hi are rewritten by the next call
    return b;
}

// deposit q into the band s (cells lo .. hi - 1 of the grid) when the whole
// stencil is inside, else into the grid g
template <int ST = 1, typename P, typename W>
__device__ __forceinline__ void dep_band(P *g, P *s, int lo, int hi, const W &c, P q) {
    const int a = min(min(c.i00, c.i01), min(c.i10, c.i11));
    const int b = max(max(c.i00, c.i01), max(c.i10, c.i11));
    if (a >= lo && b < hi) {
        atomicAdd(s + (c.i00 - lo), q * (P)c.w00);
        atomicAdd(s + (c.i01 - lo), q * (P)c.w01);
        atomicAdd(s + (c.i10 - lo), q * (P)c.w10);
        atomicAdd(s + (c.i11 - lo), q * (P)c.w11);
    } else {
        atomicAdd(g + (size_t)c.i00 * ST, q * (P)c.w00);
        atomicAdd(g + (size_t)c.i01 * ST, q * (P)c.w01);
        atomicAdd(g + (size_t)c.i10 * ST, q * (P)c.w10);
        atomicAdd(g + (size_t)c.i11 * ST, q * (P)c.w11);
    }
}

// the band's nonzero cells added to the grid, one atomic per cell
template <int ST = 1, typename P>
__device__ __forceinline__ void flush_band(P *g, const P *s, int lo, int cells) {
    for (int k = threadIdx.x; k < cells; k += blockDim.x) {
        const P v = s[k];
        if (v != P(0)) atomicAdd(g + (size_t)(lo + k) * ST, v);
    }
}

template <typename P>
__device__ __forceinline__ void zero_band(P *s, int cells) {
    for (int k = threadIdx.x; k < cells; k += blockDim.x) s[k] = P(0);
}

// n_* of the initial particles
template <typename P>
__device__ void phase_deposit_n(const EngineArgs &A, const PS<P> &Q, double *ng, Thr T) {
    const double s = A.inv_h * A.inv_h;
    for (int64_t p = T.t0; p < A.np; p += T.nt) {
        const Cic c = cic_stencil_inv(Q.x[p], Q.y[p], A.x_min, A.y_min, A.inv_h, A.N);
        cic_deposit(ng, c, Q.wd[p] * s);
    }
}

// Initial guess of a solve: the solutions of the last (up to three) slices
// extrapolated in xi to the new slice (order 0 is the plain warm start from
// the previous slice, Sec. 7.1).  w[k] multiplies the solution k slices back;
// the history of each field shifts by one as the guess replaces it.
struct Guess {
    double w0, w1, w2;
    bool active;
};

__device__ __forceinline__ Guess make_guess(int order, int have, double xt, double x0, double x1,
                                            double x2) {
    Guess g{1.0, 0.0, 0.0, order > 0 || have > 0};
    const int o = min(order, have - 1);
    if (o == 1) {
        g.w0 = (xt - x1) / (x0 - x1);
        g.w1 = (xt - x0) / (x1 - x0);
    } else if (o >= 2) {
        g.w0 = (xt - x1) * (xt - x2) / ((x0 - x1) * (x0 - x2));
        g.w1 = (xt - x0) * (xt - x2) / ((x1 - x0) * (x1 - x2));
        g.w2 = (xt - x0) * (xt - x1) / ((x2 - x0) * (x2 - x1));
    }
    return g;
}

__device__ __forceinline__ void apply_guess(double *u, double *h1, double *h2, int i,
                                            const Guess &g) {
    const double u0 = u[i], p1 = h1[i], p2 = h2[i];
    h2[i] = p1;
    h1[i] = u0;
    u[i] = g.w0 * u0 + g.w1 * p1 + g.w2 * p2;
}

// f_psi = n_* - n_ion (Eq. EqM_N8_AA) and its norm; charge sum; clear the
// moment accumulators and the next-slice density buffer
template <typename P>
__device__ void phase_psi_rhs(const EngineArgs &A, const PS<P> &Q, const double *ncur,
                              double *nnext, bool base, int j, int q, double frac, Thr T,
                              const Guess &g) {
    const int nn = A.N * A.N;
    double s = 0.0, cs = 0.0;
    if (A.a2_base) {  // |A|^2 of this slice, linear in xi between base slices
        const double *a0 = A.a2_base + (size_t)j * nn;
        const double *a1 = (j + 1 < A.n_xi) ? a0 + nn : nullptr;
        for (int i = T.t0; i < nn; i += T.nt)
            A.a2[i] = q == 0 ? a0[i] : (1.0 - frac) * a0[i] + frac * (a1 ? a1[i] : 0.0);
    }
    for (int i = T.t0; i < nn; i += T.nt) {
        if (g.active) apply_guess(A.psi, A.hist1[0], A.hist2[0], i, g);
        const double nv = (double)ncur[i];
        const double f = nv - A.n_ion[i];
        A.f_psi[i] = f;
        s += f * f;
        cs += nv;
        if constexpr (sizeof(P) == 8) {
#pragma unroll
            for (int k = 0; k < 6; ++k) Q.m[k][i] = 0.0;
        } else {
            clear_moments(A, i);
        }
        nnext[i] = 0.0;
    }
    s = block_sum(s);
    if (threadIdx.x == 0) atomicAdd(&A.sc->fnorm[0][0], s);
    if (base && A.diag_charge) {
        cs = block_sum(cs);
        if (threadIdx.x == 0) atomicAdd(&A.diag_charge[j], cs * A.h * A.h);
    }
}

// folded cell indices of an axis: the ghost's weight goes to the edge cell
__device__ __forceinline__ void fold(int right, int n, int &a, int &b) {
    a = right - 1;
    b = right;
    if (a < 0) a = -1 - a;
    if (b > n - 1) b = 2 * n - 1 - b;
    a = min(max(a, 0), n - 1);
    b = min(max(b, 0), n - 1);
}

struct CicF {
    int i00, i01, i10, i11;
    qsff::Ff w00, w01, w10, w11;
    __device__ __forceinline__ CicP<float> single() const {
        CicP<float> r;
        r.i00 = i00; r.i01 = i01; r.i10 = i10; r.i11 = i11;
        r.w00 = w00.h; r.w01 = w01.h; r.w10 = w10.h; r.w11 = w11.h;
        return r;
    }
};

__device__ __forceinline__ CicF cic_pairs(double tx, double ty, int n) {
    const qsff::AxisBits bx = qsff::axis_bits(tx), by = qsff::axis_bits(ty);
    int ax, cx, ay, cy;
    fold(bx.cell, n, ax, cx);
    fold(by.cell, n, ay, cy);
    const qsff::Ff one(1.f, 0.f), gx = one - bx.f, gy = one - by.f;
    CicF c;
    c.i00 = ay * n + ax;
    c.i01 = ay * n + cx;
    c.i10 = cy * n + ax;
    c.i11 = cy * n + cx;
    c.w00 = gy * gx;
    c.w01 = gy * bx.f;
    c.w10 = by.f * gx;
    c.w11 = by.f * bx.f;
    return c;
}

__device__ __forceinline__ qsff::Ff gather_pairs(const float2 *u, const CicF &c) {
    const float2 a = u[c.i00], b = u[c.i01], d = u[c.i10], e = u[c.i11];
    using qsff::Ff;
    return (Ff(a.x, a.y) * c.w00 + Ff(b.x, b.y) * c.w01) +
           (Ff(d.x, d.y) * c.w10 + Ff(e.x, e.y) * c.w11);
}
__device__ __forceinline__ qsff::Ff gather_pairs(const double *u, const CicF &c) {
    using namespace qsff;
    return (split(u[c.i00]) * c.w00 + split(u[c.i01]) * c.w01) +
           (split(u[c.i10]) * c.w10 + split(u[c.i11]) * c.w11);
}

// 1 + psi at a particle, not below the floor
__device__ __forceinline__ qsff::Ff one_plus_psi(qsff::Ff psi, qsff::Ff floor_, unsigned &hits) {
    qsff::Ff a = qsff::Ff(1.f, 0.f) + psi;
    if (a.h < floor_.h || (a.h == floor_.h && a.l < floor_.l)) {
        ++hits;
        a = floor_;
    }
    return a;
}

// gather psi at every particle; deposit j_perp, T, G (Eqs. Jr, FluxPres).
// gamma from the constant of motion is evaluated in float64, in the refined
// form in pairs of floats.
template <typename P>
__device__ void phase_moments(const EngineArgs &A, const PS<P> &Q, Thr T, int bid, int nblk,
                              void *smem) {
    const P s = (P)(A.inv_h * A.inv_h);
    constexpr int ST = PS<P>::stride;
    unsigned hits = 0;
    const bool sums = sums64(A);
    // privatised: this block's chunk into the six bands of sb
    const bool banded = A.band_rows > 0;
    int64_t p0 = T.t0, p1 = A.np, pst = T.nt;
    P *sb = nullptr;
    int lo = 0, hi = 0, cells = 0;
    if (banded) {
        int64_t c0, c1;
        chunk_of(A.np, bid, nblk, c0, c1);
        const Band b = band_of(A, Q.y, c0, c1, 0, A.band_rows);
        cells = b.rows * A.N;
        lo = b.r0 * A.N;
        hi = lo + cells;
        sb = (P *)((char *)smem + A.band_off);
        zero_band(sb, 6 * cells);
        __syncthreads();
        p0 = c0 + threadIdx.x;
        p1 = c1;
        pst = blockDim.x;
    }
    if constexpr (sizeof(P) == 8) {
        auto put = [&](int k, const CicP<P> &c, P q) {
            if (banded) dep_band(Q.m[k], sb + k * cells, lo, hi, c, q);
            else dep(Q.m[k], c, q);
        };
        for (int64_t p = p0; p < p1; p += pst) {
            const Cic cd = cic_stencil_inv(Q.x[p], Q.y[p], A.x_min, A.y_min, A.inv_h, A.N);
            const CicP<P> c = cic_p<P>(cd);
            const double a = guard(1.0 + cic_gather(A.psi, cd), A.psi_floor, hits);
            const P px = Q.px[p], py = Q.py[p];
            const double p2 = px * px + py * py;
            const double ia = 1.0 / a;  // one reciprocal per particle
            const P vx = px * ia, vy = py * ia;
            const P wq = Q.w[p] * s;
            // the laser's |A|^2 / 2 in the numerator of gamma (line after Eq. EoM_111)
            const double ha2 = A.a2_base ? 0.5 * cic_gather(A.a2, cd) : 0.0;
            put(M_JX, c, wq * vx);
            put(M_JY, c, wq * vy);
            put(M_TXX, c, wq * vx * vx);
            put(M_TXY, c, wq * vx * vy);
            put(M_TYY, c, wq * vy * vy);
            put(M_G, c, wq * ((1.0 + p2 + a * a + ha2) * (0.5 * ia)));  // gamma
        }
    } else {
        using qsff::Ff;
        const Ff fl = qsff::split(A.psi_floor);
        const double ox = fma(-A.x_min, A.inv_h, 0.5), oy = fma(-A.y_min, A.inv_h, 0.5);
        const int lane = threadIdx.x & 31;
        for (int64_t pw = p0 - lane; pw < p1; pw += pst) {  // whole warps
            const bool in = pw + lane < p1;
            const int64_t p = in ? pw + lane : p1 - 1;
            unsigned hit = 0;
            const CicF cf = cic_pairs(fma(Q.x[p], A.inv_h, ox), fma(Q.y[p], A.inv_h, oy), A.N);
            const CicP<P> c = cf.single();
            const Ff a = one_plus_psi(gather_pairs(A.psi2, cf), fl, hit);
            if (in) hits += hit;
            const P px = Q.px[p], py = Q.py[p];
            const Ff ia = qsff::recip(a);
            const P vx = px * ia.h, vy = py * ia.h;
            const P wq = in ? Q.w[p] * s : P(0);
            // gamma - 1 = (p^2 + psi^2 + |A|^2 / 2) / (2 (1 + psi))
            const Ff am1 = a + Ff(-1.f, 0.f);
            Ff g = qsff::two_prod(px, px) + qsff::two_prod(py, py) + am1 * am1;
            if (A.a2_base) g += gather_pairs(A.a2, cf) * 0.5f;
            g = g * (ia * 0.5f);
            const float q[6] = {wq * vx, wq * vy, wq * vx * vx, wq * vx * vy, wq * vy * vy,
                                wq * g.h};
            if (banded) {
#pragma unroll
                for (int k = 0; k < 6; ++k)
                    if (in) dep_band<ST>(Q.m[k], sb + k * cells, lo, hi, c, q[k]);
            } else if (sums) {
                if (in) dep6_float64(A, c, q);
            } else {
                dep6_pairs(A.mom32, c, q);
            }
        }
    }
    add_hits(A.sc, hits);
    if (banded) {
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 6; ++k) flush_band<ST>(Q.m[k], sb + k * cells, lo, cells);
    }
}

// central differences: zero ghosts (moments) and odd ghosts (fields)
template <int ST = 1, typename G>
__device__ __forceinline__ double dx0(const G *u, int n, int ix, int i, double inv2h) {
    const double e = ix < n - 1 ? (double)u[(size_t)(i + 1) * ST] : 0.0;
    const double w = ix > 0 ? (double)u[(size_t)(i - 1) * ST] : 0.0;
    return (e - w) * inv2h;
}
template <int ST = 1, typename G>
__device__ __forceinline__ double dy0(const G *u, int n, int iy, int i, double inv2h) {
    const double s = iy < n - 1 ? (double)u[(size_t)(i + n) * ST] : 0.0;
    const double q = iy > 0 ? (double)u[(size_t)(i - n) * ST] : 0.0;
    return (s - q) * inv2h;
}
__device__ __forceinline__ double dxo(const double *u, int n, int ix, int i, double inv2h) {
    double e = ix < n - 1 ? u[i + 1] : -u[i];
    double w = ix > 0 ? u[i - 1] : -u[i];
    return (e - w) * inv2h;
}
__device__ __forceinline__ double dyo(const double *u, int n, int iy, int i, double inv2h) {
    double s = iy < n - 1 ? u[i + n] : -u[i];
    double q = iy > 0 ? u[i - n] : -u[i];
    return (s - q) * inv2h;
}

// sources of E_z, B_z (Eqs. EqM_N8_A, Mag_z_A); j_z (Eq. Jr plus the
// driver), kappa = n_* / (1+psi) with the smoother's inverse diagonal, grad psi
template <typename P>
__device__ void phase_assemble1(const EngineArgs &A, const PS<P> &Q, const double *ncur, int j,
                                int q, double frac, Thr T, const Guess &g) {
    const int n = A.N, nn = n * n;
    constexpr int ST = PS<P>::stride;
    const double inv2h = 0.5 * A.inv_h;
    const double *J0 = A.jzb + (size_t)j * nn;
    const double *J1 = (j + 1 < A.n_xi) ? A.jzb + (size_t)(j + 1) * nn : nullptr;
    unsigned hits = 0;
    double sez = 0.0, sbz = 0.0;
    for (int i = T.t0; i < nn; i += T.nt) {
        const int iy = i / n, ix = i - iy * n;
        if (g.active) {
            apply_guess(A.ez, A.hist1[1], A.hist2[1], i, g);
            apply_guess(A.bz, A.hist1[2], A.hist2[2], i, g);
        }
        double fez = -(dx0<ST>(Q.m[M_JX], n, ix, i, inv2h) + dy0<ST>(Q.m[M_JY], n, iy, i, inv2h));
        double fbz = dx0<ST>(Q.m[M_JY], n, ix, i, inv2h) - dy0<ST>(Q.m[M_JX], n, iy, i, inv2h);
        A.f_ez[i] = fez;
        A.f_bz[i] = fbz;
        sez += fez * fez;
        sbz += fbz * fbz;
        double a = guard(1.0 + A.psi[i], A.psi_floor, hits);
        double jzb = q == 0 ? J0[i] : (1.0 - frac) * J0[i] + frac * (J1 ? J1[i] : 0.0);
        const double nv = ncur[i];
        const double ia = 1.0 / a;
        A.jz[i] = g_total(Q.mom(M_G, i), nv) * ia - nv + jzb;
        const double kap = nv * ia;
        A.kap[i] = kap;
        const int nw = qsmg::walls(ix, iy, n);
        if (A.precision == QS_FP32_REFINED) {
            const float k32 = (float)kap;
            A.k32[i] = k32;
            A.d32[i] = 1.f / ((float)(4 + nw) + A.lev_h2f[0] * k32);
        } else {
            A.invd0[i] = 1.0 / ((double)(4 + nw) + A.lev_h2[0] * kap);
        }
        A.dpx[i] = dxo(A.psi, n, ix, i, inv2h);
        A.dpy[i] = dyo(A.psi, n, iy, i, inv2h);
        if (A.dpx32) {
            A.dpx32[i] = (float)A.dpx[i];
            A.dpy32[i] = (float)A.dpy[i];
        }
        if (A.a2_base) {
            // grad(|A|^2 / 4), even ghosts (the ghost repeats the edge cell)
            const double *a2 = A.a2;
            const double e = ix < n - 1 ? a2[i + 1] : a2[i];
            const double w = ix > 0 ? a2[i - 1] : a2[i];
            const double so = iy < n - 1 ? a2[i + n] : a2[i];
            const double no = iy > 0 ? a2[i - n] : a2[i];
            A.pondx[i] = 0.25 * (e - w) * inv2h;
            A.pondy[i] = 0.25 * (so - no) * inv2h;
            if (A.chi && q == 0) A.chi[(size_t)j * nn + i] = kap;  // Eq. laser_Enve
        }
    }
    sez = block_sum(sez);
    if (threadIdx.x == 0) atomicAdd(&A.sc->fnorm[1][0], sez);
    sbz = block_sum(sbz);
    if (threadIdx.x == 0) atomicAdd(&A.sc->fnorm[1][1], sbz);
    add_hits(A.sc, hits);
}

// explicit source S of Eq. FluxCurr1_A; rhs of Eq. Main_Eq_A is -e_z x S =
// (S_y, -S_x)
template <typename P>
__device__ void phase_assemble2(const EngineArgs &A, const PS<P> &Q, const double *ncur, Thr T,
                                const Guess &g) {
    const int n = A.N, nn = n * n;
    constexpr int ST = PS<P>::stride;
    const double inv2h = 0.5 * A.inv_h;
    double sbx = 0.0, sby = 0.0;
    for (int i = T.t0; i < nn; i += T.nt) {
        const int iy = i / n, ix = i - iy * n;
        if (g.active) {
            apply_guess(A.bx, A.hist1[3], A.hist2[3], i, g);
            apply_guess(A.by, A.hist1[4], A.hist2[4], i, g);
        }
        double a = 1.0 + A.psi[i];
        if (a < A.psi_floor) a = A.psi_floor;
        const double jx = Q.mom(M_JX, i), jy = Q.mom(M_JY, i), txx = Q.mom(M_TXX, i),
                     txy = Q.mom(M_TXY, i), tyy = Q.mom(M_TYY, i),
                     G = g_total(Q.mom(M_G, i), ncur[i]), ez = A.ez[i], bz = A.bz[i];
        if (A.bz32) A.bz32[i] = (float)bz;  // B_z is final here
        const double gx = A.dpx[i], gy = A.dpy[i];
        const double ia = 1.0 / a, Gia2 = G * ia * ia;
        double sx = dx0(A.jz, n, ix, i, inv2h) - dx0<ST>(Q.m[M_TXX], n, ix, i, inv2h) -
                    dy0<ST>(Q.m[M_TXY], n, iy, i, inv2h) + Gia2 * gx -
                    (jy * bz + jx * ez + txx * gx + txy * gy) * ia;
        double sy = dy0(A.jz, n, iy, i, inv2h) - dx0<ST>(Q.m[M_TXY], n, ix, i, inv2h) -
                    dy0<ST>(Q.m[M_TYY], n, iy, i, inv2h) + Gia2 * gy +
                    (jx * bz - jy * ez - txy * gx - tyy * gy) * ia;
        if (A.a2_base) {  // -n_* grad(|A|^2/4) / (1+psi)^2 of Eq. FluxCurr1_A
            const double nia2 = ncur[i] * ia * ia;
            sx -= nia2 * A.pondx[i];
            sy -= nia2 * A.pondy[i];
        }
        A.f_bx[i] = sy;
        A.f_by[i] = -sx;
        sbx += sy * sy;
        sby += sx * sx;
    }
    sbx = block_sum(sbx);
    if (threadIdx.x == 0) atomicAdd(&A.sc->fnorm[2][0], sbx);
    sby = block_sum(sby);
    if (threadIdx.x == 0) atomicAdd(&A.sc->fnorm[2][1], sby);
}

// ---------------------------------------------------------------------------
// The same phases fused with the transforms of the direct solves: a source is
// formed where its row transform reads it, and a solution goes on to the next
// source where its inverse transform ends.  That saves three grid phases and
// the trips of six grids through L2 a slice, and in the refined form the
// sources are formed in pairs of floats, with no conversions to float64 (the
// five separate phases' FP64-pipe instructions took 37 us a 256^2 slice).
// ---------------------------------------------------------------------------
using qsff::Ff;
using qsfft::Ff2;

// source of psi (f = n_* - n_ion); charge sum; cleared accumulators
template <typename P>
__device__ void rows_psi(const EngineArgs &A, const PS<P> &Q, const double *ncur, double *nnext,
                         bool base, int j, int q, double frac, int bid, int nblk) {
    const int N = A.N, nn = N * N;
    double cs = 0.0;
    const double *a0 = A.a2_base ? A.a2_base + (size_t)j * nn : nullptr;
    const double *a1 = a0 && j + 1 < A.n_xi ? a0 + nn : nullptr;
    const bool diag = base && A.diag_charge;
    auto cell = [&](int i) {
        if (a0) A.a2[i] = q == 0 ? a0[i] : (1.0 - frac) * a0[i] + frac * (a1 ? a1[i] : 0.0);
        const double nv = ncur[i];
        if (diag) cs += nv;
        if constexpr (sizeof(P) == 8) {
#pragma unroll
            for (int k = 0; k < 6; ++k) Q.m[k][i] = 0.0;
        } else {
            clear_moments(A, i);
        }
        nnext[i] = 0.0;
        return qsff::split(nv - A.n_ion[i]);
    };
    poisson_rows<1>(A, bid, nblk, [&](int l, int x) {
        const int i = 2 * l * N + x;
        const Ff f0 = cell(i), f1 = cell(i + N);
        return qsfft::mk<Ff>(f0, f1);
    });
    if (diag) {
        cs = block_sum(cs);
        if (threadIdx.x == 0) atomicAdd(&A.diag_charge[j], cs * A.h * A.h);
    }
}

template <typename P>
__device__ void rows_psi_out(const EngineArgs &A, int bid, int nblk) {
    const int N = A.N;
    poisson_inverse<1>(A, bid, nblk, [&](int l, int x, Ff2 v) {
        const int i = 2 * l * N + x;
        A.psi[i] = qsff::join(v.x);
        A.psi[i + N] = qsff::join(v.y);
        if (sizeof(P) == 4) {
            A.psi2[i] = make_float2(v.x.h, v.x.l);
            A.psi2[i + N] = make_float2(v.y.h, v.y.l);
        }
    });
}

// grad(|A|^2 / 4) with even ghosts (the ghost repeats the edge cell)
__device__ __forceinline__ void ponderomotive(const EngineArgs &A, int ix, int iy, int i,
                                              double inv2h) {
    const int n = A.N;
    const double *a2 = A.a2;
    const double e = ix < n - 1 ? a2[i + 1] : a2[i];
    const double w = ix > 0 ? a2[i - 1] : a2[i];
    const double so = iy < n - 1 ? a2[i + n] : a2[i];
    const double no = iy > 0 ? a2[i - n] : a2[i];
    A.pondx[i] = 0.25 * (e - w) * inv2h;
    A.pondy[i] = 0.25 * (so - no) * inv2h;
}

// driver current at the cell, linear in xi between base slices
__device__ __forceinline__ double driver_jz(const double *J0, const double *J1, int i, int q,
                                            double frac) {
    return q == 0 ? J0[i] : (1.0 - frac) * J0[i] + frac * (J1 ? J1[i] : 0.0);
}

// source of E_z (c = 0) or B_z (c = 1) at a cell from the refined form's moments
__device__ __forceinline__ Ff eb_source(const EngineArgs &A, int c, int n, int ix, int iy, Ff i2h) {
    const float *const m = (const float *)A.mom32 + 8 * (size_t)(iy * n + ix);
    auto j = [&](bool in, int k, int comp) { return in ? m[8 * k + comp] : 0.f; };
    const Ff a = qsff::two_sum(j(ix < n - 1, 1, c), -j(ix > 0, -1, c)),
             b = qsff::two_sum(j(iy < n - 1, n, 1 - c), -j(iy > 0, -n, 1 - c));
    return (c ? a - b : -(a + b)) * i2h;
}

// sources of E_z, B_z; j_z, kappa and its sum, grad psi.  The refined form
// keeps j_z and grad psi as pairs of floats in the float64 grids' memory.
template <typename P>
__device__ void rows_eb(const EngineArgs &A, const PS<P> &Q, const double *ncur, int j, int q,
                        double frac, int bid, int nblk) {
    const int n = A.N, nn = n * n;
    const double inv2h = 0.5 * A.inv_h;
    const double *J0 = A.jzb + (size_t)j * nn;
    const double *J1 = (j + 1 < A.n_xi) ? J0 + nn : nullptr;
    unsigned hits = 0;
    float sums[16] = {0.f};
    const Ff fl = qsff::split(A.psi_floor), i2h = qsff::split(inv2h);
    poisson_rows<2>(A, bid, nblk, [&](int l, int ix) {
        const int iy = l, c = l & 1, i = iy * n + ix;  // this line's own row of the two
        const double nv = ncur[i];
        double kap;
        Ff2 f;
        if constexpr (sizeof(P) == 8) {
            auto src = [&](int y) {
                const int k = y * n + ix;
                const double a = dx0(Q.m[c ? M_JY : M_JX], n, ix, k, inv2h),
                             b = dy0(Q.m[c ? M_JX : M_JY], n, y, k, inv2h);
                return qsff::split(c ? a - b : -(a + b));
            };
            f = qsfft::mk<Ff>(src(l & ~1), src(l | 1));
            const double a = guard(1.0 + A.psi[i], A.psi_floor, hits), ia = 1.0 / a;
            A.jz[i] = Q.m[M_G][i] * ia - nv + driver_jz(J0, J1, i, q, frac);
            kap = nv * ia;
            A.kap[i] = kap;
            sums[0] += qsff::split(kap).h;
            A.dpx[i] = dxo(A.psi, n, ix, i, inv2h);
            A.dpy[i] = dyo(A.psi, n, iy, i, inv2h);
        } else {
            f = qsfft::mk<Ff>(eb_source(A, c, n, ix, l & ~1, i2h), eb_source(A, c, n, ix, l | 1, i2h));
            auto psi = [&](int k) {
                const float2 v = A.psi2[k];
                return Ff(v.x, v.y);
            };
            const Ff pc = psi(i), nf = qsff::split(nv);
            const Ff ia = qsff::recip(one_plus_psi(pc, fl, hits));
            const Ff jz = (nf + Ff(Q.mom(M_G, i), 0.f)) * ia - nf +
                          qsff::split(driver_jz(J0, J1, i, q, frac));
            ((float2 *)A.jz)[i] = make_float2(jz.h, jz.l);
            const Ff kf = nf * ia;
            kap = qsff::join(kf);
            A.kap[i] = kap;
            A.k32[i] = kf.h;
            sums[0] += kf.h;
            // central differences of psi with odd ghosts
            const Ff gx = ((ix < n - 1 ? psi(i + 1) : -pc) - (ix > 0 ? psi(i - 1) : -pc)) * i2h;
            const Ff gy = ((iy < n - 1 ? psi(i + n) : -pc) - (iy > 0 ? psi(i - n) : -pc)) * i2h;
            ((float2 *)A.dpx)[i] = make_float2(gx.h, gx.l);
            ((float2 *)A.dpy)[i] = make_float2(gy.h, gy.l);
            A.dpx32[i] = gx.h;
            A.dpy32[i] = gy.h;
        }
        if (A.a2_base) {
            ponderomotive(A, ix, iy, i, inv2h);
            if (A.chi && q == 0) A.chi[(size_t)j * nn + i] = kap;  // Eq. laser_Enve
        }
        return f;
    });
    sums[1] = (float)hits;
    const float t = qsfft::block_sums16(sums);
    if (threadIdx.x == 0) atomicAdd(&A.sc->ksum, (double)t);
    if (threadIdx.x == 1 && t != 0.f) atomicAdd(&A.sc->guard_hits, (unsigned long long)t);
}

// E_z, B_z from their row coefficients; explicit source S of Eq. FluxCurr1_A
// from them, the right-hand side -e_z x S = (S_y, -S_x) of Eq. Main_Eq_A with
// its norms, and its row transform: what cg_screened starts from.
template <typename P>
__device__ bool rows_eb_bp(const EngineArgs &A, const Sync &S, const PS<P> &Q, const double *ncur,
                           int bid, int nblk) {
    using T = typename std::conditional<sizeof(P) == 4, float, Ff>::type;
    using C = qsfft::V2<T>;
    const int n = A.N;
    const double inv2h = 0.5 * A.inv_h;
    double s2[2] = {0.0, 0.0};
    const Ff fl = qsff::split(A.psi_floor), i2h = qsff::split(inv2h);
    C *const cr = (C *)A.fft.cr;
    auto next = [&](int iy, int ix, Ff2 v) {
        const int i = iy * n + ix;
        const double ezd = qsff::join(v.x), bzd = qsff::join(v.y);
        A.ez[i] = ezd;
        A.bz[i] = bzd;
        double fx, fy;  // S_y, -S_x
        C r;
        if constexpr (sizeof(P) == 8) {
            double a = 1.0 + A.psi[i];
            if (a < A.psi_floor) a = A.psi_floor;
            const double jx = Q.m[M_JX][i], jy = Q.m[M_JY][i], txx = Q.m[M_TXX][i],
                         txy = Q.m[M_TXY][i], tyy = Q.m[M_TYY][i], G = Q.m[M_G][i];
            const double gx = A.dpx[i], gy = A.dpy[i];
            const double ia = 1.0 / a, Gia2 = G * ia * ia;
            double sx = dx0(A.jz, n, ix, i, inv2h) - dx0(Q.m[M_TXX], n, ix, i, inv2h) -
                        dy0(Q.m[M_TXY], n, iy, i, inv2h) + Gia2 * gx -
                        (jy * bzd + jx * ezd + txx * gx + txy * gy) * ia;
            double sy = dy0(A.jz, n, iy, i, inv2h) - dx0(Q.m[M_TXY], n, ix, i, inv2h) -
                        dy0(Q.m[M_TYY], n, iy, i, inv2h) + Gia2 * gy +
                        (jx * bzd - jy * ezd - txy * gx - tyy * gy) * ia;
            if (A.a2_base) {  // -n_* grad(|A|^2/4) / (1+psi)^2
                const double nia2 = ncur[i] * ia * ia;
                sx -= nia2 * A.pondx[i];
                sy -= nia2 * A.pondy[i];
            }
            fx = sy;
            fy = -sx;
            r = qsfft::mk<T>(qsff::split(fx), qsff::split(fy));
        } else {
            A.bz32[i] = v.y.h;  // B_z is final here
            // T_xx, T_xy, T_yy of a neighbour
            auto tt = [&](bool in, int k) {
                const float4 *m = A.mom32 + 2 * (size_t)k;
                const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
                if (!in) return z;
                const float2 d = *(const float2 *)m, b = *((const float2 *)m + 1);
                return make_float4(b.x, b.y, ((const float *)m)[4], d.x);
            };
            auto pair = [](const void *g, int k) {
                const float2 u = ((const float2 *)g)[k];
                return Ff(u.x, u.y);
            };
            const Ff zero(0.f, 0.f);
            const float4 te = tt(ix < n - 1, i + 1), tw = tt(ix > 0, i - 1),
                         ts = tt(iy < n - 1, i + n), tn = tt(iy > 0, i - n);
            const Ff dx = (ix < n - 1 ? pair(A.jz, i + 1) : zero) -
                          (ix > 0 ? pair(A.jz, i - 1) : zero) - qsff::two_sum(te.x, -tw.x) -
                          qsff::two_sum(ts.y, -tn.y);
            const Ff dy = (iy < n - 1 ? pair(A.jz, i + n) : zero) -
                          (iy > 0 ? pair(A.jz, i - n) : zero) - qsff::two_sum(te.y, -tw.y) -
                          qsff::two_sum(ts.z, -tn.z);
            const float4 m0 = A.mom32[2 * (size_t)i], m1 = A.mom32[2 * (size_t)i + 1];
            unsigned dummy = 0;
            const Ff ia = qsff::recip(one_plus_psi(pair(A.psi2, i), fl, dummy));
            const Ff nf = qsff::split(ncur[i]), gx = pair(A.dpx, i), gy = pair(A.dpy, i);
            const Ff Gia = (nf + Ff(m1.y, 0.f)) * ia;
            // the products with 1 / (1 + psi) taken out
            Ff px = Gia * gx - (v.y * m0.y + v.x * m0.x + gx * m0.z + gy * m0.w);
            Ff py = Gia * gy + (v.y * m0.x - v.x * m0.y - gx * m0.w - gy * m1.x);
            if (A.a2_base) {
                const Ff nia = nf * ia;
                px -= nia * qsff::split(A.pondx[i]);
                py -= nia * qsff::split(A.pondy[i]);
            }
            const Ff sx = dx * i2h + px * ia, sy = dy * i2h + py * ia;
            fx = qsff::join(sy);
            fy = -qsff::join(sx);
            r = make_float2(sy.h, -sx.h);
        }
        A.f_bx[i] = fx;
        A.f_by[i] = fy;
        cr[i] = r;
        s2[0] += fx * fx;
        s2[1] += fy * fy;
        return r;
    };
    const qsfft::Lines PF = fft_lines<Ff>(A), PT = fft_lines<T>(A);
    if (PF.gmax >= 2) {
        qsfft::rows_inverse_forward<Ff, T, 2>(PF, PT, bid, nblk, (const Ff2 *)A.fft.t2,
                                              (C *)A.fft.t1, next);
    } else {  // one line a block (sides above 1078): the fields first
        poisson_inverse<2>(A, bid, nblk, [&](int l, int x, Ff2 v) {
            double *const u = l & 1 ? A.bz : A.ez;
            const int i = (l & ~1) * n + x;
            u[i] = qsff::join(v.x);
            u[i + n] = qsff::join(v.y);
        });
        SYNC(34);
        qsfft::rows_forward<T, 2>(PT, bid, nblk, (C *)A.fft.t1, [&](int iy, int ix) {
            const int i = iy * n + ix;
            return next(iy, ix, qsfft::mk<Ff>(qsff::split(A.ez[i]), qsff::split(A.bz[i])));
        });
    }
    block_sum_wide(s2, A.sc->fnorm[2]);
    return true;
}

// The sums of poisson_test: residuals of psi, E_z and B_z with their sources
// formed anew, at cells q0 ... q1.  Bound by the FP64 pipe, 27 instructions a cell.
// acc: a thread's sums of the parts before (not the first) and after (not the last).
template <typename P>
__device__ __noinline__ void poisson_residuals(const EngineArgs &A, const PS<P> &Q,
                                               const double *ncur, int q0, int q1, Thr T,
                                               double *acc, bool first, bool last) {
    const int n = A.N;
    const double ih2 = A.lev_inv_h2[0], inv2h = 0.5 * A.inv_h;
    const Ff i2h = qsff::split(inv2h);
    double s[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) s[k] = first ? 0.0 : acc[k];
    for (qsmg::Walk w(q0 + T.t0, T.nt, n); w.q < q1; w.next()) {
        const int i = w.q, ix = w.col, iy = w.row;
        double f[2];
        if constexpr (sizeof(P) == 8) {
            f[0] = -(dx0(Q.m[M_JX], n, ix, i, inv2h) + dy0(Q.m[M_JY], n, iy, i, inv2h));
            f[1] = dx0(Q.m[M_JY], n, ix, i, inv2h) - dy0(Q.m[M_JX], n, iy, i, inv2h);
        } else {
            f[0] = qsff::join(eb_source(A, 0, n, ix, iy, i2h));
            f[1] = qsff::join(eb_source(A, 1, n, ix, iy, i2h));
        }
        poisson_point(A.psi, ncur[i] - A.n_ion[i], n, ix, iy, i, ih2, s, 0);
        poisson_point(A.ez, f[0], n, ix, iy, i, ih2, s, 1);
        poisson_point(A.bz, f[1], n, ix, iy, i, ih2, s, 2);
    }
    if (last) {
        block_sum_wide(s, &A.sc->pchk[0][0]);
    } else {
#pragma unroll
        for (int k = 0; k < 9; ++k) acc[k] = s[k];
    }
}

// These residuals beside the B_perp solve.  Its phases leave blocks without a line
// (G lines a block, a power of two: 24 of 152 at 128^2 to 512^2): they do a part of
// the cells in each iteration, of 3 N cells a block, which takes about as long as the
// others' two phases; what is left at the end all blocks do.  Refined blowout at
// 256^2, a slice without the residuals 197 us: all blocks in one phase +8.3 us, idle
// blocks with a part in each phase (2 N, N, N / 2 cells) +8, +6, +10, a part in each
// iteration (N, 2 N, 3 N, 4 N, 6 N) +9, +5, +4, +5, +12.  Where no block
// is idle all do them in the first phase.
template <typename P>
struct PoissonCheck {
    const EngineArgs &A;
    const PS<P> &Q;
    const double *ncur;
    int bid, nblk, rank, cnt, part, parts;
    __device__ PoissonCheck(const EngineArgs &A_, const PS<P> &Q_, const double *ncur_, int bid_,
                            int nblk_)
        : A(A_), Q(Q_), ncur(ncur_), bid(bid_), nblk(nblk_), rank(bid_), cnt(nblk_), part(0),
          parts(1) {
        const int n = A.N, G = 1 << qsfft::lines_at_once(n, nblk, A.fft.gmax);
        const int busy = (n + G - 1) / G;
        if (busy < nblk) {
            rank = bid - busy;
            cnt = nblk - busy;
            const int per = cnt * max(3 * n, 128);
            parts = (n * n + per - 1) / per;
        }
    }
    __device__ __forceinline__ int begin(int k) const {
        const int nn = A.N * A.N, len = (nn + parts - 1) / parts;
        return min(nn, k * len);
    }
    // the sums between the parts: over the line buffers, which an idle block does
    // not use
    __device__ __forceinline__ double *acc() const {
        return (double *)(qsfft::dyn_smem() + A.block_smem_offset) + 9 * (int)threadIdx.x;
    }
    __device__ bool idle() const { return cnt < nblk && rank >= 0; }
    __device__ void operator()() {
        if (part == parts) return;
        if (rank >= 0)
            poisson_residuals<P>(A, Q, ncur, begin(part), begin(part + 1), grid_thr(rank, cnt),
                                 acc(), part == 0, part + 1 == parts);
        ++part;
    }
    __device__ void rest() {
        if (part == parts) return;
        poisson_residuals<P>(A, Q, ncur, begin(part), A.N * A.N, grid_thr(bid, nblk), acc(),
                             part == 0 || rank < 0, true);
        part = parts;
    }
};

// (double)i for 0 <= i < 2^31 without a conversion: 2^52 + i is exact
__device__ __forceinline__ double whole(int i) {
    return __hiloint2double(0x43300000, i) - 4503599627370496.0;
}

// specular wall
template <typename P>
__device__ __forceinline__ void reflect(double &x, P &p, double lo, double hi) {
    if (x > hi) { x = 2.0 * hi - x; p = -p; }
    if (x < lo) { x = 2.0 * lo - x; p = -p; }
}

// The Boris-like momentum step: half kick (gamma grad psi - grad(|A|^2/4)) /
// (1+psi) + e_z x B_perp, rotation by the B_z term (e_z x p) B_z / (1+psi),
// half kick with the new gamma.
template <typename P, typename F>
__device__ __forceinline__ void boris_like(P &px, P &py, F gamma, P gx, P gy, P bx, P by, P bz,
                                           P fx, P fy, P ia, P half) {
    const P gam = gamma(px, py);
    const P pxm = px + half * ((gam * gx - fx) * ia - by);
    const P pym = py + half * ((gam * gy - fy) * ia + bx);
    const P tau = half * bz * ia;
    const P pxp = pxm - tau * pym;
    const P pyp = pym + tau * pxm;
    const P sr = P(2) * tau / (P(1) + tau * tau);
    const P pxr = pxm - sr * pyp;
    const P pyr = pym + sr * pxp;
    const P gam2 = gamma(pxr, pyr);
    px = pxr + half * ((gam2 * gx - fx) * ia - by);
    py = pyr + half * ((gam2 * gy - fy) * ia + bx);
}

// store the base slice; push every trajectory (Eqs. EoM_112_A, EoM_111);
// deposit n_* of the next slice; V_max.  gamma is evaluated in float64.
template <typename P>
__device__ void phase_push(const EngineArgs &A, const PS<P> &Q, double *nnext, bool base,
                           bool last, int j, double dxi, int pk, int sub, Thr T, int bid,
                           int nblk, void *smem) {
    const int nn = A.N * A.N;
    if (A.seg_g && sub < A.seg_cap) {  // segment store for the adjoint (float64)
        double *g = A.seg_g + (size_t)sub * SG_COUNT * nn;
        const double *ncur = Q.na == nnext ? Q.nb : Q.na;
        for (int i = T.t0; i < nn; i += T.nt) {
            g[SG_PSI * nn + i] = A.psi[i];
            g[SG_EZ * nn + i] = A.ez[i];
            g[SG_BZ * nn + i] = A.bz[i];
            g[SG_BX * nn + i] = A.bx[i];
            g[SG_BY * nn + i] = A.by[i];
            g[SG_N * nn + i] = ncur[i];
            g[SG_JX * nn + i] = (double)Q.mom(M_JX, i);
            g[SG_JY * nn + i] = (double)Q.mom(M_JY, i);
            g[SG_TXX * nn + i] = (double)Q.mom(M_TXX, i);
            g[SG_TXY * nn + i] = (double)Q.mom(M_TXY, i);
            g[SG_TYY * nn + i] = (double)Q.mom(M_TYY, i);
            g[SG_G * nn + i] = g_total(Q.mom(M_G, i), ncur[i]);
        }
        double *sp = A.seg_p + (size_t)sub * 4 * A.np;
        for (int64_t p = T.t0; p < A.np; p += T.nt) {
            sp[p] = Q.x[p];
            sp[A.np + p] = Q.y[p];
            sp[2 * A.np + p] = (double)Q.px[p];
            sp[3 * A.np + p] = (double)Q.py[p];
        }
    }
    if (base && A.hist) {
        double *h0 = A.hist + (size_t)j * nn;
        const size_t fs = (size_t)A.n_xi * nn;
        for (int i = T.t0; i < nn; i += T.nt) {
            h0[i] = A.psi[i];
            h0[fs + i] = A.ez[i];
            h0[2 * fs + i] = A.bz[i];
            h0[3 * fs + i] = A.bx[i];
            h0[4 * fs + i] = A.by[i];
        }
    }
    if (last) return;
    const double s = A.inv_h * A.inv_h;
    const P half = (P)(0.5 * dxi), dxp = (P)dxi;
    unsigned hits = 0;
    P vm = P(0);  // the square of V_max (refined form: in float32)
    // privatised n_* of the next slice: the band of the chunk's present rows
    // widened by two rows for the particles' motion
    const bool banded = A.band_rows_n > 0;
    int64_t p0 = T.t0, p1 = A.np, pst = T.nt;
    double *sb = nullptr;
    int lo = 0, hi = 0, cells = 0;
    if (banded) {
        int64_t c0, c1;
        chunk_of(A.np, bid, nblk, c0, c1);
        const Band b = band_of(A, Q.y, c0, c1, 2, A.band_rows_n);
        cells = b.rows * A.N;
        lo = b.r0 * A.N;
        hi = lo + cells;
        sb = (double *)((char *)smem + A.band_off);
        zero_band(sb, cells);
        __syncthreads();
        p0 = c0 + threadIdx.x;
        p1 = c1;
        pst = blockDim.x;
    }
    if constexpr (sizeof(P) == 8) {
        for (int64_t p = p0; p < p1; p += pst) {
            const double x = Q.x[p], y = Q.y[p];
            const Cic cd = cic_stencil_inv(x, y, A.x_min, A.y_min, A.inv_h, A.N);
            const CicP<P> c = cic_p<P>(cd);
            const double a = guard(1.0 + cic_gather(A.psi, cd), A.psi_floor, hits);
            const double ia = 1.0 / a;
            const P gx = gat<P>(A.dpx, c), gy = gat<P>(A.dpy, c), bx = gat<P>(A.bx, c),
                    by = gat<P>(A.by, c), bz = gat<P>(A.bz, c);
            P px = Q.px[p], py = Q.py[p];
            // laser (Eq. EoM_111): |A|^2 / 2 in gamma and the ponderomotive force
            // -grad(|A|^2/4) / (1+psi); zero without a laser
            double ha2 = 0.0;
            P fx = P(0), fy = P(0);
            if (A.a2_base) {
                ha2 = 0.5 * cic_gather(A.a2, cd);
                fx = gat<P>(A.pondx, c);
                fy = gat<P>(A.pondy, c);
            }
            const double q1 = 1.0 + a * a + ha2, h_ia = 0.5 * ia;
            auto gamma = [&](P u, P v) { return (q1 + u * u + v * v) * h_ia; };
            boris_like(px, py, gamma, gx, gy, bx, by, bz, fx, fy, ia, half);
            double nx = x + dxp * px * ia;
            double ny = y + dxp * py * ia;
            reflect(nx, px, A.x_min, A.x_max);
            reflect(ny, py, A.y_min, A.y_max);
            Q.x[p] = nx;
            Q.y[p] = ny;
            Q.px[p] = px;
            Q.py[p] = py;
            vm = fmax(vm, (px * px + py * py) * (ia * ia));
            const Cic c2 = cic_stencil_inv(nx, ny, A.x_min, A.y_min, A.inv_h, A.N);
            if (banded) dep_band(nnext, sb, lo, hi, c2, Q.wd[p] * s);
            else cic_deposit(nnext, c2, Q.wd[p] * s);
        }
    } else {
        using qsff::Ff;
        const Ff fl = qsff::split(A.psi_floor), one(1.f, 0.f);
        const double ox = fma(-A.x_min, A.inv_h, 0.5), oy = fma(-A.y_min, A.inv_h, 0.5);
        for (int64_t p = p0; p < p1; p += pst) {
            const double x = Q.x[p], y = Q.y[p];
            const CicF cf = cic_pairs(fma(x, A.inv_h, ox), fma(y, A.inv_h, oy), A.N);
            const CicP<P> c = cf.single();
            const Ff a = one_plus_psi(gather_pairs(A.psi2, cf), fl, hits);
            const Ff ia2 = qsff::recip(a);
            const P ia = ia2.h;
            const P gx = gat<P>(A.dpx32, c), gy = gat<P>(A.dpy32, c), bx = gat<P>(A.bx32, c),
                    by = gat<P>(A.by32, c), bz = gat<P>(A.bz32, c);
            P px = Q.px[p], py = Q.py[p];
            Ff q1 = one + a * a;
            P fx = P(0), fy = P(0);
            if (A.a2_base) {
                q1 += gather_pairs(A.a2, cf) * 0.5f;
                fx = gat<P>(A.pondx, c);
                fy = gat<P>(A.pondy, c);
            }
            const Ff h_ia = ia2 * 0.5f;
            auto gamma = [&](P u, P v) {
                return ((q1 + (qsff::two_prod(u, u) + qsff::two_prod(v, v))) * h_ia).h;
            };
            boris_like(px, py, gamma, gx, gy, bx, by, bz, fx, fy, ia, half);
            double nx = x + qsff::widen(dxp * px * ia);
            double ny = y + qsff::widen(dxp * py * ia);
            double tx = fma(nx, A.inv_h, ox), ty = fma(ny, A.inv_h, oy);
            qsff::AxisBits ax = qsff::axis_bits(tx), ay = qsff::axis_bits(ty);
            // only a particle in the half cells at the walls can have crossed one
            if ((unsigned)(ax.cell - 1) >= (unsigned)(A.N - 1) ||
                (unsigned)(ay.cell - 1) >= (unsigned)(A.N - 1)) {
                reflect(nx, px, A.x_min, A.x_max);
                reflect(ny, py, A.y_min, A.y_max);
                tx = fma(nx, A.inv_h, ox);
                ty = fma(ny, A.inv_h, oy);
                ax = qsff::axis_bits(tx);
                ay = qsff::axis_bits(ty);
            }
            Q.x[p] = nx;
            Q.y[p] = ny;
            Q.px[p] = px;
            Q.py[p] = py;
            vm = fmaxf(vm, (px * px + py * py) * (ia * ia));
            // n_* stays in float64: it must cancel n_ion to rounding
            Cic c2;
            int i0, i1, j0, j1;
            fold(ax.cell, A.N, i0, i1);
            fold(ay.cell, A.N, j0, j1);
            c2.i00 = j0 * A.N + i0;
            c2.i01 = j0 * A.N + i1;
            c2.i10 = j1 * A.N + i0;
            c2.i11 = j1 * A.N + i1;
            const double wx = tx - whole(ax.cell), wy = ty - whole(ay.cell);
            const double q = Q.wd[p] * s, qy = q * wy, qn = q - qy;
            const double q11 = qy * wx, q01 = qn * wx;
            const double q10 = qy - q11, q00 = qn - q01;
            if (banded && min(min(c2.i00, c2.i01), min(c2.i10, c2.i11)) >= lo &&
                max(max(c2.i00, c2.i01), max(c2.i10, c2.i11)) < hi) {
                atomicAdd(sb + (c2.i00 - lo), q00);
                atomicAdd(sb + (c2.i01 - lo), q01);
                atomicAdd(sb + (c2.i10 - lo), q10);
                atomicAdd(sb + (c2.i11 - lo), q11);
            } else {
                atomicAdd(nnext + c2.i00, q00);
                atomicAdd(nnext + c2.i01, q01);
                atomicAdd(nnext + c2.i10, q10);
                atomicAdd(nnext + c2.i11, q11);
            }
        }
    }
    add_hits(A.sc, hits);
    if (banded) {
        __syncthreads();
        flush_band(nnext, sb, lo, cells);
    }
    double vmax = block_max(vm);
    if (threadIdx.x == 0) {
        vmax = sqrt(vmax);
        atomicMax(&A.sc->vmax_bits[pk & 1], (unsigned long long)__double_as_longlong(vmax));
        atomicMax(&A.sc->vmax_all_bits, (unsigned long long)__double_as_longlong(vmax));
    }
}

// ---------------------------------------------------------------------------
// cell sort inside the slice loop
// ---------------------------------------------------------------------------

// exclusive scan of v over the block (any blockDim.x <= 1024); returns the
// prefix of this thread and the block total in *total
__device__ int block_exscan(int v, int *total) {
    int *const ws = (int *)qsfft::sum_scratch();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int x = v;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    __syncthreads();
    if (lane == 31) ws[wid] = x;
    __syncthreads();
    if (wid == 0) {
        const int nw = (blockDim.x + 31) >> 5;
        int t = lane < nw ? ws[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        ws[lane] = t;  // inclusive prefix of the warp sums
    }
    __syncthreads();
    *total = ws[((blockDim.x + 31) >> 5) - 1];
    return x - v + (wid > 0 ? ws[wid - 1] : 0);
}

// Stable counting sort of the plasma by (cell, id), cell = iy N + ix of the
// position's cell (floor, clamped), the order of the standalone cell sort;
// the arrays are gathered into the spare set and copied back (the slice
// loop's particle pointers stay fixed: swapping them would keep two sets of
// pointers live in registers through the whole loop).
template <typename P>
__device__ __noinline__ bool sort_plasma(const EngineArgs &A, const PS<P> &Q, const Sync &S,
                                         int bid, int nblk) {
    int32_t *const id = A.id, *const id2 = A.id2;
    P *const px2 = (P *)A.px2, *const py2 = (P *)A.py2, *const w2 = (P *)A.w2;
    const int nn = A.N * A.N;
    const Thr T = grid_thr(bid, nblk);
    for (int i = T.t0; i < nn; i += T.nt) A.s_count[i] = 0;
    SYNC(90);
    for (int64_t p = T.t0; p < A.np; p += T.nt) {
        int ix = (int)floor((Q.x[p] - A.x_min) * A.inv_h);
        int iy = (int)floor((Q.y[p] - A.y_min) * A.inv_h);
        ix = min(max(ix, 0), A.N - 1);
        iy = min(max(iy, 0), A.N - 1);
        const int c = iy * A.N + ix;
        A.s_cell[p] = c;
        atomicAdd(A.s_count + c, 1);
    }
    SYNC(91);
    // exclusive scan: each block its chunk of cells, then the chunk offsets
    const int ch = (nn + nblk - 1) / nblk;
    const int c0 = min(bid * ch, nn), c1 = min(c0 + ch, nn);
    int run = 0;
    for (int b = c0; b < c1; b += blockDim.x) {
        const int i = b + (int)threadIdx.x;
        int tot;
        const int pre = block_exscan(i < c1 ? A.s_count[i] : 0, &tot);
        if (i < c1) A.s_offset[i] = run + pre;
        run += tot;
    }
    if (threadIdx.x == 0) A.s_bsum[bid] = run;
    SYNC(92);
    __shared__ int s_base;
    if (threadIdx.x == 0) {
        int base = 0;
        for (int b = 0; b < bid; ++b) base += A.s_bsum[b];
        s_base = base;
        if (bid == nblk - 1) A.s_offset[nn] = base + run;
    }
    __syncthreads();
    for (int i = c0 + (int)threadIdx.x; i < c1; i += blockDim.x) {
        A.s_offset[i] += s_base;
        A.s_cursor[i] = A.s_offset[i];
    }
    SYNC(93);
    for (int64_t p = T.t0; p < A.np; p += T.nt)
        A.s_order[atomicAdd(A.s_cursor + A.s_cell[p], 1)] = (int32_t)p;
    SYNC(94);
    // within a cell, ascending id (segments hold a few particles)
    for (int i = T.t0; i < nn; i += T.nt) {
        const int b = A.s_offset[i], e = A.s_offset[i + 1];
        for (int k = b + 1; k < e; ++k) {
            const int32_t v = A.s_order[k], key = id[v];
            int m = k - 1;
            while (m >= b && id[A.s_order[m]] > key) {
                A.s_order[m + 1] = A.s_order[m];
                --m;
            }
            A.s_order[m + 1] = v;
        }
    }
    SYNC(95);
    const bool sep_wd = (const void *)Q.wd != (const void *)Q.w;
    for (int64_t s = T.t0; s < A.np; s += T.nt) {
        const int32_t p = A.s_order[s];
        A.x2[s] = Q.x[p];
        A.y2[s] = Q.y[p];
        px2[s] = Q.px[p];
        py2[s] = Q.py[p];
        w2[s] = Q.w[p];
        if (sep_wd) A.wd2[s] = Q.wd[p];
        id2[s] = id[p];
    }
    SYNC(96);
    for (int64_t s = T.t0; s < A.np; s += T.nt) {
        Q.x[s] = A.x2[s];
        Q.y[s] = A.y2[s];
        Q.px[s] = px2[s];
        Q.py[s] = py2[s];
        Q.w[s] = w2[s];
        if (sep_wd) Q.wd[s] = A.wd2[s];
        id[s] = id2[s];
    }
    SYNC(97);
    return true;
}

// One 3D step of one instance on `nblk` blocks (this one is `bid`): the xi
// loop of Algorithm 1.  Returns false if a barrier failed (the error word of
// the instance says why).
template <bool REF>
__device__ bool run_step(const EngineArgs &A, int bid, int nblk, const Sync &S, void *smem,
                         int *s_inv_ready) {
    if (A.trace && bid == 0 && threadIdx.x == 0) {
        A.trace[0] = 0;
        A.trace[1] = global_ns();
        A.sc->trace_n = 1;
    }
    DevScalars *sc = A.sc;
    const Thr T = grid_thr(bid, nblk);
    const bool lead = (bid == 0 && threadIdx.x == 0);
    fft_load_tables<REF>(A);

    using P = typename std::conditional<REF, float, double>::type;
    PS<P> Q;
    if constexpr (REF) {
        float *const f = (float *)A.mom32;
        Q = PS<P>{A.x, A.y, A.px32, A.py32, A.w32, A.w, A.n_a, A.n_b,
                  {f, f + 1, f + 2, f + 3, f + 4, f + 5}};
    } else {
        Q = PS<P>{A.x, A.y, A.px, A.py, A.w, A.w, A.n_a, A.n_b,
                  {A.jx, A.jy, A.txx, A.txy, A.tyy, A.G}};
    }
    // the spare particle set of the in-loop sort (not with the adjoint's
    // checkpoints or slice store: those keep the lattice's order)
    const bool sorting = A.sort_every > 0 && A.x2 && !A.ckpt && !A.seg_p;
    int n_sorts = 0;
    double *ncur = Q.na, *nnext = Q.nb;
    phase_deposit_n<P>(A, Q, ncur, T);
    if (!S(1)) return false;

    const SolveSpec Vpsi{1, 0, {A.psi, nullptr}, {A.f_psi, nullptr}, false};
    const SolveSpec Veb{2, 1, {A.ez, A.bz}, {A.f_ez, A.f_bz}, false};
    const SolveSpec Vbp{2, 2, {A.bx, A.by}, {A.f_bx, A.f_by}, true,
                        {REF ? A.bx32 : nullptr, REF ? A.by32 : nullptr}};

    int m = A.m_sched ? A.m_sched[A.j_begin] : 1;
    // per-slice scalars computed by thread 0 and read by every thread
    __shared__ struct {
        Guess g;
        double frac, dxi;
        int m;
    } s_ctl;
    __syncthreads();
    if (threadIdx.x == 0) s_ctl.dxi = A.dxi0 / m;
    __syncthreads();
    int slot = 0, pk = 0, sub = 0;
    int have = 0;                        // previous solutions available for the guess
    double gx0 = 0.0, gx1 = 0.0, gx2 = 0.0;  // their xi
    for (int j = A.j_begin; j < A.j_end; ++j) {
        if (sorting && j > A.j_begin && j % A.sort_every == 0) {
            if (!sort_plasma<P>(A, Q, S, bid, nblk)) return false;
            ++n_sorts;
            if (lead) sc->sorts = n_sorts;
        }
        if (lead && A.diag_m) {
            A.diag_m[j] = m;
            if (m > sc->max_m) sc->max_m = m;
        }
        const bool last = (j == A.n_xi - 1);
        const double dxi = s_ctl.dxi;
        if (A.ckpt && j % A.ckpt_every == 0) {  // plasma state before slice j
            double *cp = A.ckpt + (size_t)(j / A.ckpt_every) * 4 * A.np;
            for (int64_t p = T.t0; p < A.np; p += T.nt) {
                cp[p] = Q.x[p];
                cp[A.np + p] = Q.y[p];
                cp[2 * A.np + p] = (double)Q.px[p];
                cp[3 * A.np + p] = (double)Q.py[p];
            }
        }
        for (int q = 0; q < m; ++q) {
            const bool base = (q == 0);
            const double xs = j * A.dxi0 + q * dxi;  // xi of this slice (from xi_min)
            // the guess weights and the sub-step fraction by one thread
            // (float64 divides repeated by every thread cost microseconds)
            __syncthreads();
            if (threadIdx.x == 0) {
                if (!A.fft.on) s_ctl.g = make_guess(A.ws_order, have, xs, gx0, gx1, gx2);
                s_ctl.frac = q == 0 ? 0.0 : (double)q / (double)m;
            }
            __syncthreads();
            const Guess g = s_ctl.g;
            const double frac = s_ctl.frac;
            if (A.fft.on) {
                if (bid == nblk - 1) poisson_test(A);  // of the slice before
                rows_psi<P>(A, Q, ncur, nnext, base, j, q, frac, bid, nblk);
                SYNC(2);
                poisson_columns<1>(A, bid, nblk);
                SYNC(27);
                rows_psi_out<P>(A, bid, nblk);
                SYNC(28);
                phase_moments<P>(A, Q, T, bid, nblk, smem);
                SYNC(3);
                if (sums64(A)) {
                    round_moments(A, T);
                    SYNC(33);
                }
                rows_eb<P>(A, Q, ncur, j, q, frac, bid, nblk);
                SYNC(4);
                poisson_columns<2>(A, bid, nblk);
                SYNC(29);
                if (!rows_eb_bp<P>(A, S, Q, ncur, bid, nblk)) return false;
                SYNC(5);
                PoissonCheck<P> check(A, Q, ncur, bid, nblk);
                if (!mg_solve<REF>(A, S, Vbp, slot, bid, nblk, smem, s_inv_ready, true, check))
                    return false;
            } else {
                phase_psi_rhs<P>(A, Q, ncur, nnext, base, j, q, frac, T, g);
                if (!S(2)) return false;
                if (!mg_cycles<REF>(A, S, Vpsi, slot, bid, nblk, smem, s_inv_ready)) return false;
                if (REF) {  // psi as pairs, for the gathers
                    for (int i = T.t0; i < A.N * A.N; i += T.nt) {
                        const qsff::Ff v = qsff::split(A.psi[i]);
                        A.psi2[i] = make_float2(v.h, v.l);
                    }
                    if (!S(7)) return false;
                }
                phase_moments<P>(A, Q, T, bid, nblk, smem);
                if (!S(3)) return false;
                if (sums64(A)) {
                    round_moments(A, T);
                    if (!S(33)) return false;
                }
                phase_assemble1<P>(A, Q, ncur, j, q, frac, T, g);
                if (!S(4)) return false;
                if (!mg_cycles<REF>(A, S, Veb, slot, bid, nblk, smem, s_inv_ready)) return false;
                phase_assemble2<P>(A, Q, ncur, T, g);
                if (!S(5)) return false;
                if (!mg_cycles<REF>(A, S, Vbp, slot, bid, nblk, smem, s_inv_ready)) return false;
            }
            phase_push<P>(A, Q, nnext, base, last, j, dxi, pk, sub, T, bid, nblk, smem);
            ++sub;
            if (lead) {
                sc->slices += 1;
                if (!last) {
                    sc->pushes += A.np;
                    sc->vmax_bits[(pk + 1) & 1] = 0ull;
                }
                sc->fnorm[0][0] = sc->fnorm[0][1] = 0.0;
                sc->fnorm[1][0] = sc->fnorm[1][1] = 0.0;
                sc->fnorm[2][0] = sc->fnorm[2][1] = 0.0;
                sc->ksum = 0.0;
            }
            if (!S(6)) return false;
            gx2 = gx1;
            gx1 = gx0;
            gx0 = xs;
            have = min(have + 1, 3);
            if (last) break;
            double *t = ncur;
            ncur = nnext;
            nnext = t;
            ++pk;
        }
        if (last) break;
        // the next base slice's sub-steps (Sec. 5.1), by one thread
        __syncthreads();
        if (threadIdx.x == 0) {
            const double vm =
                __longlong_as_double((long long)vload(&sc->vmax_bits[(pk - 1) & 1]));
            if (lead && A.diag_vmax) A.diag_vmax[j] = vm;
            int mn;
            if (A.m_sched) {
                mn = A.m_sched[j + 1];
            } else if (vm <= A.V0) {
                mn = 1;
            } else {
                double r = ceil(vm / A.V0);
                mn = r > (double)A.refine_k ? A.refine_k : (int)r;
                if (mn < 1) mn = 1;
            }
            s_ctl.m = mn;
            s_ctl.dxi = A.dxi0 / mn;
        }
        __syncthreads();
        m = s_ctl.m;
    }
    if (A.fft.on && bid == nblk - 1) poisson_test(A);
    return true;
}

// The arguments are copied into shared memory once: the phases take them by
// reference, and a reference to a by-value kernel parameter would make a
// per-thread copy in local memory.
template <bool REF>
__global__ void __launch_bounds__(QS_ENGINE_THREADS, 1) slice_engine(const __grid_constant__ EngineArgs A0) {
    extern __shared__ __align__(16) double smem[];
    __shared__ unsigned long long s_epoch;
    __shared__ int s_inv_ready[2];
    __shared__ EngineArgs A;
    for (int k = threadIdx.x; k < (int)(sizeof(EngineArgs) / 4); k += blockDim.x)
        ((int *)&A)[k] = ((const int *)&A0)[k];
    if (threadIdx.x == 0) {
        s_epoch = 0ull;
        s_inv_ready[0] = s_inv_ready[1] = 0;
    }
    __syncthreads();
    // A launch without the configured thread-block clusters (a profiler's
    // kernel replay can drop the attribute) would reach distributed shared
    // memory of blocks that are not there: every block returns at once with
    // an error instead, before the first grid barrier.
    if (A.cl_size > 1 && (int)cooperative_groups::this_cluster().num_blocks() != A.cl_size) {
        if (threadIdx.x == 0 && atomicCAS(&A.sc->err, 0, QS_ERR_CUDA) == 0)
            A.sc->err_where = -1;
        return;
    }
    const Sync S{A.sc, &A.sc->bar_arrive, gridDim.x, A.spin_cycles, A.trace, A.trace_cap,
                 &s_epoch, blockIdx.x == 0, A.cl_size};
    run_step<REF>(A, blockIdx.x, gridDim.x, S, smem, s_inv_ready);
}

// Batched form: the launch is split into teams of `team` consecutive blocks;
// each team takes the next instance from a device-side queue, runs its whole
// 3D step behind the team's own barrier, and repeats until the queue is
// empty.  Instances may differ in size, tiles and sweeps.
template <bool REF>
__global__ void __launch_bounds__(QS_ENGINE_THREADS, 1)
    slice_engine_batched(const EngineArgs *list, int n_inst, int team, BatchState *bs) {
    extern __shared__ __align__(16) double smem[];
    __shared__ unsigned long long s_epoch;
    __shared__ int s_inv_ready[2];
    __shared__ EngineArgs sA;
    const int tid = blockIdx.x / team, bid = blockIdx.x % team;
    if (threadIdx.x == 0) s_epoch = 0ull;
    __syncthreads();
    for (;;) {
        if (bid == 0 && threadIdx.x == 0) {
            bs->team_inst[tid] = atomicAdd(&bs->next, 1);
            __threadfence();
        }
        // team barrier on the team's counter (errors of a finished instance do
        // not concern the next one, so this one checks the batch error word)
        const Sync T0{&bs->sc, &bs->team_bar[tid], (unsigned)team, list[0].spin_cycles, nullptr,
                      0, &s_epoch, false};
        if (!T0(60)) return;
        const int idx = vload(&bs->team_inst[tid]);
        if (idx >= n_inst) return;
        for (int k = threadIdx.x; k < (int)(sizeof(EngineArgs) / 4); k += blockDim.x)
            ((int *)&sA)[k] = ((const int *)(list + idx))[k];
        if (threadIdx.x == 0) s_inv_ready[0] = s_inv_ready[1] = 0;
        __syncthreads();
        const Sync S{sA.sc, &bs->team_bar[tid], (unsigned)team, sA.spin_cycles, nullptr, 0,
                     &s_epoch, false};
        if (!run_step<REF>(sA, bid, team, S, smem, s_inv_ready)) {
            // the instance failed: its blocks stop; record it for the batch
            if (bid == 0 && threadIdx.x == 0) atomicCAS(&bs->sc.err, 0, vload(&sA.sc->err));
            return;
        }
    }
}

}  // namespace
