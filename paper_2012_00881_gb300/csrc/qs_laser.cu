// Laser-envelope advance (Sec. "Description of different plasma wake
// drivers", Eq. laser_Enve): the complex envelope A of a laser with vector
// potential A exp(-i k0 xi) obeys
//     (2 i k0 d_t - 2 d_t d_xi + lap_perp) A = chi A,   chi = n_* / (1 + psi).
// Time-centred in t, the mixed derivative as the time difference of a
// backward (towards the head) difference in xi, so slices advance from the
// head j = 0 to the tail, each one a complex screened-Poisson equation
//     (lap - kappa) A^{n+1}_j = (c + chi_j - lap) A^n_j - q (A^{n+1}_{j-1} - A^n_{j-1}),
//     kappa = chi_j - c,   c = 4 (i k0 - 1/dxi) / dt,   q = 4 / (dt dxi)
// (dxi = inf: q = 0, c = 4 i k0 / dt).  chi is held at t_n; A = 0 ahead of
// the window and on the walls (odd ghosts, the slice advance's cell-centred
// 5-point Laplacian).  The paper solves it with the same multigrid as the
// wake, warm-started from the previous time step (Sec. 7.1).
//
// Solver: where the side has an odd factor of at most 7 (and max_cycles is not a
// tight cap), conjugate gradients for the complex symmetric operator
// (COCG, van der Vorst and Melissen, IEEE Trans. Magn. 26 (1990) 706) on the
// change of the slice's envelope, preconditioned with M = lap - chibar + c by
// sine transforms (qs_fft.cuh, which see for the phases and the recurrences
// in transformed rows): A z = r + (chibar - chi) z.  |c| is large, so few
// iterations are needed (256^2 blowout: 4 to 6), each two grid phases of 9.5 us,
// against seven V-cycles of nine phases (110 us a slice, before 1,070).  The iteration is in pairs of floats; its end
// forms the float64 residual and, if that is above the bound, starts again
// on it.  Otherwise, or when that does not converge:
//
// complex multigrid V(2,2) on the cell-centred grid, red-black
// Gauss-Seidel (the 5-point operator decouples the colours), 4-cell average
// restriction of the residual and of kappa, bilinear prolongation with odd
// ghosts, rediscretised coarse operators, 20 red-black sweeps on the
// coarsest level (side <= 4); each slice's solve stops when ||f - A u||_2 <=
// tol ||f||_2.  Initial guess: the slice's envelope at t_n.
//
// Execution: one persistent cooperative launch per call runs every time step
// and slice: a right-hand-side phase per slice (which also writes the
// previous slice's new envelope back), the kappa hierarchy, then the cycles.
// Levels of side <= 8 run in block 0 on __syncthreads; larger ones are
// staged tile by tile in shared memory (see "Staged grid levels" below), one
// bounded grid barrier (qs_grid_sync.cuh) per level and leg.  Grid-wide
// loops hand runs of 32 cells to the blocks in turn, so that float64 work
// spreads over every SM.
#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>
#include <new>

#include <vector>

#include "qs.h"
#include "qs_fft.cuh"
#include "qs_grid_sync.cuh"
#include "qs_launch.cuh"

namespace {

using qsync::BlockSync;
using qsync::Team;

constexpr int kMaxLevels = 14;
constexpr int kThreads = 512;
constexpr int kLocalN = 8;             // levels this small run in block 0
constexpr int kNu = 2;                 // pre- and post-sweeps, V(2, 2)
constexpr int kTileX = 32, kTileY = 16;  // largest staged output tile
constexpr int kCoarseSweeps = 20;
constexpr double kFinite = 1.7e308;     // a norm above it, or NaN, is below no bound
constexpr size_t kScalarBytes = 1024;     // room for LzScalars ahead of the grids
constexpr long long kBarrierLimit = 4000000000LL;  // clock cycles, ~2 s

struct LzScalars {
    unsigned long long bar;
    int err;
    int err_where;
    int fail;                 // a slice hit max_cycles
    int pad;
    long long cycles;         // V-cycles over all slices and steps
    double max_relres;        // largest final relative residual of a slice
    double norm[3];           // rotating residual-norm slots
    double fnorm[3];          // |f|^2 of the slices (rotating by slice count)
    double start[3][2];       // |r|^2 and sum of chi of a slice's start (likewise)
    float dots[4][16];        // dot products of the iterations (ring of 4 uses)
};

static_assert(sizeof(LzScalars) <= kScalarBytes, "scalars");

struct LzLevel {
    int n;
    double ih2;               // 1 / h^2
    double2 *u, *f, *r;       // n * n each (level 0: u is a ping-pong buffer)
    double2 *kap, *idg;       // kappa and 1 / diag(A)
};

struct LzArgs {
    LzLevel lv[kMaxLevels];
    int levels;
    int n, n_xi, steps, max_cycles;
    double tol, q;
    double2 c;
    const double *chi;        // caller: [n_xi][n][n]
    double2 *a;               // caller: [n_xi][n][n], A^n in, A^{n+steps} out
    double2 *u;               // level-0 iterate of the V-cycles
    double2 *dlt;             // A^{n+1} - A^n of the last slice done
    // direct-solve preconditioner: on, lines per block, byte offset of the
    // tables in shared memory and their source; complex scratch grids
    int fft, gmax, tab_off;
    const qsfft::Ff *tables;
    qsfft::Ff2 *tr, *t2, *tz, *tp, *cz, *cr, *cp, *cs, *ce;
    double2 *r64;
    LzScalars *sc;
};

__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cscale(double s, double2 a) { return make_double2(s * a.x, s * a.y); }
__device__ __forceinline__ double2 cinv(double2 a) {
    const double d = 1.0 / (a.x * a.x + a.y * a.y);
    return make_double2(a.x * d, -a.y * d);
}
__device__ __forceinline__ double cabs2(double2 a) { return a.x * a.x + a.y * a.y; }

// u at (i, j) with odd ghosts (zero on the walls half a cell outside).
__device__ __forceinline__ double2 ghost_at(const double2 *u, int n, int i, int j) {
    double s = 1.0;
    if (i < 0) i = 0, s = -s;
    else if (i >= n) i = n - 1, s = -s;
    if (j < 0) j = 0, s = -s;
    else if (j >= n) j = n - 1, s = -s;
    return cscale(s, u[j * n + i]);
}

__device__ __forceinline__ double2 lap_at(const double2 *u, int n, double ih2, int i, int j) {
    const double2 s = cadd(cadd(ghost_at(u, n, i - 1, j), ghost_at(u, n, i + 1, j)),
                           cadd(ghost_at(u, n, i, j - 1), ghost_at(u, n, i, j + 1)));
    return cscale(ih2, csub(s, cscale(4.0, u[j * n + i])));
}

// A u = lap u - kappa u at cell p = (i, j)
__device__ __forceinline__ double2 apply_at(const LzLevel &L, const double2 *u, int i, int j) {
    const int p = j * L.n + i;
    return csub(lap_at(u, L.n, L.ih2, i, j), cmul(L.kap[p], u[p]));
}

__device__ void set_idiag(const LzLevel &L, Team tm) {
    const int n = L.n;
    for (int p = tm.t; p < n * n; p += tm.nt) {
        const int j = p / n, i = p - j * n;
        const int w = (i == 0) + (i == n - 1) + (j == 0) + (j == n - 1);
        const double2 d = make_double2(-(4.0 + w) * L.ih2 - L.kap[p].x, -L.kap[p].y);
        L.idg[p] = cinv(d);
    }
}

// kappa of the next coarser level: average of the 4 children
__device__ void restrict_kappa(const LzLevel &F, const LzLevel &C, Team tm) {
    const int nc = C.n, nf = F.n;
    for (int p = tm.t; p < nc * nc; p += tm.nt) {
        const int J = p / nc, I = p - J * nc;
        const double2 *k = F.kap + (2 * J) * nf + 2 * I;
        C.kap[p] = cscale(0.25, cadd(cadd(k[0], k[1]), cadd(k[nf], k[nf + 1])));
    }
}

__device__ void rb_colour(const LzLevel &L, int colour, Team tm) {
    const int n = L.n, half = (n * n + 1) / 2;
    for (int k = tm.t; k < half; k += tm.nt) {
        // k-th cell of the colour: rows alternate the parity of their first cell
        const int p2 = 2 * k;
        int j = p2 / n, i = p2 - j * n;
        if (((i + j) & 1) != colour) {
            ++i;
            if (i >= n) {
                i -= n;
                ++j;
            }
        }
        if (j >= n) continue;
        const int p = j * n + i;
        const double2 res = csub(L.f[p], apply_at(L, L.u, i, j));
        L.u[p] = cadd(L.u[p], cmul(res, L.idg[p]));
    }
}

template <typename Sync>
__device__ bool smooth(const LzLevel &L, int sweeps, Team tm, const Sync &sync, int where) {
    for (int s = 0; s < sweeps; ++s)
        for (int col = 0; col < 2; ++col) {
            rb_colour(L, col, tm);
            if (!sync(where)) return false;
        }
    return true;
}

__device__ void residual(const LzLevel &L, Team tm) {
    const int n = L.n;
    for (int p = tm.t; p < n * n; p += tm.nt) {
        const int j = p / n, i = p - j * n;
        L.r[p] = csub(L.f[p], apply_at(L, L.u, i, j));
    }
}

__device__ void restrict_residual(const LzLevel &F, const LzLevel &C, Team tm) {
    const int nc = C.n, nf = F.n;
    for (int p = tm.t; p < nc * nc; p += tm.nt) {
        const int J = p / nc, I = p - J * nc;
        const double2 *r = F.r + (2 * J) * nf + 2 * I;
        C.f[p] = cscale(0.25, cadd(cadd(r[0], r[1]), cadd(r[nf], r[nf + 1])));
        C.u[p] = make_double2(0.0, 0.0);
    }
}

// fine u += bilinear interpolation of the coarse u (weights 9, 3, 3, 1 / 16)
__device__ void prolong_correct(const LzLevel &F, const LzLevel &C, Team tm) {
    const int nf = F.n, nc = C.n;
    for (int p = tm.t; p < nf * nf; p += tm.nt) {
        const int j = p / nf, i = p - j * nf;
        const int I = i >> 1, J = j >> 1;
        const int di = (i & 1) ? 1 : -1, dj = (j & 1) ? 1 : -1;
        const double2 e = cadd(cadd(cscale(9.0 / 16.0, ghost_at(C.u, nc, I, J)),
                                    cscale(3.0 / 16.0, ghost_at(C.u, nc, I + di, J))),
                               cadd(cscale(3.0 / 16.0, ghost_at(C.u, nc, I, J + dj)),
                                    cscale(1.0 / 16.0, ghost_at(C.u, nc, I + di, J + dj))));
        F.u[p] = cadd(F.u[p], e);
    }
}

// ---------------------------------------------------------------------------
// Staged grid levels.  A grid-wide level costs a grid barrier per colour
// sweep, residual, restriction and prolongation (eleven per V-cycle).  Here
// every block takes an output tile plus a halo, stages u, f, kappa and the
// inverse diagonal in shared memory and runs all the half sweeps of a leg
// there, recomputing the halo: after half sweep s only the cells at least
// s + 1 from a cut side of the region are exact, and those are the only ones
// updated.  A down leg (pre-sweeps, residual, restriction) and an up leg
// (prolongation, post-sweeps) each cost one grid barrier; the level-0 up leg
// also sums |f - A u|^2 of its tile for the stopping test.
// ---------------------------------------------------------------------------

struct Reg {
    int ox, oy, RX, RY, R;  // staged region: origin and extent
    int ax, bx, ay, by;     // its intersection with the domain
    bool cl, cr, cb, ct;    // which sides are cut (not the domain wall)
};

__device__ __forceinline__ Reg make_reg(int tx0, int ty0, int TX, int TY, int H, int n) {
    Reg g;
    g.ox = tx0 - H;
    g.oy = ty0 - H;
    g.RX = TX + 2 * H;
    g.RY = TY + 2 * H;
    g.R = g.RX * g.RY;
    g.ax = max(g.ox, 0);
    g.bx = min(g.ox + g.RX - 1, n - 1);
    g.ay = max(g.oy, 0);
    g.by = min(g.oy + g.RY - 1, n - 1);
    g.cl = g.ax > 0;
    g.cr = g.bx < n - 1;
    g.cb = g.ay > 0;
    g.ct = g.by < n - 1;
    return g;
}

// output tile of a staged level: halved (down to 8) while the level has
// fewer tiles than half the blocks, so that its work still spreads
__device__ __forceinline__ void lz_tile(int n, int nblk, int &TX, int &TY) {
    TX = kTileX;
    TY = kTileY;
    for (;;) {
        const int tiles = ((n + TX - 1) / TX) * ((n + TY - 1) / TY);
        if (2 * tiles >= nblk) break;
        if (TX >= TY && TX > 8) TX >>= 1;
        else if (TY > 8) TY >>= 1;
        else break;
    }
}

// staged arrays of a region of R cells: u, f, kappa, inverse diagonal
struct LzSmem {
    double2 *u, *f, *k, *d;
};

__device__ __forceinline__ LzSmem lz_layout(double2 *sm, int R) {
    return LzSmem{sm, sm + R, sm + 2 * R, sm + 3 * R};
}

// shared memory of the largest staged region (tile + halo 2 kNu + 1)
__host__ __device__ constexpr size_t lz_smem_bytes() {
    return (size_t)4 * (kTileX + 2 * (2 * kNu + 1)) * (kTileY + 2 * (2 * kNu + 1)) *
           sizeof(double2);
}

// 16-byte global -> shared copy, zero-filled when !valid (source size 0)
__device__ __forceinline__ void cp16(double2 *dst, const double2 *src, bool valid) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src),
                 "r"(valid ? 16 : 0)
                 : "memory");
}

__device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_all;\n" ::: "memory");
}

// (lap - kappa) u at staged cell li = (x, y) (odd ghosts: a wall adds to the
// diagonal)
__device__ __forceinline__ double2 staged_apply(const LzSmem &t, int RX, int n, double ih2, int li,
                                                int x, int y) {
    double2 nb = make_double2(0.0, 0.0);
    if (x > 0) nb = cadd(nb, t.u[li - 1]);
    if (x < n - 1) nb = cadd(nb, t.u[li + 1]);
    if (y > 0) nb = cadd(nb, t.u[li - RX]);
    if (y < n - 1) nb = cadd(nb, t.u[li + RX]);
    const int w = (x == 0) + (x == n - 1) + (y == 0) + (y == n - 1);
    const double2 lap = cscale(ih2, csub(nb, cscale(4.0 + w, t.u[li])));
    return csub(lap, cmul(t.k[li], t.u[li]));
}

// half sweeps 0 .. ns - 1 (colour s & 1) on the staged region
__device__ void staged_sweeps(const Reg &g, int n, double ih2, const LzSmem &t, int ns) {
    for (int s = 0; s < ns; ++s) {
        const int colour = s & 1;
        const int X0 = g.cl ? g.ax + s + 1 : g.ax, X1 = g.cr ? g.bx - s - 1 : g.bx;
        const int Y0 = g.cb ? g.ay + s + 1 : g.ay, Y1 = g.ct ? g.by - s - 1 : g.by;
        const int rows = Y1 - Y0 + 1, hw = (X1 - X0 + 2) >> 1;
        const int cnt = (rows > 0 && hw > 0) ? rows * hw : 0;
        for (int q = threadIdx.x; q < cnt; q += blockDim.x) {
            const int r = q / hw, y = Y0 + r;
            const int x = X0 + ((X0 + y + colour) & 1) + 2 * (q - r * hw);
            if (x > X1) continue;
            const int li = (y - g.oy) * g.RX + (x - g.ox);
            const double2 res = csub(t.f[li], staged_apply(t, g.RX, n, ih2, li, x, y));
            t.u[li] = cadd(t.u[li], cmul(res, t.d[li]));
        }
        __syncthreads();
    }
}

// stage f, kappa, 1/diag of level F and u from usrc (nullptr: zero) on g
__device__ void stage(const LzLevel &F, const Reg &g, const LzSmem &t, const double2 *usrc) {
    const int n = F.n;
    for (int q = threadIdx.x; q < g.R; q += blockDim.x) {
        const int r = q / g.RX, x = g.ox + (q - r * g.RX), y = g.oy + r;
        const bool in = x >= 0 && x < n && y >= 0 && y < n;
        const int gi = in ? y * n + x : 0;
        cp16(t.f + q, F.f + gi, in);
        cp16(t.k + q, F.kap + gi, in);
        cp16(t.d + q, F.idg + gi, in);
        if (usrc) cp16(t.u + q, usrc + gi, in);
        else t.u[q] = make_double2(0.0, 0.0);
    }
    cp_wait();
    __syncthreads();
}

// Down leg of level F -> C for this block's tiles: pre-sweeps from the
// warm start F.u (level 0) or zero, residual, restriction into C.f
// (C.u = 0).  The smoothed tile goes to F.r, not F.u: other blocks still
// stage F.u around their tiles during this leg.
__device__ void staged_down(const LzLevel &F, const LzLevel &C, bool warm, double2 *sm, int bid,
                            int nblk) {
    const int n = F.n, m = C.n;
    int TX, TY;
    lz_tile(n, nblk, TX, TY);
    const int ntx = (n + TX - 1) / TX, nty = (n + TY - 1) / TY;
    for (int tile = bid; tile < ntx * nty; tile += nblk) {
        const int tx0 = (tile % ntx) * TX, ty0 = (tile / ntx) * TY;
        const Reg g = make_reg(tx0, ty0, TX, TY, 2 * kNu + 1, n);
        const LzSmem t = lz_layout(sm, g.R);
        stage(F, g, t, warm ? F.u : nullptr);
        staged_sweeps(g, n, F.ih2, t, 2 * kNu);
        const int CX = TX / 2, CY = TY / 2;
        for (int q = threadIdx.x; q < CX * CY; q += blockDim.x) {
            const int r = q / CX;
            const int I = tx0 / 2 + (q - r * CX), J = ty0 / 2 + r;
            if (I >= m || J >= m) continue;
            double2 s = make_double2(0.0, 0.0);
            for (int b = 0; b < 2; ++b)
                for (int a = 0; a < 2; ++a) {
                    const int x = 2 * I + a, y = 2 * J + b;
                    const int li = (y - g.oy) * g.RX + (x - g.ox);
                    s = cadd(s, csub(t.f[li], staged_apply(t, g.RX, n, F.ih2, li, x, y)));
                }
            C.f[J * m + I] = cscale(0.25, s);
            C.u[J * m + I] = make_double2(0.0, 0.0);
        }
        for (int q = threadIdx.x; q < TX * TY; q += blockDim.x) {
            const int r = q / TX, x = tx0 + (q - r * TX), y = ty0 + r;
            if (x < n && y < n) F.r[y * n + x] = t.u[(y - g.oy) * g.RX + (x - g.ox)];
        }
        __syncthreads();  // the next tile reuses the staged arrays
    }
}

// Up leg of level F for this block's tiles: the pre-smoothed u (F.r, from
// the down leg) plus the bilinear prolongation of C.u, post-sweeps, the tile
// to F.u.  With `norm` (level 0) the halo is one cell wider and
// |f - A u|^2 of the tile is added to *norm_sum (this thread's share).
__device__ void staged_up(const LzLevel &F, const LzLevel &C, double2 *sm, int bid, int nblk,
                          bool norm, double *norm_sum) {
    const int n = F.n, nc = C.n;
    int TX, TY;
    lz_tile(n, nblk, TX, TY);
    const int ntx = (n + TX - 1) / TX, nty = (n + TY - 1) / TY;
    for (int tile = bid; tile < ntx * nty; tile += nblk) {
        const int tx0 = (tile % ntx) * TX, ty0 = (tile / ntx) * TY;
        const Reg g = make_reg(tx0, ty0, TX, TY, 2 * kNu + (norm ? 1 : 0), n);
        const LzSmem t = lz_layout(sm, g.R);
        stage(F, g, t, F.r);
        for (int q = threadIdx.x; q < g.R; q += blockDim.x) {
            const int r = q / g.RX, i = g.ox + (q - r * g.RX), j = g.oy + r;
            if (i < 0 || i >= n || j < 0 || j >= n) continue;
            const int I = i >> 1, J = j >> 1;
            const int di = (i & 1) ? 1 : -1, dj = (j & 1) ? 1 : -1;
            const double2 e = cadd(cadd(cscale(9.0 / 16.0, ghost_at(C.u, nc, I, J)),
                                        cscale(3.0 / 16.0, ghost_at(C.u, nc, I + di, J))),
                                   cadd(cscale(3.0 / 16.0, ghost_at(C.u, nc, I, J + dj)),
                                        cscale(1.0 / 16.0, ghost_at(C.u, nc, I + di, J + dj))));
            t.u[q] = cadd(t.u[q], e);
        }
        __syncthreads();
        staged_sweeps(g, n, F.ih2, t, 2 * kNu);
        for (int q = threadIdx.x; q < TX * TY; q += blockDim.x) {
            const int r = q / TX, x = tx0 + (q - r * TX), y = ty0 + r;
            if (x >= n || y >= n) continue;
            const int li = (y - g.oy) * g.RX + (x - g.ox);
            F.u[y * n + x] = t.u[li];
            if (norm) *norm_sum += cabs2(csub(t.f[li], staged_apply(t, g.RX, n, F.ih2, li, x, y)));
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// The coarse part (levels of side <= kLocalN) in every block's own shared
// memory, redundantly: no block waits for block 0 at a grid barrier, and the
// up leg of the first staged level prolongs from the block's own copy.  The
// coarsest level (up to kMaxExact unknowns) is solved with its exact
// inverse, formed once per slice by complex Gauss-Jordan elimination (no
// pivoting: -A has a positive definite Hermitian part, the 5-point -lap
// plus kappa with Re kappa = chi + q >= 0); larger coarsest levels take
// kCoarseSweeps red-black sweeps.
// ---------------------------------------------------------------------------
constexpr int kMaxExact = 16;
constexpr int kCoarseCells = 128;  // room for the levels of side <= kLocalN
constexpr size_t kCoarseBytes =
    (size_t)5 * kCoarseCells * sizeof(double2) + (size_t)kMaxExact * 2 * kMaxExact * sizeof(double2);

// the shared-memory hierarchy of levels loc .. Lc (pointers into sm)
__device__ void coarse_levels(const LzArgs &A, int loc, int Lc, double2 *sm, LzLevel *S) {
    double2 *p = sm;
    for (int l = loc; l <= Lc; ++l) {
        const int m = A.lv[l].n * A.lv[l].n;
        S[l].n = A.lv[l].n;
        S[l].ih2 = A.lv[l].ih2;
        S[l].u = p;
        S[l].f = p + m;
        S[l].r = p + 2 * m;
        S[l].kap = p + 3 * m;
        S[l].idg = p + 4 * m;
        p += 5 * m;
    }
}

// [A | I] -> [I | A^{-1}] for the coarsest operator A = lap - kappa
// (m = n^2 unknowns) in work (m x 2m, row-major): the inverse is the right
// half, work[i * 2m + m + j]
__device__ void coarse_inverse(const LzLevel &C, double2 *work) {
    const int n = C.n, m = n * n, W = 2 * m;
    __shared__ double2 s_piv;
    __shared__ double2 fac[kMaxExact];
    for (int e = threadIdx.x; e < m * W; e += blockDim.x) {
        const int i = e / W, j = e - i * W;
        double2 v = make_double2(0.0, 0.0);
        if (j >= m) {
            if (j - m == i) v.x = 1.0;
        } else {
            const int ix = i % n, iy = i / n, jx = j % n, jy = j / n;
            if (i == j) {
                const int w = (ix == 0) + (ix == n - 1) + (iy == 0) + (iy == n - 1);
                v = make_double2(-(4.0 + w) * C.ih2 - C.kap[i].x, -C.kap[i].y);
            } else if (abs(ix - jx) + abs(iy - jy) == 1) {
                v.x = C.ih2;
            }
        }
        work[e] = v;
    }
    __syncthreads();
    for (int k = 0; k < m; ++k) {
        if (threadIdx.x == 0) s_piv = cinv(work[k * W + k]);
        __syncthreads();
        const double2 piv = s_piv;
        for (int i = threadIdx.x; i < m; i += blockDim.x)
            fac[i] = i == k ? make_double2(0.0, 0.0) : cmul(work[i * W + k], piv);
        __syncthreads();
        for (int e = threadIdx.x; e < m * (W - k); e += blockDim.x) {
            const int i = e / (W - k), j = k + (e - i * (W - k));
            if (i != k) work[i * W + j] = csub(work[i * W + j], cmul(fac[i], work[k * W + j]));
        }
        __syncthreads();
        for (int j = k + threadIdx.x; j < W; j += blockDim.x) work[k * W + j] = cmul(work[k * W + j], piv);
        __syncthreads();
    }
}

template <typename Sync>
__device__ bool down(const LzLevel *H, int from, int to, Team tm, const Sync &sync) {
    for (int l = from; l < to; ++l) {
        if (!smooth(H[l], 2, tm, sync, 10 + l)) return false;
        residual(H[l], tm);
        if (!sync(30 + l)) return false;
        restrict_residual(H[l], H[l + 1], tm);
        if (!sync(50 + l)) return false;
    }
    return true;
}

template <typename Sync>
__device__ bool up(const LzLevel *H, int from, int to, Team tm, const Sync &sync) {
    for (int l = from; l >= to; --l) {
        prolong_correct(H[l], H[l + 1], tm);
        if (!sync(70 + l)) return false;
        if (!smooth(H[l], 2, tm, sync, 90 + l)) return false;
    }
    return true;
}

// ---------------------------------------------------------------------------
// Direct-solve preconditioned iterations
// ---------------------------------------------------------------------------
using qsff::Ff;
using qsfft::Ff2;

__device__ __forceinline__ Ff2 split2(double2 v) {
    return qsfft::mk<Ff>(qsff::split(v.x), qsff::split(v.y));
}
__device__ __forceinline__ double2 join2(Ff2 v) {
    return make_double2(qsff::join(v.x), qsff::join(v.y));
}
// a + b s for a complex float s
__device__ __forceinline__ Ff2 axpy(Ff2 a, float2 s, Ff2 b) {
    return qsfft::mk<Ff>(a.x + (b.x * s.x + b.y * -s.y), a.y + (b.y * s.x + b.x * s.y));
}
__device__ __forceinline__ float2 fmul(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// 1 / a, scaled: late in an iteration |a|^2 is below float32's range
__device__ __forceinline__ float2 finv(float2 a) {
    const float m = 1.f / fmaxf(fabsf(a.x), fabsf(a.y)), x = a.x * m, y = a.y * m;
    const float d = m / (x * x + y * y);
    return make_float2(x * d, -y * d);
}

// Adds the block's 16 sums to dots[use & 3] and clears the slots two uses ahead.
__device__ void lz_reduce(LzScalars *sc, float v[16], int use) {
    const float t = qsfft::block_sums16(v);
    if (threadIdx.x < 16) {
        if (t != 0.f) atomicAdd(&sc->dots[use & 3][threadIdx.x], t);
        if (blockIdx.x == 0) sc->dots[(use + 2) & 3][threadIdx.x] = 0.f;
    }
}

// The change of slice j's envelope into A.dlt.  On entry A.dlt is the previous
// slice's change (added to the caller's array here).  Returns 1 (converged),
// 0 (not: A.u = A^n + the change so far, for the V-cycles), 3 (not finite), -1
// (a barrier failed).  its: iterations; relres: the final relative residual (thread 0).
__device__ int slice_direct(const LzArgs &A, const qsync::GridBarrier<LzScalars> &gsync, int j,
                            long long g, long long &kglob, int &use, int &its, double &relres) {
    LzScalars *sc = A.sc;
    const int n = A.n, nn = n * n;
    const qsfft::Lines P{n, A.gmax, 0, A.tab_off};
    const LzLevel &L0 = A.lv[0];
    const double2 *aj = A.a + (size_t)j * nn;
    const double *chij = A.chi + (size_t)j * nn;
    __shared__ float2 s_al, s_be, s_ig, s_ia;
    __shared__ float s_ss, s_target;  // (scaled) |A p|^2; |r|^2 that ends a round
    __shared__ double s_r0, s_thr;
    __shared__ int s_go;
    its = 0;
    // source f (its norm sets the bound) and the residual of A^n, in which the
    // large c A^n cancels: r = 2 chi A^n - 2 lap A^n - q (change of slice j - 1)
    double st[3] = {0.0, 0.0, 0.0};
    qsfft::rows_forward<Ff, 2>(P, blockIdx.x, gridDim.x, A.tr, [&](int y, int x) {
        const int p = y * n + x;
        const double2 ao = aj[p], lap = lap_at(aj, n, L0.ih2, x, y);
        const double chi = chij[p];
        double2 h = csub(cscale(chi, ao), lap);
        double2 f = cadd(cmul(A.c, ao), h);
        double2 r = cadd(h, h);
        if (j > 0) {
            const double2 d = A.dlt[p], gq = cscale(A.q, d);
            f = csub(f, gq);
            r = csub(r, gq);
            double2 *prev = A.a + (size_t)(j - 1) * nn + p;
            *prev = cadd(*prev, d);
        }
        L0.f[p] = f;
        A.r64[p] = r;
        st[0] += cabs2(f);
        st[1] += cabs2(r);
        st[2] += chi;
        const Ff2 rf = split2(r);
        A.cr[p] = rf;
        return rf;
    });
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        sc->fnorm[(g + 1) % 3] = 0.0;
        sc->start[(g + 1) % 3][0] = sc->start[(g + 1) % 3][1] = 0.0;
    }
    qsync::block_sum_add<kThreads>(st, 1, &sc->fnorm[g % 3]);
    qsync::block_sum_add<kThreads>(st + 1, 2, sc->start[g % 3]);
    if (!gsync(1)) return -1;
    if (threadIdx.x == 0) {
        const double f2 = qsync::vload(&sc->fnorm[g % 3]);
        s_r0 = qsync::vload(&sc->start[g % 3][0]);
        s_thr = A.tol * A.tol * f2;
        s_go = s_r0 <= s_thr && s_r0 <= kFinite;
        relres = f2 > 0.0 ? sqrt(s_r0 / f2) : 0.0;
    }
    __syncthreads();
    const bool done = s_go != 0;
    const double chibar = qsync::vload(&sc->start[g % 3][1]) / (double)nn;
    const Ff cb = qsff::split(chibar);
    // M = lap - chibar + c = lap - (chibar - c)
    const Ff2 shift = qsfft::mk<Ff>(qsff::split(chibar - A.c.x), qsff::split(-A.c.y));
    auto dk = [&](int p) { return cb - qsff::split(chij[p]); };
    // power of two near 1 / |r|: the sums are of scaled values
    const int ex = (int)((__double_as_longlong(s_r0) >> 52) & 0x7ff);
    const int k2 = ex == 0 || ex == 0x7ff ? 0 : min(max((ex - 1023) / 2, -120), 120);
    const float scale = __int_as_float((127 - k2) << 23);
    const double scale2 = (double)scale * (double)scale;
    if (done) {
        const qsync::Team grid = qsync::spread_team();
        for (int p = grid.t; p < nn; p += grid.nt) A.dlt[p] = make_double2(0.0, 0.0);
        return gsync(2) ? 1 : -1;
    }
    const int cap = min(4 * A.max_cycles, 48);
    // float32 for the test on the path of every iteration, set once a round
    auto set_target = [&] {
        s_target = fmaxf((float)(fmax(1e-24 * s_r0, 0.09 * s_thr) * scale2), 1e-37f);
    };
    if (threadIdx.x == 0) set_target();
    for (int round = 0;; ++round) {
        float2 al = make_float2(0.f, 0.f), be = al;
        int inner = 0;
        for (;;) {
            qsfft::columns<Ff, 2>(P, blockIdx.x, gridDim.x, A.t2, shift, [&](int y, int l) {
                const int p = y * n + l;
                Ff2 r = A.tr[p];
                if (inner > 0) {
                    Ff2 s = A.tz[p];
                    if (inner > 1) s = axpy(s, be, A.tp[p]);
                    A.tp[p] = s;
                    r = axpy(r, make_float2(-al.x, -al.y), s);
                    A.tr[p] = r;
                }
                return r;
            });
            if (!gsync(7)) return -1;
            float d[16] = {0.f};
            qsfft::rows_inverse_forward<Ff, Ff, 1>(
                P, P, blockIdx.x, gridDim.x, A.t2, A.tz, [&](int y, int x, Ff2 z) {
                    const int p = y * n + x;
                    const Ff k = dk(p);
                    Ff2 r = A.cr[p], s = qsfft::mk<Ff>(Ff(0.f, 0.f), Ff(0.f, 0.f));
                    if (inner > 0) {  // the update of the last iteration
                        const Ff2 zo = A.cz[p];
                        Ff2 q = zo, e = s;
                        s = qsfft::mk<Ff>(r.x + k * zo.x, r.y + k * zo.y);
                        if (inner > 1) {
                            q = axpy(q, be, A.cp[p]);
                            s = axpy(s, be, A.cs[p]);
                            e = A.ce[p];
                        }
                        e = axpy(e, al, q);
                        r = axpy(r, make_float2(-al.x, -al.y), s);
                        A.cp[p] = q;
                        A.cs[p] = s;
                        A.ce[p] = e;
                        A.cr[p] = r;
                    }
                    A.cz[p] = z;
                    const Ff2 w = qsfft::mk<Ff>(r.x + k * z.x, r.y + k * z.y);
                    const float rx = r.x.h * scale, ry = r.y.h * scale, zx = z.x.h * scale,
                                zy = z.y.h * scale, wx = w.x.h * scale, wy = w.y.h * scale,
                                sx = s.x.h * scale, sy = s.y.h * scale;
                    d[0] += rx * zx - ry * zy;  // r z
                    d[1] += rx * zy + ry * zx;
                    d[2] += zx * wx - zy * wy;  // z A z
                    d[3] += zx * wy + zy * wx;
                    d[4] += wx * rx + wy * ry;  // A z conj(r)
                    d[5] += wy * rx - wx * ry;
                    d[6] += sx * rx + sy * ry;  // A p conj(r), the last p
                    d[7] += sy * rx - sx * ry;
                    d[8] += sx * wx + sy * wy;  // A p conj(A z)
                    d[9] += sy * wx - sx * wy;
                    d[10] += wx * wx + wy * wy;
                    d[11] += rx * rx + ry * ry;
                    return w;
                });
            lz_reduce(sc, d, use);
            if (!gsync(8)) return -1;
            if (threadIdx.x == 0) {
                const volatile float *v = sc->dots[use & 3];
                const float2 ga = make_float2(v[0], v[1]), de = make_float2(v[2], v[3]);
                const float2 zero = make_float2(0.f, 0.f);
                float2 b = zero, a = zero, ia = zero, ig = zero;
                // solved to float32's smallest numbers: stands still
                if (fmaxf(fabsf(ga.x), fabsf(ga.y)) >= 1e-36f) {
                    ig = finv(ga);
                    if (inner > 0) b = fmul(ga, s_ig);
                    ia = fmul(de, ig);
                    if (inner > 0) {
                        const float2 t = fmul(b, s_ia);
                        ia = make_float2(ia.x - t.x, ia.y - t.y);
                    }
                    if (fmaxf(fabsf(ia.x), fabsf(ia.y)) >= 1e-30f) a = finv(ia);
                }
                s_ig = ig;
                s_ia = ia;
                s_al = a;
                s_be = b;
                // |r - a s|^2 with s = w + b s_old; the sums are good to about
                // 1e-7 of |r|^2: no smaller value is believed
                const float so = inner > 0 ? s_ss : 0.f;
                const float2 ws = fmul(b, make_float2(v[8], v[9]));
                const float2 rs = fmul(b, make_float2(v[6], v[7]));
                const float ss = v[10] + 2.f * ws.x + (b.x * b.x + b.y * b.y) * so;
                const float2 ars = fmul(a, make_float2(v[4] + rs.x, v[5] + rs.y));
                const float rr = v[11];
                float nr = rr - 2.f * ars.x + (a.x * a.x + a.y * a.y) * ss;
                nr = nr < 2e-7f * rr ? 2e-7f * rr : nr;
                s_ss = ss;
                s_go = nr > s_target;  // a NaN ends the round
            }
            ++use;
            __syncthreads();
            al = s_al;
            be = s_be;
            const bool go = s_go != 0;  // rewritten two grid barriers on
            ++its;
            ++inner;
            if (!go || its >= cap || inner >= 24) break;
        }
        // change += e, r <- r - A e in float64, with its norm
        auto e_at = [&](int p) {
            Ff2 q = A.cz[p], e = qsfft::mk<Ff>(Ff(0.f, 0.f), Ff(0.f, 0.f));
            if (inner > 1) {
                q = axpy(q, be, A.cp[p]);
                e = A.ce[p];
            }
            return join2(axpy(e, al, q));
        };
        double rn = 0.0;
        if (blockIdx.x == 0 && threadIdx.x == 0) sc->norm[(kglob + 1) % 3] = 0.0;
        qsfft::rows_forward<Ff, 2>(P, blockIdx.x, gridDim.x, A.tr, [&](int y, int x) {
            const int p = y * n + x;
            const double2 e = e_at(p), zero = make_double2(0.0, 0.0);
            const double2 s = cadd(cadd(x > 0 ? e_at(p - 1) : zero, x < n - 1 ? e_at(p + 1) : zero),
                                   cadd(y > 0 ? e_at(p - n) : zero, y < n - 1 ? e_at(p + n) : zero));
            const int w = 4 + (x == 0) + (x == n - 1) + (y == 0) + (y == n - 1);
            const double2 lap = cscale(L0.ih2, csub(s, cscale((double)w, e)));
            const double2 le = cadd(lap, cmul(make_double2(A.c.x - chij[p], A.c.y), e));
            const double2 r = csub(A.r64[p], le);
            A.r64[p] = r;
            const double2 dn = round > 0 ? cadd(A.dlt[p], e) : e;
            A.dlt[p] = dn;
            A.u[p] = cadd(aj[p], dn);
            rn += cabs2(r);
            const Ff2 rf = split2(r);
            A.cr[p] = rf;
            return rf;
        });
        qsync::block_sum_add<kThreads>(&rn, 1, &sc->norm[kglob % 3]);
        if (!gsync(9)) return -1;
        if (threadIdx.x == 0) {
            const double r2 = qsync::vload(&sc->norm[kglob % 3]);
            const double f2 = qsync::vload(&sc->fnorm[g % 3]);
            const bool slow = !(r2 <= 0.0625 * s_r0);
            s_go = !(r2 <= kFinite) ? 3 : r2 <= s_thr ? 1 : (slow || its >= cap) ? 0 : 2;
            s_r0 = r2;
            set_target();
            relres = f2 > 0.0 ? sqrt(r2 / f2) : 0.0;
        }
        ++kglob;
        __syncthreads();
        const int r = s_go;
        __syncthreads();
        if (r != 2) return r;
    }
}

__global__ void __launch_bounds__(kThreads, 1) laser_kernel(const __grid_constant__ LzArgs P) {
    double2 *const lz_dyn = (double2 *)qsfft::dyn_smem();  // the staged regions
    __shared__ LzArgs A;
    __shared__ unsigned long long epoch;
    if (threadIdx.x == 0) {
        A = P;
        epoch = 0;
    }
    __syncthreads();
    LzScalars *sc = A.sc;
    const qsync::GridBarrier<LzScalars> gsync{sc, &epoch, kBarrierLimit};
    const Team grid = qsync::spread_team();
    const Team blk{(int)threadIdx.x, (int)blockDim.x};
    const int n = A.n, nn = n * n, Lc = A.levels - 1;
    int loc = 0;  // first level of the coarse part
    while (loc < Lc && A.lv[loc].n > kLocalN) ++loc;
    // the coarse part's levels in shared memory, after the staged regions
    // (used when loc > 0; the host checks that they fit)
    __shared__ LzLevel S[kMaxLevels];
    double2 *const csm = lz_dyn + lz_smem_bytes() / sizeof(double2);
    const bool exact = A.lv[Lc].n * A.lv[Lc].n <= kMaxExact;
    double2 *const cwork = csm + 5 * kCoarseCells;  // [I | A^{-1}] of the coarsest level
    int coarse_cells = 0;
    for (int l = loc; l <= Lc; ++l) coarse_cells += A.lv[l].n * A.lv[l].n;
    const bool local = loc > 0 && coarse_cells <= kCoarseCells;
    if (threadIdx.x == 0 && local) coarse_levels(A, loc, Lc, csm, S);
    __syncthreads();
    long long kglob = 0;  // residual-norm computations so far (slot kglob % 3)
    long long g = 0;      // slices so far

    if (A.fft) {
        const int words = 6 * n + 4 * (n / 2 + 1);  // floats of [tw][dct][lam], as pairs
        float *const t = (float *)((char *)lz_dyn + A.tab_off);
        for (int k = threadIdx.x; k < words; k += blockDim.x) t[k] = ((const float *)A.tables)[k];
        if (threadIdx.x == 0) A.lv[0].u = A.u;
        __syncthreads();
    }
    int use = 0;  // uses of the dot products' ring
    for (int step = 0; step < A.steps; ++step) {
        for (int j = 0; j < A.n_xi; ++j, ++g) {
            double2 *U = A.u;
            if (threadIdx.x == 0) A.lv[0].u = U;
            __syncthreads();
            const LzLevel &L0 = A.lv[0];
            const double2 *aj = A.a + (size_t)j * nn;
            const double *chij = A.chi + (size_t)j * nn;
            const bool direct = A.fft != 0;
            int before = 0;  // what the iterations count as
            if (direct) {
                int its = 0;
                double rel = 0.0;
                const int r = slice_direct(A, gsync, j, g, kglob, use, its, rel);
                if (r < 0) return;
                before = (its + 3) / 4;
                if (r == 1) {
                    if (blockIdx.x == 0 && threadIdx.x == 0) {
                        sc->cycles += before;
                        if (rel > sc->max_relres) sc->max_relres = rel;
                    }
                    continue;
                }
                // the V-cycles go on from its iterate, or start from A^n
                for (int p = grid.t; p < nn; p += grid.nt) {
                    L0.kap[p] = make_double2(chij[p] - A.c.x, -A.c.y);
                    if (r == 3) U[p] = aj[p];
                }
            } else {
                // right-hand side, warm start, kappa and 1/diag of level 0; the
                // previous slice's new envelope goes to the caller's array
                double fn = 0.0;
                // slot (g + 1) % 3 was last read two slices ago, before a barrier
                if (blockIdx.x == 0 && threadIdx.x == 0) sc->fnorm[(g + 1) % 3] = 0.0;
                for (int p = grid.t; p < nn; p += grid.nt) {
                    const int jj = p / n, i = p - jj * n;
                    const double2 ao = aj[p];
                    const double chi = chij[p];
                    double2 f = csub(cmul(make_double2(A.c.x + chi, A.c.y), ao),
                                     lap_at(aj, n, L0.ih2, i, jj));
                    if (j > 0) {
                        const double2 d = A.dlt[p];
                        f = csub(f, cscale(A.q, d));
                        double2 *prev = A.a + (size_t)(j - 1) * nn + p;
                        *prev = cadd(*prev, d);
                    }
                    L0.f[p] = f;
                    U[p] = ao;
                    L0.kap[p] = make_double2(chi - A.c.x, -A.c.y);
                    fn += cabs2(f);
                }
                qsync::block_sum_add<kThreads>(&fn, 1, &sc->fnorm[g % 3]);
            }
            set_idiag(L0, grid);
            if (!gsync(1)) return;
            for (int l = 1; l <= Lc; ++l) {
                if (l <= loc) {
                    restrict_kappa(A.lv[l - 1], A.lv[l], grid);
                    if (!gsync(2)) return;
                    set_idiag(A.lv[l], grid);
                } else if (blockIdx.x == 0) {
                    restrict_kappa(A.lv[l - 1], A.lv[l], blk);
                    __syncthreads();
                    set_idiag(A.lv[l], blk);
                    __syncthreads();
                }
            }
            // initial residual, then V-cycles until converged; each cycle's
            // level-0 up leg sums the residual of its result
            int cyc = 0;
            {
                double rn = 0.0;
                if (blockIdx.x == 0 && threadIdx.x == 0) sc->norm[(kglob + 1) % 3] = 0.0;
                for (int p = grid.t; p < nn; p += grid.nt) {
                    const int jj = p / n, i = p - jj * n;
                    rn += cabs2(csub(L0.f[p], apply_at(L0, U, i, jj)));
                }
                qsync::block_sum_add<kThreads>(&rn, 1, &sc->norm[kglob % 3]);
                if (!gsync(4)) return;
            }
            for (;;) {
                const double r2 = qsync::vload(&sc->norm[kglob % 3]);
                const double f2 = qsync::vload(&sc->fnorm[g % 3]);
                ++kglob;
                const bool bad = !(r2 <= kFinite);  // more cycles don't mend it
                const bool conv = !bad && r2 <= A.tol * A.tol * f2;
                if (conv || bad || cyc >= A.max_cycles) {
                    if (blockIdx.x == 0 && threadIdx.x == 0) {
                        sc->cycles += before + cyc;
                        const double rel = f2 > 0.0 ? sqrt(r2 / f2) : 0.0;
                        if (rel > sc->max_relres) sc->max_relres = rel;
                        if (!conv) sc->fail = 1;
                    }
                    break;
                }
                ++cyc;
                if (blockIdx.x == 0 && threadIdx.x == 0) sc->norm[(kglob + 1) % 3] = 0.0;
                double rn = 0.0;
                if (loc == 0) {  // a grid this small: block 0 alone, then the residual
                    if (blockIdx.x == 0) {
                        const BlockSync bs;
                        if (Lc == 0) {
                            smooth(A.lv[0], kCoarseSweeps, blk, bs, 5);
                        } else {
                            down(A.lv, 0, Lc, blk, bs);
                            smooth(A.lv[Lc], kCoarseSweeps, blk, bs, 5);
                            up(A.lv, Lc - 1, 0, blk, bs);
                        }
                    }
                    if (!gsync(3)) return;
                    for (int p = grid.t; p < nn; p += grid.nt) {
                        const int jj = p / n, i = p - jj * n;
                        rn += cabs2(csub(L0.f[p], apply_at(L0, U, i, jj)));
                    }
                } else {
                    for (int l = 0; l < loc; ++l) {
                        staged_down(A.lv[l], A.lv[l + 1], l == 0, lz_dyn, blockIdx.x, gridDim.x);
                        if (!gsync(10 + l)) return;
                    }
                    if (!local) {  // block 0 in global memory
                        if (blockIdx.x == 0) {
                            const BlockSync bs;
                            down(A.lv, loc, Lc, blk, bs);
                            smooth(A.lv[Lc], kCoarseSweeps, blk, bs, 5);
                            up(A.lv, Lc - 1, loc, blk, bs);
                        }
                        if (!gsync(3)) return;
                    } else {  // the coarse part, redundantly in every block's shared memory
                        const BlockSync bs;
                        const LzLevel &G = A.lv[loc];
                        const int m0 = G.n * G.n;
                        for (int p = threadIdx.x; p < m0; p += blockDim.x) {
                            cp16(S[loc].f + p, G.f + p, true);
                            S[loc].u[p] = make_double2(0.0, 0.0);
                        }
                        if (cyc == 1) {  // kappa and 1/diag change once per slice
                            for (int l = loc; l <= Lc; ++l)
                                for (int p = threadIdx.x; p < S[l].n * S[l].n; p += blockDim.x) {
                                    cp16(S[l].kap + p, A.lv[l].kap + p, true);
                                    cp16(S[l].idg + p, A.lv[l].idg + p, true);
                                }
                        }
                        cp_wait();
                        __syncthreads();
                        if (cyc == 1 && exact) coarse_inverse(S[Lc], cwork);
                        down(S, loc, Lc, blk, bs);
                        if (exact) {
                            const int mc = S[Lc].n * S[Lc].n;
                            const double2 *inv = cwork + mc;  // row i at inv + 2 mc i
                            for (int i = threadIdx.x; i < mc; i += blockDim.x) {
                                double2 s = make_double2(0.0, 0.0);
                                for (int k = 0; k < mc; ++k)
                                    s = cadd(s, cmul(inv[2 * mc * i + k], S[Lc].f[k]));
                                S[Lc].u[i] = s;
                            }
                            __syncthreads();
                        } else {
                            smooth(S[Lc], kCoarseSweeps, blk, bs, 5);
                        }
                        up(S, Lc - 1, loc, blk, bs);
                    }
                    for (int l = loc - 1; l >= 0; --l) {
                        staged_up(A.lv[l], (local && l + 1 == loc) ? S[loc] : A.lv[l + 1], lz_dyn,
                                  blockIdx.x, gridDim.x, l == 0, &rn);
                        if (l > 0 && !gsync(30 + l)) return;
                    }
                }
                qsync::block_sum_add<kThreads>(&rn, 1, &sc->norm[kglob % 3]);
                if (!gsync(4)) return;
            }
            for (int p = grid.t; p < nn; p += grid.nt) A.dlt[p] = csub(U[p], aj[p]);
            if (!gsync(5)) return;
        }
        // the last slice's new envelope
        double2 *const last = A.a + (size_t)(A.n_xi - 1) * nn;
        for (int p = grid.t; p < nn; p += grid.nt) last[p] = cadd(last[p], A.dlt[p]);
        if (!gsync(6)) return;
    }
}

int cuda_status(cudaError_t e) {
    if (e == cudaSuccess) return QS_OK;
    cudaGetLastError();
    return e == cudaErrorMemoryAllocation ? QS_ERR_OOM : QS_ERR_CUDA;
}

}  // namespace

struct qs_laser {
    int n = 0, n_xi = 0;
    double width = 0.0, dxi = 0.0;
    cudaStream_t stream = nullptr;
    int grid_blocks = 0;
    size_t smem = 0;
    LzArgs args{};
    void *dev = nullptr;
    void *pinned = nullptr;
};

extern "C" int qs_laser_create(int n, double width, int n_xi, double k0, double dt, double dxi,
                               void *cuda_stream, qs_laser **out) {
    if (!out) return QS_ERR_ARG;
    *out = nullptr;
    if (n < 2 || n > 8192 || n_xi < 1 || !(width > 0.0) || !std::isfinite(width)) return QS_ERR_ARG;
    if (!(k0 > 0.0) || !std::isfinite(k0) || !(dt > 0.0) || !std::isfinite(dt)) return QS_ERR_ARG;
    if (!(dxi > 0.0)) return QS_ERR_ARG;  // +inf allowed: no xi coupling
    qs_laser *s = new (std::nothrow) qs_laser();
    if (!s) return QS_ERR_OOM;
    s->n = n;
    s->n_xi = n_xi;
    s->width = width;
    s->dxi = dxi;
    s->stream = static_cast<cudaStream_t>(cuda_stream);
    LzArgs &A = s->args;
    A.n = n;
    A.n_xi = n_xi;
    const double q = std::isinf(dxi) ? 0.0 : 4.0 / (dt * dxi);
    A.q = q;
    A.c = make_double2(-q, 4.0 * k0 / dt);
    // levels: halve while the side is even and above 4
    int sides[kMaxLevels];
    int levels = 0;
    for (int m = n;;) {
        sides[levels++] = m;
        if (m % 2 || m <= 4 || levels == kMaxLevels) break;
        m /= 2;
    }
    A.levels = levels;
    int odd = n;
    while (odd % 2 == 0) odd /= 2;
    const size_t line = (size_t)(n + n / 8 + 1) * sizeof(qsfft::Ff2);  // padded
    bool fft = n % 2 == 0 && n >= 8 && n <= 2048 && odd <= 7;
    size_t elems = 2 * (size_t)n * n;  // u, dlt
    const size_t tab_pairs = 3 * (size_t)n + 2 * (size_t)(n / 2 + 1);
    for (int l = 0; l < levels; ++l) elems += 5 * (size_t)sides[l] * sides[l];
    const size_t extra = fft ? 10 * (size_t)n * n + (tab_pairs + 1) / 2 : 0;
    int st = cuda_status(cudaMalloc(&s->dev, kScalarBytes + (elems + extra) * sizeof(double2)));
    if (st == QS_ERR_OOM && fft) {  // the V-cycles need none of the transforms' grids
        fft = false;
        s->dev = nullptr;
        st = cuda_status(cudaMalloc(&s->dev, kScalarBytes + elems * sizeof(double2)));
    }
    if (st == QS_OK) st = cuda_status(cudaMallocHost(&s->pinned, sizeof(LzScalars)));
    if (st != QS_OK) {
        qs_laser_destroy(s);
        return st;
    }
    char *base = static_cast<char *>(s->dev);
    A.sc = reinterpret_cast<LzScalars *>(base);
    double2 *p = reinterpret_cast<double2 *>(base + kScalarBytes);
    A.u = p;
    p += (size_t)n * n;
    A.dlt = p;
    p += (size_t)n * n;
    s->smem = lz_smem_bytes() + kCoarseBytes;
    if (fft) {
        A.r64 = p;
        p += (size_t)n * n;
        for (qsfft::Ff2 **q : {&A.tr, &A.t2, &A.tz, &A.tp, &A.cz, &A.cr, &A.cp, &A.cs, &A.ce}) {
            *q = reinterpret_cast<qsfft::Ff2 *>(p);
            p += (size_t)n * n;
        }
        A.tables = reinterpret_cast<const qsfft::Ff *>(p);
        std::vector<qsfft::Ff> tab = qsfft::host_tables(n, width / n);
        // on the object's stream, which may not wait for the default one
        st = cuda_status(cudaMemcpyAsync(p, tab.data(), tab.size() * sizeof(qsfft::Ff),
                                         cudaMemcpyHostToDevice, s->stream));
        if (st == QS_OK) st = cuda_status(cudaStreamSynchronize(s->stream));
        if (st != QS_OK) {
            qs_laser_destroy(s);
            return st;
        }
        p += (tab_pairs + 1) / 2;
        A.gmax = 1;
        while (A.gmax < 8 && 4 * A.gmax * line <= 76 * 1024) A.gmax *= 2;
        // the lines lie over the staged regions, the tables after everything
        if (2 * A.gmax * line > s->smem) s->smem = 2 * A.gmax * line;
        s->smem = (s->smem + 255) & ~(size_t)255;
        A.tab_off = (int)s->smem;
        s->smem += tab_pairs * sizeof(qsfft::Ff);
        A.fft = s->smem <= 220 * 1024;
        if (!A.fft) s->smem = lz_smem_bytes() + kCoarseBytes;
    }
    for (int l = 0; l < levels; ++l) {
        LzLevel &L = A.lv[l];
        const size_t m = (size_t)sides[l] * sides[l];
        const double h = width / sides[l];
        L.n = sides[l];
        L.ih2 = 1.0 / (h * h);
        L.u = p;  // level 0's u is replaced by A.u
        p += m;
        L.f = p;
        p += m;
        L.r = p;
        p += m;
        L.kap = p;
        p += m;
        L.idg = p;
        p += m;
    }
    int dev = 0, sms = 0, per_sm = 0;
    st = cuda_status(cudaGetDevice(&dev));
    if (st == QS_OK) st = cuda_status(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    if (st == QS_OK)
        st = cuda_status(qs_raise_smem_limit((const void *)laser_kernel));
    if (st == QS_OK)
        st = cuda_status(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, laser_kernel, kThreads,
                                                                       s->smem));
    if (st == QS_OK && per_sm < 1) st = QS_ERR_CUDA;
    if (st != QS_OK) {
        qs_laser_destroy(s);
        return st;
    }
    s->grid_blocks = sms;
    *out = s;
    return QS_OK;
}

extern "C" int qs_laser_advance(qs_laser *s, const double *d_chi, double *d_a, int steps,
                                double tol, int max_cycles, int64_t *cycles, double *max_relres) {
    if (!s || !d_chi || !d_a || steps < 0 || max_cycles < 1 || !(tol > 0.0)) return QS_ERR_ARG;
    if (steps == 0) {
        if (cycles) *cycles = 0;
        if (max_relres) *max_relres = 0.0;
        return QS_OK;
    }
    LzArgs A = s->args;
    A.chi = d_chi;
    A.a = reinterpret_cast<double2 *>(d_a);
    A.steps = steps;
    A.tol = tol;
    A.max_cycles = max_cycles;
    // a cap of a few V-cycles keeps its meaning: V-cycles; so does a tolerance below the
    // rounding of A, to which the iterations' residual (of A's change) is blind
    if (max_cycles < 4 || tol < 0x1p-52) A.fft = 0;
    int st = cuda_status(cudaMemsetAsync(A.sc, 0, sizeof(LzScalars), s->stream));
    if (st != QS_OK) return st;
    void *params[] = {&A};
    st = cuda_status(cudaLaunchCooperativeKernel((const void *)laser_kernel, dim3(s->grid_blocks),
                                                 dim3(kThreads), params, s->smem, s->stream));
    if (st != QS_OK) return st;
    st = cuda_status(cudaMemcpyAsync(s->pinned, A.sc, sizeof(LzScalars), cudaMemcpyDeviceToHost,
                                     s->stream));
    if (st == QS_OK) st = cuda_status(cudaStreamSynchronize(s->stream));
    if (st != QS_OK) return st;
    const LzScalars *h = static_cast<const LzScalars *>(s->pinned);
    if (h->err) return h->err;
    if (cycles) *cycles = h->cycles;
    if (max_relres) *max_relres = h->max_relres;
    return h->fail ? QS_ERR_NOT_CONVERGED : QS_OK;
}

extern "C" void qs_laser_destroy(qs_laser *s) {
    if (!s) return;
    if (s->dev) cudaFree(s->dev);
    if (s->pinned) cudaFreeHost(s->pinned);
    delete s;
}

// Grid of an envelope object (for the laser-driven 3D step, which checks that
// the slice loop and the envelope share cells, box and slices).
void qs_laser_shape(const qs_laser *s, int *n, double *width, int *n_xi, double *dxi) {
    *n = s->n;
    *width = s->width;
    *n_xi = s->n_xi;
    *dxi = s->dxi;
}
