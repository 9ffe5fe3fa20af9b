// Device machinery shared by the slice engine and the adjoint engine: the
// bounded grid barrier, block reductions, the direct and conjugate-gradient
// solves by sine transforms, and the multigrid solves (float64 V-cycles; refined
// form: float64 residual, float32 staged V-cycles, float64 correction).  Everything is in an unnamed namespace: each translation unit
// that includes this header gets its own copy.
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

#include "qs_cluster.cuh"
#include "qs_fft.cuh"
#include "qs_tile.cuh"

namespace {

#define SYNC(where)                 \
    do {                            \
        if (!S(where)) return false; \
    } while (0)

__device__ __forceinline__ int vload(const int *p) { return *(const volatile int *)p; }
__device__ __forceinline__ float vload(const float *p) { return *(const volatile float *)p; }
__device__ __forceinline__ double vload(const double *p) { return *(const volatile double *)p; }
__device__ __forceinline__ unsigned long long vload(const unsigned long long *p) {
    return *(const volatile unsigned long long *)p;
}

__device__ __forceinline__ int64_t global_ns() {
    int64_t t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void red_release_add_u64(unsigned long long *p, unsigned long long v) {
    asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Grid-wide barrier for a cooperative launch (all blocks co-resident).  Each
// block counts the barriers it has passed (its epoch); on arrival its thread
// 0 adds 1 to a monotonic counter with a release reduction (no round trip)
// and polls with acquire loads until the counter reaches epoch * nblk.  The
// error word is read beside the counter, never before the arrival or between
// two polls, where its trip to L2 would lie on every phase's path: a block that
// gave up does not arrive, so the others are still polling when they see it.
// A refined slice at 256^2 (23 barriers) took 213 us with both in the way, 204
// without.
struct Sync {
    DevScalars *sc;             // the instance's scalars (error word, trace count)
    unsigned long long *bar;    // monotonic arrival counter of the blocks in the team
    unsigned nblk;              // blocks in the team
    long long limit;
    int64_t *trace;
    int trace_cap;
    unsigned long long *epoch;  // this block's barrier count (shared memory)
    bool tracer;                // this block records the phase trace
    int cl = 1;                 // cluster size of the launch (> 1: clusters run
                                // the multigrid cycles, see qs_cluster.cuh)
    // Arrival without the wait, of a block that neither reads what the others wrote
    // before this barrier nor writes before the next one, where it waits.
    __device__ void arrive() const {
        __syncthreads();
        if (threadIdx.x == 0) {
            *epoch += 1;
            red_release_add_u64(bar, 1ull);
        }
    }
    __device__ bool operator()(int where) const {
        __shared__ int s_ok;
        __syncthreads();
        if (threadIdx.x == 0) {
            int ok = 1;
            const unsigned long long target = (*epoch + 1) * nblk;
            *epoch += 1;
            red_release_add_u64(bar, 1ull);
            const long long t0 = clock64();
            for (;;) {
                const int err = vload(&sc->err);
                if (ld_acquire_u64(bar) >= target) break;
                if (err != 0) {
                    ok = 0;
                    break;
                }
                if (clock64() - t0 > limit) {
                    if (atomicCAS(&sc->err, 0, QS_ERR_TIMEOUT) == 0) sc->err_where = where;
                    ok = 0;
                    break;
                }
            }
            s_ok = ok;
            if (trace && tracer) {
                const unsigned long long k = sc->trace_n;
                if (k < (unsigned long long)trace_cap) {
                    trace[2 * k] = where;
                    trace[2 * k + 1] = global_ns();
                    sc->trace_n = k + 1;
                }
            }
        }
        __syncthreads();
        if (cl > 1) {
            // The blocks of a cluster take one decision: after a timed-out
            // wait some blocks may see the barrier complete and others the
            // error word, and a block that went on into a cluster solve
            // would wait at a cluster barrier for one that has left.
            namespace cg = cooperative_groups;
            cg::cluster_group clu = cg::this_cluster();
            __shared__ int s_oks[16];
            if (threadIdx.x == 0)
                clu.map_shared_rank(s_oks, 0)[clu.block_rank()] = s_ok;
            clu.sync();
            if (threadIdx.x == 0) {
                const int *all = clu.map_shared_rank(s_oks, 0);
                int ok = 1;
                for (int b = 0; b < cl; ++b) ok &= all[b] != 0;
                s_ok = ok;
            }
            clu.sync();  // s_oks is rewritten at the next barrier
        }
        return s_ok != 0;
    }
};

using qsmg::Thr;
// The first index of this thread in the grid-wide loops
// `for (i = t0; i < count; i += nt)`.  Runs of 32 consecutive indices go to
// the blocks in turn (run w * nblk + b to warp w of block b), so that a loop
// shorter than the launch (a coarse level, a 64^2 grid, the cells of a small
// grid) still spreads over every SM, while each warp's accesses stay
// contiguous.  float64 work is throughput-bound on GB300 (about two FMA per
// clock per SM): the same loop on the first few blocks alone took several
// times longer.  t0 ranges over a permutation of [0, nt) (blockDim.x is a
// multiple of 32), so every index is visited exactly once.
__device__ __forceinline__ Thr grid_thr(int bid, int nblk) {
    const int w = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
    return Thr{((w * nblk + bid) << 5) + lane, nblk * (int)blockDim.x};
}

// sum over the block; valid in thread 0
__device__ double block_sum(double v) {
    double *const red = (double *)qsfft::sum_scratch();
    for (int o = 16; o; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) red[wid] = v;
    __syncthreads();
    double t = 0.0;
    if (wid == 0) {
        int nw = (blockDim.x + 31) >> 5;
        t = lane < nw ? red[lane] : 0.0;
        for (int o = 16; o; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    }
    return t;
}
// four float32 sums over the block in one pass (one block barrier); valid in
// thread 0
__device__ void block_sum4f(float v[4]) {
    float (*const red4)[4] = (float (*)[4])qsfft::sum_scratch();
#pragma unroll
    for (int k = 0; k < 4; ++k)
        for (int o = 16; o; o >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < 4; ++k) red4[wid][k] = v[k];
    __syncthreads();
    if (wid == 0) {
        const int nw = (blockDim.x + 31) >> 5;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            float t = lane < nw ? red4[lane][k] : 0.f;
            for (int o = 16; o; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
            v[k] = t;
        }
    }
    __syncthreads();  // red4 is reused by the next call
}

// Adds the block's sums of v[0 .. K) (>= 0; squares) to dst[0 .. K).  The
// values keep float64's range and the sums float32's precision, each warp's
// with a power of two of its own: a norm may be of 1e-30 or of 1e+30, which
// squares in float32 are not.  (A float64 sum is 10 additions of 64 cycles a
// warp and value.)
template <int K>
__device__ void block_sum_wide(const double (&v)[K], double *dst) {
    constexpr int nw = QS_ENGINE_THREADS / 32;
    static_assert(K <= 9 && nw <= qsfft::kSumWarps, "scratch");
    float (*const sm)[nw] = (float (*)[nw])qsfft::sum_scratch();
    int (*const se)[nw] = (int (*)[nw])(qsfft::sum_scratch() + K * nw);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();  // the scratch may still be read
#pragma unroll
    for (int c = 0; c < K; ++c) {
        const unsigned hi = (unsigned)__double2hiint(v[c]);
        const int e = (int)(hi >> 20) & 0x7ff, E = __reduce_max_sync(0xffffffffu, e);
        float m = 0.f;
        if (e == 0x7ff) m = (float)v[c];  // infinite or NaN
        else if (e > 0 && E - e <= 60)
            m = qsff::split(__hiloint2double((int)(hi + ((unsigned)(1023 - E) << 20)),
                                             __double2loint(v[c]))).h;
        for (int o = 16; o; o >>= 1) m += __shfl_xor_sync(0xffffffffu, m, o);
        if (lane == 0) {
            sm[c][wid] = m;
            se[c][wid] = E;
        }
    }
    __syncthreads();
    for (int c = wid; c < K; c += nw) {
        const int e = lane < nw ? se[c][lane] : 0, E = __reduce_max_sync(0xffffffffu, e);
        float m = lane < nw ? sm[c][lane] : 0.f;
        if (E - e > 60) m = 0.f;
        else m *= __int_as_float((127 + e - E) << 23);
        for (int o = 16; o; o >>= 1) m += __shfl_xor_sync(0xffffffffu, m, o);
        if (lane == 0 && m != 0.f) {
            const double w = qsff::widen(m);
            const int x = ((__double2hiint(w) >> 20) & 0x7ff) + E - 1023;
            double t = w;  // not finite
            if (E != 0x7ff)
                t = x >= 0x7ff ? __longlong_as_double(0x7ff0000000000000LL)
                               : __hiloint2double((__double2hiint(w) & 0xfffff) | (x << 20),
                                                  __double2loint(w));
            atomicAdd(dst + c, t);
        }
    }
}

__device__ float block_max(float v) {
    float *const redf = qsfft::sum_scratch();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int o = 16; o; o >>= 1) v = fmaxf(v, __shfl_down_sync(0xffffffffu, v, o));
    __syncthreads();
    if (lane == 0) redf[wid] = v;
    __syncthreads();
    float t = 0.f;
    if (wid == 0) {
        t = lane < ((int)blockDim.x >> 5) ? redf[lane] : 0.f;
        for (int o = 16; o; o >>= 1) t = fmaxf(t, __shfl_down_sync(0xffffffffu, t, o));
    }
    return t;
}
__device__ double block_max(double v) {
    double *const red = (double *)qsfft::sum_scratch();
    for (int o = 16; o; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) red[wid] = v;
    __syncthreads();
    double t = 0.0;
    if (wid == 0) {
        int nw = (blockDim.x + 31) >> 5;
        t = lane < nw ? red[lane] : 0.0;
        for (int o = 16; o; o >>= 1) t = fmax(t, __shfl_down_sync(0xffffffffu, t, o));
    }
    return t;
}

// ---------------------------------------------------------------------------
// multigrid solves (1 or 2 components sharing the operator)
// ---------------------------------------------------------------------------
using qsmg::Hier;
using qsmg::Lvl;

struct SolveSpec {
    int nc;
    int kind;  // 0 psi, 1 (Ez,Bz), 2 (Bx,By): index into fnorm / vcycles
    double *u[2];
    double *f[2];
    bool screened;
    float *u32[2] = {nullptr, nullptr};  // refined form: float32 copy of the solution
};

// The hierarchy descriptors live in shared memory, one copy per block:
// thread l fills level l (a per-thread copy indexed by level would sit in
// local memory and be re-read from L1/L2 on every access).
__device__ void hier64(const EngineArgs &A, const SolveSpec &V, Hier<double> &H) {
    H.L = A.nlev;
    for (int l = threadIdx.x; l < A.nlev; l += blockDim.x) {
        Lvl<double> &v = H.lv[l];
        v.n = A.lev_n[l];
        v.h2 = A.lev_h2[l];
        v.inv_h2 = A.lev_inv_h2[l];
        v.h2t = A.lev_h2[l];
        v.inv_h2t = A.lev_inv_h2[l];
        v.omega = A.omega;
        for (int c = 0; c < 2; ++c) {
            v.u[c] = l == 0 ? V.u[c] : A.lev[l].u[c];
            v.f[c] = l == 0 ? V.f[c] : A.lev[l].f[c];
        }
        v.k = V.screened ? (l == 0 ? A.kap : A.lev[l].kap) : nullptr;
        v.d = V.screened ? (l == 0 ? A.invd0 : A.lev[l].d) : nullptr;
    }
}

__device__ void hier32(const EngineArgs &A, const SolveSpec &V, Hier<float> &H) {
    H.L = A.nlev;
    for (int l = threadIdx.x; l < A.nlev; l += blockDim.x) {
        Lvl<float> &v = H.lv[l];
        v.n = A.lev_n[l];
        v.h2 = A.lev_h2[l];
        v.inv_h2 = A.lev_inv_h2[l];
        v.h2t = A.lev_h2f[l];
        v.inv_h2t = A.lev_inv_h2f[l];
        v.omega = (float)A.omega;
        for (int c = 0; c < 2; ++c) {
            v.u[c] = l == 0 ? A.e32[c] : A.lev32[l].u[c];
            v.f[c] = l == 0 ? A.r32[0][c] : A.lev32[l].f[c];
        }
        v.k = V.screened ? (l == 0 ? A.k32 : A.lev32[l].k) : nullptr;
        v.d = V.screened ? (l == 0 ? A.d32 : A.lev32[l].d) : nullptr;
    }
}

// Level-0 red-black half sweep of the float32 correction that also adds the
// final correction into the float64 iterate: u64 += e at the points this
// thread updates and at the points of the other colour (not written here).
template <int NC>
__device__ void relax_half_finalize(const Lvl<float> L, int color, Thr R, double *fin0,
                                    double *fin1) {
    const int n = L.n;
    const float h2 = L.h2t;
    float *const u0 = L.u[0];
    float *const u1 = L.u[NC - 1];
    const float *const f0 = L.f[0];
    const float *const f1 = L.f[NC - 1];
    const int npts = n * n;
    for (qsmg::Walk w(R.t0, R.nt, n); w.q < npts; w.next()) {
        const int ix = w.col, iy = w.row;
        const int i = w.q;
        if (((ix + iy) & 1) == color) {
            const float di = L.d ? L.d[i] : qsmg::const_inv_diag<float>(qsmg::walls(ix, iy, n));
            qsmg::gs_point<float, NC>(u0, u1, f0, f1, h2, di, L.omega, n, ix, iy);
        }
        fin0[i] += (double)u0[i];
        if (NC > 1) fin1[i] += (double)u1[i];
    }
}

// One V-cycle on hierarchy H.  Levels of side > block_level_n are relaxed by
// the whole grid, the rest by block 0 in shared memory.  With `fin0` set (the
// refined form) the float32 correction is added into the float64 iterate
// during the last level-0 phase.
template <typename T, int NC>
__device__ bool vcycle(const EngineArgs &A, const Sync &S, const Hier<T> &H, int bid, int nblk,
                       void *smem, qsmg::CoarseInv ci, double *fin0, double *fin1) {
    const int L = H.L;
    int lg = 0;
    while (lg < L - 1 && H.lv[lg].n > A.block_level_n) ++lg;
    const Thr T0 = grid_thr(bid, nblk);
    for (int l = 0; l < lg; ++l) {
        const Lvl<T> F = H.lv[l], C = H.lv[l + 1];
        for (int s = 0; s < A.nu1; ++s) {
            qsmg::relax_half<T, NC>(F, 0, T0);
            SYNC(10);
            qsmg::relax_half<T, NC>(F, 1, T0);
            SYNC(11);
        }
        qsmg::restrict_res<T, NC>(F, C, T0);
        SYNC(12);
    }
    if (bid == 0) qsmg::block_vcycle<T, NC>(H, lg, A.nu1c, A.nu2, smem, ci);
    SYNC(13);
    if constexpr (sizeof(T) == 4) {
        if (fin0 && (lg == 0 || A.nu2 == 0)) {
            // no fused level-0 sweep: add the correction in a phase of its own
            for (int l = lg - 1; l >= 0; --l) {
                qsmg::prolong_add<T, NC>(H.lv[l], H.lv[l + 1], T0);
                SYNC(14);
            }
            const int nn = H.lv[0].n * H.lv[0].n;
            const float *e0 = H.lv[0].u[0];
            const float *e1 = H.lv[0].u[NC - 1];
            for (int q = T0.t0; q < nn; q += T0.nt) {
                fin0[q] += (double)e0[q];
                if (NC > 1) fin1[q] += (double)e1[q];
            }
            SYNC(17);
            return true;
        }
    }
    for (int l = lg - 1; l >= 0; --l) {
        const Lvl<T> F = H.lv[l], C = H.lv[l + 1];
        qsmg::prolong_add<T, NC>(F, C, T0);
        SYNC(14);
        for (int s = 0; s < A.nu2; ++s) {
            qsmg::relax_half<T, NC>(F, 0, T0);
            SYNC(15);
            if constexpr (sizeof(T) == 4) {
                if (fin0 && l == 0 && s == A.nu2 - 1) {
                    relax_half_finalize<NC>(F, 1, T0, fin0, fin1);
                    SYNC(16);
                    continue;
                }
            }
            qsmg::relax_half<T, NC>(F, 1, T0);
            SYNC(16);
        }
    }
    return true;
}

// Output tile of a staged level of side n: the configured tile, halved
// (the longer side first, down to 8) while the level has fewer than nblk/2
// tiles, so that coarser grid-wide levels still spread over the blocks and
// each block's region stays small.
__device__ __forceinline__ void level_tile(const EngineArgs &A, int n, int nblk, int &TX,
                                           int &TY) {
    TX = A.tile_x;
    TY = A.tile_y;
    for (;;) {
        const int tiles = ((n + TX - 1) / TX) * ((n + TY - 1) / TY);
        if (2 * tiles >= nblk) break;
        if (TX >= TY && TX > 8) TX >>= 1;
        else if (TY > 8) TY >>= 1;
        else break;
    }
}

// Refined form: one float32 V-cycle on the correction.  The grid-wide levels
// are staged tile by tile on the way down (one grid barrier per level);
// every block then solves the coarse levels itself in shared memory (no
// barrier); one phase runs every up leg and the level-0 update of the
// float64 iterate u and residual r (r <- r - A e) and accumulates ||r||^2,
// ||u||^2 into norms_out (the slot of the convergence test).
// *fused_done reports whether that happened: grids too small to stage fall
// back to the plain cycle, which leaves the residual to a separate pass.
template <int NC>
__device__ bool vcycle_staged(const EngineArgs &A, const Sync &S, const Hier<float> &H, int bid,
                              int nblk, void *smem, qsmg::CoarseInv ci, double *fin0,
                              double *fin1, const qstile::Fused *fused, double *norms_out,
                              double *norms_clear, bool *fused_done) {
    const int L = H.L;
    int lg = 0;
    while (lg < L - 1 && H.lv[lg].n > A.block_level_n) ++lg;
    *fused_done = false;
    if (lg == 0) return vcycle<float, NC>(A, S, H, bid, nblk, smem, ci, fin0, fin1);
    // shared memory: the coarse part's levels first, the staged tile after them
    float *sm = (float *)((char *)smem + A.tile_smem_offset);
    const qsmg::Marks mk{bid == 0 ? A.trace : nullptr, &A.sc->trace_n, A.trace_cap};
    for (int l = 0; l < lg; ++l) {
        int TX, TY;
        level_tile(A, H.lv[l].n, nblk, TX, TY);
        // the correction starts from zero; its pre-smoothed tile goes to
        // the level's own array (the up cascade reads it there)
        qstile::down_level<float, NC>(H.lv[l], H.lv[l + 1], A.nu1, TX, TY, sm, bid, nblk,
                                      H.lv[l].u, nullptr, mk);
        mk(62);
        SYNC(30);
    }
    qsmg::block_vcycle<float, NC>(H, lg, A.nu1c, A.nu2, smem, ci, false, mk);
    const int mg2 = H.lv[lg].n * H.lv[lg].n;
    // every up leg and the level-0 update in one phase
    int TX, TY;
    level_tile(A, H.lv[0].n, nblk, TX, TY);
    // ||r||^2, ||u||^2 of the tile in float32: the stopping test needs a
    // few digits of them
    float nrm[4] = {0.f, 0.f, 0.f, 0.f};
    qstile::up_cascade_fused<NC>(H, lg, (const float *)smem, (const float *)smem + 2 * mg2,
                                 A.nu2, TX, TY, sm, bid, nblk, *fused, nrm, mk);
    block_sum4f(nrm);
    if (threadIdx.x == 0)
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            atomicAdd(norms_out + c, (double)nrm[c]);
            atomicAdd(norms_out + 2 + c, (double)nrm[2 + c]);
        }
    if (bid == 0 && threadIdx.x == 0)
        for (int e = 0; e < 4; ++e) norms_clear[e] = 0.0;
    mk(67);
    *fused_done = true;
    SYNC(32);
    return true;
}

// Float64 form: one V-cycle with the grid-wide levels staged tile by tile
// (qs_tile.cuh): a down leg per level (pre-sweeps from the iterate at level
// 0, from zero below, residual, restriction; the pre-smoothed tile to the
// level's scratch pair), the coarse levels by block 0, an up leg per level
// (prolongation, post-sweeps) reading the scratch pair; the level-0 up leg
// also sums ||f - A u||^2 and ||u||^2 of its tile into norms_out for the
// stopping test.  One grid barrier per level and leg instead of one per
// colour sweep, restriction and prolongation.
template <int NC>
__device__ bool vcycle_staged64(const EngineArgs &A, const Sync &S, const Hier<double> &H,
                                int bid, int nblk, void *smem, qsmg::CoarseInv ci,
                                double *norms_out, double *norms_clear) {
    const int L = H.L;
    int lg = 0;
    while (lg < L - 1 && H.lv[lg].n > A.block_level_n) ++lg;
    double *sm = (double *)((char *)smem + A.tile_smem_offset);
    for (int l = 0; l < lg; ++l) {
        int TX, TY;
        level_tile(A, H.lv[l].n, nblk, TX, TY);
        qstile::down_level<double, NC>(H.lv[l], H.lv[l + 1], A.nu1, TX, TY, sm, bid, nblk,
                                       A.lev[l].s, l == 0 ? H.lv[0].u : nullptr);
        SYNC(40);
    }
    if (bid == 0) qsmg::block_vcycle<double, NC>(H, lg, A.nu1c, A.nu2, smem, ci);
    SYNC(41);
    double nrm[4] = {0.0, 0.0, 0.0, 0.0};
    for (int l = lg - 1; l >= 0; --l) {
        int TX, TY;
        level_tile(A, H.lv[l].n, nblk, TX, TY);
        qstile::up_level<double, NC>(H.lv[l], H.lv[l + 1], A.lev[l].s, A.nu2, TX, TY, sm, bid,
                                     nblk, l == 0, nrm);
        if (l > 0) SYNC(42);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const double t = block_sum(nrm[k]);
        if (threadIdx.x == 0 && (k & 1) < NC) atomicAdd(norms_out + k, t);
    }
    if (bid == 0 && threadIdx.x == 0)
        for (int e = 0; e < 4; ++e) norms_clear[e] = 0.0;
    SYNC(43);
    return true;
}

// ||f - A u||^2 and ||u||^2 per component at level 0 in float64, accumulated
// into out[c] and out[2 + c].  For the refined form the residual also becomes
// the float32 right-hand side of the next inner cycle, whose correction
// starts at zero.
template <int NC>
__device__ void residual_norm(const EngineArgs &A, const SolveSpec &V, double *out, Thr T,
                              bool to32, float *const *r32) {
    const int n = A.N;
    const double inv_h2 = A.lev_inv_h2[0];
    const double *const kap = V.screened ? A.kap : nullptr;
    const double *const u0 = V.u[0];
    const double *const u1 = V.u[NC - 1];
    const double *const f0 = V.f[0];
    const double *const f1 = V.f[NC - 1];
    float *const r0 = r32[0];
    float *const r1 = r32[NC - 1];
    float *const e0 = A.e32[0];
    float *const e1 = A.e32[NC - 1];
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    for (qsmg::Walk w(T.t0, T.nt, n); w.q < n * n; w.next()) {
        const int k = w.q;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const double *u = c ? u1 : u0;
            const double r = (c ? f1 : f0)[k] - qsmg::apply_op<double>(u, kap, n, inv_h2, w.col, w.row);
            s[c] += r * r;
            s[2 + c] += u[k] * u[k];
            if (to32) {
                (c ? r1 : r0)[k] = (float)r;
                (c ? e1 : e0)[k] = 0.f;
                A.r64[c][k] = r;
            }
        }
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        double t = block_sum(s[c]);
        if (threadIdx.x == 0) atomicAdd(out + c, t);
        t = block_sum(s[2 + c]);
        if (threadIdx.x == 0) atomicAdd(out + 2 + c, t);
    }
}

// ---------------------------------------------------------------------------
// V-cycles inside thread-block clusters (qs_cluster.cuh): one cluster per
// component, cluster k = blocks [k C, (k + 1) C) of the launch.
// ---------------------------------------------------------------------------

// The cluster's view of its hierarchy: distributed level l (l < Y.ld) and
// the local levels of block 0.
template <typename T>
struct ClusterView {
    void *cb;  // the cluster region of this block's shared memory
    const qsclu::Layout *Y;
    int rank, C;
    bool scr;
    __device__ qsclu::DLvl<T> dl(const EngineArgs &A, cooperative_groups::cluster_group &cl,
                                 int l) const {
        qsclu::DLvl<T> D;
        D.n = Y->n[l];
        D.R = Y->R[l];
        D.row0 = rank * D.R;
        D.u = qsclu::arr<T>(cb, *Y, l, 0);
        D.f = qsclu::arr<T>(cb, *Y, l, 1);
        D.k = scr ? qsclu::arr<T>(cb, *Y, l, 2) : nullptr;
        D.d = scr ? qsclu::arr<T>(cb, *Y, l, 3) : nullptr;
        D.up_u = rank > 0 ? cl.map_shared_rank(D.u, rank - 1) : nullptr;
        D.dn_u = rank < C - 1 ? cl.map_shared_rank(D.u, rank + 1) : nullptr;
        D.h2 = (T)A.lev_h2[l];
        D.inv_h2 = (T)A.lev_inv_h2[l];
        D.omega = (T)A.omega;
        return D;
    }
    __device__ Lvl<T> lv(const EngineArgs &A, int l) const {
        Lvl<T> v;
        v.u[0] = v.u[1] = qsclu::arr<T>(cb, *Y, l, 0);
        v.f[0] = v.f[1] = qsclu::arr<T>(cb, *Y, l, 1);
        v.k = scr ? qsclu::arr<T>(cb, *Y, l, 2) : nullptr;
        v.d = scr ? qsclu::arr<T>(cb, *Y, l, 3) : nullptr;
        v.n = Y->n[l];
        v.h2 = A.lev_h2[l];
        v.inv_h2 = A.lev_inv_h2[l];
        v.h2t = (T)A.lev_h2[l];
        v.inv_h2t = (T)A.lev_inv_h2[l];
        v.omega = (T)A.omega;
        return v;
    }
};

// One V(nu1, nu2) cycle of the cluster's component on the hierarchy held in
// its shared memory (level 0's u and f already there).  with_k: restrict
// kappa too (the first cycle of a solve).
template <typename T>
__device__ void cluster_vcycle(const EngineArgs &A, cooperative_groups::cluster_group &cl,
                               const ClusterView<T> &V, qsmg::CoarseInv ci, bool with_k,
                               const qsmg::Marks &mk) {
    const qsclu::Layout &Y = *V.Y;
    const int ld = Y.ld, L = Y.L;
    for (int l = 0; l < ld; ++l) {
        const qsclu::DLvl<T> D = V.dl(A, cl, l);
        const int nu = D.n > A.block_level_n ? A.nu1 : A.nu1c;
        for (int s = 0; s < nu; ++s) {
            qsclu::d_relax<T>(D, 0);
            cl.sync();
            qsclu::d_relax<T>(D, 1);
            cl.sync();
        }
        const int m = Y.n[l + 1];
        T *cu, *cf, *ck = nullptr, *cd = nullptr;
        int crow0;
        if (l + 1 < ld) {  // into this block's strip of the next level
            cu = qsclu::arr<T>(V.cb, Y, l + 1, 0);
            cf = qsclu::arr<T>(V.cb, Y, l + 1, 1);
            if (V.scr) {
                ck = qsclu::arr<T>(V.cb, Y, l + 1, 2);
                cd = qsclu::arr<T>(V.cb, Y, l + 1, 3);
            }
            crow0 = D.row0 >> 1;
        } else {  // into block 0's whole first local level
            cu = cl.map_shared_rank(qsclu::arr<T>(V.cb, Y, ld, 0), 0);
            cf = cl.map_shared_rank(qsclu::arr<T>(V.cb, Y, ld, 1), 0);
            if (V.scr) {
                ck = cl.map_shared_rank(qsclu::arr<T>(V.cb, Y, ld, 2), 0);
                cd = cl.map_shared_rank(qsclu::arr<T>(V.cb, Y, ld, 3), 0);
            }
            crow0 = 0;
        }
        qsclu::d_restrict<T>(D, m, crow0, cu, cf, ck, cd, (T)A.lev_h2[l + 1], with_k);
        cl.sync();
        mk(71 + l);
    }
    if (V.rank == 0) {  // the local levels, all of block 0's warps
        const Thr B{(int)threadIdx.x, (int)blockDim.x};
        for (int l = ld; l < L - 1; ++l) {
            const Lvl<T> F = V.lv(A, l), Cc = V.lv(A, l + 1);
            const int nu = F.n > A.block_level_n ? A.nu1 : A.nu1c;
            for (int s = 0; s < nu; ++s) {
                qsmg::relax_half<T, 1>(F, 0, B);
                __syncthreads();
                qsmg::relax_half<T, 1>(F, 1, B);
                __syncthreads();
            }
            qsmg::restrict_res<T, 1>(F, Cc, B, with_k);
            __syncthreads();
        }
        qsmg::coarse_solve<T, 1>(V.lv(A, L - 1), (double *)((char *)V.cb + Y.work), ci);
        for (int l = L - 2; l >= ld; --l) {
            const Lvl<T> F = V.lv(A, l), Cc = V.lv(A, l + 1);
            qsmg::prolong_add<T, 1>(F, Cc, B);
            __syncthreads();
            for (int s = 0; s < A.nu2; ++s) {
                qsmg::relax_half<T, 1>(F, 0, B);
                __syncthreads();
                qsmg::relax_half<T, 1>(F, 1, B);
                __syncthreads();
            }
        }
    }
    cl.sync();
    mk(78);
    for (int l = ld - 1; l >= 0; --l) {
        const qsclu::DLvl<T> D = V.dl(A, cl, l);
        if (l + 1 == ld)
            qsclu::d_prolong_w<T>(D, cl.map_shared_rank(qsclu::arr<T>(V.cb, Y, ld, 0), 0),
                                  Y.n[ld]);
        else
            qsclu::d_prolong_d<T>(D, V.dl(A, cl, l + 1));
        cl.sync();
        for (int s = 0; s < A.nu2; ++s) {
            qsclu::d_relax<T>(D, 0);
            cl.sync();
            qsclu::d_relax<T>(D, 1);
            cl.sync();
        }
        mk(81 + l);
    }
}

// Float64 form: the solve of component bid / C by its cluster, to the grid
// path's stopping test; fn: ||f||^2 per component (thread 0).  Blocks of
// other clusters return at once; the caller's grid barrier follows.
__device__ __noinline__ void mg_solve_cluster64(const EngineArgs &A, const SolveSpec &V, int bid,
                                   void *smem_base, qsmg::CoarseInv ci, const double *fn) {
    namespace cg = cooperative_groups;
    const int C = A.cl_size, comp = bid / C;
    if (comp >= V.nc) return;
    cg::cluster_group cl = cg::this_cluster();
    __shared__ qsclu::Layout Y;
    __shared__ int s_conv;
    __shared__ double s_rel;
    if (threadIdx.x == 0) Y = qsclu::cluster_layout(A.lev_n, A.nlev, C, sizeof(double));
    __syncthreads();
    const ClusterView<double> cv{(char *)smem_base + A.cl_smem_offset, &Y,
                                 (int)cl.block_rank(), C, V.screened};
    const double *const gu = V.u[comp];
    const double *const gf = V.f[comp];
    {  // level 0: this block's rows of the warm start, the source and kappa
        const qsclu::DLvl<double> D = cv.dl(A, cl, 0);
        const size_t g0 = (size_t)D.row0 * D.n;
        for (int q = threadIdx.x; q < D.R * D.n; q += blockDim.x) {
            D.u[q] = gu[g0 + q];
            D.f[q] = gf[g0 + q];
            if (cv.scr) {
                D.k[q] = A.kap[g0 + q];
                D.d[q] = A.invd0[g0 + q];
            }
        }
    }
    cl.sync();
    double *const slots0 = cl.map_shared_rank((double *)((char *)cv.cb + Y.slots), 0);
    const double fl = 1e-13 * A.lev_inv_h2[0];
    const qsmg::Marks mk{A.trace, &A.sc->trace_n, A.trace_cap};  // block 0, thread 0
    int it = 0;
    bool conv = false;
    for (;;) {
        if (it > 0) {  // ||f - A u||^2 and ||u||^2 of the component
            const qsclu::DLvl<double> D = cv.dl(A, cl, 0);
            double s[2] = {0.0, 0.0};
            for (int q = threadIdx.x; q < D.R * D.n; q += blockDim.x) {
                const int ly = q / D.n, x = q - ly * D.n;
                const double r = qsclu::d_res(D, x, D.row0 + ly, q);
                s[0] += r * r;
                s[1] += D.u[q] * D.u[q];
            }
            for (int e = 0; e < 2; ++e) {
                const double t = block_sum(s[e]);
                if (threadIdx.x == 0) slots0[cv.rank * 2 + e] = t;
            }
            cl.sync();
            __shared__ double s_tot[2];
            if (threadIdx.x < 32) {  // warp 0: one remote load per lane, then a warp sum
                for (int e = 0; e < 2; ++e) {
                    double v = 0.0;
                    for (int b = threadIdx.x; b < C; b += 32) v += slots0[b * 2 + e];
                    for (int o = 16; o; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
                    if (threadIdx.x == 0) s_tot[e] = v;
                }
            }
            if (threadIdx.x == 0) {
                const double f2 = fn[comp];
                double thr = fmax(A.mg_tol * A.mg_tol * f2, A.mg_atol * A.mg_atol);
                thr = fmax(thr, fl * fl * s_tot[1]);
                s_conv = f2 == 0.0 ? 1 : !(s_tot[0] <= 1.7e308) ? 2 : s_tot[0] <= thr;
                s_rel = f2 > 0.0 ? sqrt(s_tot[0] / f2) : 0.0;
            }
            __syncthreads();
            conv = s_conv == 1;
            mk(70);
            if (s_conv || it >= A.mg_max_vcycles) break;
        }
        cluster_vcycle<double>(A, cl, cv, ci, it == 0, mk);
        ++it;
    }
    {  // this block's rows of the solution
        const qsclu::DLvl<double> D = cv.dl(A, cl, 0);
        const size_t g0 = (size_t)D.row0 * D.n;
        double *const u = V.u[comp];
        for (int q = threadIdx.x; q < D.R * D.n; q += blockDim.x) u[g0 + q] = D.u[q];
    }
    if (cv.rank == 0 && threadIdx.x == 0) {
        DevScalars *sc = A.sc;
        atomicMax(&sc->cl_cycles, it);
        atomicMax((unsigned long long *)&sc->max_relres,
                  (unsigned long long)__double_as_longlong(s_rel));
        if (!conv) sc->not_converged = 1;
    }
    cl.sync();  // no block leaves while another may still read its shared memory
}

// Refined form, the cluster part of an outer iteration: the float32 V-cycle
// of the correction e (from zero) with the float32 residual as right-hand
// side, by the cluster of component bid / C; e is written to A.e32[comp].
__device__ __noinline__ void cluster_inner_cycle(const EngineArgs &A, const SolveSpec &V, int bid,
                                    void *smem_base, qsmg::CoarseInv ci, bool first) {
    namespace cg = cooperative_groups;
    const int C = A.cl_size, comp = bid / C;
    if (comp >= V.nc) return;
    cg::cluster_group cl = cg::this_cluster();
    __shared__ qsclu::Layout Y;
    if (threadIdx.x == 0) Y = qsclu::cluster_layout(A.lev_n, A.nlev, C, sizeof(float));
    __syncthreads();
    const ClusterView<float> cv{(char *)smem_base + A.cl_smem_offset, &Y,
                                (int)cl.block_rank(), C, V.screened};
    const qsmg::Marks mk{A.trace, &A.sc->trace_n, A.trace_cap};
    {
        const qsclu::DLvl<float> D = cv.dl(A, cl, 0);
        const size_t g0 = (size_t)D.row0 * D.n;
        const float *const r = A.r32[0][comp];
        for (int q = threadIdx.x; q < D.R * D.n; q += blockDim.x) {
            D.u[q] = 0.f;
            D.f[q] = r[g0 + q];
            if (first && cv.scr) {  // kappa is fixed during a solve
                D.k[q] = A.k32[g0 + q];
                D.d[q] = A.d32[g0 + q];
            }
        }
    }
    cl.sync();
    cluster_vcycle<float>(A, cl, cv, ci, first, mk);
    {
        const qsclu::DLvl<float> D = cv.dl(A, cl, 0);
        const size_t g0 = (size_t)D.row0 * D.n;
        float *const e = A.e32[comp];
        for (int q = threadIdx.x; q < D.R * D.n; q += blockDim.x) e[g0 + q] = D.u[q];
    }
    cl.sync();
}

// Refined form, the grid-wide part of an outer iteration: in float64,
// u += e and r <- r - (lap_h - kappa) e (= f - A(u + e)), with the 5-point
// sum of the float32 e formed exactly as a float32 pair (error-free sums and
// an FMA product) before it is widened; r32 = (float) r for the next cycle;
// the float32 copy of u where asked; ||r||^2, ||u||^2 into norms_out.
template <int NC>
__device__ __noinline__ void update_from_e(const EngineArgs &A, const SolveSpec &V, Thr T,
                              double *norms_out) {
    const int n = A.N;
    const double inv_h2 = A.lev_inv_h2[0];
    const double *const kap = V.screened ? A.kap : nullptr;
    float nrm[4] = {0.f, 0.f, 0.f, 0.f};
    for (qsmg::Walk w(T.t0, T.nt, n); w.q < n * n; w.next()) {
        const int x = w.col, y = w.row, i = w.q;
        const float cw = (float)(4 + qsmg::walls(x, y, n));
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const float *e = A.e32[c];
            const float ef = e[i];
            float hi = 0.f, lo = 0.f;
            if (x > 0) qstile::two_sum_acc(hi, lo, e[i - 1]);
            if (x < n - 1) qstile::two_sum_acc(hi, lo, e[i + 1]);
            if (y > 0) qstile::two_sum_acc(hi, lo, e[i - n]);
            if (y < n - 1) qstile::two_sum_acc(hi, lo, e[i + n]);
            const float pc = __fmul_rn(cw, ef);
            const float pe = __fmaf_rn(cw, ef, -pc);  // cw ef = pc + pe exactly
            qstile::two_sum_acc(hi, lo, -pc);
            lo = __fsub_rn(lo, pe);
            const double ec = (double)ef;
            double ae = ((double)hi + (double)lo) * inv_h2;
            if (kap) ae -= kap[i] * ec;
            const double u = V.u[c][i] + ec;
            const double r = A.r64[c][i] - ae;
            const float rf = (float)r, uf = (float)u;
            V.u[c][i] = u;
            A.r64[c][i] = r;
            A.r32[0][c][i] = rf;
            if (V.u32[c]) V.u32[c][i] = uf;
            nrm[c] = __fmaf_rn(rf, rf, nrm[c]);
            nrm[2 + c] = __fmaf_rn(uf, uf, nrm[2 + c]);
        }
    }
    block_sum4f(nrm);
    if (threadIdx.x == 0)
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            atomicAdd(norms_out + c, (double)nrm[c]);
            atomicAdd(norms_out + 2 + c, (double)nrm[2 + c]);
        }
}

// Refined form in clusters: each outer iteration is one float32 V-cycle of
// the correction per component, by that component's cluster, then the
// float64 update of u and r by the whole grid (two grid barriers).  A
// separate function: inlined, its registers made the slice engine spill.
__device__ __noinline__ bool mg_solve_ref_cluster(const EngineArgs &A, const Sync &S,
                                                  const SolveSpec &V, int &slot, int bid,
                                                  int nblk, void *smem_base, qsmg::CoarseInv ci,
                                                  const double *s_fn) {
    DevScalars *sc = A.sc;
    const Thr T = grid_thr(bid, nblk);
    __shared__ int s_conv;
    // Refined form in clusters: each outer iteration is one float32
    // V-cycle of the correction per component, by that component's
    // cluster, then the float64 update of u and r by the whole grid.
    if (V.nc == 1) residual_norm<1>(A, V, sc->rnorm[slot & 3], T, true, A.r32[0]);
    else residual_norm<2>(A, V, sc->rnorm[slot & 3], T, true, A.r32[0]);
    if (bid == 0 && threadIdx.x == 0)
        for (int e = 0; e < 4; ++e) sc->rnorm[(slot + 2) & 3][e] = 0.0;
    SYNC(21);
    double rel = 0.0;
    int it = 0;
    bool conv = false;
    for (;;) {
        if (threadIdx.x == 0) {
            const double fl = 1e-13 * A.lev_inv_h2[0];
            int cv = 1, stop = 0;
            rel = 0.0;
            for (int c = 0; c < V.nc; ++c) {
                const double fn = s_fn[c];
                if (fn == 0.0) continue;
                const double rn = vload(&sc->rnorm[slot & 3][c]);
                const double un = vload(&sc->rnorm[slot & 3][2 + c]);
                double thr = fmax(A.mg_tol * A.mg_tol * fn, A.mg_atol * A.mg_atol);
                thr = fmax(thr, fl * fl * un);
                if (!(rn <= thr)) cv = 0;
                if (!(rn <= 1.7e308)) stop = 1;
                rel = fmax(rel, sqrt(rn / fn));
            }
            s_conv = stop ? 2 : cv;
        }
        __syncthreads();
        const int sv = s_conv;
        __syncthreads();
        conv = sv == 1;
        ++slot;
        if (sv || it >= A.mg_max_vcycles) break;
        cluster_inner_cycle(A, V, bid, smem_base, ci, it == 0);
        SYNC(24);
        if (V.nc == 1) update_from_e<1>(A, V, T, sc->rnorm[slot & 3]);
        else update_from_e<2>(A, V, T, sc->rnorm[slot & 3]);
        if (bid == 0 && threadIdx.x == 0)
            for (int e = 0; e < 4; ++e) sc->rnorm[(slot + 2) & 3][e] = 0.0;
        SYNC(25);
        ++it;
    }
    if (bid == 0 && threadIdx.x == 0) {
        sc->vcycles[V.kind] += it;
        if (rel > sc->max_relres) sc->max_relres = rel;
        if (!conv) sc->not_converged = 1;
    }
    if (V.u32[0] && it == 0) {  // converged at once: the float32 copy of u
        const int nn = A.N * A.N;
        for (int c = 0; c < V.nc; ++c)
            for (int k = T.t0; k < nn; k += T.nt) V.u32[c][k] = (float)V.u[c][k];
        SYNC(23);
    }
    return true;
}

// ---------------------------------------------------------------------------
// direct solves by sine transforms (qs_fft.cuh)
// ---------------------------------------------------------------------------

// Copies the transform tables to shared memory, once per launch or instance:
// as pairs of floats for the Poisson solves (and the float64 form's iterations),
// as float32 for the refined form's iterations.
template <bool REF>
__device__ void fft_load_tables(const EngineArgs &A) {
    if (!A.fft.on) return;
    using qsff::Ff;
    const int N = A.N, H = N / 2 + 1;
    qsfft::Ff2 *tw = (qsfft::Ff2 *)(qsfft::dyn_smem() + A.fft.tab_off);
    Ff *lam = (Ff *)(tw + N + H);
    float2 *tw32 = (float2 *)(lam + N);
    float *lam32 = (float *)(tw32 + N + H);
    auto conv = [](double2 v) { return qsfft::mk<Ff>(qsff::split(v.x), qsff::split(v.y)); };
    for (int k = threadIdx.x; k < N; k += blockDim.x) {
        tw[k] = conv(A.fft.tw64[k]);
        if (k < H) tw[N + k] = conv(A.fft.dct64[k]);
        lam[k] = qsff::split(A.fft.lam64[k]);
        if (REF) {
            tw32[k] = A.fft.tw32[k];
            if (k < H) tw32[N + k] = A.fft.dct32[k];
            lam32[k] = A.fft.lam32[k];
        }
    }
    __syncthreads();
}

template <typename T>
__device__ __forceinline__ qsfft::Lines fft_lines(const EngineArgs &A) {
    const int n = A.N, h = n / 2 + 1;
    const int tab = A.fft.tab_off + (sizeof(T) == 4 ? (n + h) * 16 + n * 8 : 0);
    return qsfft::Lines{n, A.fft.gmax, A.block_smem_offset, tab};
}

// The five-point sum of e times h^2, neighbours minus (4 + walls) e.  float32
// values: exact to the rounding of a float64, by error-free float32 sums and
// an FMA product, without float64 arithmetic on the five values.
__device__ __forceinline__ double five_point(float c, float w, float e, float n, float s,
                                             float k) {
    float hi = 0.f, lo = 0.f;
    qstile::two_sum_acc(hi, lo, w);
    qstile::two_sum_acc(hi, lo, e);
    qstile::two_sum_acc(hi, lo, n);
    qstile::two_sum_acc(hi, lo, s);
    const float pc = __fmul_rn(k, c);
    const float pe = __fmaf_rn(k, c, -pc);  // k c = pc + pe exactly
    qstile::two_sum_acc(hi, lo, -pc);
    lo = __fsub_rn(lo, pe);
    return qsff::join(qsff::quick(hi, lo));
}
// pairs: in float64 (the cancellation of the sum would show the pairs' last bits)
__device__ __forceinline__ double five_point(qsff::Ff c, qsff::Ff w, qsff::Ff e, qsff::Ff n,
                                             qsff::Ff s, float k) {
    using qsff::join;
    return (join(w) + join(e)) + (join(n) + join(s)) - qsff::widen(k) * join(c);
}

// float64 to and from the storage type of an iteration
template <typename T>
__device__ __forceinline__ T narrow(double v) {
    const qsff::Ff p = qsff::split(v);
    if constexpr (sizeof(T) == 4) return p.h;
    else return p;
}
__device__ __forceinline__ double value(float v) { return qsff::widen(v); }
__device__ __forceinline__ double value(qsff::Ff v) { return qsff::join(v); }
__device__ __forceinline__ float head(float v) { return v; }
__device__ __forceinline__ float head(qsff::Ff v) { return v.h; }

// Sums of 16 values over the block into out[0 .. 15] (global); clears the ring's slots two uses ahead.
template <typename O>
__device__ void reduce16(DevScalars *sc, float v[16], O *out, int slot, int bid) {
    const float t = qsfft::block_sums16(v);
    if (threadIdx.x < 16) {
        if (t != 0.f) atomicAdd(out + threadIdx.x, (O)t);
        if (bid == 0) {
            sc->cgd[(slot + 2) & 3][threadIdx.x] = 0.f;
            if (threadIdx.x < 4) sc->rnorm[(slot + 2) & 3][threadIdx.x] = 0.0;
        }
    }
}

// Scalars of an iterative solve, one copy per block.  Lane c of the first warp
// writes those of component c; block barriers stand between uses.  They stand
// on every phase's critical path, and a float64 instruction takes 64 cycles
// there: what only steers the iteration is float32 (a step size only has to be
// the same for all vectors).  With the tests in float64 on one thread an
// iteration at 64^2 took 17.2 us instead of 16.5, a slice of the refined form
// at 256^2 219 instead of 213.
struct IterScalars {
    float scale[2];           // powers of two near 1 / ||f|| (sums are of scaled values)
    double thr[2], r0[2];     // stopping bound, residual a round starts from (squared, scaled)
    float target[2], fs[2];   // ||r||^2 that ends a round; ||f||^2 (scaled)
    // of the last iteration: 1 / (r, z), 1 / alpha, step sizes, ||A p||^2 (scaled)
    float ig[2], ia[2], al[2], be[2], ss[2];
    float kbar;
    int go;
    int bad;  // the last residual is not finite
};

// `red` times the residual a round starts from, or just below the bound
__device__ __forceinline__ float round_target(double red, double r0, double thr) {
    return fmaxf((float)fmax(red * r0, 0.09 * thr), 1e-37f);
}

// Source scales and stopping bounds; go: 1 if any component needs work, 0 if
// none does, 2 if a source is beyond what the iterations' float32 exponents hold
// (||f|| above 2^100: N^2 times it passes through the transforms) or not finite.
__device__ void iter_begin(const EngineArgs &A, const SolveSpec &V, IterScalars &I, double red) {
    __syncthreads();
    if (threadIdx.x < 32) {
        const int c = threadIdx.x;
        bool work = false, beyond = false;
        if (c < 2) {
            const double fn = c < V.nc ? vload(&A.sc->fnorm[V.kind][c]) : 0.0;
            const int ex = (int)((__double_as_longlong(fn) >> 52) & 0x7ff);
            const int k = ex == 0 || ex == 0x7ff ? 0 : (ex - 1023) / 2;
            const int kc = min(max(k, -120), 120);
            beyond = ex == 0x7ff || k > 100;
            I.scale[c] = __int_as_float((127 - kc) << 23);
            const double s2 = __longlong_as_double((long long)(1023 - 2 * kc) << 52);
            const double thr = fmax(A.mg_tol * A.mg_tol * fn, A.mg_atol * A.mg_atol) * s2;
            const double r0 = fn * s2;
            I.thr[c] = thr;
            I.r0[c] = r0;
            I.target[c] = round_target(red, r0, thr);
            I.fs[c] = (float)r0;
            work = !(r0 <= thr);
        }
        const unsigned any = __ballot_sync(0xffffffffu, work);
        const unsigned out = __ballot_sync(0xffffffffu, beyond);
        if (c == 0) {
            I.kbar = V.screened ? qsff::split(vload(&A.sc->ksum)).h / (float)(A.N * A.N) : 0.f;
            I.go = out ? 2 : any != 0;
        }
    }
    __syncthreads();
}

// After u += e and the new residual's norms (rnorm[slot]): converged (1), too
// slow or out of iterations (0), or another round (-2).
__device__ int iter_check(const EngineArgs &A, const SolveSpec &V, IterScalars &I, int slot,
                          int bid, bool last, double red) {
    DevScalars *sc = A.sc;
    if (threadIdx.x < 32) {
        const int c = threadIdx.x;
        bool open = false, slow = false, bad = false;
        float rel = 0.f;
        if (c < V.nc) {
            const double fl = 1e-13 * A.lev_inv_h2[0];
            const double rn = vload(&sc->rnorm[slot & 3][c]);
            const double un = vload(&sc->rnorm[slot & 3][2 + c]);
            open = !(rn <= fmax(I.thr[c], fl * fl * un));
            slow = open && !(rn <= 0.0625 * I.r0[c]);
            bad = !(rn <= 1.7e308);
            I.r0[c] = rn;
            I.target[c] = round_target(red, rn, I.thr[c]);
            if (I.fs[c] > 0.f) rel = sqrtf((float)rn / I.fs[c]);
        }
        const unsigned nopen = __ballot_sync(0xffffffffu, open);
        const unsigned nslow = __ballot_sync(0xffffffffu, slow);
        const unsigned nbad = __ballot_sync(0xffffffffu, bad);
        rel = fmaxf(rel, __shfl_sync(0xffffffffu, rel, 1));
        if (c == 0) {
            if (bid == 0 && !nopen && (double)rel > sc->max_relres) sc->max_relres = (double)rel;
            I.go = !nopen ? 1 : (nslow || last) ? 0 : -2;
            I.bad = nbad != 0;
        }
    }
    __syncthreads();
    const int r = I.go;
    __syncthreads();  // rewritten by the next test
    return r;
}

__device__ void zero_solution(const EngineArgs &A, const SolveSpec &V, int bid, int nblk) {
    const Thr T0 = grid_thr(bid, nblk);
    for (int c = 0; c < V.nc; ++c)
        for (int i = T0.t0; i < A.N * A.N; i += T0.nt) {
            V.u[c][i] = 0.0;
            if (V.u32[c]) V.u32[c][i] = 0.f;
        }
}

// Adds |r|^2, |u|^2, |f|^2 of lap_h u = f at a cell to s[3 k ...]: r in float64.
__device__ __forceinline__ void poisson_point(const double *u, double f, int n, int ix, int iy,
                                              int i, double ih2, double (&s)[9], int k) {
    const int nw = qsmg::walls(ix, iy, n);
    const double d = nw == 0 ? 4.0 : nw == 1 ? 5.0 : 6.0, c = u[i];
    const double w = ix > 0 ? u[i - 1] : 0.0, e = ix < n - 1 ? u[i + 1] : 0.0;
    const double a = iy > 0 ? u[i - n] : 0.0, b = iy < n - 1 ? u[i + n] : 0.0;
    const double r = fma(-ih2, fma(-d, c, (w + e) + (a + b)), f);
    s[3 * k] += r * r;
    s[3 * k + 1] += c * c;
    s[3 * k + 2] += f * f;
}

// The direct solves' stopping test, after the fact, from the sums of the slice
// before (cleared here): they leave a residual of 2 to 3e-14 ||u|| / h^2 (26 sides from
// 8 to 2048; smooth, dipole, noisy and mixed sources; of ||f|| that is 1e-14 to
// 2e-9), under the bound that the V-cycles stop at.  What fails it is not finite or
// beyond float32's exponents.  One block, a barrier after the sums.
__device__ void poisson_test(const EngineArgs &A) {
    DevScalars *sc = A.sc;
    const int k = threadIdx.x;
    if (k >= 3) return;
    const double rn = vload(&sc->pchk[k][0]), un = vload(&sc->pchk[k][1]),
                 fn = vload(&sc->pchk[k][2]);
    sc->pchk[k][0] = sc->pchk[k][1] = sc->pchk[k][2] = 0.0;
    if (fn == 0.0) return;
    const double fl = 1e-13 * A.lev_inv_h2[0];
    const double thr = fmax(fmax(A.mg_tol * A.mg_tol * fn, A.mg_atol * A.mg_atol), fl * fl * un);
    if (!(rn <= thr && rn <= 1.7e308)) sc->not_converged = 1;
    if (sc->pworst[k][1] == 0.0 || rn * sc->pworst[k][1] > sc->pworst[k][0] * fn) {
        sc->pworst[k][0] = rn;
        sc->pworst[k][1] = fn;
    }
}

// lap_h u = f for one field, or two at once, in three grid phases, in pairs of
// floats.  (In float64 the phases are bound by the FP64 pipe: two fields at 256^2
// 37 us, pairs 28; at 512^2 96 and 57.)  Two fields keep lines of their own: B_z is often orders of magnitude below E_z, and as
// the imaginary part beside it its residual was 4e-10 of its source on a 64^2
// linear wake, 3e-8 on a 256^2 blowout.  load(line, x) gives rows 2p and 2p + 1 of a
// field at the line's point and store(line, x, value) takes the solution.
template <int NC, typename L>
__device__ __forceinline__ void poisson_rows(const EngineArgs &A, int bid, int nblk, L load) {
    qsfft::rows_forward<qsff::Ff, 1, NC>(fft_lines<qsff::Ff>(A), bid, nblk,
                                         (qsfft::Ff2 *)A.fft.t1, load);
}
template <int NC>
__device__ __noinline__ void poisson_columns(const EngineArgs &A, int bid, int nblk) {
    const qsfft::Ff2 *const t1 = (const qsfft::Ff2 *)A.fft.t1;
    const int N = A.N;
    qsfft::columns<qsff::Ff, 1, NC>(
        fft_lines<qsff::Ff>(A), bid, nblk, (qsfft::Ff2 *)A.fft.t2, qsff::Ff(0.f, 0.f),
        [&](int y, int l) { return t1[qsfft::column_at<NC>(y, l, N)]; });
    if (bid == 0 && threadIdx.x == 0) A.sc->vcycles[NC - 1] += 1;
}
template <int NC, typename F>
__device__ __forceinline__ void poisson_inverse(const EngineArgs &A, int bid, int nblk, F store) {
    qsfft::rows_inverse<qsff::Ff, 1, NC>(fft_lines<qsff::Ff>(A), bid, nblk,
                                         (const qsfft::Ff2 *)A.fft.t2, store);
}

template <int NC>
__device__ bool direct_poisson(const EngineArgs &A, const Sync &S, const SolveSpec &V, int bid,
                               int nblk) {
    const int N = A.N;
    // field and first row of a line
    auto field = [](int l) { return NC == 2 ? l & 1 : 0; };
    auto row = [](int l) { return NC == 2 ? l & ~1 : 2 * l; };
    poisson_rows<NC>(A, bid, nblk, [&](int l, int x) {
        const double *const f = V.f[field(l)];
        const size_t i = (size_t)row(l) * N + x;
        return qsfft::mk<qsff::Ff>(qsff::split(f[i]), qsff::split(f[i + N]));
    });
    SYNC(26);
    poisson_columns<NC>(A, bid, nblk);
    SYNC(27);
    poisson_inverse<NC>(A, bid, nblk, [&](int l, int x, qsfft::Ff2 v) {
        double *const u = V.u[field(l)];
        const size_t i = (size_t)row(l) * N + x;
        u[i] = qsff::join(v.x);
        u[i + N] = qsff::join(v.y);
    });
    SYNC(28);
    return true;
}

// (lap_h - kappa) u = f for the two components of B_perp by conjugate
// gradients preconditioned with M = lap_h - kbar, kbar the mean of kappa, whose
// inverse is a direct solve by sine transforms.  A z = M z + (kbar - kappa) z =
// r + (kbar - kappa) z, so the operator costs one product a cell.  M^-1 A is a
// compact perturbation of the identity, so the iteration converges
// superlinearly: 4 to 8 steps to 1e-10 on the 256^2 blowout (kappa 0 ... 18),
// 18 to 25 in a channel with kappa 1 ... 11, from a zero guess (the guess
// extrapolated from three slices carries their macroparticle noise: its
// residual is above the source's at the window's head).
//
// An iteration is two grid phases.  Rows: the last update of p, A p, e and r
// (with the step sizes that the previous barrier brought), z = M^-1 r from its
// row coefficients, A z, the dot products, and the row transform of A z at
// once, before the step sizes are known: the row transforms of r and A p
// follow the same recurrences, which the column phase applies to its own
// elements.  (With the update and the forward transform behind the dot
// products' barrier an iteration was three phases.)  ||r||^2 follows from the
// dot products too, so that the end of a round costs no phase.
//
// Refined form: float32 iterations on the residual equation, to 1e-5 of the
// residual they start from; then u += e, r <- r - A e in float64 and again.
// Float64 form: in pairs of floats to the tolerance (in float64 the two phases
// of an iteration took 21 and 20 us at 256^2, bound by the FP64 pipe; pairs:
// 11.7 and 10.9 us); the same step then checks it.  Both stop on the float64 residual.
// The sums are of values scaled by a power of two near 1 / ||f||, so that
// float32 cannot underflow in them.
// prepared: the source's row transform and copy are in tr and cr already.
// side(): work besides the solve, once an iteration (and side.rest() by the caller
// after it); side.idle(): this block has no line, so that it need not wait for the
// columns and has both phases of the iteration for that work.
// Returns 1 (converged), 0 (not within its cap: u holds the last iterate and
// the V-cycles take over), -1 (a barrier failed).
template <bool REF, typename X>
__device__ int cg_screened(const EngineArgs &A, const Sync &S, const SolveSpec &V, int &slot,
                           int bid, int nblk, bool prepared, X &side) {
    using T = typename std::conditional<REF, float, qsff::Ff>::type;
    using C = qsfft::V2<T>;
    DevScalars *sc = A.sc;
    const qsfft::Lines P = fft_lines<T>(A);
    const int N = A.N;
    C *const tr = (C *)A.fft.t1, *const t2 = (C *)A.fft.t2, *const tz = (C *)A.fft.tz,
             *const tp = (C *)A.fft.tp;
    C *const cz = (C *)A.fft.cz, *const cr = (C *)A.fft.cr, *const cp = (C *)A.fft.cp,
             *const cs = (C *)A.fft.cs, *const ce = (C *)A.fft.ce;
    __shared__ IterScalars I;
    const double red = REF ? 1e-10 : 1e-26;  // a round's reduction, squared
    iter_begin(A, V, I, red);
    if (I.go == 2) return 0;
    if (!I.go) {  // both sources are rounding noise or zero
        zero_solution(A, V, bid, nblk);
        return S(50) ? 1 : -1;
    }
    const T kbar(I.kbar);
    const float sc0 = I.scale[0], sc1 = I.scale[1];
    auto dk = [&](size_t i) {  // kbar - kappa
        if constexpr (REF) return kbar - A.k32[i];
        else return kbar - qsff::split(A.kap[i]);
    };
    if (!prepared) {
        qsfft::rows_forward<T, 2>(P, bid, nblk, tr, [&](int y, int x) {
            const size_t i = (size_t)y * N + x;
            const C r = qsfft::mk<T>(narrow<T>(V.f[0][i]), narrow<T>(V.f[1][i]));
            cr[i] = r;
            return r;
        });
        if (!S(51)) return -1;
    }
    const int cap = min(A.mg_max_vcycles, 48);
    int it = 0, result = -2;
    for (int round = 0; result == -2; ++round) {
        float al0 = 0.f, al1 = 0.f, be0 = 0.f, be1 = 0.f;
        int inner = 0;
        for (;;) {
            qsfft::columns<T, 2>(P, bid, nblk, t2, kbar, [&](int y, int l) {
                const size_t i = (size_t)y * N + l;
                C r = tr[i];
                if (inner > 0) {
                    C s = tz[i];
                    if (inner > 1) {
                        const C so = tp[i];
                        s.x += so.x * be0;
                        s.y += so.y * be1;
                    }
                    tp[i] = s;
                    r.x -= s.x * al0;
                    r.y -= s.y * al1;
                    tr[i] = r;
                }
                return r;
            });
            if (side.idle()) S.arrive();
            else if (!S(52)) return -1;
            float d[16] = {0.f};
            qsfft::rows_inverse_forward<T, T, 1>(P, P, bid, nblk, t2, tz, [&](int y, int x, C z) {
                const size_t i = (size_t)y * N + x;
                const T k = dk(i);
                C r = cr[i], s = qsfft::mk<T>(T(0.f), T(0.f));
                if (inner > 0) {  // the update of the last iteration
                    const C zo = cz[i];
                    C p = zo, e;
                    s = qsfft::mk<T>(r.x + k * zo.x, r.y + k * zo.y);
                    if (inner > 1) {
                        const C po = cp[i], so = cs[i];
                        e = ce[i];
                        p.x += po.x * be0;
                        p.y += po.y * be1;
                        s.x += so.x * be0;
                        s.y += so.y * be1;
                        e.x += p.x * al0;
                        e.y += p.y * al1;
                    } else {
                        e = qsfft::mk<T>(p.x * al0, p.y * al1);
                    }
                    r.x -= s.x * al0;
                    r.y -= s.y * al1;
                    cp[i] = p;
                    cs[i] = s;
                    ce[i] = e;
                    cr[i] = r;
                }
                cz[i] = z;
                const C w = qsfft::mk<T>(r.x + k * z.x, r.y + k * z.y);
                const float rx = head(r.x) * sc0, ry = head(r.y) * sc1, zx = head(z.x) * sc0,
                            zy = head(z.y) * sc1, wx = head(w.x) * sc0, wy = head(w.y) * sc1,
                            sx = head(s.x) * sc0, sy = head(s.y) * sc1;
                d[0] += rx * zx;
                d[1] += ry * zy;
                d[2] += zx * wx;
                d[3] += zy * wy;
                d[4] += rx * wx;
                d[5] += ry * wy;
                d[6] += rx * sx;
                d[7] += ry * sy;
                d[8] += wx * wx;
                d[9] += wy * wy;
                d[10] += wx * sx;
                d[11] += wy * sy;
                d[12] += rx * rx;
                d[13] += ry * ry;
                return w;
            });
            reduce16(sc, d, sc->cgd[slot & 3], slot, bid);
            side();
            if (!S(53)) return -1;
            if (threadIdx.x < 32) {  // one lane a component
                const int c = threadIdx.x;
                bool open = false;
                if (c < 2) {
                    const float *g = sc->cgd[slot & 3];
                    const float ga = vload(g + c), de = vload(g + 2 + c);
                    const float rw = vload(g + 4 + c), rs = vload(g + 6 + c),
                                ww = vload(g + 8 + c), ws = vload(g + 10 + c),
                                rr = vload(g + 12 + c);
                    float be = 0.f, al = 0.f, ia = 0.f, ig = 0.f;
                    // a component that is solved to float32's smallest numbers
                    // stands still (1 / ga would be infinite)
                    if (fabsf(ga) >= 1e-36f) {
                        ig = 1.f / ga;
                        be = inner > 0 ? ga * I.ig[c] : 0.f;
                        ia = de * ig - be * (inner > 0 ? I.ia[c] : 0.f);
                        al = fabsf(ia) >= 1e-30f ? 1.f / ia : 0.f;
                    }
                    I.ig[c] = ig;
                    I.ia[c] = ia;
                    I.al[c] = al;
                    I.be[c] = be;
                    // ||r - al s||^2 with s = w + be s_old.  The sums are good to
                    // about 1e-7 of ||r||^2: no smaller value is believed.
                    const float so = inner > 0 ? I.ss[c] : 0.f;
                    const float ss = ww + be * (2.f * ws + be * so);
                    I.ss[c] = ss;
                    const float nr = rr - al * (2.f * (rw + be * rs) - al * ss);
                    // a NaN ends the round: its float64 residual decides
                    open = (nr < 2e-7f * rr ? 2e-7f * rr : nr) > I.target[c];
                }
                const unsigned nopen = __ballot_sync(0xffffffffu, open);
                if (c == 0) I.go = nopen != 0;
            }
            ++slot;
            __syncthreads();
            al0 = I.al[0];
            al1 = I.al[1];
            be0 = I.be[0];
            be1 = I.be[1];
            const bool go = I.go != 0;  // rewritten two grid barriers on
            ++it;
            ++inner;
            if (!go || it >= cap || inner >= 24) break;
        }
        // u += e, r <- r - A e in float64 with the norms of the stopping test;
        // the new right-hand side goes through its row transform on the way.
        // e is e + al p with the last step, at the cell and its neighbours.
        auto e_at = [&](size_t i) {
            C p = cz[i];
            if (inner == 1) return qsfft::mk<T>(p.x * al0, p.y * al1);
            const C po = cp[i], eo = ce[i];
            p.x += po.x * be0;
            p.y += po.y * be1;
            return qsfft::mk<T>(eo.x + p.x * al0, eo.y + p.y * al1);
        };
        float n[16] = {0.f};
        const double ih2 = A.lev_inv_h2[0];
        qsfft::rows_forward<T, 2>(P, bid, nblk, tr, [&](int y, int x) {
            const size_t i = (size_t)y * N + x;
            const C zero = qsfft::mk<T>(T(0.f), T(0.f));
            const C e = e_at(i);
            const C ew = x > 0 ? e_at(i - 1) : zero, ee = x < N - 1 ? e_at(i + 1) : zero;
            const C en = y > 0 ? e_at(i - N) : zero, es = y < N - 1 ? e_at(i + N) : zero;
            const float cw = (float)(4 + qsmg::walls(x, y, N));
            const double kap = A.kap[i];
            double u0 = value(e.x), u1 = value(e.y), q0, q1;
            const double a0 = five_point(e.x, ew.x, ee.x, en.x, es.x, cw) * ih2 - kap * u0;
            const double a1 = five_point(e.y, ew.y, ee.y, en.y, es.y, cw) * ih2 - kap * u1;
            if (round == 0) {
                q0 = V.f[0][i];
                q1 = V.f[1][i];
            } else {
                u0 += V.u[0][i];
                u1 += V.u[1][i];
                q0 = A.r64[0][i];
                q1 = A.r64[1][i];
            }
            const double r0 = q0 - a0, r1 = q1 - a1;
            V.u[0][i] = u0;
            V.u[1][i] = u1;
            const float h0 = narrow<float>(u0), h1 = narrow<float>(u1);
            if (V.u32[0]) {
                V.u32[0][i] = h0;
                V.u32[1][i] = h1;
            }
            A.r64[0][i] = r0;
            A.r64[1][i] = r1;
            const C r = qsfft::mk<T>(narrow<T>(r0), narrow<T>(r1));
            cr[i] = r;
            const float v0 = h0 * sc0, v1 = h1 * sc1, n0 = head(r.x) * sc0, n1 = head(r.y) * sc1;
            n[0] += n0 * n0;
            n[1] += n1 * n1;
            n[2] += v0 * v0;
            n[3] += v1 * v1;
            return r;
        });
        reduce16(sc, n, A.sc->rnorm[slot & 3], slot, bid);
        if (!S(55)) return -1;
        result = iter_check(A, V, I, slot, bid, it >= cap, red);
        ++slot;
    }
    if (bid == 0 && threadIdx.x == 0) sc->vcycles[V.kind] += it;
    // nothing for the cycles to go on from
    if (result == 0 && I.bad) zero_solution(A, V, bid, nblk);
    return result;
}

// The sums of poisson_test for a solve of mg_solve's.
template <int NC>
__device__ void poisson_sums(const EngineArgs &A, const SolveSpec &V, Thr T) {
    const double ih2 = A.lev_inv_h2[0];
    double s[9] = {0.0};
    for (qsmg::Walk w(T.t0, T.nt, A.N); w.q < A.N * A.N; w.next())
#pragma unroll
        for (int c = 0; c < NC; ++c)
            poisson_point(V.u[c], V.f[c][w.q], A.N, w.col, w.row, w.q, ih2, s, c);
    if constexpr (NC == 1) {
        const double t[3] = {s[0], s[1], s[2]};
        block_sum_wide(t, A.sc->pchk[0]);
    } else {
        const double t[6] = {s[0], s[1], s[2], s[3], s[4], s[5]};
        block_sum_wide(t, A.sc->pchk[1]);
    }
}

// The screened smoother's inverse diagonal, needed only when the V-cycles
// take over from the conjugate gradients.
__device__ void screened_diagonal(const EngineArgs &A, Thr T) {
    const int n = A.N;
    for (qsmg::Walk w(T.t0, T.nt, n); w.q < n * n; w.next()) {
        const int nw = qsmg::walls(w.col, w.row, n);
        if (A.precision == QS_FP32_REFINED)
            A.d32[w.q] = 1.f / ((float)(4 + nw) + A.lev_h2f[0] * A.k32[w.q]);
        else
            A.invd0[w.q] = 1.0 / ((double)(4 + nw) + A.lev_h2[0] * A.kap[w.q]);
    }
}

struct Nothing {
    __device__ bool idle() const { return false; }
    __device__ void operator()() const {}
    __device__ void rest() const {}
};

// Iterate until, for every component,
//   ||f - A u|| <= max(tol ||f||, 1e-13 ||u|| / h^2, atol)
// (the second bound is a small multiple of the rounding level of the
// float64 residual; atol stops solves whose source is rounding noise).
// Float64 form: V-cycles on u.  Refined form: float64 residual, float32
// V-cycle on the correction, float64 update (iterative refinement).
template <bool REF>
__device__ __noinline__ bool mg_cycles(const EngineArgs &A, const Sync &S, const SolveSpec &V, int &slot,
                          int bid, int nblk, void *smem_base, int *inv_ready) {
    DevScalars *sc = A.sc;
    // shared memory: [coarsest inverses][coarse levels + work][staged tile]
    void *smem = (char *)smem_base + A.block_smem_offset;
    const int mc = A.lev_n[A.nlev - 1] * A.lev_n[A.nlev - 1];
    const qsmg::CoarseInv ci{(double *)smem_base + (V.screened ? mc * mc : 0),
                             inv_ready + (V.screened ? 1 : 0)};
    if (V.screened) {  // kappa changed: the screened inverse must be rebuilt
        __syncthreads();
        if (threadIdx.x == 0) inv_ready[1] = 0;
        __syncthreads();
    }
    // The scalar bookkeeping of the solve (source norms, the convergence
    // test) is done by thread 0 alone and broadcast through shared memory:
    // float64 divides and square roots repeated by every thread would cost
    // microseconds on GB300's float64 pipe.
    __shared__ double s_fn[2];
    __shared__ int s_zero_mask, s_conv;
    __syncthreads();
    if (threadIdx.x == 0) {
        int mask = 0;
        for (int c = 0; c < V.nc; ++c) {
            s_fn[c] = vload(&sc->fnorm[V.kind][c]);
            if (s_fn[c] == 0.0) mask |= 1 << c;
        }
        s_zero_mask = mask;
    }
    __syncthreads();
    const int zero_mask = s_zero_mask;
    const Thr T = grid_thr(bid, nblk);
    if (zero_mask) {
        const int nn = A.N * A.N;
        for (int c = 0; c < V.nc; ++c)
            if (zero_mask & (1 << c))
                for (int k = T.t0; k < nn; k += T.nt) {
                    V.u[c][k] = 0.0;
                    if (V.u32[c]) V.u32[c][k] = 0.f;
                }
        SYNC(20);
    }
    if (zero_mask == (1 << V.nc) - 1) return true;
#ifndef QS_NO_CLUSTER_SOLVES
    if (!REF && A.cl_size > 1) {  // one cluster per component solves alone
        mg_solve_cluster64(A, V, bid, smem_base, ci, s_fn);
        SYNC(22);
        if (bid == 0 && threadIdx.x == 0) {
            A.sc->vcycles[V.kind] += A.sc->cl_cycles;
            A.sc->cl_cycles = 0;
        }
        return true;
    }
#endif
#ifndef QS_NO_CLUSTER_SOLVES
    if (REF && A.cl_size > 1)
        return mg_solve_ref_cluster(A, S, V, slot, bid, nblk, smem_base, ci, s_fn);
#endif
    // one of the two, by the form
    __shared__ __align__(16) unsigned char
        hier_mem[sizeof(Hier<double>) > sizeof(Hier<float>) ? sizeof(Hier<double>)
                                                            : sizeof(Hier<float>)];
    Hier<double> &H64 = *(Hier<double> *)hier_mem;
    Hier<float> &H32 = *(Hier<float> *)hier_mem;
    __syncthreads();
    if (REF) hier32(A, V, H32);
    else hier64(A, V, H64);
    __syncthreads();
    bool conv = false;
    double rel = 0.0;  // thread 0 only
    int it = 0;
    bool norms_ready = false;  // the last cycle already produced this slot's norms
    // The fused residual update writes the next float32 right-hand side into
    // the other buffer of a pair: the current one is still read as halo by
    // other blocks while it is written.
    int rbuf = 0;
    bool u32_fresh = false;  // the last cycle wrote the float32 copy of u
    for (;;) {
        if (REF || it > 0) {
            if (!norms_ready) {
                if (V.nc == 1) residual_norm<1>(A, V, sc->rnorm[slot & 3], T, REF, H32.lv[0].f);
                else residual_norm<2>(A, V, sc->rnorm[slot & 3], T, REF, H32.lv[0].f);
                if (bid == 0 && threadIdx.x == 0)
                    for (int e = 0; e < 4; ++e) sc->rnorm[(slot + 2) & 3][e] = 0.0;
                SYNC(21);
            }
            if (threadIdx.x == 0) {
                const double fl = 1e-13 * A.lev_inv_h2[0];
                // a residual that is not finite is not below any bound, and
                // further cycles don't mend it
                int cv = 1, stop = 0;
                rel = 0.0;
                for (int c = 0; c < V.nc; ++c) {
                    const double fn = s_fn[c];
                    if (fn == 0.0) continue;
                    const double rn = vload(&sc->rnorm[slot & 3][c]);
                    const double un = vload(&sc->rnorm[slot & 3][2 + c]);
                    double thr = fmax(A.mg_tol * A.mg_tol * fn, A.mg_atol * A.mg_atol);
                    thr = fmax(thr, fl * fl * un);
                    if (!(rn <= thr)) cv = 0;
                    if (!(rn <= 1.7e308)) stop = 1;
                    rel = fmax(rel, sqrt(rn / fn));
                }
                s_conv = stop ? 2 : cv;
            }
            __syncthreads();
            const int sv = s_conv;
            __syncthreads();  // s_conv is rewritten by the next test
            conv = sv == 1;
            ++slot;
            if (sv || it >= A.mg_max_vcycles) break;
        }
        bool ok;
        norms_ready = false;
        if (REF) {
            const qstile::Fused fz{{V.u[0], V.u[V.nc - 1]},
                                   {A.r64[0], A.r64[V.nc - 1]},
                                   {A.r32[1 - rbuf][0], A.r32[1 - rbuf][V.nc - 1]},
                                   {V.u32[0], V.u32[V.nc - 1]},
                                   V.screened ? A.kap : nullptr,
                                   A.lev_inv_h2[0]};
            double *nout = sc->rnorm[slot & 3], *nclr = sc->rnorm[(slot + 2) & 3];
            if (V.nc == 1)
                ok = A.tile_x > 0
                         ? vcycle_staged<1>(A, S, H32, bid, nblk, smem, ci, V.u[0], V.u[0], &fz,
                                            nout, nclr, &norms_ready)
                         : vcycle<float, 1>(A, S, H32, bid, nblk, smem, ci, V.u[0], V.u[0]);
            else
                ok = A.tile_x > 0
                         ? vcycle_staged<2>(A, S, H32, bid, nblk, smem, ci, V.u[0], V.u[1], &fz,
                                            nout, nclr, &norms_ready)
                         : vcycle<float, 2>(A, S, H32, bid, nblk, smem, ci, V.u[0], V.u[1]);
        } else if (A.tile_x > 0 && H64.lv[0].n > A.block_level_n) {
            double *nout = sc->rnorm[slot & 3], *nclr = sc->rnorm[(slot + 2) & 3];
            ok = V.nc == 1 ? vcycle_staged64<1>(A, S, H64, bid, nblk, smem, ci, nout, nclr)
                           : vcycle_staged64<2>(A, S, H64, bid, nblk, smem, ci, nout, nclr);
            norms_ready = true;  // the level-0 up leg summed the stopping test's norms
        } else {
            ok = V.nc == 1 ? vcycle<double, 1>(A, S, H64, bid, nblk, smem, ci, nullptr, nullptr)
                           : vcycle<double, 2>(A, S, H64, bid, nblk, smem, ci, nullptr, nullptr);
        }
        if (!ok) return false;
        u32_fresh = REF && norms_ready;
        if (REF && norms_ready) {  // all blocks are past the cycle's last barrier
            rbuf ^= 1;
            if (threadIdx.x == 0)
                for (int c = 0; c < 2; ++c) H32.lv[0].f[c] = A.r32[rbuf][c];
            __syncthreads();
        }
        ++it;
    }
    if (bid == 0 && threadIdx.x == 0) {
        sc->vcycles[V.kind] += it;
        if (rel > sc->max_relres) sc->max_relres = rel;
        if (!conv) sc->not_converged = 1;
    }
    if (V.u32[0] && !u32_fresh) {  // no cycle, or a cycle without the fused update
        const int nn = A.N * A.N;
        for (int c = 0; c < V.nc; ++c)
            for (int k = T.t0; k < nn; k += T.nt) V.u32[c][k] = (float)V.u[c][k];
        SYNC(23);
    }
    return true;
}

// A field solve: by transforms and iterations, else by V-cycles.
template <bool REF, typename X = const Nothing>
__device__ bool mg_solve(const EngineArgs &A, const Sync &S, const SolveSpec &V, int &slot,
                         int bid, int nblk, void *smem_base, int *inv_ready,
                         bool prepared = false, X &side = Nothing()) {
    if (A.fft.on) {
        if (!V.screened)
            return V.nc == 1 ? direct_poisson<1>(A, S, V, bid, nblk)
                             : direct_poisson<2>(A, S, V, bid, nblk);
        const int r = cg_screened<REF>(A, S, V, slot, bid, nblk, prepared, side);
        if (r < 0) return false;
        side.rest();  // before the cycles take the shared memory
        if (r > 0) return true;
        screened_diagonal(A, grid_thr(bid, nblk));
        // The cycles move `slot` on without clearing the dot products' ring: the
        // next slice's iterations would add to what these left in it.
        if (bid == 0 && threadIdx.x < 64)
            A.sc->cgd[threadIdx.x >> 4][threadIdx.x & 15] = 0.f;
        SYNC(56);
    }
    return mg_cycles<REF>(A, S, V, slot, bid, nblk, smem_base, inv_ready);
}

__device__ __forceinline__ double guard(double a, double floor_, unsigned &hits) {
    if (a < floor_) {
        ++hits;
        return floor_;
    }
    return a;
}

__device__ void add_hits(DevScalars *sc, unsigned hits) {
    double t = block_sum((double)hits);
    if (threadIdx.x == 0 && t > 0.0) atomicAdd(&sc->guard_hits, (unsigned long long)t);
}

}  // namespace
