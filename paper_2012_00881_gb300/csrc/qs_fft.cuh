// Sine transforms of grid lines by the threads of one block, and the three
// phases of a direct solve of (lap_h - kbar) u = f on the cell-centred grid.
//
// With odd ghosts the 5-point Laplacian is diagonal in sin(pi (k+1) (i+1/2) / N)
// along each axis.  Writing k = N - 1 - j turns that transform into the cosine
// transform of (-1)^i f_i, whose N-point complex FFT (the even samples
// ascending, then the odd ones descending) is rotated by w_j = e^{-i pi j / 2N}
// (Makhoul's algorithm, IEEE Trans. ASSP 28 (1980) 27).  The transform is
// linear over the complex numbers, so two real fields, or two rows of one
// field, go through one complex line:
//   A = w_j V_j,  B = conj(w_j) V_{N-j}:  2 C_j = A + B,  2 C_{N-j} = i (A - B),
// and back
//   V_j = conj(w_j) (C_j - i C_{N-j}),    V_{N-j} = w_j (C_j + i C_{N-j}).
// The FFT is a Stockham radix-4 / radix-2 chain in shared memory with one odd
// radix (3, 5 or 7) last, which covers every grid side the library takes.
//
// A direct solve is three grid phases: rows forward, columns forward - divide -
// inverse, rows inverse, each a read and a write of the grid through L2.  What
// bounds them: in float64 the FP64 pipe (two FMA a clock and SM; about 8,500
// instructions a 256-point complex line), in float32 the two L2 round trips and
// the grid barrier of each phase.
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

namespace qsfft {

template <typename T>
using V2 = typename std::conditional<sizeof(T) == 8, double2, float2>::type;

template <typename T>
__device__ __forceinline__ V2<T> mk(T x, T y) {
    V2<T> v;
    v.x = x;
    v.y = y;
    return v;
}
template <typename V>
__device__ __forceinline__ V cadd(V a, V b) {
    a.x += b.x;
    a.y += b.y;
    return a;
}
template <typename V>
__device__ __forceinline__ V csub(V a, V b) {
    a.x -= b.x;
    a.y -= b.y;
    return a;
}
// a w, or a conj(w) with CONJ
template <bool CONJ, typename V>
__device__ __forceinline__ V cmul(V a, V w) {
    V r;
    if (CONJ) {
        r.x = a.x * w.x + a.y * w.y;
        r.y = a.y * w.x - a.x * w.y;
    } else {
        r.x = a.x * w.x - a.y * w.y;
        r.y = a.y * w.x + a.x * w.y;
    }
    return r;
}

// Tables and line buffers of a block.  tw[k] = e^{-2 pi i k / N}, k < N;
// dct[j] = e^{-i pi j / 2N}, j <= N/2; lam[j] = -(2 + 2 cos(pi j / N)) / h^2,
// the eigenvalue of cosine index j.  a, b: G lines of N complex values each.
template <typename T>
struct Lines {
    int N, gmax;
    const V2<T> *tw, *dct;
    const T *lam;
    V2<T> *a, *b;
};

// index t over lines of n items: (line, item); few lines per block, so a
// subtraction loop is cheaper than a division
struct Split {
    int g, j, n;
    __device__ Split(int n_) : g(0), j((int)threadIdx.x), n(n_) { wrap(); }
    __device__ void wrap() {
        while (j >= n) {
            j -= n;
            ++g;
        }
    }
    __device__ void next() {
        j += (int)blockDim.x;
        wrap();
    }
};

// One Stockham pass of radix R over gl lines: the sub-transforms done so far
// have length Ns (a power of two).
template <typename T, int R, bool INV>
__device__ __forceinline__ void pass(const Lines<T> &P, const V2<T> *src, V2<T> *dst, int Ns,
                                     int gl) {
    using V = V2<T>;
    const int nb = P.N / R, step = nb / Ns;
    for (Split s(nb); s.g < gl; s.next()) {
        const int j = s.j, k = j & (Ns - 1);
        const V *x = src + s.g * P.N;
        V *y = dst + s.g * P.N + (j - k) * R + k;
        V v[R];
        v[0] = x[j];
#pragma unroll
        for (int r = 1; r < R; ++r) {
            v[r] = x[j + r * nb];
            if (Ns > 1) v[r] = cmul<INV>(v[r], P.tw[k * r * step]);
        }
        if constexpr (R == 2) {
            y[0] = cadd(v[0], v[1]);
            y[Ns] = csub(v[0], v[1]);
        } else if constexpr (R == 4) {
            const V s02 = cadd(v[0], v[2]), d02 = csub(v[0], v[2]);
            const V s13 = cadd(v[1], v[3]), d13 = csub(v[1], v[3]);
            // -i d13 forward, +i d13 inverse
            const V q = INV ? mk<T>(-d13.y, d13.x) : mk<T>(d13.y, -d13.x);
            y[0] = cadd(s02, s13);
            y[Ns] = cadd(d02, q);
            y[2 * Ns] = csub(s02, s13);
            y[3 * Ns] = csub(d02, q);
        } else {
#pragma unroll
            for (int o = 0; o < R; ++o) {
                V t = v[0];
#pragma unroll
                for (int r = 1; r < R; ++r) t = cadd(t, cmul<INV>(v[r], P.tw[((o * r) % R) * nb]));
                y[o * Ns] = t;
            }
        }
    }
}

// The transform of the gl lines in P.a; returns the buffer that holds the
// result (the other one is free).  Every thread of the block; the caller has
// synchronised the block after filling P.a.
template <typename T, bool INV>
__device__ V2<T> *fft(const Lines<T> &P, int gl) {
    V2<T> *src = P.a, *dst = P.b;
    int Ns = 1, n = P.N;
    // float64: a pass on fewer than 128 radix-4 butterflies would leave some of
    // the SM's four FP64 units idle; radix 2 has twice as many, each less than
    // half the work (256 points, one line: 4.1k against 7.2k pipe cycles)
    const bool r4 = sizeof(T) == 4 || gl * P.N >= 512;
    auto done = [&](int R) {
        V2<T> *t = src;
        src = dst;
        dst = t;
        Ns *= R;
        n /= R;
        __syncthreads();
    };
    while (r4 && (n & 3) == 0) {
        pass<T, 4, INV>(P, src, dst, Ns, gl);
        done(4);
    }
    while ((n & 1) == 0) {
        pass<T, 2, INV>(P, src, dst, Ns, gl);
        done(2);
    }
    if (n == 3) {
        pass<T, 3, INV>(P, src, dst, Ns, gl);
        done(3);
    } else if (n == 5) {
        pass<T, 5, INV>(P, src, dst, Ns, gl);
        done(5);
    } else if (n == 7) {
        pass<T, 7, INV>(P, src, dst, Ns, gl);
        done(7);
    }
    return src;
}

// Lines a block takes at a time: as few as spread nl lines over nblk blocks in
// one round (a power of two), at most gmax.
__device__ __forceinline__ int lines_at_once(int nl, int nblk, int gmax) {
    int g = 1;
    while (g < gmax && g * nblk < nl) g <<= 1;
    return g;
}

// Where sample i of a line sits in the FFT input; odd samples change sign.
__device__ __forceinline__ int slot_of(int i, int N) { return (i & 1) ? N - 1 - (i >> 1) : i >> 1; }

// Rows forward.  Two components (NC = 2): line y is the complex row of both.
// One component: line p is rows 2p (real part) and 2p + 1.  load(line, x) gives
// the samples; the coefficients (times 2) go to `out`, complex [y][j] or real
// [y][j].
template <typename T, int NC, typename F>
__device__ void rows_forward(const Lines<T> &P, int bid, int nblk, V2<T> *out, F load) {
    using V = V2<T>;
    const int N = P.N, nl = NC == 2 ? N : N / 2;
    const int G = lines_at_once(nl, nblk, P.gmax);
    for (int l0 = bid * G; l0 < nl; l0 += nblk * G) {
        const int gl = min(G, nl - l0);
        for (Split s(N); s.g < gl; s.next()) {
            V v = load(l0 + s.g, s.j);
            if (s.j & 1) v = mk<T>(-v.x, -v.y);
            P.a[s.g * N + slot_of(s.j, N)] = v;
        }
        __syncthreads();
        const V *r = fft<T, false>(P, gl);
        for (Split s(N / 2 + 1); s.g < gl; s.next()) {
            const int j = s.j;
            const V *x = r + s.g * N;
            V c, d;
            if (j == 0) {
                c = cadd(x[0], x[0]);
                d = c;
            } else {
                const V w = P.dct[j];
                const V A = cmul<false>(x[j], w), B = cmul<true>(x[N - j], w);
                const V m = csub(A, B);
                c = cadd(A, B);
                d = mk<T>(-m.y, m.x);
            }
            const bool two = j > 0 && 2 * j < N;
            if constexpr (NC == 2) {
                V *o = out + (size_t)(l0 + s.g) * N;
                o[j] = c;
                if (two) o[N - j] = d;
            } else {
                T *o = (T *)out + (size_t)(2 * (l0 + s.g)) * N;
                o[j] = c.x;
                o[N + j] = c.y;
                if (two) {
                    o[N - j] = d.x;
                    o[2 * N - j] = d.y;
                }
            }
        }
        __syncthreads();
    }
}

// 1 / d for d != 0: float32 directly, float64 by two Newton steps from the
// float32 reciprocal (a float64 divide is a long sequence on the FP64 pipe)
__device__ __forceinline__ float recip(float d) { return 1.f / d; }
__device__ __forceinline__ double recip(double d) {
    double r = (double)(1.f / (float)d);
    r = r * fma(-d, r, 2.0);
    r = r * fma(-d, r, 2.0);
    return r;
}

// Columns: forward, times 1 / (4 N^2 (lam_x + lam_y - kbar)), inverse.  The
// one-component array seen as complex pairs puts columns 2p and 2p + 1 into
// line p.  in and out may not overlap.
template <typename T, int NC>
__device__ void columns(const Lines<T> &P, int bid, int nblk, const V2<T> *in, V2<T> *out,
                        T kbar) {
    using V = V2<T>;
    const int N = P.N, nl = NC == 2 ? N : N / 2;
    const int G = lines_at_once(nl, nblk, P.gmax);
    const int sh = 31 - __clz(G);
    const T c4 = T(0.25) / ((T)N * (T)N);
    for (int l0 = bid * G; l0 < nl; l0 += nblk * G) {
        const int gl = min(G, nl - l0);
        for (int t = threadIdx.x; t < (N << sh); t += blockDim.x) {
            const int y = t >> sh, g = t & (G - 1);
            if (g >= gl) continue;
            V v = in[(size_t)y * nl + l0 + g];
            if (y & 1) v = mk<T>(-v.x, -v.y);
            P.a[g * N + slot_of(y, N)] = v;
        }
        __syncthreads();
        Lines<T> Q = P;
        Q.a = fft<T, false>(P, gl);
        Q.b = Q.a == P.a ? P.b : P.a;
        for (Split s(N / 2 + 1); s.g < gl; s.next()) {
            const int j = s.j, l = l0 + s.g;
            const T lx0 = P.lam[NC == 2 ? l : 2 * l] - kbar;
            const T lx1 = NC == 2 ? lx0 : P.lam[2 * l + 1] - kbar;
            auto scaled = [&](V c, int jj) {
                const T ly = P.lam[jj];
                const T s0 = c4 * recip(lx0 + ly);
                const T s1 = NC == 2 ? s0 : c4 * recip(lx1 + ly);
                return mk<T>(c.x * s0, c.y * s1);
            };
            V *x = Q.a + s.g * N;
            if (j == 0) {
                x[0] = scaled(cadd(x[0], x[0]), 0);
                continue;
            }
            const V w = P.dct[j];
            const V A = cmul<false>(x[j], w), B = cmul<true>(x[N - j], w);
            const V c = scaled(cadd(A, B), j), m = csub(A, B);
            // -i C_{N-j} with C_{N-j} = i m scaled: the parts swap twice
            V d = scaled(mk<T>(-m.y, m.x), N - j);
            d = mk<T>(d.y, -d.x);
            x[j] = cmul<true>(cadd(c, d), w);
            if (2 * j < N) x[N - j] = cmul<false>(csub(c, d), w);
        }
        __syncthreads();
        const V *r = fft<T, true>(Q, gl);
        for (int t = threadIdx.x; t < (N << sh); t += blockDim.x) {
            const int y = t >> sh, g = t & (G - 1);
            if (g >= gl) continue;
            V v = r[g * N + slot_of(y, N)];
            if (y & 1) v = mk<T>(-v.x, -v.y);
            out[(size_t)y * nl + l0 + g] = v;
        }
        __syncthreads();
    }
}

// Rows inverse: store(line, x, value) takes the solution's samples.
template <typename T, int NC, typename F>
__device__ void rows_inverse(const Lines<T> &P, int bid, int nblk, const V2<T> *in, F store) {
    using V = V2<T>;
    const int N = P.N, nl = NC == 2 ? N : N / 2;
    const int G = lines_at_once(nl, nblk, P.gmax);
    for (int l0 = bid * G; l0 < nl; l0 += nblk * G) {
        const int gl = min(G, nl - l0);
        for (Split s(N / 2 + 1); s.g < gl; s.next()) {
            const int j = s.j, l = l0 + s.g;
            auto coef = [&](int jj) {
                if constexpr (NC == 2) {
                    return in[(size_t)l * N + jj];
                } else {
                    const T *o = (const T *)in + (size_t)(2 * l) * N;
                    return mk<T>(o[jj], o[N + jj]);
                }
            };
            V *x = P.a + s.g * N;
            const V c = coef(j);
            if (j == 0) {
                x[0] = c;
                continue;
            }
            const V w = P.dct[j], e = coef(N - j);
            const V d = mk<T>(e.y, -e.x);  // -i C_{N-j}
            x[j] = cmul<true>(cadd(c, d), w);
            if (2 * j < N) x[N - j] = cmul<false>(csub(c, d), w);
        }
        __syncthreads();
        const V *r = fft<T, true>(P, gl);
        for (Split s(N); s.g < gl; s.next()) {
            V v = r[s.g * N + slot_of(s.j, N)];
            if (s.j & 1) v = mk<T>(-v.x, -v.y);
            store(l0 + s.g, s.j, v);
        }
        __syncthreads();
    }
}

}  // namespace qsfft
