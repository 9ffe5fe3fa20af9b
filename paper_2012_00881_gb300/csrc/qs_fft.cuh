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
// bounds them, in float32 and in pairs of floats: instruction fetches, the two
// L2 round trips and the grid barrier of each phase (256^2, two fields: 8 to 10 us
// a phase; in float64, bound by its pipe, 12).
#pragma once

#include <cuda_runtime.h>

#include <cmath>
#include <type_traits>
#include <vector>

#include "qs_ff.cuh"

namespace qsfft {

using qsff::Ff;

// complex numbers of a storage type
struct __align__(16) Ff2 {
    Ff x, y;
};
template <typename T>
struct Cplx {
    using type = float2;
};
template <>
struct Cplx<Ff> {
    using type = Ff2;
};
template <typename T>
using V2 = typename Cplx<T>::type;

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

// The block's dynamic shared memory (every kernel's extern array is this one):
// buffers and tables are passed as byte offsets into it, so that all accesses
// compile to shared-memory instructions across calls.
__device__ __forceinline__ char *dyn_smem() {
    extern __shared__ __align__(16) double smem[];
    return (char *)smem;
}
template <typename T>
__device__ __forceinline__ V2<T> *cplx_at(int off) {
    return (V2<T> *)(dyn_smem() + off);
}

// e^{-2 pi i num / den}, 0 <= num < den, on the host: the angle reduced to
// [0, pi / 4], so that the tables are exact to rounding and symmetric.
inline double2 host_unit(long long num, long long den) {
    const int oct = (int)(num * 8 / den);
    const long long a = oct & 1 ? (oct + 1) * den - 8 * num : 8 * num - oct * den;
    const double t = 3.14159265358979323846 * (double)a / (4.0 * (double)den);
    const double c = std::cos(t), s = std::sin(t);
    const double re[8] = {c, s, -s, -c, -c, -s, s, c}, im[8] = {s, c, c, s, -s, -c, -c, -s};
    return double2{re[oct], -im[oct]};
}
// eigenvalue of cosine index j: -(2 + 2 cos(pi j / n)) / h^2
inline double host_lam(int j, int n, double h) {
    const double c = std::cos(0.5 * 3.14159265358979323846 * j / n);
    return -4.0 * c * c / (h * h);
}
// [tw][dct][lam] of a side, as pairs (two a complex number)
inline std::vector<Ff> host_tables(int n, double h) {
    std::vector<Ff> t;
    auto put = [&](double2 v) {
        t.push_back(Ff(v.x));
        t.push_back(Ff(v.y));
    };
    for (int k = 0; k < n; ++k) put(host_unit(k, n));
    for (int k = 0; 2 * k <= n; ++k) put(host_unit(k, 4LL * n));
    for (int k = 0; k < n; ++k) t.push_back(Ff(host_lam(k, n, h)));
    return t;
}

// Line buffers and tables of a block, all in shared memory: a, b hold gmax
// lines of N complex values each; at tab: tw[k] = e^{-2 pi i k / N}, k < N;
// dct[j] = e^{-i pi j / 2N}, j <= N/2; lam[j] = -(2 + 2 cos(pi j / N)) / h^2, the
// eigenvalue of cosine index j.
struct Lines {
    int N, gmax, a, tab;
};
template <typename T>
__device__ __forceinline__ const V2<T> *dct_table(int tab, int N) {
    return cplx_at<T>(tab) + N;
}
template <typename T>
__device__ __forceinline__ const T *lam_table(int tab, int N) {
    return (const T *)(cplx_at<T>(tab) + N + N / 2 + 1);
}

// Where point i of a line sits in its buffer: one free element after every 128
// bytes, so that the strided writes of a radix-8 pass fall into different
// banks (512 points, four lines: 1,150 -> 350 cycles a pass).
template <typename T>
__host__ __device__ __forceinline__ constexpr int pad(int i) {
    return i + (i >> (sizeof(T) == 8 ? 3 : 4));
}
// elements of a padded line of N points
template <typename T>
__host__ __device__ __forceinline__ constexpr int line_len(int N) {
    return pad<T>(N - 1) + 1;
}

template <typename T>
__device__ __forceinline__ int buf_b(const Lines &P) {
    return P.a + P.gmax * line_len<T>(P.N) * (int)sizeof(V2<T>);
}
// A thread's items of a line-wise loop: the block's warps are dealt to G (a power
// of two) lines in turn, so that a loop with few items still uses all four
// schedulers (and FP64 units) of the SM; an index computed by division or by a
// loop costs 250 cycles a pass, this one a few.
struct Deal {
    int g, j0, stride;
    __device__ __forceinline__ explicit Deal(int lgG) {
        const int w = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
        g = w & ((1 << lgG) - 1);
        j0 = ((w >> lgG) << 5) + lane;
        stride = (int)blockDim.x >> lgG;
    }
};

// -i v
template <typename V>
__device__ __forceinline__ V mul_i(V v) {
    V r;
    r.x = v.y;
    r.y = -v.x;
    return r;
}
template <typename V>
__device__ __forceinline__ V conj(V v) {
    v.y = -v.y;
    return v;
}

template <typename V>
__device__ __forceinline__ void dft4(V &a, V &b, V &c, V &d) {
    const V s02 = cadd(a, c), d02 = csub(a, c);
    const V s13 = cadd(b, d), q = mul_i(csub(b, d));
    a = cadd(s02, s13);
    b = cadd(d02, q);
    c = csub(s02, s13);
    d = csub(d02, q);
}

// One Stockham pass of radix R over gl lines of N points: the sub-transforms
// done so far have length Ns = N / n (a power of two).
template <typename T, int R>
__device__ __forceinline__ void pass(const V2<T> *src, V2<T> *dst, const V2<T> *tw, int N, int n,
                                     int Ns, const Deal &D, int gl) {
    using V = V2<T>;
    const int nb = (unsigned)N / R, step = (unsigned)n / R, line = D.g * line_len<T>(N);
    for (int j = D.g < gl ? D.j0 : nb; j < nb; j += D.stride) {
        const int k = j & (Ns - 1), ks = k * step, o = (j - k) * R + k;
        const V *x = src + line;
        V *y = dst + line;
        V v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = x[pad<T>(j + r * nb)];
        if (Ns > 1) {
            if constexpr (std::is_same<T, float>::value && (R == 4 || R == 8)) {
                // powers of one twiddle: its multiples' table entries lie in
                // few banks (512 points, four lines: 1,400 cycles a pass)
                const V w1 = tw[ks], w2 = cmul<false>(w1, w1), w3 = cmul<false>(w2, w1);
                v[1] = cmul<false>(v[1], w1);
                v[2] = cmul<false>(v[2], w2);
                v[3] = cmul<false>(v[3], w3);
                if constexpr (R == 8) {
                    const V w4 = cmul<false>(w2, w2);
                    v[4] = cmul<false>(v[4], w4);
                    v[5] = cmul<false>(v[5], cmul<false>(w4, w1));
                    v[6] = cmul<false>(v[6], cmul<false>(w4, w2));
                    v[7] = cmul<false>(v[7], cmul<false>(w4, w3));
                }
            } else {
#pragma unroll
                for (int r = 1; r < R; ++r) v[r] = cmul<false>(v[r], tw[r * ks]);
            }
        }
        auto put = [&](int r, V q) { y[pad<T>(o + r * Ns)] = q; };
        if constexpr (R == 2) {
            put(0, cadd(v[0], v[1]));
            put(1, csub(v[0], v[1]));
        } else if constexpr (R == 4) {
            dft4(v[0], v[1], v[2], v[3]);
#pragma unroll
            for (int r = 0; r < 4; ++r) put(r, v[r]);
        } else if constexpr (R == 8) {
            // even and odd halves, the odd one turned by multiples of pi / 4
            dft4(v[0], v[2], v[4], v[6]);
            dft4(v[1], v[3], v[5], v[7]);
            const T h = T(0.70710678118654752440);
            const V q1 = mul_i(v[3]), q3 = mul_i(v[7]);
            const V o1 = mk<T>(h * (v[3].x + q1.x), h * (v[3].y + q1.y));
            const V o2 = mul_i(v[5]);
            const V o3 = mk<T>(h * (q3.x - v[7].x), h * (q3.y - v[7].y));
            put(0, cadd(v[0], v[1]));
            put(1, cadd(v[2], o1));
            put(2, cadd(v[4], o2));
            put(3, cadd(v[6], o3));
            put(4, csub(v[0], v[1]));
            put(5, csub(v[2], o1));
            put(6, csub(v[4], o2));
            put(7, csub(v[6], o3));
        } else {
#pragma unroll
            for (int q = 0; q < R; ++q) {
                V t = v[0];
#pragma unroll
                for (int r = 1; r < R; ++r) t = cadd(t, cmul<false>(v[r], tw[((q * r) % R) * nb]));
                put(q, t);
            }
        }
    }
    __syncthreads();
}

// The transform (e^{-2 pi i jk/N}) of the gl lines at offset `a`; returns the
// offset of the buffer that holds the result, a or b.  The inverse transform is
// its conjugate of the conjugate.  Every thread of the block; the caller has
// synchronised the block after filling the lines.
//
// One copy of the code, out of line, with one instance of each radix and sizes
// in registers: the slice engine runs a few thousand instructions of each phase
// once and moves on, so that its phases are bound by instruction fetches as much
// as by data (with constant sizes a 256-point transform of two lines alone takes
// 1,050 cycles, with these 1,640, but a slice of the engine takes 219 us
// instead of 232).  float32: radix 8, with 4 or 4 x 4 for the rest.  Pairs:
// radix 4, whose 300 instructions on two warps a 256-point line finish sooner
// than radix 8's 900 on one.
template <typename T>
__device__ __noinline__ int fft(int a, int b, int tab, int N, int lgG, int gl) {
    const V2<T> *tw = cplx_at<T>(tab);
    const Deal D(lgG);
    int Ns = 1, n = N;
    auto run = [&](auto radix) {
        constexpr int R = decltype(radix)::value;
        pass<T, R>(cplx_at<T>(a), cplx_at<T>(b), tw, N, n, Ns, D, gl);
        const int t = a;
        a = b;
        b = t;
        Ns *= R;
        n = (unsigned)n / R;
    };
    int k = __ffs(n) - 1;  // factors of two left
    if constexpr (std::is_same<T, float>::value) {
#pragma unroll 1
        for (; k >= 3 && k != 4; k -= 3) run(std::integral_constant<int, 8>());
    }
#pragma unroll 1
    for (; k >= 2; k -= 2) run(std::integral_constant<int, 4>());
    if (k) run(std::integral_constant<int, 2>());
    if (n == 3) run(std::integral_constant<int, 3>());
    else if (n == 5) run(std::integral_constant<int, 5>());
    else if (n == 7) run(std::integral_constant<int, 7>());
    return a;
}

// Lines of real fields: one field (S = 1), whose line p is rows (in the column
// phase, columns) 2p and 2p + 1, or two (S = 2), each with lines of its own, so
// that a small field keeps its own relative accuracy beside a large one (as the
// two parts of one complex line the larger one's rounding reaches the other).
// Their lines lie one after the other, field c's rows at c N^2; row line 2p + c
// is line p of field c, column line c N / 2 + p likewise.
template <int S>
__device__ __forceinline__ size_t row_base(int line, int N) {
    if constexpr (S == 1) return (size_t)(2 * line) * N;
    return ((size_t)(line & 1) * N + (line & ~1)) * N;
}
// row y of column line `line`, in complex numbers
template <int S>
__device__ __forceinline__ size_t column_at(int y, int line, int N) {
    const size_t at = (size_t)y * (N / 2) + line;
    return S == 2 && line >= N / 2 ? at + (size_t)(N - 1) * (N / 2) : at;
}
template <int NC, int S>
__device__ __forceinline__ int lines_of(int N) {
    static_assert(NC == 1 || S == 1, "stacked fields are real");
    return NC == 2 || S == 2 ? N : N / 2;
}

// log2 of the lines a block takes at a time: as few as spread nl lines over nblk
// blocks in one round, at most gmax.
__device__ __forceinline__ int lines_at_once(int nl, int nblk, int gmax) {
    int lg = 0;
    while ((1 << lg) < gmax && (nblk << lg) < nl) ++lg;
    return lg;
}

// Where sample i of a line sits in the FFT input; odd samples change sign.
__device__ __forceinline__ int slot_of(int i, int N) { return (i & 1) ? N - 1 - (i >> 1) : i >> 1; }
// sample i from the conjugate of the inverse transform
template <typename V>
__device__ __forceinline__ V sample(V v, int i) {
    if (i & 1) v.x = -v.x;
    else v.y = -v.y;
    return v;
}

// The second half of rows_forward: transform of the filled lines l0 ... and
// the coefficients (times 2) to `out`.
template <typename T, int NC, int S>
__device__ __noinline__ void rows_forward_rest(int a, int b, int tab, int N, int l0, int lgG, int gl,
                                               V2<T> *out) {
    using V = V2<T>;
    const Deal D(lgG);
    __syncthreads();
    const V *r = cplx_at<T>(fft<T>(a, b, tab, N, lgG, gl));
    const V *dct = dct_table<T>(tab, N);
    for (int j = D.g < gl ? D.j0 : N; 2 * j <= N; j += D.stride) {
        const V *x = r + D.g * line_len<T>(N);
        V c, d;
        if (j == 0) {
            c = cadd(x[0], x[0]);
            d = c;
        } else {
            const V w = dct[j];
            const V A = cmul<false>(x[pad<T>(j)], w), B = cmul<true>(x[pad<T>(N - j)], w);
            const V m = csub(A, B);
            c = cadd(A, B);
            d = mk<T>(-m.y, m.x);
        }
        const bool two = j > 0 && 2 * j < N;
        if constexpr (NC == 2) {
            V *o = out + (size_t)(l0 + D.g) * N;
            o[j] = c;
            if (two) o[N - j] = d;
        } else {
            T *o = (T *)out + row_base<S>(l0 + D.g, N);
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

// Rows forward.  Two components (NC = 2): line y is the complex row of both.
// One component: line p is rows 2p (real part) and 2p + 1.  load(line, x) gives
// the samples; the coefficients go to `out`, complex [y][j] or real [y][j].
template <typename T, int NC, int S = 1, typename F>
__device__ __forceinline__ void rows_forward(const Lines &P, int bid, int nblk, V2<T> *out,
                                             F load) {
    using V = V2<T>;
    const int N = P.N, nl = lines_of<NC, S>(N);
    const int lgG = lines_at_once(nl, nblk, P.gmax), G = 1 << lgG;
    const Deal D(lgG);
    V *const a = cplx_at<T>(P.a);
    for (int l0 = bid * G; l0 < nl; l0 += nblk * G) {
        const int gl = min(G, nl - l0);
        for (int x = D.g < gl ? D.j0 : N; x < N; x += D.stride) {
            V v = load(l0 + D.g, x);
            if (x & 1) v = mk<T>(-v.x, -v.y);
            a[D.g * line_len<T>(N) + pad<T>(slot_of(x, N))] = v;
        }
        rows_forward_rest<T, NC, S>(P.a, buf_b<T>(P), P.tab, N, l0, lgG, gl, out);
    }
}

using qsff::recip;
__device__ __forceinline__ float recip(float d) { return 1.f / d; }

// The rest of `columns` after its lines are filled: forward, times
// 1 / (4 N^2 (lam_x + lam_y - kbar)), inverse, and the store.  kbar: a real
// number, or a complex one (two components as one complex field).
template <typename T, int NC, int S, typename K>
__device__ __noinline__ void columns_rest(int a, int b, int tab, int N, int l0, int lgG, int gl,
                                          V2<T> *out, K kbar) {
    constexpr bool cplx = !std::is_same<K, T>::value;
    static_assert(!cplx || NC == 2, "a complex shift needs a complex field");
    using V = V2<T>;
    const int G = 1 << lgG;
    const Deal D(lgG);
    const T c4 = recip(T(4 * N * N));
    const V *const dct = dct_table<T>(tab, N);
    const T *const lam = lam_table<T>(tab, N);
    __syncthreads();
    const int f = fft<T>(a, b, tab, N, lgG, gl);
    for (int j = D.g < gl ? D.j0 : N; 2 * j <= N; j += D.stride) {
        int l = l0 + D.g;
        if (S == 2 && l >= N / 2) l -= N / 2;
        T kr;
        if constexpr (cplx) kr = kbar.x;
        else kr = kbar;
        const T lx0 = lam[NC == 2 ? l : 2 * l] - kr;
        const T lx1 = NC == 2 ? lx0 : lam[2 * l + 1] - kr;
        auto scaled = [&](V c, int jj) {
            const T ly = lam[jj];
            if constexpr (cplx) {  // 1 / (d - i k) = (d + i k) / (d^2 + k^2)
                const T d = lx0 + ly, g = c4 * recip(d * d + kbar.y * kbar.y);
                return cmul<false>(c, mk<T>(d * g, kbar.y * g));
            }
            const T s0 = c4 * recip(lx0 + ly);
            const T s1 = NC == 2 ? s0 : c4 * recip(lx1 + ly);
            return mk<T>(c.x * s0, c.y * s1);
        };
        V *x = cplx_at<T>(f) + D.g * line_len<T>(N);
        if (j == 0) {
            x[0] = conj(scaled(cadd(x[0], x[0]), 0));
            continue;
        }
        const V w = dct[j];
        const V A = cmul<false>(x[pad<T>(j)], w), B = cmul<true>(x[pad<T>(N - j)], w);
        const V c = scaled(cadd(A, B), j), m = csub(A, B);
        // -i C_{N-j} with C_{N-j} = i m scaled: the parts swap twice
        V d = scaled(mk<T>(-m.y, m.x), N - j);
        d = mk<T>(d.y, -d.x);
        x[pad<T>(j)] = conj(cmul<true>(cadd(c, d), w));
        if (2 * j < N) x[pad<T>(N - j)] = conj(cmul<false>(csub(c, d), w));
    }
    __syncthreads();
    const V *r = cplx_at<T>(fft<T>(f, f == a ? b : a, tab, N, lgG, gl));
    for (int t = threadIdx.x; t < (N << lgG); t += blockDim.x) {
        const int y = t >> lgG, g = t & (G - 1);
        if (g >= gl) continue;
        const V v = r[g * line_len<T>(N) + pad<T>(slot_of(y, N))];
        out[NC == 2 ? (size_t)y * N + l0 + g : column_at<S>(y, l0 + g, N)] = sample(v, y);
    }
    __syncthreads();
}

// Columns: load(y, line) gives the row coefficients; the solution's row
// coefficients go to `out`.  The one-component array seen as complex pairs puts
// columns 2p and 2p + 1 into line p.
template <typename T, int NC, int S = 1, typename K, typename F>
__device__ __forceinline__ void columns(const Lines &P, int bid, int nblk, V2<T> *out, K kbar,
                                        F load) {
    using V = V2<T>;
    const int N = P.N, nl = lines_of<NC, S>(N);
    const int lgG = lines_at_once(nl, nblk, P.gmax), G = 1 << lgG;
    V *const a = cplx_at<T>(P.a);
    for (int l0 = bid * G; l0 < nl; l0 += nblk * G) {
        const int gl = min(G, nl - l0);
        for (int t = threadIdx.x; t < (N << lgG); t += blockDim.x) {
            const int y = t >> lgG, g = t & (G - 1);
            if (g >= gl) continue;
            V v = load(y, l0 + g);
            if (y & 1) v = mk<T>(-v.x, -v.y);
            a[g * line_len<T>(N) + pad<T>(slot_of(y, N))] = v;
        }
        columns_rest<T, NC, S, K>(P.a, buf_b<T>(P), P.tab, N, l0, lgG, gl, out, kbar);
    }
}

// The first half of rows_inverse: coefficients of lines l0 ... to samples;
// returns the offset of the buffer that holds their conjugates (see sample).
template <typename T, int NC, int S>
__device__ __noinline__ int rows_inverse_first(int a, int b, int tab, int N, int l0, int lgG, int gl,
                                               const V2<T> *in) {
    using V = V2<T>;
    const V *const dct = dct_table<T>(tab, N);
    const Deal D(lgG);
    for (int j = D.g < gl ? D.j0 : N; 2 * j <= N; j += D.stride) {
        const int l = l0 + D.g;
        auto coef = [&](int jj) {
            if constexpr (NC == 2) {
                return in[(size_t)l * N + jj];
            } else {
                const T *o = (const T *)in + row_base<S>(l, N);
                return mk<T>(o[jj], o[N + jj]);
            }
        };
        V *x = cplx_at<T>(a) + D.g * line_len<T>(N);
        const V c = coef(j);
        if (j == 0) {
            x[0] = conj(c);
            continue;
        }
        const V w = dct[j], e = coef(N - j);
        const V d = mk<T>(e.y, -e.x);  // -i C_{N-j}
        x[pad<T>(j)] = conj(cmul<true>(cadd(c, d), w));
        if (2 * j < N) x[pad<T>(N - j)] = conj(cmul<false>(csub(c, d), w));
    }
    __syncthreads();
    return fft<T>(a, b, tab, N, lgG, gl);
}

// Rows inverse: store(line, x, value) takes the solution's samples.
template <typename T, int NC, int S = 1, typename F>
__device__ __forceinline__ void rows_inverse(const Lines &P, int bid, int nblk, const V2<T> *in,
                                             F store) {
    using V = V2<T>;
    const int N = P.N, nl = lines_of<NC, S>(N);
    const int lgG = lines_at_once(nl, nblk, P.gmax), G = 1 << lgG;
    const Deal D(lgG);
    for (int l0 = bid * G; l0 < nl; l0 += nblk * G) {
        const int gl = min(G, nl - l0);
        const V *r = cplx_at<T>(
            rows_inverse_first<T, NC, S>(P.a, buf_b<T>(P), P.tab, N, l0, lgG, gl, in));
        for (int x = D.g < gl ? D.j0 : N; x < N; x += D.stride) {
            store(l0 + D.g, x, sample(r[D.g * line_len<T>(N) + pad<T>(slot_of(x, N))], x));
        }
        __syncthreads();
    }
}

// Rows inverse and, of what next(row, x, value) makes of the samples of two
// fields, rows forward of two components again, in another storage type if asked.
// The fields are the parts of complex rows (S = 1) or stacked (S = 2: a block
// takes pairs of lines, rows 2p and 2p + 1 of both fields; needs P.gmax >= 2).
template <typename T, typename U, int S, typename F>
__device__ __forceinline__ void rows_inverse_forward(const Lines &P, const Lines &PU, int bid,
                                                     int nblk, const V2<T> *in, V2<U> *out,
                                                     F next) {
    using V = V2<T>;
    const int N = P.N, b = buf_b<T>(P);
    const int lgG = max(S - 1, lines_at_once(N, nblk, P.gmax)), G = 1 << lgG;
    const Deal D(lgG);
    for (int l0 = bid * G; l0 < N; l0 += nblk * G) {
        const int gl = min(G, N - l0);
        const int f = rows_inverse_first<T, 3 - S, S>(P.a, b, P.tab, N, l0, lgG, gl, in);
        const int o = f == P.a ? b : P.a;  // the free buffer: no smaller than U needs
        const V *r = cplx_at<T>(f) + (S == 2 ? D.g & ~1 : D.g) * line_len<T>(N);
        V2<U> *q = cplx_at<U>(o) + D.g * line_len<U>(N);
        for (int x = D.g < gl ? D.j0 : N; x < N; x += D.stride) {
            const int at = slot_of(x, N);
            V v = sample(r[pad<T>(at)], x);
            if constexpr (S == 2) {
                const V c = sample(r[line_len<T>(N) + pad<T>(at)], x);
                v = D.g & 1 ? mk<T>(v.y, c.y) : mk<T>(v.x, c.x);
            }
            V2<U> w = next(l0 + D.g, x, v);
            if (x & 1) w = mk<U>(-w.x, -w.y);
            q[pad<U>(at)] = w;
        }
        rows_forward_rest<U, 2, 1>(o, f, PU.tab, N, l0, lgG, gl, out);
    }
}

// Shared scratch of the block's sums (up to 16 warps); a block barrier stands
// between two uses.
constexpr int kSumWarps = 16;
static __device__ __forceinline__ float *sum_scratch() {
    __shared__ __align__(16) float scratch[18 * kSumWarps];
    return scratch;
}

// Sums of 16 values over the block: thread t < 16 returns the sum of v[t].  Each
// shuffle halves the values a lane holds: 16 shuffles instead of 80.
static __device__ float block_sums16(float v[16]) {
    float (*const red)[17] = (float (*)[17])sum_scratch();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (int)blockDim.x >> 5;
#pragma unroll
    for (int o = 16; o >= 2; o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int k = 0; k < o / 2; ++k) {
            const float give = up ? v[k] : v[k + o / 2];
            const float keep = up ? v[k + o / 2] : v[k];
            v[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
    // lane bits 4..1 select the value: bit 4 its half, and so on
    if ((lane & 1) == 0) red[wid][lane >> 1] = v[0];
    __syncthreads();
    float t = 0.f;
    if (threadIdx.x < 16)
        for (int w = 0; w < nw; ++w) t += red[w][threadIdx.x];
    return t;
}

}  // namespace qsfft
