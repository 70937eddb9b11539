// Mixed-radix complex FFT of a tile of lines held in shared memory, FP32.
//
// A tile holds its lines of n points as tile[i * rs + line] (line fastest; or any two strides), so
// that a warp's accesses of one radix step are contiguous whatever the radix.  Stockham's autosort form:
// step with radix r after a product L of earlier radices takes, for b in [0, n/r), the points
// b + s n/r (s < r), twiddles them by exp(-2 pi i q s / (L r)), q = b mod L, applies the r-point
// DFT and writes the points (b / L) L r + q + s L of the other buffer; one barrier per step,
// results in natural order.  Radices 2..10, 12 and 16 are unrolled in registers (composite
// ones by Cooley-Tukey over their factors); any other prime factor takes a direct O(r) sum per
// output, so every extent is accepted.  The inverse is the forward transform with real and
// imaginary parts swapped before and after.
#pragma once

#include <cuda_runtime.h>

namespace of {

constexpr int FFT_MAX_N = 2048;      // points of one line (two tiles of lines in shared memory)
constexpr int FFT_MAX_STAGES = 12;

#define OF_HD __host__ __device__ __forceinline__

struct FftPlan {
    int n, nst;
    bool unrolled;                   // every radix is
    int r[FFT_MAX_STAGES];           // radix of each step
    int L[FFT_MAX_STAGES];           // product of the radices before it
    int T[FFT_MAX_STAGES];           // n / r
    int tl[FFT_MAX_STAGES];          // n / (r L): twiddle step
    unsigned mL[FFT_MAX_STAGES];     // floor(2^32 / L) + 1 (0 for L = 1): b / L = mulhi(b, mL)
    unsigned mT[FFT_MAX_STAGES];     // the same for T
    const float2* tw;                // exp(-2 pi i k / n), k < n
};

OF_HD bool fft_unrolled(int r) { return (r >= 2 && r <= 10) || r == 12 || r == 16; }

OF_HD unsigned fft_mulhi(unsigned a, unsigned b) {
#ifdef __CUDA_ARCH__
    return __umulhi(a, b);
#else
    return (unsigned)(((unsigned long long)a * b) >> 32);
#endif
}
OF_HD int fft_div(int v, unsigned magic) { return magic ? (int)fft_mulhi((unsigned)v, magic) : v; }

OF_HD float2 cxadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
OF_HD float2 cxsub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
OF_HD float2 cxmul(float2 a, float2 b) { return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }

// exp(-2 pi i k / N) as compile-time constants (Taylor series after reduction to |t| <= pi / 4)
template <int N>
struct FftRoots {
    float c[N], s[N];
    static constexpr double taylor(double t, bool odd) {
        double term = odd ? t : 1.0, sum = term;
        for (int k = odd ? 1 : 0; k < 24; k += 2) {
            term *= -t * t / ((k + 1.0) * (k + 2.0));
            sum += term;
        }
        return sum;
    }
    constexpr FftRoots() : c(), s() {
        for (int k = 0; k < N; ++k) {
            // angle 2 pi k / N = (pi / 2) quarter + t, 8 k = 2 quarter N + rest with |rest| <= N
            const int quarter = (4 * k + N / 2) / N;
            const double t = 6.283185307179586476925 * ((double)k / N - 0.25 * quarter);
            const double ct = taylor(t, false), st = taylor(t, true);
            const int h = quarter % 4;
            c[k] = (float)(h == 0 ? ct : h == 1 ? -st : h == 2 ? -ct : st);
            s[k] = (float)(h == 0 ? -st : h == 1 ? -ct : h == 2 ? st : ct);
        }
    }
};

// v times the compile-time root (c, s)
OF_HD float2 cxroot(float2 v, float c, float s) {
    if (s == 0.f && c == 1.f) return v;
    if (s == 0.f && c == -1.f) return make_float2(-v.x, -v.y);
    if (c == 0.f && s == -1.f) return make_float2(v.y, -v.x);
    if (c == 0.f && s == 1.f) return make_float2(-v.y, v.x);
    return make_float2(v.x * c - v.y * s, v.x * s + v.y * c);
}

template <int R> struct Dft;
template <> struct Dft<2> {
    static OF_HD void run(float2 (&v)[2]) {
        const float2 a = v[0], b = v[1];
        v[0] = cxadd(a, b);
        v[1] = cxsub(a, b);
    }
};
template <> struct Dft<4> {
    static OF_HD void run(float2 (&v)[4]) {
        const float2 a = cxadd(v[0], v[2]), b = cxsub(v[0], v[2]);
        const float2 c = cxadd(v[1], v[3]), d = cxsub(v[1], v[3]);
        v[0] = cxadd(a, c);
        v[2] = cxsub(a, c);
        v[1] = make_float2(b.x + d.y, b.y - d.x);   // b - i d
        v[3] = make_float2(b.x - d.y, b.y + d.x);
    }
};
// odd R: pairs s_k = v_k + v_{R-k}, d_k = v_k - v_{R-k}
template <int R> struct DftOdd {
    static OF_HD void run(float2 (&v)[R]) {
        constexpr FftRoots<R> W{};
        constexpr int H = R / 2;
        float2 s[H], d[H];
#pragma unroll
        for (int k = 0; k < H; ++k) {
            s[k] = cxadd(v[k + 1], v[R - 1 - k]);
            d[k] = cxsub(v[k + 1], v[R - 1 - k]);
        }
        const float2 v0 = v[0];
        float2 sum = v0;
#pragma unroll
        for (int k = 0; k < H; ++k) sum = cxadd(sum, s[k]);
        v[0] = sum;
#pragma unroll
        for (int m = 1; m <= H; ++m) {
            float2 re = v0, im = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < H; ++k) {
                const int t = (m * (k + 1)) % R;
                re.x += W.c[t] * s[k].x;
                re.y += W.c[t] * s[k].y;
                im.x += W.s[t] * d[k].x;
                im.y += W.s[t] * d[k].y;
            }
            // re + i im and re - i im
            v[m] = make_float2(re.x - im.y, re.y + im.x);
            v[R - m] = make_float2(re.x + im.y, re.y - im.x);
        }
    }
};
template <> struct Dft<3> : DftOdd<3> {};
template <> struct Dft<5> : DftOdd<5> {};
template <> struct Dft<7> : DftOdd<7> {};
// R = A B: n = B n1 + n2, k = k1 + A k2
template <int A, int B> struct DftPair {
    static OF_HD void run(float2 (&v)[A * B]) {
        constexpr FftRoots<A * B> W{};
        float2 y[B][A];
#pragma unroll
        for (int n2 = 0; n2 < B; ++n2) {
            float2 a[A];
#pragma unroll
            for (int n1 = 0; n1 < A; ++n1) a[n1] = v[B * n1 + n2];
            Dft<A>::run(a);
#pragma unroll
            for (int k1 = 0; k1 < A; ++k1) y[n2][k1] = cxroot(a[k1], W.c[(n2 * k1) % (A * B)], W.s[(n2 * k1) % (A * B)]);
        }
#pragma unroll
        for (int k1 = 0; k1 < A; ++k1) {
            float2 b[B];
#pragma unroll
            for (int n2 = 0; n2 < B; ++n2) b[n2] = y[n2][k1];
            Dft<B>::run(b);
#pragma unroll
            for (int k2 = 0; k2 < B; ++k2) v[k1 + A * k2] = b[k2];
        }
    }
};
template <> struct Dft<6> : DftPair<2, 3> {};
template <> struct Dft<8> : DftPair<4, 2> {};
template <> struct Dft<9> : DftPair<3, 3> {};
template <> struct Dft<10> : DftPair<2, 5> {};
template <> struct Dft<12> : DftPair<4, 3> {};
template <> struct Dft<16> : DftPair<4, 4> {};

// One butterfly of an unrolled step: line `line`, index b, from src(line, i) to dst(line, i, v)
template <int R, class Src, class Dst>
OF_HD void fft_butterfly(const Src& src, const Dst& dst, const float2* tw, int L, int T, int tl, unsigned mL, int line,
                         int b) {
    const int p = fft_div(b, mL), q = b - p * L;
    float2 v[R];
#pragma unroll
    for (int s = 0; s < R; ++s) v[s] = src(line, b + s * T);
    if (L > 1) {
        const int step = q * tl;
#pragma unroll
        for (int s = 1; s < R; ++s) v[s] = cxmul(v[s], tw[s * step]);
    }
    Dft<R>::run(v);
    const int o = p * L * R + q;
#pragma unroll
    for (int s = 0; s < R; ++s) dst(line, o + s * L, v[s]);
}

// The last step of a transform, mid(i, X_i) on its results, and the first step of a transform of
// those (whose first radix is the same): index b's results b + s T are that step's inputs.
template <int R, class Src, class Mid, class Dst>
OF_HD void fft_turn(const Src& src, const Mid& mid, const Dst& dst, const float2* tw, int T, int line, int b) {
    float2 v[R];
#pragma unroll
    for (int s = 0; s < R; ++s) v[s] = src(line, b + s * T);
    if (T > 1) {
#pragma unroll
        for (int s = 1; s < R; ++s) v[s] = cxmul(v[s], tw[s * b]);
    }
    Dft<R>::run(v);
#pragma unroll
    for (int s = 0; s < R; ++s) v[s] = mid(b + s * T, v[s]);
    Dft<R>::run(v);
#pragma unroll
    for (int s = 0; s < R; ++s) dst(line, b * R + s, v[s]);
}

// One output of a step with a large prime radix r: u = s T + b
template <class Src, class Dst>
OF_HD void fft_direct_output(const Src& src, const Dst& dst, const float2* tw, int n, int r, int L, int T, int tl,
                             unsigned mL, unsigned mT, int line, int u) {
    const int s = fft_div(u, mT), b = u - s * T;
    const int p = fft_div(b, mL), q = b - p * L;
    const int step = (s * T + q * tl) % n;
    float2 acc = make_float2(0.f, 0.f);
    int k = 0;
    for (int t = 0; t < r; ++t) {
        const float2 x = src(line, b + t * T), w = tw[k];
        acc.x = fmaf(x.x, w.x, fmaf(-x.y, w.y, acc.x));
        acc.y = fmaf(x.x, w.y, fmaf(x.y, w.x, acc.y));
        k += step;
        if (k >= n) k -= n;
    }
    dst(line, p * L * r + q + s * L, acc);
}

// Points of a tile in shared memory: point i of a line at p[i * rs + line * ls]
struct FftTile {
    float2* p;
    int rs, ls = 1;
    OF_HD float2 operator()(int line, int i) const { return p[i * rs + line * ls]; }
    OF_HD void operator()(int line, int i, float2 v) const { p[i * rs + line * ls] = v; }
};

// The lines of a tile, and how a work item splits into a line (fastest) and the rest: a power of two
// of them, or any number m
struct FftPow2 {
    int lg;
    OF_HD int lines() const { return 1 << lg; }
    OF_HD int rest(int w) const { return w >> lg; }
};
struct FftAny {
    int m;
    unsigned magic;   // floor(2^32 / m) + 1 (0 for m = 1): exact for items below 2^16
    OF_HD int lines() const { return m; }
    OF_HD int rest(int w) const { return fft_div(w, magic); }
};

// f(constant R) for the unrolled radix r
#define OF_FFT_RADIX(r, CALL)                                                                   \
    switch (r) {                                                                                \
        case 2: { constexpr int R = 2; CALL; } break;                                           \
        case 3: { constexpr int R = 3; CALL; } break;                                           \
        case 4: { constexpr int R = 4; CALL; } break;                                           \
        case 5: { constexpr int R = 5; CALL; } break;                                           \
        case 6: { constexpr int R = 6; CALL; } break;                                           \
        case 7: { constexpr int R = 7; CALL; } break;                                           \
        case 8: { constexpr int R = 8; CALL; } break;                                           \
        case 9: { constexpr int R = 9; CALL; } break;                                           \
        case 10: { constexpr int R = 10; CALL; } break;                                         \
        case 12: { constexpr int R = 12; CALL; } break;                                         \
        case 16: { constexpr int R = 16; CALL; } break;                                         \
        default: break;                                                                         \
    }

// One unrolled step for the work items first, first + stride, ... (item = butterfly of a line)
template <class Map, class Src, class Dst>
OF_HD void fft_step(const FftPlan& P, int st, const Src& src, const Dst& dst, const float2* tw, const Map& map,
                    int first, int stride) {
    const int nl = map.lines(), items = P.T[st] * nl;
    OF_FFT_RADIX(P.r[st], for (int w = first; w < items; w += stride) {
        const int b = map.rest(w);
        fft_butterfly<R>(src, dst, tw, P.L[st], P.T[st], P.tl[st], P.mL[st], w - b * nl, b);
    })
}
// fft_turn with the last step of P
template <class Map, class Src, class Mid, class Dst>
OF_HD void fft_turn_step(const FftPlan& P, const Src& src, const Mid& mid, const Dst& dst, const float2* tw,
                         const Map& map, int first, int stride) {
    const int st = P.nst - 1, nl = map.lines(), items = P.T[st] * nl;
    OF_FFT_RADIX(P.r[st], for (int w = first; w < items; w += stride) {
        const int b = map.rest(w);
        fft_turn<R>(src, mid, dst, tw, P.T[st], w - b * nl, b);
    })
}
// Any step between two tiles of the same strides: unrolled, or one output per item
template <class Map>
OF_HD void fft_any_step(const FftPlan& P, int st, const FftTile& in, const FftTile& out, const float2* tw,
                        const Map& map, int first, int stride) {
    if (fft_unrolled(P.r[st])) {
        fft_step(P, st, in, out, tw, map, first, stride);
    } else {
        const int nl = map.lines(), items = P.n * nl;
        for (int w = first; w < items; w += stride) {
            const int u = map.rest(w);
            fft_direct_output(in, out, tw, P.n, P.r[st], P.L[st], P.T[st], P.tl[st], P.mL[st], P.mT[st], w - u * nl, u);
        }
    }
}

// The plan of n = r[0] r[1] .. r[k - 1], in that order
inline void fft_plan_of(int n, int k, const int* r, FftPlan& P) {
    P.n = n;
    P.nst = k;
    P.unrolled = true;
    P.tw = nullptr;
    auto magic = [](int d) { return d == 1 ? 0u : (unsigned)((1ull << 32) / (unsigned)d + 1); };
    for (int s = 0, L = 1; s < k; L *= r[s++]) {
        P.unrolled = P.unrolled && fft_unrolled(r[s]);
        P.r[s] = r[s];
        P.L[s] = L;
        P.T[s] = n / r[s];
        P.tl[s] = n / (r[s] * L);
        P.mL[s] = magic(L);
        P.mT[s] = magic(P.T[s]);
    }
}

// Radices of n: the fewest steps, small radices among equals
inline bool fft_make_plan(int n, FftPlan& P) {
    if (n < 1 || n > FFT_MAX_N) return false;
    struct Best { double cost; int r; };
    // cost[m] over the divisors of n: cheapest sequence of radices with product m
    static const int radices[] = {16, 12, 10, 9, 8, 7, 6, 5, 4, 3, 2};
    double cost[FFT_MAX_N + 1];
    int first[FFT_MAX_N + 1];
    for (int m = 0; m <= n; ++m) { cost[m] = 1e30; first[m] = 0; }
    cost[1] = 0.0;
    for (int m = 2; m <= n; ++m) {
        if (n % m) continue;
        auto take = [&](int r, double c) {
            if (m % r == 0 && cost[m / r] + c < cost[m]) { cost[m] = cost[m / r] + c; first[m] = r; }
        };
        for (int r : radices) take(r, 1.0 + 0.04 * r);
        for (int r = 11; r <= m; r += 2) {
            bool prime = true;
            for (int d = 3; d * d <= r; d += 2) prime = prime && r % d != 0;
            if (prime) take(r, 1.0 + 0.3 * r);
        }
    }
    int r[FFT_MAX_STAGES], k = 0;
    for (int m = n; m > 1; m /= first[m]) {
        if (k == FFT_MAX_STAGES || first[m] < 2) return false;
        r[k++] = first[m];
    }
    fft_plan_of(n, k, r, P);
    return true;
}

}  // namespace of
