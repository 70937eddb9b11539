// Direct FP32 solves with translation-invariant operators on the periodic grid.
//
// The order-2N Laplacian of Eq. FD:Laplacian commutes with lattice translations, so the discrete
// Fourier transform diagonalises it: -L_h has the eigenvalue l(k) = l_x + l_y + l_z with
// l_a = sum_p 4 w_p sin^2(p theta_a / 2).  One forward transform, a division by the symbol
// (l for Poisson, a l + Q for the shifted systems, (l + s0) / (l + s1)^2 for the NLCG's
// preconditioner) and one inverse transform therefore apply the exact inverse.  In FP32 that is
// the correction of one refinement pass of the mixed-precision solves: the FP64 residual of
// each pass drops by the FP32 rounding (1e-4 .. 1e-6), where a multigrid-preconditioned Krylov
// pass took 4 .. 30 iterations of ~17 dependent launches for the same drop.
//
// Five launches (three on small planes, which x and y share): x forward, y forward, z forward * symbol * z inverse, y inverse, x inverse,
// each moving the half spectrum once (4 B per point and direction; 8 B for complex fields).
// Real fields: two x rows are the real and imaginary part of one line, separated into
// their half spectra (n1 / 2 + 1 points) on the way out and combined again on the way back.
// A block transforms a tile of TX = 16 lines (128-byte segments of global memory for the y and
// z lines) in shared memory, of_fft.cuh.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <vector>

#include "of_fft.cuh"
#include "of_krylov.cuh"

namespace of {

struct Fft {
    bool ok = false;
    FftPlan plan[3], z_back;   // z_back: the radices of plan[2] reversed
    const float* sym[3];     // l_a(k), k < n_a
    double lmax = 0.0;       // the largest eigenvalue of -L_h
};

void fft_destroy(Fft* f) { delete f; }

static Fft& fft_of(of_grid* g) {
    if (!g->fft) g->fft = new Fft();
    return *g->fft;
}

bool fft_available(of_grid* g) {
    return g->d.n1 <= FFT_MAX_N && g->d.n2 <= FFT_MAX_N && g->d.n3 <= FFT_MAX_N;
}

// Plans, twiddles and symbol tables (host FP64, rounded once), built with the first direct solve
static Fft& fft_tables(of_grid* g) {
    Fft& f = fft_of(g);
    if (f.ok) return f;
    const int n[3] = {g->d.n1, g->d.n2, g->d.n3};
    std::vector<float> host;
    size_t off[6];
    f.lmax = 0.0;
    for (int a = 0; a < 3; ++a) {
        OF_REQUIRE(fft_make_plan(n[a], f.plan[a]), OF_EINVAL, "direct solve: no transform of %d points", n[a]);
        off[a] = host.size();
        for (int k = 0; k < n[a]; ++k) {
            const double t = -2.0 * M_PI * k / n[a];
            host.push_back((float)std::cos(t));
            host.push_back((float)std::sin(t));
        }
        off[3 + a] = host.size();
        double top = 0.0;
        for (int k = 0; k < n[a]; ++k) {
            double l = 0.0;
            for (int p = 1; p <= g->N; ++p) {
                const double s = std::sin(M_PI * (double)((long long)p * k % n[a]) / n[a]);
                l += 4.0 * g->w64.w[a][p] * s * s;
            }
            host.push_back((float)l);
            top = std::max(top, l);
        }
        f.lmax += top;
        if (host.size() & 1) host.push_back(0.f);   // the twiddles of the next axis are float2
    }
    float* dev = (float*)ws(g, WS_FFTT, sizeof(float) * host.size());
    OF_CUDA(cudaMemcpyAsync(dev, host.data(), sizeof(float) * host.size(), cudaMemcpyHostToDevice, g->stream));
    OF_CUDA(cudaStreamSynchronize(g->stream));   // the host vector goes out of scope
    for (int a = 0; a < 3; ++a) {
        f.plan[a].tw = (const float2*)(dev + off[a]);
        f.sym[a] = dev + off[3 + a];
    }
    int back[FFT_MAX_STAGES];
    for (int s = 0; s < f.plan[2].nst; ++s) back[s] = f.plan[2].r[f.plan[2].nst - 1 - s];
    fft_plan_of(n[2], f.plan[2].nst, back, f.z_back);
    f.ok = true;
    return f;
}

// ------------------------------------------------------------- FP64 <-> scaled FP32 by bits
// v 2^-sh rounded to FP32 (values below its normal range become zero) and back: by integer
// arithmetic on the bits, as GB300 converts and multiplies FP64 at 2 per clock and SM.
__device__ __forceinline__ float narrow_scaled(double v, int sh) {
    const int hi = __double2hiint(v);
    const unsigned lo = (unsigned)__double2loint(v);
    const int e = ((hi >> 20) & 0x7ff) - (1023 - 127) - sh;
    const unsigned sign = (unsigned)hi & 0x80000000u;
    unsigned m = (((unsigned)hi & 0xfffffu) << 3) | (lo >> 29);
    m += ((unsigned)max(e, 0) << 23) + ((lo >> 28) & 1u);   // round half away; a carry moves the exponent
    m = e >= 255 ? 0x7f800000u : m;
    return __uint_as_float(e <= 0 ? sign : (sign | m));
}
__device__ __forceinline__ double widen_scaled(float v, int sh) {
    const unsigned b = __float_as_uint(v);
    const int e = (int)((b >> 23) & 0xffu);
    const unsigned hi = (b & 0x80000000u) | ((unsigned)(e + (1023 - 127) + sh) << 20) | ((b & 0x7fffffu) >> 3);
    return e == 0 ? 0.0 : __hiloint2double((int)hi, (int)(b << 29));
}

// ------------------------------------------------------------------- loads and stores
// The residual enters a correction divided by the state's scale 2^sh, and the correction is
// added to the solution times it.
__device__ __forceinline__ int scale_exponent(const KState* st) {
    return ((__double2hiint(st->scale) >> 20) & 0x7ff) - 1023;
}
struct LdReal32 {
    const float* p;
    __device__ void begin() {}
    __device__ float at(long long i) const { return p[i]; }
};
struct LdReal64 {
    const double* p;
    const KState* st;
    int sh;
    __device__ void begin() { sh = scale_exponent(st); }
    __device__ float at(long long i) const { return narrow_scaled(p[i], sh); }
};
struct LdCplx64 {
    const double2* p;
    const KState* st;
    int sh;
    __device__ void begin() { sh = scale_exponent(st); }
    __device__ float2 at(long long i) const {
        const double2 v = p[i];
        return make_float2(narrow_scaled(v.x, sh), narrow_scaled(v.y, sh));
    }
};
struct StReal32 {
    float* p;
    __device__ void begin() {}
    __device__ void put(long long i, float v) const { p[i] = v; }
};
struct StAccum64 {
    double* p;
    const KState* st;
    int sh;
    __device__ void begin() { sh = scale_exponent(st); }
    __device__ void put(long long i, float v) const { p[i] += widen_scaled(v, sh); }
};
struct StAccumCplx64 {
    double2* p;
    const KState* st;
    int sh;
    __device__ void begin() { sh = scale_exponent(st); }
    __device__ void put(long long i, float2 v) const {
        double2 x = p[i];
        x.x += widen_scaled(v.x, sh);
        x.y += widen_scaled(v.y, sh);
        p[i] = x;
    }
};

// ----------------------------------------------------------------------------- kernels
constexpr int FFT_THREADS = 256;

__device__ __forceinline__ float2* fft_smem_tables(const FftPlan& P) {
    extern __shared__ float2 fft_smem[];
    for (int k = threadIdx.x; k < P.n; k += blockDim.x) fft_smem[k] = P.tw[k];
    return fft_smem;
}

// All steps of the tile in a (other buffer b); returns the buffer that holds the result.  The
// caller's writes to a are made visible here.
template <class Map>
__device__ __forceinline__ float2* fft_tile(const FftPlan& P, float2* a, float2* b, const float2* tw, int rs, int ls,
                                            const Map& map) {
    __syncthreads();
    for (int st = 0; st < P.nst; ++st) {
        fft_any_step(P, st, FftTile{a, rs, ls}, FftTile{b, rs, ls}, tw, map, threadIdx.x, blockDim.x);
        __syncthreads();
        float2* t = a;
        a = b;
        b = t;
    }
    return a;
}

// x lines forward.  Real: line l of the tile is rows 2 (TX blk + l) and + 1; out gets nh = n / 2 + 1
// points per row.  Complex: line l is row TX blk + l, nh = n.
template <bool CPLX, class LD>
__global__ void __launch_bounds__(FFT_THREADS) k_fft_x_forward(FftPlan P, int lg, long long rows, int nh, LD ld,
                                                               float2* __restrict__ out, const double* done) {
    pdl_enter();
    if (*done != 0.0) return;
    ld.begin();
    const int TX = 1 << lg, rs = TX + 1, n = P.n;
    const float2* tw = fft_smem_tables(P);
    float2* A = const_cast<float2*>(tw) + n;
    float2* Bf = A + n * rs;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const long long row0 = (long long)blockIdx.x * TX * (CPLX ? 1 : 2);
    for (int l = warp; l < TX; l += nw) {
        if constexpr (CPLX) {
            const long long r = row0 + l;
            if (r >= rows) continue;
#pragma unroll 4
            for (int i = lane; i < n; i += 32) A[i * rs + l] = ld.at(r * n + i);
        } else {
            const long long r = row0 + 2 * l;
            if (r >= rows) continue;
            const bool two = r + 1 < rows;
#pragma unroll 4
            for (int i = lane; i < n; i += 32)
                A[i * rs + l] = make_float2(ld.at(r * n + i), two ? ld.at((r + 1) * n + i) : 0.f);
        }
    }
    const float2* R = fft_tile(P, A, Bf, tw, rs, 1, FftPow2{lg});
    for (int l = warp; l < TX; l += nw) {
        if constexpr (CPLX) {
            const long long r = row0 + l;
            if (r >= rows) continue;
#pragma unroll 4
            for (int k = lane; k < n; k += 32) out[r * nh + k] = R[k * rs + l];
        } else {
            const long long r = row0 + 2 * l;
            if (r >= rows) continue;
            const bool two = r + 1 < rows;
#pragma unroll 2
            for (int k = lane; k < nh; k += 32) {
                const float2 c = R[k * rs + l], d = R[(k == 0 ? 0 : n - k) * rs + l];
                // the spectra of the real and the imaginary part
                out[r * nh + k] = make_float2(0.5f * (c.x + d.x), 0.5f * (c.y - d.y));
                if (two) out[(r + 1) * nh + k] = make_float2(0.5f * (c.y + d.y), 0.5f * (d.x - c.x));
            }
        }
    }
}

// x lines inverse (forward transform of swapped values, swapped back on the way out)
template <bool CPLX, class ST>
__global__ void __launch_bounds__(FFT_THREADS) k_fft_x_inverse(FftPlan P, int lg, long long rows, int nh,
                                                               const float2* __restrict__ in, ST st,
                                                               const double* done) {
    pdl_enter();
    if (*done != 0.0) return;
    st.begin();
    const int TX = 1 << lg, rs = TX + 1, n = P.n;
    const float2* tw = fft_smem_tables(P);
    float2* A = const_cast<float2*>(tw) + n;
    float2* Bf = A + n * rs;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const long long row0 = (long long)blockIdx.x * TX * (CPLX ? 1 : 2);
    for (int l = warp; l < TX; l += nw) {
        if constexpr (CPLX) {
            const long long r = row0 + l;
            if (r >= rows) continue;
#pragma unroll 4
            for (int k = lane; k < n; k += 32) {
                const float2 v = in[r * nh + k];
                A[k * rs + l] = make_float2(v.y, v.x);
            }
        } else {
            const long long r = row0 + 2 * l;
            if (r >= rows) continue;
            const bool two = r + 1 < rows;
#pragma unroll 4
            for (int k = lane; k < nh; k += 32) {
                float2 a = in[r * nh + k], b = two ? in[(r + 1) * nh + k] : make_float2(0.f, 0.f);
                const int m = k == 0 ? 0 : n - k;
                if (m == k) a.y = b.y = 0.f;   // the spectrum of a real row is real there
                // a + i b at k, conj(a) + i conj(b) at n - k, real and imaginary part swapped
                A[k * rs + l] = make_float2(a.y + b.x, a.x - b.y);
                if (m != k) A[m * rs + l] = make_float2(b.x - a.y, a.x + b.y);
            }
        }
    }
    const float2* R = fft_tile(P, A, Bf, tw, rs, 1, FftPow2{lg});
    for (int l = warp; l < TX; l += nw) {
        if constexpr (CPLX) {
            const long long r = row0 + l;
            if (r >= rows) continue;
#pragma unroll 4
            for (int i = lane; i < n; i += 32) {
                const float2 v = R[i * rs + l];
                st.put(r * n + i, make_float2(v.y, v.x));
            }
        } else {
            const long long r = row0 + 2 * l;
            if (r >= rows) continue;
            const bool two = r + 1 < rows;
#pragma unroll 4
            for (int i = lane; i < n; i += 32) {
                const float2 v = R[i * rs + l];
                st.put(r * n + i, v.y);
                if (two) st.put((r + 1) * n + i, v.x);
            }
        }
    }
}

// y lines: column c of `cols` starts at (c / group) * gstride + c % group, its points are `stride`
// apart (group = nh, gstride = n2 nh, stride = nh)
struct FftCols {
    long long cols, group, gstride, stride;
};

// The points of this thread's column in global memory, real and imaginary part swapped or not;
// columns beyond the last read zeros and store nothing
struct FftGlobal {
    float2* p;
    long long stride;
    bool act, swap;
    __device__ float2 operator()(int, int i) const {
        if (!act) return make_float2(0.f, 0.f);
        const float2 v = p[i * stride];
        return swap ? make_float2(v.y, v.x) : v;
    }
    __device__ void operator()(int, int i, float2 v) const {
        if (act) p[i * stride] = swap ? make_float2(v.y, v.x) : v;
    }
};

// Whether a tile's first step reads and its last step writes global memory, so that a transform of
// two steps passes shared memory once (320^3: y 83 -> 51 us, z 115 -> 86; 192^3 complex 28 -> 18 and
// 41 -> 35; 96^3: y 4.4 -> 3.6).  Not with a prime factor above 10, and not where the steps have fewer
// than 128 butterflies per tile: there all threads copying is the shorter chain (96^3 in tiles of 8
// lines: z 7.0 against 5.6 us).
__device__ __forceinline__ bool fft_straight(const FftPlan& P, int lg) {
    return P.unrolled && P.nst > 1 && (P.T[0] << lg) >= 128;
}

// A tile's lines from global memory and back.  tile: two tiles.
__device__ __forceinline__ void fft_lines(const FftPlan& P, const FftGlobal& G, float2* tile, const float2* tw,
                                          int lg) {
    const int t = threadIdx.x, nt = blockDim.x, rs = 1 << lg, line = t & (rs - 1);
    float2 *A = tile, *B = tile + (P.n << lg);
    if (fft_straight(P, lg)) {
        fft_step(P, 0, G, FftTile{A, rs}, tw, FftPow2{lg}, t, nt);
        __syncthreads();
        for (int st = 1; st + 1 < P.nst; ++st) {
            fft_step(P, st, FftTile{A, rs}, FftTile{B, rs}, tw, FftPow2{lg}, t, nt);
            __syncthreads();
            float2* x = A;
            A = B;
            B = x;
        }
        fft_step(P, P.nst - 1, FftTile{A, rs}, G, tw, FftPow2{lg}, t, nt);
    } else {
#pragma unroll 4
        for (int i = t >> lg; i < P.n; i += nt >> lg) A[(i << lg) + line] = G(line, i);
        const float2* R = fft_tile(P, A, B, tw, rs, 1, FftPow2{lg});
        for (int i = t >> lg; i < P.n; i += nt >> lg) G(line, i, R[(i << lg) + line]);
    }
}

// (one kernel for both directions: each launch starts with a cold instruction cache)
__global__ void __launch_bounds__(FFT_THREADS) k_fft_y(FftPlan P, int lg, FftCols C, float2* F, bool inverse,
                                                       const double* done) {
    pdl_enter();
    if (*done != 0.0) return;
    const float2* tw = fft_smem_tables(P);
    const long long col = ((long long)blockIdx.x << lg) + (threadIdx.x & ((1 << lg) - 1));
    const long long grp = col / C.group, base = grp * C.gstride + (col - grp * C.group);
    fft_lines(P, FftGlobal{F + base, C.stride, col < C.cols, inverse}, const_cast<float2*>(tw) + P.n, tw, lg);
}

// symbol of the inverse: kind 0: 1 / l (0 for the constant mode); 1: 1 / (l + s1);
// 2: (l + s0) / (l + s1)^2; 3: 1 / (a l + Q), 0 where |a l + Q|^2 <= s0.  norm = 1 / (n1 n2 n3).
// s0 of kind 3 is (2^-20 S)^2, S = |a| l_max + |Q|: a symbol below that is known in FP32, to a few 2^-24
// of S, with less than two digits, and the FP32 rounding of a solution that holds S / |a l + Q| times the
// residual changes the residual by more than 1/16: such a mode, which could make a pass raise the
// residual by orders, is left to the Krylov solvers.
struct FftFilter {
    int kind;
    float a, qr, qi, s0, s1, norm;
    const float *lx, *ly, *lz;
    // v times the symbol at eigenvalue l, real and imaginary part swapped
    __device__ __forceinline__ float2 apply(float l, float2 v) const {
        if (kind == 3) {
            const float dr = fmaf(a, l, qr), di = qi;
            const float den = fmaf(dr, dr, di * di);
            const float m = den > s0 ? norm / den : 0.f;
            const float gr = dr * m, gi = -di * m;
            return make_float2(gr * v.y + gi * v.x, gr * v.x - gi * v.y);
        }
        float m;
        if (kind == 0) {
            m = l > 0.f ? norm / l : 0.f;
        } else {
            const float q = 1.f / (l + s1);
            m = norm * q;
            if (kind == 2) m *= (l + s0) * q;
        }
        return make_float2(m * v.y, m * v.x);
    }
};

// z lines: forward (plan P), times the symbol, inverse (plan Q, the radices of P reversed: its first
// step starts from the results the last step of P leaves in registers)
__global__ void __launch_bounds__(FFT_THREADS) k_fft_z_filter(FftPlan P, FftPlan Q, int lg, long long cols, int nh,
                                                              float2* F, FftFilter f, const double* done) {
    pdl_enter();
    if (*done != 0.0) return;
    const float2* tw = fft_smem_tables(P);
    float2* A = const_cast<float2*>(tw) + P.n;
    float2* B = A + (P.n << lg);
    const int t = threadIdx.x, nt = blockDim.x, rs = 1 << lg, line = t & (rs - 1);
    const long long col = ((long long)blockIdx.x << lg) + line;
    const bool act = col < cols;
    const int ky = act ? (int)(col / nh) : 0, kx = act ? (int)(col - (long long)ky * nh) : 0;
    const float lxy = f.lx[kx] + f.ly[ky];
    const FftGlobal in{F + col, cols, act, false};
    const FftGlobal out{F + col, cols, act, true};
    auto filter = [&](int i, float2 v) { return f.apply(lxy + f.lz[i], v); };
    auto swap_tiles = [&]() {
        __syncthreads();
        float2* x = A;
        A = B;
        B = x;
    };
    if (fft_straight(P, lg)) {
        fft_step(P, 0, in, FftTile{B, rs}, tw, FftPow2{lg}, t, nt);
        swap_tiles();
        for (int st = 1; st + 1 < P.nst; ++st) {
            fft_step(P, st, FftTile{A, rs}, FftTile{B, rs}, tw, FftPow2{lg}, t, nt);
            swap_tiles();
        }
        fft_turn_step(P, FftTile{A, rs}, filter, FftTile{B, rs}, tw, FftPow2{lg}, t, nt);
        swap_tiles();
        for (int st = 1; st + 1 < Q.nst; ++st) {
            fft_step(Q, st, FftTile{A, rs}, FftTile{B, rs}, tw, FftPow2{lg}, t, nt);
            swap_tiles();
        }
        fft_step(Q, Q.nst - 1, FftTile{A, rs}, out, tw, FftPow2{lg}, t, nt);
    } else {
#pragma unroll 4
        for (int i = t >> lg; i < P.n; i += nt >> lg) A[(i << lg) + line] = in(line, i);
        for (int pass = 0; pass < 2; ++pass) {
            float2* R = fft_tile(P, A, B, tw, rs, 1, FftPow2{lg});
            for (int i = t >> lg; i < P.n; i += nt >> lg) {
                const float2 v = R[(i << lg) + line];
                if (pass) out(line, i, v);
                else R[(i << lg) + line] = filter(i, v);
            }
            B = R == A ? B : A;
            A = R;
        }
    }
}

// ------------------------------------------------------------------- x and y in one launch
// A z plane per block, for planes whose two buffers fit shared memory: the x lines (real: pairs of
// rows) and then the y lines of the half spectrum without a pass over global memory between.
constexpr int FFT_PLANE_THREADS = 512;

struct FftPlane {
    FftPlan px, py;
    FftAny mx, my;      // lines of the two phases
    int rx, ry;         // strides of a point: x phase [i][line], y phase [row][k]
    int buf;            // points of one buffer
    int n2, nh;
};

template <bool CPLX, class LD>
__global__ void __launch_bounds__(FFT_PLANE_THREADS) k_fft_xy_forward(FftPlane G, LD ld, float2* __restrict__ out,
                                                                      const double* done) {
    pdl_enter();
    if (*done != 0.0) return;
    ld.begin();
    const int n1 = G.px.n, n2 = G.n2, nh = G.nh;
    float2* tx = fft_smem_tables(G.px);
    float2* ty = tx + n1;
    for (int k = threadIdx.x; k < n2; k += blockDim.x) ty[k] = G.py.tw[k];
    float2 *A = ty + n2, *B = A + G.buf;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const long long row0 = (long long)blockIdx.x * n2;
    for (int l = warp; l < G.mx.m; l += nw) {
        const long long r = CPLX ? row0 + l : row0 + 2 * l;
        const bool two = !CPLX && 2 * l + 1 < n2;
#pragma unroll 4
        for (int i = lane; i < n1; i += 32) {
            if constexpr (CPLX) A[i * G.rx + l] = ld.at(r * n1 + i);
            else A[i * G.rx + l] = make_float2(ld.at(r * n1 + i), two ? ld.at((r + 1) * n1 + i) : 0.f);
        }
    }
    float2* R = fft_tile(G.px, A, B, tx, G.rx, 1, G.mx);
    float2* Y = R == A ? B : A;
    const float2* Z;
    int zi, zl;   // strides of a row and of k in Z
    if constexpr (CPLX) {   // the x phase's lines are the y phase's points
        Z = fft_tile(G.py, R, Y, ty, 1, G.rx, G.my);
        zi = 1;
        zl = G.rx;
    } else {
        for (int l = warp; l < G.mx.m; l += nw)
            for (int k = lane; k < nh; k += 32) {
                const float2 c = R[k * G.rx + l], d = R[(k == 0 ? 0 : n1 - k) * G.rx + l];
                Y[2 * l * G.ry + k] = make_float2(0.5f * (c.x + d.x), 0.5f * (c.y - d.y));
                if (2 * l + 1 < n2) Y[(2 * l + 1) * G.ry + k] = make_float2(0.5f * (c.y + d.y), 0.5f * (d.x - c.x));
            }
        Z = fft_tile(G.py, Y, R, ty, G.ry, 1, G.my);
        zi = G.ry;
        zl = 1;
    }
    for (int j = warp; j < n2; j += nw)
#pragma unroll 4
        for (int k = lane; k < nh; k += 32) out[(row0 + j) * nh + k] = Z[j * zi + k * zl];
}

template <bool CPLX, class ST>
__global__ void __launch_bounds__(FFT_PLANE_THREADS) k_fft_xy_inverse(FftPlane G, const float2* __restrict__ in, ST st,
                                                                      const double* done) {
    pdl_enter();
    if (*done != 0.0) return;
    st.begin();
    const int n1 = G.px.n, n2 = G.n2, nh = G.nh;
    float2* tx = fft_smem_tables(G.px);
    float2* ty = tx + n1;
    for (int k = threadIdx.x; k < n2; k += blockDim.x) ty[k] = G.py.tw[k];
    float2 *A = ty + n2, *B = A + G.buf;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const long long row0 = (long long)blockIdx.x * n2;
    const int zi = CPLX ? 1 : G.ry, zl = CPLX ? G.rx : 1;   // complex: already the x phase's tile
    for (int j = warp; j < n2; j += nw)
#pragma unroll 4
        for (int k = lane; k < nh; k += 32) {
            const float2 v = in[(row0 + j) * nh + k];
            A[j * zi + k * zl] = make_float2(v.y, v.x);
        }
    float2* R = fft_tile(G.py, A, B, ty, zi, zl, G.my);
    float2* X = R == A ? B : A;
    const float2* Z;
    if constexpr (CPLX) {
        Z = fft_tile(G.px, R, X, tx, G.rx, 1, G.mx);
    } else {
        for (int l = warp; l < G.mx.m; l += nw)
            for (int k = lane; k < nh; k += 32) {
                float2 a = R[2 * l * G.ry + k];   // swapped
                float2 b = 2 * l + 1 < n2 ? R[(2 * l + 1) * G.ry + k] : make_float2(0.f, 0.f);
                const int m = k == 0 ? 0 : n1 - k;
                if (m == k) a.x = b.x = 0.f;      // the spectrum of a real row is real there
                X[k * G.rx + l] = make_float2(a.x + b.y, a.y - b.x);
                if (m != k) X[m * G.rx + l] = make_float2(b.y - a.x, a.y + b.x);
            }
        Z = fft_tile(G.px, X, R, tx, G.rx, 1, G.mx);
    }
    for (int l = warp; l < G.mx.m; l += nw) {
        const long long r = CPLX ? row0 + l : row0 + 2 * l;
        const bool two = !CPLX && 2 * l + 1 < n2;
#pragma unroll 4
        for (int i = lane; i < n1; i += 32) {
            const float2 v = Z[i * G.rx + l];
            if constexpr (CPLX) {
                st.put(r * n1 + i, make_float2(v.y, v.x));
            } else {
                st.put(r * n1 + i, v.y);
                if (two) st.put((r + 1) * n1 + i, v.x);
            }
        }
    }
}

// ------------------------------------------------------------------------------- host
// raises a kernel's dynamic shared memory limit where it needs that (once per thread and device)
static void allow_smem(of_grid* g, const void* kernel, size_t smem) {
    if (smem <= 40 * 1024) return;
    static thread_local std::vector<std::pair<const void*, int>> raised;
    const std::pair<const void*, int> key(kernel, g->device);
    if (std::find(raised.begin(), raised.end(), key) != raised.end()) return;
    OF_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
    raised.push_back(key);
}

// x and y share a launch for planes of at most this shared memory (real 72^2, complex 52^2), of
// which there are at least 16: two launches less pay while a launch is all latency (Poisson solve
// 24^3 119 -> 106 us, 32^3 118 -> 109, 45 x 50 x 54 139 -> 131), but one block per plane leaves SMs idle
// that the larger planes need (96^3 198 -> 202).
constexpr size_t FFT_PLANE_SMEM = 48 * 1024;
constexpr int FFT_MIN_PLANES = 16;

// log2 of the lines per tile: 16 while four blocks per SM fit beside each other in shared memory
// (56 KB each) and every SM has one, else 8, and 4 for very long lines or very few.  320^3: x
// 93 / 231 -> 72 / 142 us, y 118 -> 83, z 167 -> 115 from 16 to 8 lines; 192^3 complex: y 28, z 41 with
// 16, 32 and 45 with 8.  8 lines below four blocks per SM took the x lines of one 96^3 solve from
// 5.5 / 6.3 to 4.8 / 5.3 us but 12 cells on eight streams from 1.87 to 2.09 ms.
static int tile_lg(int n, long long lines) {
    const long long sms = num_sms();
    if (n * 35LL * (long long)sizeof(float2) <= 56 * 1024 && (lines >> 4) >= sms) return 4;
    return n <= 1024 && (lines >> 3) >= sms ? 3 : 2;
}

template <bool CPLX, class LD, class ST>
static void fft_apply(of_grid* g, LD ld, ST st, FftFilter f, const double* done) {
    Fft& T = fft_tables(g);
    const Dims& d = g->d;
    const int nh = CPLX ? d.n1 : d.n1 / 2 + 1;
    const long long rows = (long long)d.n2 * d.n3;
    float2* F = (float2*)ws(g, WS_FFT, sizeof(float2) * (size_t)rows * nh);
    f.norm = (float)(1.0 / (double)d.n);
    f.lx = T.sym[0];
    f.ly = T.sym[1];
    f.lz = T.sym[2];
    const double word = 4.0 * (CPLX ? 2 : 1) * (double)d.n;
    ProfScope ps(g, PC_FFT, 10.0 * word + 3.0 * 2.0 * word);
    auto blocks = [](long long lines, int lg) { return (unsigned)((lines + (1 << lg) - 1) >> lg); };
    // x forward
    const long long xl = CPLX ? rows : (rows + 1) / 2;
    const int lgx = tile_lg(d.n1, xl), lgy = tile_lg(d.n2, (long long)nh * d.n3), lgz = tile_lg(d.n3, (long long)nh * d.n2);
    const size_t sx = sizeof(float2) * (size_t)d.n1 * (1 + 2 * ((1 << lgx) + 1));
    const size_t sy = sizeof(float2) * (size_t)d.n2 * (1 + 2 * (1 << lgy));
    const size_t sz = sizeof(float2) * (size_t)d.n3 * (1 + 2 * (1 << lgz));
    const FftCols cy{(long long)nh * d.n3, nh, (long long)d.n2 * nh, nh};
    const long long zc = (long long)nh * d.n2;
    allow_smem(g, (const void*)k_fft_x_forward<CPLX, LD>, sx);
    allow_smem(g, (const void*)k_fft_x_inverse<CPLX, ST>, sx);
    allow_smem(g, (const void*)k_fft_y, sy);
    allow_smem(g, (const void*)k_fft_z_filter, sz);
    FftPlane G;
    G.px = T.plan[0];
    G.py = T.plan[1];
    G.mx.m = CPLX ? d.n2 : (d.n2 + 1) / 2;
    G.my.m = G.nh = nh;
    G.n2 = d.n2;
    for (FftAny* m : {&G.mx, &G.my}) m->magic = m->m == 1 ? 0u : (unsigned)((1ull << 32) / (unsigned)m->m + 1);
    G.rx = G.mx.m | 1;   // odd: a warp's points of one line fall into different banks
    G.ry = nh | 1;
    const long long buf = CPLX ? (long long)d.n1 * G.rx : std::max((long long)d.n1 * G.rx, (long long)d.n2 * G.ry);
    const size_t sp = sizeof(float2) * (size_t)(d.n1 + d.n2 + 2 * buf);
    G.buf = (int)buf;
    const bool planes = d.n2 > 1 && d.n3 >= FFT_MIN_PLANES && sp <= FFT_PLANE_SMEM &&
                        (long long)d.n1 * G.mx.m < 65536 && (long long)d.n2 * nh < 65536;
    if (planes) {
        allow_smem(g, (const void*)k_fft_xy_forward<CPLX, LD>, sp);
        allow_smem(g, (const void*)k_fft_xy_inverse<CPLX, ST>, sp);
        launch_pdl(k_fft_xy_forward<CPLX, LD>, d.n3, FFT_PLANE_THREADS, sp, g->stream, G, ld, F, done);
    } else {
        launch_pdl(k_fft_x_forward<CPLX, LD>, blocks(xl, lgx), FFT_THREADS, sx, g->stream, T.plan[0], lgx, rows, nh, ld, F, done);
        if (d.n2 > 1)
            launch_pdl(k_fft_y, blocks(cy.cols, lgy), FFT_THREADS, sy, g->stream, T.plan[1], lgy, cy, F, false, done);
    }
    launch_pdl(k_fft_z_filter, blocks(zc, lgz), FFT_THREADS, sz, g->stream, T.plan[2], T.z_back, lgz, zc, nh, F, f, done);
    if (planes) {
        launch_pdl(k_fft_xy_inverse<CPLX, ST>, d.n3, FFT_PLANE_THREADS, sp, g->stream, G, (const float2*)F, st, done);
    } else {
        if (d.n2 > 1)
            launch_pdl(k_fft_y, blocks(cy.cols, lgy), FFT_THREADS, sy, g->stream, T.plan[1], lgy, cy, F, true, done);
        launch_pdl(k_fft_x_inverse<CPLX, ST>, blocks(xl, lgx), FFT_THREADS, sx, g->stream, T.plan[0], lgx, rows, nh,
                   (const float2*)F, st, done);
    }
}

void fft_correct(of_grid* g, const double* r, double* x, const KState* st) {
    FftFilter f{};
    fft_apply<false>(g, LdReal64{r, st, 0}, StAccum64{x, st, 0}, f, &st->done);
}

void fft_correct_shifted(of_grid* g, const double2* r, double2* x, double a, double2 Q, const KState* st) {
    FftFilter f{};
    f.kind = 3;
    f.a = (float)a;
    f.qr = (float)Q.x;
    f.qi = (float)Q.y;
    const double least = std::ldexp(std::fabs(a) * fft_tables(g).lmax + std::hypot(Q.x, Q.y), -20);
    f.s0 = (float)(least * least);
    fft_apply<true>(g, LdCplx64{r, st, 0}, StAccumCplx64{x, st, 0}, f, &st->done);
}

void fft_inverse_real(of_grid* g, const float* r, float* z, double shift, double low, const double* done) {
    FftFilter f{};
    f.kind = low > 0.0 ? 2 : 1;
    f.s0 = (float)low;
    f.s1 = (float)shift;
    fft_apply<false>(g, LdReal32{r}, StReal32{z}, f, done);
}

}  // namespace of
