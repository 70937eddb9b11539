// FP64 Laplacian sweeps summed exactly in 64-bit fixed point on the integer pipes.
//
// GB300 issues 2 FP64 operations per clock and SM but 60 mad.wide.s32 (32 x 32 + 64 bits): the
// order-12 sum of an FP64 field, 37 FP64 operations per point, is bound by the FP64 pipe at
// 13 GPts/s.  The weights of Eq. FD:Laplacian are integers over a common denominator,
//   N = 6: w_p h^2 = {1425600, -222750, 44000, -7425, 864, -50} / 831600, centre -2480478 / 831600,
// so with the field in fixed point, X = x 2^k in 60 bits, the sum over the neighbours is an exact
// integer sum, each weight multiplying the two 32-bit limbs of the 64-bit sum of the neighbours
// at its distance (six with equal spacings, two else): about 8 integer operations per distance and
// no FP64 operation until one conversion and one multiplication per point (per axis when the
// spacings differ).
//
// Brick of 16 units x 8 rows x 8 planes per block of 128 threads, a unit being two neighbouring
// doubles of a row (two real points, or one complex point).  The brick and its x-y halo are staged
// once in shared memory as fixed point; each thread takes the z halo of its own column straight
// from global memory.  The block's range is 4/3 or more of the largest of its z halo and of eight
// staged rows spread over the brick, and is set anew, from all values, where a staged one lies beyond
// it; a value that is not finite makes the block take FP64 arithmetic instead.  So does every point
// whose own value and whose six next ones (in z those of the brick) are all below 2^53 units of the
// fixed point (2^-7 of its range), where 60 bits would keep fewer than the 53 of FP64.  At the others a staged value is cut off by at most 2^-53 of the largest of those
// seven, and the sum is no less accurate than the FP64 one (on random and smooth stencils just above
// the limit the RMS error is 0.3 .. 1 of it at orders 6 and 12, up to 1.5 at order 2 where the centre
// alone is small).  A complex value counts by the larger of its parts.  Ordinary fields take the integer
// path but for a few points where value and slope are small together (about ten in an electrostatic
// potential on 96^3), fields that fall by powers of ten across a brick take FP64 arithmetic.
//
// Measured on a GB300 (order 12): 96^3 69.1 us in FP64 arithmetic -> 12.9, 192^3 514 -> 99, 320^3 2.4 ms ->
// 0.43 (76 GPts/s), of which the looks at each point's neighbours, and the code they add, are 0.3, 8 and 40 us;
// where nearly every
// point takes FP64 arithmetic after all (a Gaussian in the middle of 96^3) 69.  Bound by instruction issue
// and latency at 12 warps per SM (168 registers; 4.9 staged values per point with their conversions, ~8
// integer operations per distance).  Tried before the looks (12.7 us, 80 GPts/s at 320^3): both loads and
// conversions of two slots in flight 13.8 us / 74 GPts/s (spills), two blocks per SM without spills
// 16.1 / 80, 4 planes per brick 16.1 / 70, 16 rows 16.3 / 81, 16 rows of 4 planes 18.2 / 69.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "of_stencil.cuh"

namespace of {

#define OF_FIX_HD __host__ __device__ __forceinline__

// W_p (p = 0: the centre, once per axis) and the common denominator
template <int N> OF_FIX_HD constexpr int fix_weight(int p) {
    if (N == 1) return p == 0 ? -2 : 1;
    if (N == 3) return p == 0 ? -490 : p == 1 ? 270 : p == 2 ? -27 : 2;
    return p == 0 ? -2480478 : p == 1 ? 1425600 : p == 2 ? -222750 : p == 3 ? 44000 : p == 4 ? -7425 : p == 5 ? 864 : -50;
}
// low bits left out of the integer sum's conversion: the sum is at most 2^60 times the 12, 3264 or
// 17.6e6 of three axes' absolute weights, below 2^(63 + SH)
OF_FIX_HD constexpr int fix_shift(int N) { return N == 1 ? 2 : N == 3 ? 10 : 22; }
inline double fix_denominator(int N) { return N == 1 ? 1.0 : N == 3 ? 180.0 : 831600.0; }

// double -> fixed point with exponent E (biased, >= 128): the mantissa as a 60-bit integer shifted
// right by E - e (towards zero), in units of 2^(E - 1082); |x| < 2^(E - 1022).  Subnormals are 0.
OF_FIX_HD long long fix_from_bits(int hi, unsigned lo, int E) {
    const int e = (hi >> 20) & 0x7ff;
    const unsigned long long m = ((unsigned long long)(((unsigned)hi & 0xfffffu) | 0x100000u) << 32) | lo;
    const int s = E - e < 63 ? E - e : 63;   // 63 leaves nothing of 60 bits
    const long long v = (long long)((m << 7) >> s), sign = (long long)(hi >> 31);
    return (v ^ sign) - sign;
}

// magnitude of v's high word: |v| > 2^53 - 2^32 where it is at least FIX_FINE
OF_FIX_HD unsigned fix_mag(long long v) {
    const int h = (int)(v >> 32);
    return (unsigned)(h < 0 ? -h : h);
}
constexpr unsigned FIX_FINE = 1u << 21;

// A sum s of neighbours (64 bits) times W, by its two 32-bit limbs: the sum of W s is h 2^32 + p - n
struct FixAcc {
    long long h = 0;
    unsigned long long p = 0, n = 0;
    OF_FIX_HD void add(long long s, int W) {
        const int hi = (int)(s >> 32);
        const unsigned lo = (unsigned)s;
        h += (long long)hi * W;
        if (W > 0) p += (unsigned long long)lo * (unsigned)W;
        else n += (unsigned long long)lo * (unsigned)(-W);
    }
    // the sum times 2^-SH, rounded to FP64; 2^(63 + SH) is above the largest sum
    template <int SH>
    OF_FIX_HD double value() const {
        const long long lo = (long long)(p - n);
        const long long t = h + (lo >> 32);
        return (double)(long long)(((unsigned long long)t << (32 - SH)) | ((unsigned long long)(unsigned)lo >> SH));
    }
};

// A sweep's field: a plain one (op.field()), or one the op forms on load, two doubles at a time
// (op.pair(i0, i1, vec), neighbours or, vec, one 16-byte load; op.bits(): the OR of its addresses).
template <class Op, class = void>
struct HasPair { static constexpr bool value = false; };
template <class Op>
struct HasPair<Op, decltype((void)std::declval<const Op&>().pair(0u, 0u, true), void())> {
    static constexpr bool value = true;
};
__device__ __forceinline__ double2 fix_pair(const double* x, unsigned i0, unsigned i1, bool vec) {
    if (vec) return *reinterpret_cast<const double2*>(x + i0);
    return make_double2(x[i0], x[i1]);
}
template <class Op>
__device__ __forceinline__ double2 fix_load(const Op& op, unsigned i0, unsigned i1, bool vec) {
    if constexpr (HasPair<Op>::value) return op.pair(i0, i1, vec);
    else return fix_pair(op.field(), i0, i1, vec);
}
// What an op reads beside the field at a unit's points (op.pre(i, act0, act1), two neighbouring points
// of a real field or one of a complex one): loaded a plane ahead, for op.store_pre.
template <class Op, class = void>
struct HasPre { static constexpr bool value = false; };
template <class Op>
struct HasPre<Op, decltype((void)std::declval<const Op&>().pre(0LL, true, true), void())> {
    static constexpr bool value = true;
};
template <class Op>
uintptr_t fix_bits(const Op& op) {
    if constexpr (HasPair<Op>::value) return op.bits();
    else return (uintptr_t)op.field();
}

constexpr int FX_UX = 16, FX_BY = 8, FX_THREADS = FX_UX * FX_BY;
// Units of a warp that its lanes take together in FP64 arithmetic.  Eight in the complex Krylov sweep: its tile
// (72 KB) and its two sums leave three blocks per SM 592 bytes more each (with 32 units, at two blocks, FP64
// COCG on 192^3 took 36.8 ms instead of 33.5).
template <bool CPLX, class Op> constexpr int fix_items() { return CPLX && !HasPre<Op>::value ? 8 : 32; }

struct FixScale {
    double s[3];   // 2^fix_shift / (D h_a^2)
};

template <int N, bool CPLX>
constexpr int fix_row_width() { return 32 + 2 * (CPLX ? 2 * N : ((N + 1) & ~1)); }
template <int N, bool CPLX, int BZ>
constexpr size_t fix_smem_bytes() {
    return sizeof(long long) * (size_t)BZ * (FX_BY + 2 * N) * fix_row_width<N, CPLX>();
}

// The Laplacian at the planes k < nz of a thread's two columns, from the fixed-point column (z) and
// tile (own: this unit's first value in the tile's first plane): put(k, l0, l1), after
// ahead(k + 1).  With equal
// spacings the six neighbours at distance p are summed before the two multiplications by W_p
// (s0 = s1 = s2); else each axis has its sum and its scale.
template <int N, bool CPLX, bool ISO, int BZ, class Ahead, class Put>
__device__ __forceinline__ void fix_planes(const longlong2 (&col)[BZ + 2 * N], const long long* own, int nz, double s0,
                                           double s1, double s2, Ahead&& ahead, Put&& put) {
    constexpr int RW = fix_row_width<N, CPLX>(), CPL = (FX_BY + 2 * N) * RW, SH = fix_shift(N);
    constexpr int HX = (N + 1) & ~1;
#pragma unroll
    for (int k = 0; k < BZ; ++k) {
        if (k >= nz) break;
        ahead(k + 1);
        const long long* b = own + k * CPL;
        const longlong2 c = col[N + k];
        long long xv[2 * HX + 2];   // real: row values -HX .. HX + 1 around the unit
        if constexpr (!CPLX) {
#pragma unroll
            for (int m = 0; m <= HX; ++m) {
                const longlong2 t = *reinterpret_cast<const longlong2*>(b - HX + 2 * m);
                xv[2 * m] = t.x;
                xv[2 * m + 1] = t.y;
            }
        }
        auto xsum = [&](int p) {
            if constexpr (CPLX) {
                const longlong2 u = *reinterpret_cast<const longlong2*>(b + 2 * p);
                const longlong2 v = *reinterpret_cast<const longlong2*>(b - 2 * p);
                return make_longlong2(u.x + v.x, u.y + v.y);
            } else {
                return make_longlong2(xv[HX + p] + xv[HX - p], xv[HX + 1 + p] + xv[HX + 1 - p]);
            }
        };
        auto ysum = [&](int p) {
            const longlong2 u = *reinterpret_cast<const longlong2*>(b + p * RW);
            const longlong2 v = *reinterpret_cast<const longlong2*>(b - p * RW);
            return make_longlong2(u.x + v.x, u.y + v.y);
        };
        auto zsum = [&](int p) {
            return make_longlong2(col[N + k + p].x + col[N + k - p].x, col[N + k + p].y + col[N + k - p].y);
        };
        double l0 = 0.0, l1 = 0.0;
        if constexpr (ISO) {
            FixAcc a0, a1;
            a0.add(c.x, 3 * fix_weight<N>(0));
            a1.add(c.y, 3 * fix_weight<N>(0));
#pragma unroll
            for (int p = 1; p <= N; ++p) {
                const longlong2 x = xsum(p), y = ysum(p), z = zsum(p);
                a0.add(x.x + y.x + z.x, fix_weight<N>(p));
                a1.add(x.y + y.y + z.y, fix_weight<N>(p));
            }
            l0 = s0 * a0.template value<SH>();
            l1 = s0 * a1.template value<SH>();
        } else {
            auto axis = [&](auto&& sum, double s) {
                FixAcc a0, a1;
                a0.add(c.x, fix_weight<N>(0));
                a1.add(c.y, fix_weight<N>(0));
#pragma unroll
                for (int p = 1; p <= N; ++p) {
                    const longlong2 t = sum(p);
                    a0.add(t.x, fix_weight<N>(p));
                    a1.add(t.y, fix_weight<N>(p));
                }
                l0 = fma(s, a0.template value<SH>(), l0);
                l1 = fma(s, a1.template value<SH>(), l1);
            };
            axis(xsum, s0);
            axis(ysum, s1);
            axis(zsum, s2);
        }
        put(k, l0, l1);
    }
}

// Those of the planes `small` (bits), in which the thread's unit is below `least`, in which a point of
// it and its six neighbours all are; the neighbours in z only within the brick.
template <int N, bool CPLX, int BZ>
__device__ __forceinline__ unsigned fix_coarse(const long long* own, unsigned small, unsigned least) {
    constexpr int RW = fix_row_width<N, CPLX>(), CPL = (FX_BY + 2 * N) * RW;
    unsigned coarse = 0;
#pragma unroll 1
    for (; small; small &= small - 1u) {
        const int k = __ffs((int)small) - 1;
        const long long* b = own + k * CPL;
        unsigned m0 = 0, m1 = 0;
        auto near = [&](const long long* p) {
            const longlong2 v = *reinterpret_cast<const longlong2*>(p);
            m0 |= fix_mag(v.x);
            m1 |= fix_mag(v.y);
        };
        near(b + RW);
        near(b - RW);
        near(k + 1 < BZ ? b + CPL : b);
        near(k > 0 ? b - CPL : b);
        if constexpr (CPLX) {
            near(b + 2);
            near(b - 2);
            m0 = m1 = m0 | m1;
        } else {
            m0 |= fix_mag(b[-1]);
            m1 |= fix_mag(b[2]);
        }
        coarse |= min(m0, m1) < least ? 1u << k : 0u;
    }
    return coarse;
}

// One sweep over this block's bricks: op.store or op.store_pre at every point.
template <int N, bool CPLX, bool ISO, int BZ, class Op>
__device__ __forceinline__ void fix_sweep(const Dims& d, const Weights<double>& W, const FixScale& fs, bool vec, int bx,
                                          int by, int bricks, Op& op) {
    constexpr int HX = CPLX ? 2 * N : ((N + 1) & ~1);   // staged halo doubles each side in x
    constexpr int RW = fix_row_width<N, CPLX>();
    constexpr int ROWS = FX_BY + 2 * N;
    constexpr int CPL = ROWS * RW;
    // slots: the core columns of every staged row (16 chunks of two doubles), then the x halo of the
    // core rows (PH lanes per side, of which HX / 2 hold a chunk)
    constexpr int PH = (HX / 2 + 3) / 4 * 4;
    constexpr int SLOTS = ROWS * FX_UX + FX_BY * 2 * PH;
    constexpr int SPT = (SLOTS + FX_THREADS - 1) / FX_THREADS;
    constexpr int ITEMS = fix_items<CPLX, Op>();
    constexpr bool ALL = SPT * BZ <= 8;   // thin bricks: every slot's loads in flight at once
    extern __shared__ __align__(16) long long fix_smem[];
    __shared__ int yoff[ROWS], zoff[BZ + 2 * N], xoff[RW];   // periodic offsets in doubles (< 2^31)
    __shared__ int wtop[2][FX_THREADS / 32];
    __shared__ unsigned char items[FX_THREADS / 32][ITEMS];
    __shared__ __align__(16) double2 taken[FX_THREADS / 32][ITEMS];
    const int tx = threadIdx.x, ty = threadIdx.y, tid = tx + FX_UX * ty;
    const int RF = CPLX ? 2 * d.n1 : d.n1, PF = RF * d.n2;
    // Staged row and first column of each of this thread's slots.  The first FX_BY rows of the order
    // are spread evenly over the staged rows, so that the first slot's values (from which, with
    // the z halo, the block's exponent comes) sample the whole brick.
    auto slot = [&](int m, int& row, int& col) {
        const int sl = tid + m * FX_THREADS;
        row = -1;
        col = 0;
        if (sl < ROWS * FX_UX) {
            int j = sl / FX_UX;
            auto spread = [](int i) { return (i * (ROWS - 1) + 3) / (FX_BY - 1); };
            if (j < FX_BY) {
                row = spread(j);
            } else {
                j -= FX_BY;   // the j-th row that is not one of those
                for (int i = 0; i < FX_BY; ++i) j += spread(i) <= j;
                row = j;
            }
            col = HX + 2 * (sl % FX_UX);
        } else if (sl < SLOTS) {
            const int q = sl - ROWS * FX_UX, side = (q / PH) & 1, c = q % PH;
            if (c < HX / 2) {
                row = N + q / (2 * PH);
                col = 2 * c + (side ? HX + 32 : 0);
            }
        }
    };
    int srow[SPT], scol[SPT];
#pragma unroll
    for (int m = 0; m < SPT; ++m) slot(m, srow[m], scol[m]);
    // two doubles of a chunk: one 16-byte load where rows and the field allow it (a chunk
    // starts at an even double and is contiguous across the wrap when rows are even)
    auto load2 = [&](int base, int x0, int x1, bool v) -> double2 {
        return fix_load(op, (unsigned)(base + x0), (unsigned)(base + x1), v);
    };
    auto expo = [](double a) { return (__double2hiint(a) >> 20) & 0x7ff; };

    for (int brick = blockIdx.x; brick < bricks; brick += gridDim.x) {
        const int kb = brick / (bx * by), rem = brick - kb * bx * by, jb = rem / bx, ib = rem - jb * bx;
        const int x0 = ib * 32, y0 = jb * FX_BY, z0 = kb * BZ;
        __syncthreads();   // the previous brick's readers of the tables and the tile
        for (int t = tid; t < BZ + 2 * N; t += FX_THREADS) zoff[t] = wrap_index(z0 - N + t, d.n3) * PF;
        for (int t = tid; t < ROWS; t += FX_THREADS) yoff[t] = wrap_index(y0 - N + t, d.n2) * RF;
        for (int t = tid; t < RW; t += FX_THREADS) {
            if constexpr (CPLX) xoff[t] = 2 * wrap_index((x0 - HX) / 2 + (t >> 1), d.n1) + (t & 1);
            else xoff[t] = wrap_index(x0 - HX + t, d.n1);
        }
        __syncthreads();
        // the z halo of this thread's own column and its first slot in every plane, the sample that the
        // block's exponent comes from
        const int own = yoff[N + ty], oc0 = xoff[HX + 2 * tx], oc1 = xoff[HX + 2 * tx + 1];
        longlong2 col[BZ + 2 * N];
        double2 v[ALL ? SPT : 1][BZ];
        auto load_slot = [&](int m, double2 (&v)[BZ]) {
            if (srow[m] < 0) return;
            const int o = yoff[srow[m]], c0 = xoff[scol[m]], c1 = xoff[scol[m] + 1];
            // (the branch around the loads: in each of them it made the compiler issue both forms)
            if (vec) {
#pragma unroll
                for (int k = 0; k < BZ; ++k) v[k] = load2(zoff[N + k] + o, c0, c1, true);
            } else {
#pragma unroll
                for (int k = 0; k < BZ; ++k) v[k] = load2(zoff[N + k] + o, c0, c1, false);
            }
        };
        double2 zr[2 * N];
        if (vec) {
#pragma unroll
            for (int j = 0; j < 2 * N; ++j) zr[j] = load2(zoff[j < N ? j : j + BZ] + own, oc0, oc1, true);
        } else {
#pragma unroll
            for (int j = 0; j < 2 * N; ++j) zr[j] = load2(zoff[j < N ? j : j + BZ] + own, oc0, oc1, false);
        }
#pragma unroll
        for (int m = 0; m < (ALL ? SPT : 1); ++m) load_slot(m, v[m]);
        auto block_max = [&](int v, int (&slot)[FX_THREADS / 32]) {
            const int w = __reduce_max_sync(0xffffffffu, v);
            if ((tid & 31) == 0) slot[tid >> 5] = w;
            __syncthreads();
            int t = 0;
#pragma unroll
            for (int k = 0; k < FX_THREADS / 32; ++k) t = max(t, slot[k]);
            return t;
        };
        int first = 0;   // the largest exponent and mantissa of the sample
        auto sample = [&](double2 q) {
            first = max(first, max(__double2hiint(q.x) & 0x7fffffff, __double2hiint(q.y) & 0x7fffffff));
        };
#pragma unroll
        for (int j = 0; j < 2 * N; ++j) sample(zr[j]);
#pragma unroll
        for (int m = 0; m < (ALL ? SPT : 1); ++m)
            if (srow[m] >= 0) {
#pragma unroll
                for (int k = 0; k < BZ; ++k) sample(v[m][k]);
            }
        // 2^(E - 1022) is 4/3 of the sample's largest or more; 128: what is that small takes FP64
        int E = max((block_max(first, wtop[0]) + 0x80000) >> 20, 128);
        auto fix = [&](double2 q) {
            return make_longlong2(fix_from_bits(__double2hiint(q.x), (unsigned)__double2loint(q.x), E),
                                  fix_from_bits(__double2hiint(q.y), (unsigned)__double2loint(q.y), E));
        };
        // beyond the sample: the largest exponent; and, where the sample is that small, all values' bits
        int top = 0, bits = 0;
        auto mark = [&](double2 q) {
            bits |= __double2hiint(q.x) | __double2loint(q.x) | __double2hiint(q.y) | __double2loint(q.y);
        };
        if (E == 128) {
#pragma unroll
            for (int j = 0; j < 2 * N; ++j) mark(zr[j]);
        }
#pragma unroll
        for (int m = 0; m < SPT; ++m) {
            double2 (&q)[BZ] = v[ALL ? m : 0];
            if (!ALL && m > 0) load_slot(m, q);
            if (srow[m] >= 0) {
                long long* dst = fix_smem + srow[m] * RW + scol[m];
#pragma unroll
                for (int k = 0; k < BZ; ++k) {
                    if (!ALL && m > 0) top = max(top, max(expo(q[k].x), expo(q[k].y)));
                    *reinterpret_cast<longlong2*>(dst + k * CPL) = fix(q[k]);
                }
                if (E == 128) {
#pragma unroll
                    for (int k = 0; k < BZ; ++k) mark(q[k]);
                }
            }
        }
        // the largest exponent beyond the sample, with 2^16 where a bit is set anywhere (or the sample not small)
        const int all = block_max(top | (bits != 0 || E > 128 ? 1 << 16 : 0), wtop[1]);
        if ((all & 0xffff) > E && (all & 0xffff) <= 2046) {
            // a staged value above the sample's range: once more, with its exponent (a short loop: cold code)
            E = all & 0xffff;
#pragma unroll 1
            for (int m = 0; m < SPT; ++m) {
                int row, c;
                slot(m, row, c);
                if (row < 0) continue;
#pragma unroll 1
                for (int k = 0; k < BZ; ++k) {
                    const int o = zoff[N + k] + yoff[row];
                    *reinterpret_cast<longlong2*>(fix_smem + k * CPL + row * RW + c) =
                        fix(fix_load(op, (unsigned)(o + xoff[c]), (unsigned)(o + xoff[c + 1]), false));
                }
            }
            __syncthreads();
        }
#pragma unroll
        for (int j = 0; j < 2 * N; ++j) col[j < N ? j : j + BZ] = fix(zr[j]);
        const int y = y0 + ty, xe = x0 + 2 * tx;         // first double of this thread's unit
        const bool act0 = y < d.n2 && xe < RF, act1 = act0 && xe + 1 < RF;
        const long long i0 = (long long)y * d.n1 + (CPLX ? xe / 2 : xe);
        const int nz = min(BZ, d.n3 - z0);
        auto fetch = [&](int k) {
            if constexpr (HasPre<Op>::value) return op.pre((long long)(z0 + k) * d.n1 * d.n2 + i0, act0, act1);
            else return 0;
        };
        auto store = [&](int k, auto&& p, double l0, double l1) {
            const long long i = (long long)(z0 + k) * d.n1 * d.n2 + i0;
            if constexpr (HasPre<Op>::value) {
                op.store_pre(i, p, l0, l1, act0, act1);
            } else if constexpr (CPLX) {
                if (act0) op.store(i, op.load(i), make_double2(l0, l1));
            } else {
                if (act0) op.store(i, op.load(i), l0);
                if (act1) op.store(i + 1, op.load(i + 1), l1);
            }
        };
        // FP64 arithmetic straight from global memory (code that is cold when it runs, and one block holds up a
        // sweep of a small grid: short loops, and the op's own code only where points are many)
        constexpr int XS = CPLX ? 2 : 1;
        auto at = [&](int j, int r, int c) {
            const int o = zoff[j] + yoff[r];
            return fix_load(op, (unsigned)(o + xoff[c]), (unsigned)(o + xoff[c + 1]), false);
        };
        const int lane = tid & 31, warp = tid >> 5;
        unsigned coarse = act0 ? (1u << nz) - 1u : 0u;   // planes left to FP64 arithmetic
        if (E <= 2046 && (all & 0xffff) <= E) {
            const long long* own_s = fix_smem + (ty + N) * RW + HX + 2 * tx;
#pragma unroll
            for (int k = 0; k < BZ; ++k) col[N + k] = *reinterpret_cast<const longlong2*>(own_s + k * CPL);
            const unsigned least = all ? FIX_FINE : 0u;
            // planes in which the unit's first and second value are below the limit; a complex value counts once
            unsigned s0 = 0, s1 = 0;
#pragma unroll
            for (int k = 0; k < BZ; ++k) {
                const unsigned m0 = fix_mag(col[N + k].x), m1 = fix_mag(col[N + k].y);
                s0 |= (CPLX ? m0 | m1 : m0) < least ? 1u << k : 0u;
                s1 |= !CPLX && m1 < least ? 1u << k : 0u;
            }
            if constexpr (CPLX) s1 = s0;
            int mine = 0, total = 0;
            // what the neighbours that this lane and those beside it hold leave to a closer look: both of the
            // unit (complex: the next lane's), next in z, one of the two in y
            const unsigned sy = __shfl_xor_sync(0xffffffffu, s0 | s1 << 16, FX_UX);
            auto column = [](unsigned s) { return (s << 1 | 1u) & (s >> 1 | 1u << (BZ - 1)); };
            unsigned small = s0 & s1 & ((column(s0) & sy) | (column(s1) & sy >> 16));
            if constexpr (CPLX) small &= __shfl_xor_sync(0xffffffffu, s0, 1);
            // a warp in which eight units pass none of this in any plane leaves all its points
            bool leave = __popc(__ballot_sync(0xffffffffu, small == (1u << BZ) - 1u)) >= 8;
            if (!leave && __any_sync(0xffffffffu, small != 0)) {
                const unsigned c = fix_coarse<N, CPLX, BZ>(own_s, small, least) & coarse;
                const int count = __popc(c);
                total = __reduce_add_sync(0xffffffffu, count);
                leave = total > ITEMS;
                if (!leave && total > 0) {   // eight lanes to a unit, four units at a time
                    mine = count;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int v = __shfl_up_sync(0xffffffffu, mine, o);
                        if (lane >= o) mine += v;
                    }
                    mine -= count;
                    int q = mine;
                    for (unsigned r = c; r; r &= r - 1u) items[warp][q++] = (unsigned char)((__ffs((int)r) - 1) * 32 + lane);
                    __syncwarp();
#pragma unroll 1
                    for (int q0 = 0; q0 < total; q0 += 4) {
                        const int qi = min(q0 + (lane >> 3), total - 1), e = items[warp][qi], k = N + (e >> 5);
                        const int cx = HX + 2 * (e & (FX_UX - 1)), ry = N + (warp * 32 + (e & 31)) / FX_UX;
                        double2 acc = make_double2(0.0, 0.0);
#pragma unroll
                        for (int t0 = 0; t0 <= 6 * N; t0 += 8) {   // 2N taps of each axis, the centre
                            const int t = t0 + (lane & 7), a = t / (2 * N), h = t - a * 2 * N, p = h / 2 + 1, o = h & 1 ? -p : p;
                            if (t > 6 * N) continue;
                            const double2 v = at(k + (a == 2 ? o : 0), ry + (a == 1 ? o : 0), cx + (a == 0 ? o * XS : 0));
                            const double w = a == 3 ? W.centre : W.w[a][p];
                            acc.x = fma(w, v.x, acc.x);
                            acc.y = fma(w, v.y, acc.y);
                        }
#pragma unroll
                        for (int o = 4; o > 0; o >>= 1) {
                            acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o);
                            acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
                        }
                        if ((lane & 7) == 0) taken[warp][qi] = acc;
                    }
                    __syncwarp();
                    small = c;
                }
            }
            if (total == 0) small = 0;   // now the planes whose values stand in `taken`
            if (!leave) {
                coarse = 0;
                const double unit = __hiloint2double((E - 1082 + 1023) << 20, 0);
                auto cur = fetch(0), next = cur;
                fix_planes<N, CPLX, ISO, BZ>(
                    col, own_s, nz, fs.s[0] * unit, fs.s[1] * unit, fs.s[2] * unit,
                    [&](int k) {
                        if (k < nz) next = fetch(k);
                    },
                    [&](int k, double l0, double l1) {
                        if ((small >> k) & 1u) {
                            const double2 v = taken[warp][mine++];
                            l0 = v.x;
                            l1 = v.y;
                        }
                        store(k, cur, l0, l1);
                        cur = next;
                    });
                __syncwarp();   // before the next brick's values
            }
        }
        const int cx = HX + 2 * tx, ry = N + ty;
#pragma unroll 1
        for (; coarse; coarse &= coarse - 1u) {
            const int k = __ffs((int)coarse) - 1;
            double2 acc = at(N + k, ry, cx);
            acc = make_double2(W.centre * acc.x, W.centre * acc.y);
            auto tap = [&](double w, double2 a, double2 b) {
                acc.x = fma(w, a.x + b.x, acc.x);
                acc.y = fma(w, a.y + b.y, acc.y);
            };
#pragma unroll 1
            for (int p = 1; p <= N; ++p) {
                tap(W.w[2][p], at(N + k + p, ry, cx), at(N + k - p, ry, cx));
                tap(W.w[0][p], at(N + k, ry, cx + p * XS), at(N + k, ry, cx - p * XS));
                tap(W.w[1][p], at(N + k, ry + p, cx), at(N + k, ry - p, cx));
            }
            store(k, fetch(k), acc.x, acc.y);
        }
    }
}

template <int N, bool CPLX, bool ISO, int BZ, class Op>
__global__ void __launch_bounds__(FX_THREADS, N == 1 ? 4 : 3)
fix_kernel(Dims d, Weights<double> W, FixScale fs, bool vec, int bx, int by, int bricks, Op op) {
    pdl_enter();
    if (!op.begin()) return;
    fix_sweep<N, CPLX, ISO, BZ>(d, W, fs, vec, bx, by, bricks, op);
    op.end();
}

// Spacings equal but for the rounding of h = L / n (which moves 1 / h^2 by up to 2^-52 an axis, and its
// own three operations by as much again) count as equal: their mean for the three axes, so that the
// sums of all axes share one conversion (96^3: order 12 18.9 -> 12.7 us, order 2 14.3 -> 7.4, when measured).
inline FixScale fix_scale(of_grid* g) {
    FixScale fs;
    for (int a = 0; a < 3; ++a) fs.s[a] = std::ldexp(1.0, fix_shift(g->N)) / (fix_denominator(g->N) * g->h[a] * g->h[a]);
    const double lo = std::min({fs.s[0], fs.s[1], fs.s[2]}), hi = std::max({fs.s[0], fs.s[1], fs.s[2]});
    if (hi - lo <= std::ldexp(lo, -50)) fs.s[0] = fs.s[1] = fs.s[2] = lo + 0.5 * (hi - lo);
    return fs;
}

template <int N, bool CPLX, bool ISO, int BZ, class Op>
void launch_fix_kernel(of_grid* g, const FixScale& fs, Op op) {
    const Dims& d = g->d;
    const long long RF = CPLX ? 2LL * d.n1 : d.n1;
    const bool vec = RF % 2 == 0 && (fix_bits(op) & 15) == 0;
    const int bx = (int)((RF + 31) / 32), by = (d.n2 + FX_BY - 1) / FX_BY;
    const int bricks = bx * by * ((d.n3 + BZ - 1) / BZ);
    // one block per brick, up to the reductions' limit
    const unsigned grid = (unsigned)std::min(bricks, OF_MAX_RED_BLOCKS);
    constexpr size_t smem = fix_smem_bytes<N, CPLX, BZ>();
    if constexpr (smem > 40 * 1024) {
        static thread_local int configured_device = -1;
        if (configured_device != g->device) {
            OF_CUDA(cudaFuncSetAttribute(fix_kernel<N, CPLX, ISO, BZ, Op>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem));
            configured_device = g->device;
        }
    }
    launch_pdl(fix_kernel<N, CPLX, ISO, BZ, Op>, dim3(grid), dim3(FX_UX, FX_BY), smem, g->stream, d, g->w64, fs, vec,
               bx, by, bricks, op);
}

// Bricks of 8 planes, or of 2 where those leave most SMs without a block (32^3: 16 bricks of 8
// planes 8.1 us, 64 of 2 planes 4.0 us)
template <int N, bool CPLX, bool ISO, class Op>
void launch_fix_depth(of_grid* g, const FixScale& fs, Op op) {
    const Dims& d = g->d;
    const long long bricks = ((CPLX ? 2LL : 1LL) * d.n1 + 31) / 32 * ((d.n2 + FX_BY - 1) / FX_BY) * ((d.n3 + 7) / 8);
    if (bricks < num_sms()) launch_fix_kernel<N, CPLX, ISO, 2>(g, fs, op);
    else launch_fix_kernel<N, CPLX, ISO, 8>(g, fs, op);
}

// Sweeps an FP64 field of the grid (the doubles of a real or, CPLX, an interleaved complex field;
// op.load / op.store as for the other sweeps) with the fixed-point kernel.
template <bool CPLX, class Op>
void launch_field(of_grid* g, Op op) {
    if ((CPLX ? 2 : 1) * g->d.n >= (1LL << 31)) {   // beyond the kernel's 32-bit offsets
        using T = typename std::conditional<CPLX, double2, double>::type;
        launch_stencil<T, CPLX ? 1 : 2>(g, g->w64, op);
        return;
    }
    const int cls = OpInfo<Op>::cls >= 0 ? OpInfo<Op>::cls : PC_STENCIL_F64;
    ProfScope ps(g, cls, (double)OpInfo<Op>::words * (CPLX ? 16.0 : 8.0) * (double)g->d.n);
    const FixScale fs = fix_scale(g);
    const bool iso = fs.s[0] == fs.s[1] && fs.s[1] == fs.s[2];
    switch (g->N * 2 + (iso ? 1 : 0)) {
        case 2: launch_fix_depth<1, CPLX, false>(g, fs, op); break;
        case 3: launch_fix_depth<1, CPLX, true>(g, fs, op); break;
        case 6: launch_fix_depth<3, CPLX, false>(g, fs, op); break;
        case 7: launch_fix_depth<3, CPLX, true>(g, fs, op); break;
        case 12: launch_fix_depth<6, CPLX, false>(g, fs, op); break;
        case 13: launch_fix_depth<6, CPLX, true>(g, fs, op); break;
        default: OF_REQUIRE(false, OF_EINVAL, "unsupported finite-difference half order %d", g->N);
    }
}

}  // namespace of
