// Plain FP64 CG in one cooperative launch, for grids whose bricks (of_fix.cuh) are all resident.
//
// On such grids an iteration is a chain of latencies: sweep and update as two launches took 24 us
// at 45 x 50 x 54, of which the arithmetic is a few.  Here the blocks stay: each iteration is
// the sweep p = r + beta p_in, A p, p^T A p over the block's own bricks, a grid barrier, the update
// of its own points, another barrier.  Every block adds all blocks' partial sums itself, in one
// order, so that all hold the same alpha, beta and stopping decision without a third barrier.
// us per iteration, two launches / this kernel, order 12: 12^3 24.2 / 17.4, 32^3 23.3 / 16.0, 45 x 50 x 54
// 27.1 / 22.6, 64^3 33.5 / 26.1, 80 x 57 x 57 36.9 / 30.7; 45 x 50 x 54 at order 6: 24.3 / 19.9, of which the sweep
// 7.3, the update 2.9 and the two sums with their barriers 4.7 each (chains of FP64 additions of 64
// cycles per warp, and four L2 latencies).  96^3 has more bricks than are resident.
// Other blocks' r and p are read past L1 (__ldcg), which is not coherent within a launch.
// The barrier's wait is bounded: a block that gives up raises a flag that the others poll, all
// return, and the solve reports OF_ETIMEOUT.
#include <algorithm>

#include "of_krylov.cuh"

namespace of {

struct OpCg {
    const double* r;
    const double* pin;
    double* pout;
    double* Ap;
    double a, q, beta, acc;
    __device__ double load(long long i) const { return fma(beta, __ldcg(pin + i), __ldcg(r + i)); }
    __device__ double2 pair(unsigned i0, unsigned i1, bool vec) const {
        double2 rv, pv;
        if (vec) {
            rv = __ldcg(reinterpret_cast<const double2*>(r + i0));
            pv = __ldcg(reinterpret_cast<const double2*>(pin + i0));
        } else {
            rv = make_double2(__ldcg(r + i0), __ldcg(r + i1));
            pv = make_double2(__ldcg(pin + i0), __ldcg(pin + i1));
        }
        return make_double2(fma(beta, pv.x, rv.x), fma(beta, pv.y, rv.y));
    }
    __device__ void store(long long i, double c, double lap) {
        pout[i] = c;
        const double v = fma(q, c, -a * lap);
        Ap[i] = v;
        acc = fma(c, v, acc);
    }
};

__device__ __forceinline__ unsigned long long cg_now() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// All blocks' sum of v (every thread's share), the same bits in every block; false: gave up (at once,
// without polling, for wait_ns = 0).  `target`: arrivals that end this barrier.
__device__ __forceinline__ bool cg_total(double v, double* partials, unsigned* bar, unsigned target,
                                         unsigned long long wait_ns, double& total) {
    __shared__ double sums[1];
    __shared__ int ok;
    const int tid = threadIdx.x + FX_UX * threadIdx.y, nb = gridDim.x;
    const double one[1] = {v};
    block_sums<1>(one, sums);
    __syncthreads();   // with it, every thread's stores are ordered before the arrival
    if (tid == 0) {
        __stcg(partials + blockIdx.x, sums[0]);
        __threadfence();
        atomicAdd(bar, 1u);
        volatile unsigned* count = bar;
        volatile unsigned* quit = bar + 1;
        int got = 0;
        unsigned long long t0 = 0;
        for (int k = 0; wait_ns != 0 && k < (1 << 26); ++k) {
            if ((int)(*count - target) >= 0) { got = 1; break; }   // (both wrap: 2^32 / 2 blocks iterations)
            if ((k & 255) == 255) {
                if (*quit) break;
                if (t0 == 0) t0 = cg_now();
                else if (cg_now() - t0 > wait_ns) break;
            }
        }
        if (!got) *quit = 1u;
        __threadfence();
        ok = got;
    }
    __syncthreads();
    if (!ok) return false;
    double t[4] = {0.0, 0.0, 0.0, 0.0};   // OF_MAX_RED_BLOCKS is above what can be resident
    for (int b = tid; b < nb; b += 4 * FX_THREADS)
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (b + j * FX_THREADS < nb) t[j] += __ldcg(partials + b + j * FX_THREADS);
    const double part[1] = {(t[0] + t[1]) + (t[2] + t[3])};
    block_sums<1>(part, sums);
    __syncthreads();
    total = sums[0];
    return true;
}

template <int N, bool ISO, int BZ>
__global__ void __launch_bounds__(FX_THREADS, BZ == 2 ? 3 : 2)
cg_kernel(Dims d, Weights<double> W, FixScale fs, bool vec, int bx, int by, int bricks, double* __restrict__ x, double* r,
          double* pa, double* pb, double* Ap, double a, double q, KState* st, double* partials, unsigned* bar,
          unsigned long long wait_ns) {
    if (st->done != 0.0) return;
    const double tol2 = st->tol2, maxit = st->maxit;
    double beta = st->beta_re, rho = st->rho_re, rr = st->rr, iters = st->iters;
    double pAp = 0.0, alpha = 0.0, breakdown = 0.0;
    OpCg op{r, pa, pb, Ap, a, q, 0.0, 0.0};
    unsigned target = 0;
    bool ok = true;
    for (bool done = false; !done;) {
        op.beta = beta;
        op.acc = 0.0;
        fix_sweep<N, false, ISO, BZ>(d, W, fs, vec, bx, by, bricks, op);
        target += gridDim.x;
        ok = cg_total(op.acc, partials, bar, target, wait_ns, pAp);
        if (!ok) break;
        if (!(pAp > 0.0)) {
            breakdown = 1.0;
            break;
        }
        alpha = rho * pAp / (pAp * pAp);   // as cdiv rounds it
        double acc = 0.0;
        for (int brick = blockIdx.x; brick < bricks; brick += gridDim.x) {
            const int kb = brick / (bx * by), rem = brick - kb * bx * by, jb = rem / bx;
            const int xe = (rem - jb * bx) * 32 + 2 * threadIdx.x, y = jb * FX_BY + threadIdx.y, z0 = kb * BZ;
            if (y >= d.n2 || xe >= d.n1) continue;
            const int nz = min(BZ, d.n3 - z0);
            const bool two = xe + 1 < d.n1;
            constexpr int G = BZ < 4 ? BZ : 4;   // planes whose loads are in flight together
            for (int k0 = 0; k0 < nz; k0 += G) {
                double v[4][2 * G];
#pragma unroll
                for (int k = 0; k < G; ++k) {
                    const long long i = ((long long)(z0 + k0 + k) * d.n2 + y) * d.n1 + xe;
#pragma unroll
                    for (int c = 0; c < 2; ++c)
                        if (k0 + k < nz && (c == 0 || two)) {
                            v[0][2 * k + c] = x[i + c];
                            v[1][2 * k + c] = __ldcg(r + i + c);
                            v[2][2 * k + c] = __ldcg(op.pout + i + c);
                            v[3][2 * k + c] = __ldcg(Ap + i + c);
                        }
                }
#pragma unroll
                for (int k = 0; k < G; ++k) {
                    const long long i = ((long long)(z0 + k0 + k) * d.n2 + y) * d.n1 + xe;
#pragma unroll
                    for (int c = 0; c < 2; ++c)
                        if (k0 + k < nz && (c == 0 || two)) {
                            x[i + c] = fma(alpha, v[2][2 * k + c], v[0][2 * k + c]);
                            const double w = fma(-alpha, v[3][2 * k + c], v[1][2 * k + c]);
                            r[i + c] = w;
                            acc = fma(w, w, acc);
                        }
                }
            }
        }
        target += gridDim.x;
        ok = cg_total(acc, partials + OF_MAX_RED_BLOCKS, bar, target, wait_ns, rr);
        if (!ok) break;
        iters += 1.0;
        if (rr <= tol2 || iters >= maxit) {
            done = true;
        } else if (!(fabs(rho) > 0.0)) {
            breakdown = 1.0;
            done = true;
        } else {
            beta = rr * rho / (rho * rho);
        }
        rho = rr;
        double* t = const_cast<double*>(op.pin);
        op.pin = op.pout;
        op.pout = t;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0 && threadIdx.y == 0) {
        st->rr = rr;
        st->rho_re = rho;
        st->pAp_re = pAp;
        st->alpha_re = alpha;
        st->beta_re = beta;
        st->iters = iters;
        st->breakdown = ok ? breakdown : 2.0;
        st->done = 1.0;
    }
}

struct CgLaunch {
    of_grid* g;
    FixScale fs;
    double *x, *r, *pa, *pb, *Ap;
    double a, q;
    int st_off;
    KState* h;   // the state read back
};

template <int N, bool ISO, int BZ>
static bool cg_launch(const CgLaunch& c) {
    of_grid* g = c.g;
    constexpr size_t smem = fix_smem_bytes<N, false, BZ>();
    static thread_local int device = -1, resident = 0;
    if (device != g->device) {
        OF_CUDA(cudaFuncSetAttribute(cg_kernel<N, ISO, BZ>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        OF_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&resident, cg_kernel<N, ISO, BZ>, FX_THREADS, smem));
        device = g->device;
    }
    Dims d = g->d;
    int bx = (d.n1 + 31) / 32, by = (d.n2 + FX_BY - 1) / FX_BY;
    const long long all = (long long)bx * by * ((d.n3 + BZ - 1) / BZ);
    if (all > std::min((long long)resident * num_sms(), (long long)OF_MAX_RED_BLOCKS)) return false;
    int bricks = (int)all;
    bool vec = d.n1 % 2 == 0 && (((uintptr_t)c.r | (uintptr_t)c.pa | (uintptr_t)c.pb) & 15) == 0;
    double *x = c.x, *r = c.r, *pa = c.pa, *pb = c.pb, *Ap = c.Ap, *partials = g->s.partials;
    double a = c.a, q = c.q;
    KState* st = kstate(g, c.st_off);
    unsigned* bar = g->s.counter + 1;   // arrivals, and the flag of a block that gave up
    OF_CUDA(cudaMemsetAsync(bar, 0, 2 * sizeof(unsigned), g->stream));
    Weights<double> W = g->w64;
    FixScale fs = c.fs;
    unsigned long long wait_ns = g->wait_ns;
    void* args[] = {&d, &W, &fs, &vec, &bx, &by, &bricks, &x, &r, &pa, &pb, &Ap, &a, &q, &st, &partials, &bar, &wait_ns};
    ProfScope ps(g, PC_CG_F64, 0.0);
    const cudaError_t err = cudaLaunchCooperativeKernel((const void*)cg_kernel<N, ISO, BZ>, dim3(bricks),
                                                        dim3(FX_UX, FX_BY), args, smem, g->stream);
    // a context that is given part of the SMs, or none of whose launches may be cooperative, refuses: the
    // solve then runs as separate launches
    if (err == cudaErrorCooperativeLaunchTooLarge || err == cudaErrorNotSupported) {
        cudaGetLastError();
        return false;
    }
    OF_CUDA(err);
    __atomic_add_fetch(&g_launch_count, 1ull, __ATOMIC_RELAXED);
    ps.end_timing();
    fetch_scalars(g, c.st_off, KSTATE_DOUBLES, (double*)c.h);
    OF_REQUIRE(c.h->breakdown != 2.0, OF_ETIMEOUT, "FP64 CG: a grid barrier was not passed within the wait limit");
    ps.bytes = 10.0 * sizeof(double) * (double)d.n * c.h->iters;
    return true;
}

// Bricks of 2 planes where all are resident (shorter phases: 45 x 50 x 54 at order 6 19.9 us per iteration
// against 23.5 with 98 bricks of 8), else of 8
template <int N, bool ISO>
static bool cg_depth(const CgLaunch& c) {
    return cg_launch<N, ISO, 2>(c) || cg_launch<N, ISO, 8>(c);
}

bool cg_resident(of_grid* g, int st_off, double* x, double* r, double* pa, double* pb, double* Ap, double a, double q,
                 KState* h) {
    const CgLaunch c{g, fix_scale(g), x, r, pa, pb, Ap, a, q, st_off, h};
    const bool iso = c.fs.s[0] == c.fs.s[1] && c.fs.s[1] == c.fs.s[2];
    switch (g->N * 2 + (iso ? 1 : 0)) {
        case 2: return cg_depth<1, false>(c);
        case 3: return cg_depth<1, true>(c);
        case 6: return cg_depth<3, false>(c);
        case 7: return cg_depth<3, true>(c);
        case 12: return cg_depth<6, false>(c);
        case 13: return cg_depth<6, true>(c);
        default: return false;
    }
}

}  // namespace of
