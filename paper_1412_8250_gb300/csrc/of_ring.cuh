// FP32 sweeps of large grids whose field is read as it is (op.field()).
//
// A block of 32 x 8 threads walks a 64 x 32 tile of the x-y plane along z; each thread owns two
// x-neighbouring points in four adjacent rows and keeps their 2N + 1 z-neighbours in registers
// (rotated by compile-time index).  The planes of the tile with their periodic x and y halo pass
// through a ring in shared memory, filled by asynchronous copies N + AHEAD planes before they are
// computed: plane z serves the x and y taps of z, and its own points enter the register queue
// when z - N is computed, so each plane is fetched from global memory once.
// What bounds it is the shared-memory pipe: per 8 points 24 64-bit reads for the x taps, 12 for
// the y taps (four rows share one column) and 4 for the queue, 0.31 wavefronts per point; with two
// rows per thread, and the queue's and the tile's planes fetched apart through registers, it was
// 0.48 and two fetches, and odd n1 took a scalar kernel.  320^3, order 12: 95 -> 71 us
// (462 GPts/s, 68 us in a row of calls; HBM's floor is 39), order 6 128 -> 56, order 2 95 -> 53; 319 x 320 x 320 178 -> 93.
// The blocks share all (tile, plane) pairs evenly; a run of planes costs 2N more of its own points
// at its start, hence the rule on planes per block in launch_ring.
#pragma once

#include "of_stencil.cuh"

namespace of {

template <class Op, class = void>
struct HasField32 { static constexpr bool value = false; };
template <class Op>
struct HasField32<Op, std::enable_if_t<std::is_same<decltype(std::declval<const Op&>().field()), const float*>::value>> {
    static constexpr bool value = true;
};

constexpr int RG_TX = 64, RG_TY = 32, RG_ROWS = 4, RG_THREADS = 256, RG_AHEAD = 4;
template <int N> constexpr int ring_hx() { return (N + 3) & ~3; }
template <int N> constexpr int ring_slots() { return N + RG_AHEAD + 1; }
template <int N> constexpr int ring_plane() { return (RG_TY + 2 * N) * (RG_TX + 2 * ring_hx<N>()); }
template <int N> constexpr size_t ring_smem() { return sizeof(float) * ring_slots<N>() * ring_plane<N>(); }

// VEC: floats per copy (4, 2 or 1): n1 a multiple of it and the field aligned to it
template <int N, int VEC, class Op>
__global__ void __launch_bounds__(RG_THREADS, 1) ring_kernel(Dims d, Weights<float> W, long long tiles, int tilesx, Op op) {
    constexpr int HX = ring_hx<N>(), SX = RG_TX + 2 * HX, SY = RG_TY + 2 * N, S = ring_slots<N>();
    constexpr int CX = SX / VEC, CH = CX * SY, PER = (CH + RG_THREADS - 1) / RG_THREADS;
    constexpr int Q = 2 * N + 1, R = RG_ROWS;
    extern __shared__ __align__(16) float ring[];
    pdl_enter();
    if (!op.begin()) return;
    const int tid = threadIdx.x, lane = tid & 31, row0 = (tid >> 5) * R;
    const int n1 = d.n1, n2 = d.n2, n3 = d.n3;
    const long long plane = (long long)n1 * n2;
    const float* f = op.field();
    const uint32_t ring0 = (uint32_t)__cvta_generic_to_shared(ring);
    unsigned long long wz2[N + 1], wy2[N + 1];
#pragma unroll
    for (int p = 0; p <= N; ++p) {
        wz2[p] = pk2(make_float2(W.w[2][p], W.w[2][p]));
        wy2[p] = pk2(make_float2(W.w[1][p], W.w[1][p]));
    }
    const unsigned long long centre2 = pk2(make_float2(W.centre, W.centre));
    // this block's (tile, plane) pairs
    const long long all = tiles * n3;
    long long at = all * blockIdx.x / gridDim.x;
    const long long end = all * (blockIdx.x + 1) / gridDim.x;
    while (at < end) {
        const long long tile = at / n3;
        const int z0 = (int)(at - tile * n3);
        const int cz = (int)min((long long)(n3 - z0), end - at);
        at += cz;
        const int x0 = (int)(tile % tilesx) * RG_TX, y0 = (int)(tile / tilesx) * RG_TY;
        // staged chunks of this thread: in-plane offsets
        int off[PER];
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            const int e = min(tid + k * RG_THREADS, CH - 1);
            const int sy = e / CX, c = e - sy * CX;
            off[k] = wrap_index(y0 - N + sy, n2) * n1 + wrap_index(x0 - HX + VEC * c, n1);
        }
        const int x = x0 + 2 * lane;
        const bool in0 = x < n1, in1 = !in0 || x + 1 < n1;   // !in1: the row's last point, f(x + 1) is its first
        int rowoff[R];
        bool act[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int y = y0 + row0 + r;
            act[r] = in0 && y < n2;
            rowoff[r] = wrap_index(y, n2) * n1 + (in0 ? x : 0);   // rows past the end are the others' y neighbours
        }
        __syncthreads();   // the last run's reads of the ring
        int put = 0;       // slot and plane of the next copy
        long long zput = (long long)z0 * plane;
        auto stage = [&](bool any) {
            if (any) {
                const uint32_t dst = ring0 + put * (ring_plane<N>() * 4) + tid * (VEC * 4);
                const float* src = f + zput;
#pragma unroll
                for (int k = 0; k < PER; ++k)
                    if (tid + k * RG_THREADS < CH) {
                        if constexpr (VEC == 4)
                            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                                         :: "r"(dst + k * RG_THREADS * VEC * 4), "l"(src + off[k]) : "memory");
                        else
                            asm volatile("cp.async.ca.shared.global [%0], [%1], %2;"
                                         :: "r"(dst + k * RG_THREADS * VEC * 4), "l"(src + off[k]), "n"(VEC * 4) : "memory");
                    }
                put = put + 1 == S ? 0 : put + 1;
                zput += plane;
                if (zput >= (long long)n3 * plane) zput -= (long long)n3 * plane;
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        const int total = cz + N;   // planes z0 .. z0 + cz + N - 1
        int staged = 0;
        for (; staged < N + RG_AHEAD; ++staged) stage(staged < total);
        unsigned long long q[R][Q];
#pragma unroll
        for (int j = 0; j < 2 * N; ++j) {
            const long long zo = (long long)wrap_index(z0 - N + j, n3) * plane;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float* s = f + zo + rowoff[r];
                if constexpr (VEC > 1) q[r][j] = pk2(__ldg(reinterpret_cast<const float2*>(s)));
                else q[r][j] = pk2(make_float2(__ldg(s), __ldg(in1 ? s + 1 : s + 1 - n1)));
            }
        }
        int cur = 0, top = N % S;   // slots of the planes t and t + N
        const int at0 = (row0 + N) * SX + HX + 2 * lane;
        for (int tb = 0; tb < cz; tb += Q) {
#pragma unroll
            for (int k = 0; k < Q; ++k) {
                const int t = tb + k;
                if (t >= cz) break;
                asm volatile("cp.async.wait_group %0;" :: "n"(RG_AHEAD - 1) : "memory");
                __syncthreads();
                stage(staged < total);
                ++staged;
                const float* pc = ring + cur * ring_plane<N>() + at0;
                const float* pt = ring + top * ring_plane<N>() + at0;
                cur = cur + 1 == S ? 0 : cur + 1;
                top = top + 1 == S ? 0 : top + 1;
                unsigned long long acc[R];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    q[r][(2 * N + k) % Q] = *reinterpret_cast<const unsigned long long*>(pt + r * SX);
                    acc[r] = fma2(centre2, q[r][(N + k) % Q], 0ull);
#pragma unroll
                    for (int p = 1; p <= N; ++p)
                        acc[r] = fma2(wz2[p], add2(q[r][(N + p + k) % Q], q[r][(N - p + k) % Q]), acc[r]);
                }
                unsigned long long col[R + 2 * N];   // rows row0 - N .. row0 + R - 1 + N
#pragma unroll
                for (int j = 0; j < R + 2 * N; ++j)
                    if (j < N || j >= N + R) col[j] = *reinterpret_cast<const unsigned long long*>(pc + (j - N) * SX);
#pragma unroll
                for (int r = 0; r < R; ++r) col[N + r] = q[r][(N + k) % Q];
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int p = 1; p <= N; ++p)
                        acc[r] = fma2(wy2[p], add2(col[N + r + p], col[N + r - p]), acc[r]);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    constexpr int H = (N + 1) & ~1;
                    float v[2 * H + 2];   // points x - H .. x + 1 + H
#pragma unroll
                    for (int m = 0; m <= H; ++m) {
                        const float2 w = 2 * m == H ? upk2(q[r][(N + k) % Q])
                                                    : *reinterpret_cast<const float2*>(pc + r * SX - H + 2 * m);
                        v[2 * m] = w.x;
                        v[2 * m + 1] = w.y;
                    }
                    float2 a = upk2(acc[r]);
#pragma unroll
                    for (int p = 1; p <= N; ++p) {
                        a.x = fmaf(W.w[0][p], v[H + p] + v[H - p], a.x);
                        a.y = fmaf(W.w[0][p], v[H + 1 + p] + v[H + 1 - p], a.y);
                    }
                    if (act[r]) {
                        const float2 c = upk2(q[r][(N + k) % Q]);
                        const long long i = (long long)(z0 + t) * plane + rowoff[r];
                        if (VEC > 1) op_store2(op, i, c, a);
                        else {
                            op.store(i, c.x, a.x);
                            if (in1) op.store(i + 1, c.y, a.y);
                        }
                    }
                }
            }
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    op.end();
}

template <int N, int VEC, class Op>
void launch_ring_vec(of_grid* g, const Weights<float>& W, Op op) {
    static thread_local int configured_device = -1;
    if (configured_device != g->device) {
        OF_CUDA(cudaFuncSetAttribute(ring_kernel<N, VEC, Op>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)ring_smem<N>()));
        configured_device = g->device;
    }
    const int tx = (g->d.n1 + RG_TX - 1) / RG_TX;
    const long long tiles = (long long)tx * ((g->d.n2 + RG_TY - 1) / RG_TY);
    const int grid = (int)std::min(tiles * g->d.n3, (long long)num_sms());
    ProfScope ps(g, PC_STENCIL_F32, 2.0 * sizeof(float) * (double)g->d.n);
    launch_pdl(ring_kernel<N, VEC, Op>, dim3(grid), dim3(RG_THREADS), ring_smem<N>(), g->stream, g->d, W, tiles, tx, op);
}

// An FP32 sweep; `out` is where it stores (for its alignment).
template <class Op>
void launch_field32(of_grid* g, Op op, const float* out) {
    static_assert(HasField32<Op>::value, "a plain FP32 field");
    const long long tiles = (long long)((g->d.n1 + RG_TX - 1) / RG_TX) * ((g->d.n2 + RG_TY - 1) / RG_TY);
    // From 6 planes per block on, and where more than half of the tiles' points are the grid's
    // (us, this kernel / the others; order 12 unless said): 96^3 8.5 / 5.4, 128^3 7.8 / 10.6, 160^3
    // 15 / 16, order 2 at 96^3 4.7 / 3.7 and at 128^3 4.9 / 7.3, 61 x 201 x 333 22 / 28.
    const bool fits = tiles * g->d.n3 >= 6LL * num_sms() && 2LL * g->d.n1 * g->d.n2 > tiles * (RG_TX * RG_TY);
    if (fits && (long long)g->d.n1 * g->d.n2 < (1LL << 31)) {
        const uintptr_t a = reinterpret_cast<uintptr_t>(op.field()) | reinterpret_cast<uintptr_t>(out);
        const int vec = g->d.n1 % 4 == 0 && a % 16 == 0 ? 4 : (g->d.n1 % 2 == 0 && a % 8 == 0 ? 2 : 1);
#define OF_RING(N)                                                        \
    do {                                                                  \
        if (vec == 4) launch_ring_vec<N, 4>(g, g->w32, op);               \
        else if (vec == 2) launch_ring_vec<N, 2>(g, g->w32, op);          \
        else launch_ring_vec<N, 1>(g, g->w32, op);                        \
    } while (0)
        switch (g->N) {
            case 1: OF_RING(1); return;
            case 3: OF_RING(3); return;
            case 6: OF_RING(6); return;
            default: break;
        }
#undef OF_RING
    }
    launch_stencil<float, 2>(g, g->w32, op);
}

}  // namespace of
