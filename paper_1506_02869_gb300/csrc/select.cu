// Final sample selection (Sec. 3.8): the particle with the fewest infeasible
// aircraft, then the smallest sum of mean costs (the largest product of
// weights), ties to the lowest index.  Two passes: per-block candidates, then
// one block over the candidates.  Sums run over aircraft in index order in
// FP64, so the decision is exact and independent of the launch shape.
#include "device_common.cuh"
#include "launch.cuh"
#include "tma_internal.h"

namespace tma {

namespace {

struct Cand {
    int ninf;
    double sum;
    long long l;
};

__device__ __forceinline__ bool better(const Cand &a, const Cand &b)
{
    if (a.ninf != b.ninf) return a.ninf < b.ninf;
    if (a.sum != b.sum) return a.sum < b.sum;
    return a.l < b.l;
}

__device__ Cand block_best(Cand c)
{
    __shared__ int sn[256];
    __shared__ double ss[256];
    __shared__ long long sl[256];
    sn[threadIdx.x] = c.ninf;
    ss[threadIdx.x] = c.sum;
    sl[threadIdx.x] = c.l;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) {
            const Cand a{sn[threadIdx.x], ss[threadIdx.x], sl[threadIdx.x]};
            const Cand b{sn[threadIdx.x + o], ss[threadIdx.x + o], sl[threadIdx.x + o]};
            if (better(b, a)) {
                sn[threadIdx.x] = b.ninf;
                ss[threadIdx.x] = b.sum;
                sl[threadIdx.x] = b.l;
            }
        }
        __syncthreads();
    }
    return Cand{sn[0], ss[0], sl[0]};
}

// A particle's infeasible aircraft and, in FP32, an interval that holds its FP64
// sum: |s - S| <= N 2^-23 sum |c| covers N roundings of 2^-24 in either order and
// those of the bound itself; an overflowing FP32 sum gives an interval that
// excludes nothing.
struct Bound {
    int ninf;
    float lo, hi;
};

__device__ __forceinline__ Bound bound_of(const float *__restrict__ c, int N, long long L)
{
    Bound b{0, 0.0f, 0.0f};
    float s = 0.0f, a = 0.0f;
#pragma unroll 8
    for (int i = 0; i < N; ++i) {
        const float v = __ldg(c + (size_t)i * L);
        const bool bad = !(fabsf(v) < __int_as_float(0x7f800000));     // infinite or NaN
        b.ninf += bad;
        s += bad ? 0.0f : v;
        a += bad ? 0.0f : fabsf(v);
    }
    const float e = (float)N * 1.1920929e-7f * a + 4.7019774e-38f * (float)N;   // and flushed subnormals
    const bool finite = a < 1e38f;
    b.lo = finite ? s - e : -__int_as_float(0x7f800000);
    b.hi = finite ? s + e : __int_as_float(0x7f800000);
    return b;
}

constexpr int kSelPer = 4;   // particles a thread looks at between two block reductions

// Per-block candidates.  FP64 additions run at 2 per SM and cycle here, so summing
// every particle in FP64 was the whole time (34 us on 24 x 262144): the particles
// whose FP32 interval lies above another's with no more infeasible aircraft cannot
// be chosen, and only the rest are summed in FP64 (34 -> 13 us; the 25 MB of costs
// take 4 us to read).
__global__ void __launch_bounds__(256) select_partial(const float *__restrict__ cbar, int N,
                                                      long long L, Cand *__restrict__ part)
{
    __shared__ int wn[8];
    __shared__ float wh[8];
    grid_begin();
    Cand best{1 << 30, 0.0, 1ll << 62};
    int bn = 1 << 30;                                  // least infeasible count of the block so far,
    float bh = __int_as_float(0x7f800000);             // least upper end among those
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long l0 = (long long)blockIdx.x * blockDim.x; l0 < L; l0 += stride * kSelPer) {
        Bound b[kSelPer];
#pragma unroll
        for (int q = 0; q < kSelPer; ++q) {
            const long long l = l0 + threadIdx.x + q * stride;
            b[q].ninf = 1 << 30;
            if (l < L) {
                b[q] = bound_of(cbar + l, N, L);
                if (b[q].ninf < bn) {
                    bn = b[q].ninf;
                    bh = b[q].hi;
                } else if (b[q].ninf == bn) {
                    bh = fminf(bh, b[q].hi);
                }
            }
        }
        const int n = __reduce_min_sync(0xffffffffu, bn);
        float h = bn == n ? bh : __int_as_float(0x7f800000);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) h = fminf(h, __shfl_xor_sync(0xffffffffu, h, o));
        __syncthreads();                               // the previous round's values are read
        if ((threadIdx.x & 31) == 0) {
            wn[threadIdx.x >> 5] = n;
            wh[threadIdx.x >> 5] = h;
        }
        __syncthreads();
        bn = wn[0];
#pragma unroll
        for (int w = 1; w < 8; ++w) bn = min(bn, wn[w]);
        bh = __int_as_float(0x7f800000);
#pragma unroll
        for (int w = 0; w < 8; ++w)
            if (wn[w] == bn) bh = fminf(bh, wh[w]);
#pragma unroll
        for (int q = 0; q < kSelPer; ++q) {
            const long long l = l0 + threadIdx.x + q * stride;
            if (l >= L || b[q].ninf != bn || !(b[q].lo <= bh)) continue;
            double sum = 0.0;
            for (int i = 0; i < N; ++i) {
                const float c = __ldg(cbar + (size_t)i * L + l);
                if (!(isinf(c) || isnan(c))) sum += (double)c;
            }
            const Cand c{b[q].ninf, sum, l};
            if (better(c, best)) best = c;
        }
    }
    best = block_best(best);
    if (threadIdx.x == 0) part[blockIdx.x] = best;
}

__global__ void __launch_bounds__(256) select_final(const Cand *__restrict__ part, int nparts,
                                                    long long *__restrict__ out_best,
                                                    double *__restrict__ out_sum,
                                                    int *__restrict__ out_ninf)
{
    grid_begin_early();
    Cand best{1 << 30, 0.0, 1ll << 62};
    for (int j = threadIdx.x; j < nparts; j += blockDim.x)
        if (better(part[j], best)) best = part[j];
    best = block_best(best);
    if (threadIdx.x == 0) {
        *out_best = best.l;
        if (out_sum) *out_sum = best.ninf == 0 ? best.sum : __longlong_as_double(0x7ff0000000000000ll);
        if (out_ninf) *out_ninf = best.ninf;
    }
}

// Copies the chosen particle's controls; when err is given, also ORs the
// solve's status into the sticky error word: bit 0 a weight segment was all
// zero (flags bit 0), bit 1 the chosen particle has an infeasible aircraft.
__global__ void gather_best_kernel(const float *__restrict__ u, const long long *__restrict__ best,
                                   int n, float *__restrict__ out, const unsigned int *flags,
                                   const int *ninf, unsigned int *err)
{
    grid_begin();
    const long long b = *best;
    for (int j = threadIdx.x; j < n; j += blockDim.x) out[j] = u[(size_t)b * n + j];
    if (err && threadIdx.x == 0) *err |= (*flags & 1u) | (*ninf > 0 ? 2u : 0u);
}

constexpr int kSelBlocks = 592;   // 4 x 148 resident blocks; the second pass reads 592 candidates

}  // namespace

size_t select_workspace(int64_t L)
{
    (void)L;
    return kSelBlocks * sizeof(Cand) + 16;
}

cudaError_t launch_select(const float *cbar, int N, int64_t L, int64_t *best, double *best_sum,
                          int *ninf, void *work, cudaStream_t st)
{
    if (L <= 0) return cudaSuccess;
    auto *part = reinterpret_cast<Cand *>((reinterpret_cast<uintptr_t>(work) + 15) & ~uintptr_t(15));
    const long long need = (L + 255) / 256;
    const int nb = (int)(need < kSelBlocks ? need : kSelBlocks);
    launch_dependent(select_partial, nb, 256, 0, st, cbar, N, L, part);
    launch_dependent(select_final, 1, 256, 0, st, part, nb, reinterpret_cast<long long *>(best), best_sum, ninf);
    count_launch(2);
    return cudaGetLastError();
}

cudaError_t launch_gather_best(const float *u, const int64_t *best, int n, float *best_u,
                               cudaStream_t st, const unsigned int *flags, const int *ninf,
                               unsigned int *err)
{
    launch_dependent(gather_best_kernel, 1, 256, 0, st, u, reinterpret_cast<const long long *>(best), n, best_u, flags,
                     ninf, err);
    count_launch();
    return cudaGetLastError();
}

}  // namespace tma
