// Wind-field generation (Sec. 3.9.1): W(0) = Qhat v(0), W(k+1) = a W(k) + Q v(k+1)
// with Qhat = sigma (L_xy kron L_z) and Q = sqrt(1 - a^2) Qhat.  Because the
// recursion is linear, W(k) = sigma (L_xy kron L_z) B(k) with
// B(0) = v(0), B(k) = a B(k-1) + sqrt(1 - a^2) v(k).
//
// Kernel 1 draws v (Philox stream 3, Box-Muller), runs the AR(1) recursion
// over k and applies the small vertical factor L_z, writing
// Btmp[q][((m H + k) nz + iz) 2 + c] for horizontal node q.
// Kernel 2 applies the horizontal factor as one lower-triangular matrix
// product over q (an FP32 register-tiled GEMM) and writes the rollout's packed
// layout: float4 per node, its own value and the difference to the node one
// level up, so that the trilinear interpolation needs four aligned 16-byte
// loads and no subtraction in the vertical direction; the plain values too
// when the caller wants them.
#include "launch.cuh"
#include "wind_normals.cuh"

namespace tma {

namespace {

template <int LANES>
__global__ void __launch_bounds__(128) wind_normals_ar_kernel(const WindC w, const DynState *__restrict__ dyn,
                                                              float *__restrict__ Btmp)
{
    grid_begin();
    const long long t = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / LANES;
    const int iz = threadIdx.x % LANES;
    const bool on = t < (long long)w.M * w.nxy && iz < w.nz;
    const long long tc = min(t, (long long)w.M * w.nxy - 1);
    const int m = (int)(tc / w.nxy);
    const int q = (int)(tc - (long long)m * w.nxy);
    wind_normals_column<LANES>(w, w.key0, w.key1, w.stream, dyn->mpc_step, m, q, iz, on,
                               Btmp + (size_t)q * w.ldb + (size_t)m * w.H * (size_t)(2 * w.nz));
}

__device__ __forceinline__ void cp_async16(float *dst, const float *src, bool on)
{
    // zero-filled when off
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(on ? 16 : 0)
                 : "memory");
}

// The product's tiles are kTile x kTile.
constexpr int kTile = 64, kGemmThreads = kTile * kTile / 64;

// Columns of a tile that are used: whole vertical columns of nodes (2 nz values
// each, so that a node's upper neighbour is in the tile) and a multiple of 4
// (16-byte copies).  All 64 for 2, 4, 8 and 16 levels, 36 for 9, 44 to 60 for the
// others: the rest of such a tile's product is thrown away (64 x 64 x 9 grid, 4
// samples, 30 steps: 1070 us, where 8 levels take 575; 1514 and 1375 us with the
// 128 x 128 tiles that used every column).
__host__ __device__ constexpr int wind_tile_cols(int nz)
{
    const int unit = nz % 2 == 0 ? 2 * nz : 4 * nz;
    return kTile / unit * unit;
}

// C[p][col] = sum_{q <= p} At[q][p] Btmp[q][col], q ascending in one chain of
// fused multiply-adds per output, sigma C into the packed layout.  64 x 64 tiles,
// 8 x 8 outputs per thread (64 threads: the two warps of a block wait for
// little, and small fields fill the chip; 128 x 128 tiles of 256 threads were 8-30 %
// slower from 5 samples of a 32 x 32 x 8 grid over 90 steps on), K in steps of 8
// through a ring of four stages filled by cp.async; a pair of columns per
// two-lane FP32 instruction (each lane the IEEE single operation), which halves
// the issue slots of the products.  At is the factor transposed and zero-padded
// to multiples of 128, Btmp zero-padded to as many rows, so the main loop needs
// guards for the last columns only.  Row tiles run from the last (longest sums)
// to the first.  Bound: the FP32 units (2.6e11 products and sums for 16 samples of
// a 64 x 64 x 8 grid over 60 steps, 3.2 ms at their peak): that field with its
// plain values takes 4.20 ms (normals included) against 9.47 ms with a
// single-buffered loop, a second pass that formed the differences and a strided
// copy for the plain values.
constexpr int kStages = 4, kKStep = 8;

__global__ void __launch_bounds__(kGemmThreads, 6)
    wind_gemm_kernel(const WindC w, const float *__restrict__ At, int lda, const float *__restrict__ Bm, int n_ctiles,
                     int n_rtiles, float4 *__restrict__ W, float *__restrict__ Wown, bool pairs)
{
    constexpr int T = kTile, kThreads = kGemmThreads;
    constexpr int kPad = T + 2;          // rows an odd number of 8-byte words apart: no bank conflicts along rows
    constexpr int kRing = kStages * kKStep * 2 * T, kOut = T * kPad;
    __shared__ __align__(16) float sh[kRing > kOut ? kRing : kOut];
    grid_begin();
    const int t = threadIdx.x;
    const int tx = t % (T / 8), ty = t / (T / 8);
    const int rt = n_rtiles - 1 - (int)(blockIdx.x / n_ctiles);
    const int cols = wind_tile_cols(w.nz);
    const int row0 = rt * T, col0 = (int)(blockIdx.x % n_ctiles) * cols;
    const int steps = (min(w.nxy, row0 + T) + kKStep - 1) / kKStep;
    float2 acc[8][4];
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = make_float2(0.0f, 0.0f);

    // stage s: A rows [kKStep][T], then B rows [kKStep][T]
    auto fill = [&](int step) {
        if (step < steps) {
            float *A = sh + (step % kStages) * kKStep * 2 * T, *B = A + kKStep * T;
#pragma unroll
            for (int e = t; e < kKStep * T / 4; e += kThreads) {
                const int k = e / (T / 4), c = e % (T / 4) * 4;
                const size_t q = (size_t)(step * kKStep + k);
                cp_async16(A + k * T + c, At + q * lda + row0 + c, true);
                const bool on = col0 + c < w.ldb;
                cp_async16(B + k * T + c, Bm + q * w.ldb + (on ? col0 + c : 0), on);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int s = 0; s < kStages - 1; ++s) fill(s);
    for (int step = 0; step < steps; ++step) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
        __syncthreads();                 // this step's stage is filled, the previous step's is free
        fill(step + kStages - 1);
        const float *A = sh + (step % kStages) * kKStep * 2 * T + ty * 8;
        const float *B = sh + (step % kStages) * kKStep * 2 * T + kKStep * T + tx * 4;
#pragma unroll
        for (int kk = 0; kk < kKStep; ++kk) {
            const float4 a0 = *reinterpret_cast<const float4 *>(A + kk * T);
            const float4 a1 = *reinterpret_cast<const float4 *>(A + kk * T + 4);
            const float4 b0 = *reinterpret_cast<const float4 *>(B + kk * T);
            const float4 b1 = *reinterpret_cast<const float4 *>(B + kk * T + T / 2);
            const float ar[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            const float2 br[4] = {make_float2(b0.x, b0.y), make_float2(b0.z, b0.w), make_float2(b1.x, b1.y),
                                  make_float2(b1.z, b1.w)};
#pragma unroll
            for (int a = 0; a < 8; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[a][b] = __ffma2_rn(make_float2(ar[a], ar[a]), br[b], acc[a][b]);
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");

    // through shared memory into the packed records: for each field mk and level,
    // consecutive threads take consecutive rows (nodes along y)
    const int two_nz = 2 * w.nz;
    const int mk0 = col0 / two_nz, n_mk = min(cols, w.ncol - col0) / two_nz;
    const float sg = w.sigma;
    __syncthreads();
#pragma unroll
    for (int a = 0; a < 8; ++a) {
        float2 *o = reinterpret_cast<float2 *>(sh + (ty * 8 + a) * kPad + tx * 4);
        o[0] = acc[a][0];
        o[1] = acc[a][1];
        o[T / 4] = acc[a][2];
        o[T / 4 + 1] = acc[a][3];
    }
    __syncthreads();
    const int rows = min(T, w.nxy - row0);
    const int row = t % T, p = row0 + row;
    if (row < rows) {
        const size_t rec = (size_t)(p / w.ny) * w.out.pitch + p % w.ny;
        const float *src = sh + row * kPad;
        for (int c = t / T; c < n_mk * (w.nz - 1); c += kThreads / T) {
            const int mk = c / (w.nz - 1), iz = c - mk * (w.nz - 1);
            const float2 lo = *reinterpret_cast<const float2 *>(src + mk * two_nz + 2 * iz);
            const float2 hi = *reinterpret_cast<const float2 *>(src + mk * two_nz + 2 * iz + 2);
            const float2 own = make_float2(__fmul_rn(sg, lo.x), __fmul_rn(sg, lo.y));
            W[(size_t)(mk0 + mk) * w.out.P + (size_t)iz * w.out.plane + rec] =
                make_float4(own.x, own.y, __fsub_rn(__fmul_rn(sg, hi.x), own.x),
                            __fsub_rn(__fmul_rn(sg, hi.y), own.y));
        }
    }
    if (Wown) {
        // the caller's layout [mk][row][level][2]: consecutive threads take consecutive
        // levels; a pair in one store when the caller's pointer allows it
        for (int n = t; n < n_mk * rows * w.nz; n += kThreads) {
            const int iz = n % w.nz, q = n / w.nz, mk = q / rows, r = q - mk * rows;
            const float2 v = *reinterpret_cast<const float2 *>(sh + r * kPad + mk * two_nz + 2 * iz);
            float *o = Wown + 2 * (((size_t)(mk0 + mk) * w.nxy + row0 + r) * w.nz + iz);
            const float2 own = make_float2(__fmul_rn(sg, v.x), __fmul_rn(sg, v.y));
            if (pairs) {
                *reinterpret_cast<float2 *>(o) = own;
            } else {
                o[0] = own.x;
                o[1] = own.y;
            }
        }
    }
}

}  // namespace

cudaError_t launch_wind_normals_ar(const WindC &w, const DynState *dyn, float *Btmp,
                                   cudaStream_t st)
{
    if (w.M <= 0 || w.nxy <= 0) return cudaSuccess;
    const int lanes = wind_column_lanes(w.nz);
    const unsigned grid = (unsigned)(((long long)w.M * w.nxy * lanes + 127) / 128);
    switch (lanes) {
    case 2: launch_dependent(wind_normals_ar_kernel<2>, grid, 128, 0, st, w, dyn, Btmp); break;
    case 4: launch_dependent(wind_normals_ar_kernel<4>, grid, 128, 0, st, w, dyn, Btmp); break;
    case 8: launch_dependent(wind_normals_ar_kernel<8>, grid, 128, 0, st, w, dyn, Btmp); break;
    default: launch_dependent(wind_normals_ar_kernel<16>, grid, 128, 0, st, w, dyn, Btmp); break;
    }
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_wind_gemm(const WindC &w, const float *Lxy_t, int lda, const float *Btmp,
                             float *W, cudaStream_t st, float *W_own)
{
    const int cols = wind_tile_cols(w.nz);
    const int ct = (w.ncol + cols - 1) / cols, rt = (w.nxy + kTile - 1) / kTile;
    launch_dependent(wind_gemm_kernel, ct * rt, kGemmThreads, 0, st, w, Lxy_t, lda, Btmp, ct, rt,
                     reinterpret_cast<float4 *>(W), W_own, reinterpret_cast<uintptr_t>(W_own) % sizeof(float2) == 0);
    count_launch();
    return cudaGetLastError();
}

}  // namespace tma
