// The wind field's normals with their recursion in time and vertical factor
// (Sec. 3.9.1), shared by the single-scenario and the batched launch.
#pragma once

#include "device_common.cuh"
#include "tma_internal.h"

namespace tma {

// Lanes of a vertical column: the power of two that holds its nz levels.
__host__ __device__ constexpr int wind_column_lanes(int nz)
{
    return nz <= 2 ? 2 : (nz <= 4 ? 4 : (nz <= 8 ? 8 : 16));
}

// One (sample, horizontal node, level) per thread, the levels of a column in
// LANES neighbouring lanes: draws v (Philox, Box-Muller), B(0) = v(0), B(k) = a
// B(k-1) + b v(k), and the vertical factor from the lower levels' B through
// shuffles.  o: the column's row of Btmp at (sample, step 0, level 0, component
// 0); a step's nz pairs are contiguous, so a column's lanes store 8 nz bytes.
// A thread per level keeps the chip busy on few samples (the draws of a column
// one after the other were its whole time) and makes the stores coalesced.
template <int LANES>
__device__ __forceinline__ void wind_normals_column(const WindC &w, uint32_t k0, uint32_t k1, uint32_t stream,
                                                    uint32_t mpc, int m, int q, int iz, bool on, float *o)
{
    const int nz = w.nz;
    float lz[LANES];
#pragma unroll
    for (int jz = 0; jz < LANES; ++jz) lz[jz] = jz <= iz && iz < nz ? w.Lz[iz * TMA_MAX_GRID_Z + jz] : 0.0f;
    float bx = 0.0f, by = 0.0f;
    for (int k = 0; k < w.H; ++k) {
        const uint4 r = draw(k0, k1, (uint32_t)(q * nz + iz), (uint32_t)m << 8, (uint32_t)k, stream, 0u, mpc);
        const float2 n = box_muller(r.x, r.y);
        if (k == 0) {
            bx = n.x;
            by = n.y;
        } else {
            bx = fmaf(w.a, bx, w.b * n.x);
            by = fmaf(w.a, by, w.b * n.y);
        }
        float ax = 0.0f, ay = 0.0f;
#pragma unroll
        for (int jz = 0; jz < LANES; ++jz) {
            const float vx = __shfl_sync(0xffffffffu, bx, jz, LANES), vy = __shfl_sync(0xffffffffu, by, jz, LANES);
            if (jz <= iz) {
                ax = fmaf(lz[jz], vx, ax);
                ay = fmaf(lz[jz], vy, ay);
            }
        }
        if (on) *reinterpret_cast<float2 *>(o + 2 * iz) = make_float2(ax, ay);
        o += 2 * nz;
    }
}

}  // namespace tma
