// The wind-dependent half of the two-kernel rollout (rollout_traj.cu), shared with
// the gradient (adjoint.cu): the trajectories' records and one sample's forward pass
// over them.
#pragma once

#include "launch.cuh"
#include "rollout_tile.cuh"

namespace tma {

// Records of a slab of particles, in tiles of TP particles, B = N TP threads:
// element ((tile H + k) B + t), t = i TP + j, for every array.
struct TrajOut {
    float4 *air;       // z after step k, v cos(gamma) (its sign bit: heading and speed fit the landing sector), cos chi, sin chi
    float *chi;        // arrivals: heading after step k
    float *fuel;       // arrivals: fuel burned after step k
    uint4 *mask;       // partner masks of the steps of chunk c: element ((tile nc + c) B + t), nc = ceil(H / 4)
    float4 *state;     // the gradient's: z, v, fuel burned, chi after step k (else nullptr)
    unsigned *bad;     // the gradient's: [tile][TP], not 0: infeasible under some sample (else nullptr)
    float4 *fin;       // [tile][B]: sum |Z - z|, sum |v - vD|, fuel burned, stopping step (int; H: none)
};

// First step of the horizon this aircraft flies, and whether it is in the
// problem at all (the rolling window; else 0 and false).
__device__ __forceinline__ int entry_step(const ProblemC &P, int t_enter, const DynState *__restrict__ dyn, int i,
                                          uint32_t mpc, bool &out)
{
    out = false;
    if (!P.rolling) return 0;
    const long long d = (long long)t_enter - (long long)mpc;
    const int k_in = d > 0 ? (int)min(d, (long long)P.H) : 0;
    out = ((dyn->finished >> i) & 1u) != 0u || k_in >= P.H;
    return k_in;
}

// Partner of mask bit b of aircraft i: the pairs it would own in the one-sample
// tile (i + 1 + b, b < n_own) come first, then those it would receive (i - 1 -
// (b - n_own)), so that penalties are summed in that tile's order.
__device__ __forceinline__ int partner_of(int i, int b, int n_own, int N)
{
    const unsigned r = (unsigned)(b < n_own ? i + 1 + b : i + N - 1 + n_own - b);
    return (int)min(r, r - (unsigned)N);       // mod N: r - N wraps to a large value when r < N
}

constexpr int kStepsPerBarrier = 4;   // steps whose positions are exchanged behind one barrier: a chunk

__host__ __device__ constexpr int n_chunks(int H) { return (H + kStepsPerBarrier - 1) / kStepsPerBarrier; }

// Shared memory of a block (32-bit words): positions float2 [2 (chunk parity)]
// [kStepsPerBarrier][N][TP], their bounds over the chunk float4 [2][N][TP]; soft:
// the altitudes as the positions; hard: separation flags [N][TP]; wind mode 1: the
// particles' wind state [2][kStepsPerBarrier][16][TP].
__host__ __device__ constexpr int wind_rollout_words(int N, int tp, bool soft, bool own_wind)
{
    return (2 * kStepsPerBarrier * N * (soft ? 3 : 2) + 8 * N + (soft ? 0 : N) +
            (own_wind ? 2 * kStepsPerBarrier * 16 : 0)) * tp;
}

__device__ __forceinline__ float sgnf(float a) { return a > 0.0f ? 1.0f : (a < 0.0f ? -1.0f : 0.0f); }

// Derivative of one pair's separation penalty (weight w = 2 mu sigma(beta g) / M)
// with respect to this aircraft's position, from the differences own - partner.
__device__ __forceinline__ void pair_grad(const ProblemC &P, float w, float dx, float dy, float dz,
                                          float &sx, float &sy, float &sz)
{
    const float dh = sqrtf(fmaf(dx, dx, dy * dy));
    const float ghh = fmaf(-dh, P.Sh_inv, 1.0f);
    const float gvv = fmaf(-fabsf(dz), P.Sv_inv, 1.0f);
    if (ghh <= gvv) {
        if (dh > 0.0f) {
            const float eh = w * P.Sh_inv / dh;
            sx = fmaf(-eh, dx, sx);
            sy = fmaf(-eh, dy, sy);
        }
    } else {
        sz = fmaf(-w * P.Sv_inv, sgnf(dz), sz);
    }
}

// The penalty of a pair and the logistic weight of its derivative, from one
// exponential of -|beta g| (0, 0 when either aircraft is not flying: its
// published altitude is far away).
__device__ __forceinline__ float2 pair_penalty(const ProblemC &P, float dx, float dy, float dz)
{
    const float dh = sqrtf(fmaf(dx, dx, dy * dy));
    const float gmin = fminf(fmaf(-dh, P.Sh_inv, 1.0f), fmaf(-fabsf(dz), P.Sv_inv, 1.0f));
    const float bg = P.sp_beta * gmin;
    const float e = __expf(-fabsf(bg));
    return make_float2((fmaxf(bg, 0.0f) + log1p_unit(e)) * P.sp_inv_beta,
                       (bg >= 0.0f ? 1.0f : e) / (1.0f + e));
}

// What one sample's pass leaves of one aircraft of one particle.
struct Flown {
    Kahan sA, sB;          // bearing and (arrivals) glide-angle deviations
    float sN, soft;        // noise term, separation penalty
    int k_end;             // first step not flown: stopped by a limit, or after the landing
    bool landed, sepv;
};

// What the gradient keeps of the pass: for its slab's element (step, thread) the
// position after the step and, where a partner was within reach, the derivative of
// the penalty with respect to it; a bit per step of a chunk says where that is.
struct FlightLog {
    float2 *xy;
    float2 *polar;     // arrivals: bearing and glide angle there
    float4 *sep;
    unsigned *near;
};

// One sample m's pass of aircraft i (type, entry step k_in, stopping step kd) of
// particle l in a block of N TP threads: sh is its wind_rollout_words buffer, Wm
// the sample's field; every thread of the block calls it.  With Log the penalties'
// derivatives (sep_c: the weight of a pair's penalty in the objective, twice over
// the aircraft, over the samples) and the positions are written to `log`, whose
// elements are those of the records for tile `log_tile`.
template <int TP, bool OwnWind, bool Soft, bool Log>
__device__ __forceinline__ Flown wind_forward(const ProblemC &P, const DynState *__restrict__ dyn,
                                              const float4 *__restrict__ Wm, const TrajOut &R, float *sh, int tile,
                                              int t, long long l, int m, int J, uint32_t mpc, int type, float target,
                                              int k_in, int kd, const FlightLog &log, int log_tile, float sep_c)
{
    constexpr int KB = kStepsPerBarrier;
    const int N = P.N, H = P.H, B = N * TP;
    const int i = t / TP, j = t % TP;
    const int n_own = ((N - 1) >> 1) + (((N & 1) == 0 && i < (N >> 1)) ? 1 : 0);

    float2 *pos = reinterpret_cast<float2 *>(sh);                               // [2][KB][N][TP]
    float4 *box = reinterpret_cast<float4 *>(sh + 4 * KB * B);                  // [2][N][TP]
    float *zs = sh + 4 * KB * B + 8 * B;                                        // soft: [2][KB][N][TP]
    int *vflag = reinterpret_cast<int *>(zs);                                   // hard: [N][TP]
    float *pw = zs + (Soft ? 2 * KB * B : B);                                   // mode 1: [2][KB][16][TP]
    if constexpr (!Soft) vflag[t] = 0;

    float x = dyn->x0[i][0], y = dyn->x0[i][1], z = dyn->x0[i][2];
    Kahan sA, sB;              // bearing and (arrivals) glide-angle deviations
    float sN = 0.0f, soft = 0.0f;
    int k_end = kd;            // first step not flown: stopped by a limit, or after the landing
    bool landed = false, sepv = false;

    // wind mode 1: the state B(k) of the particle's field at step k, drawn by the
    // warps of the tile in turn (a row is always advanced by the same thread)
    auto own_wind_step = [&](int k) {
        float *dst = pw + (((k / KB) & 1) * KB + k % KB) * 16 * TP + j;
        const float *src = pw + ((((k + 2 * KB - 1) / KB) & 1) * KB + (k + KB - 1) % KB) * 16 * TP + j;   // B(k-1)
        for (int r = i; r < 4; r += N) {
            const uint4 d = draw_rk(P.rk, (uint32_t)l, (uint32_t)(4 * m + r), (uint32_t)k, 9u, 0u, mpc);
            const float2 v0 = box_muller_fast(d.x, d.y), v1 = box_muller_fast(d.z, d.w);
            const float v[4] = {v0.x, v0.y, v1.x, v1.y};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int row = (4 * r + e) * TP;
                dst[row] = k == 0 ? v[e] : fmaf(P.wind_a, src[row], P.wind_b * v[e]);
            }
        }
    };
    if constexpr (OwnWind) {
        for (int k = 0; k < min(KB, H); ++k) own_wind_step(k);
        __syncthreads();
    }

    const float4 *Wk = Wm;
    unsigned o = (unsigned)tile * H * B + t;                   // the workspace bound keeps the records within 32 bits
    unsigned olog = (unsigned)log_tile * H * B + t;
    const float far2 = Soft ? P.sp_far_h2 : P.Sh2;
    for (int k0 = 0; k0 < H; k0 += KB) {
        const int par = (k0 / KB) & 1;
        float2 *buf = pos + par * KB * B;
        float *zbuf = zs + par * KB * B;
        float4 *bx = box + par * B;
        const bool up = k0 < k_end && k0 + KB > k_in;               // flying in this chunk at all
#pragma unroll 1
        for (int e0 = 0; e0 < KB; e0 += 2) {
            float2 nrm[2];
            if (up) {
                const uint4 r = draw_rk(P.rk, (uint32_t)l, (uint32_t)i | ((uint32_t)m << 8), (uint32_t)((k0 + e0) >> 1),
                                        0u, (uint32_t)J, mpc);
                nrm[0] = box_muller_fast(r.x, r.y);
                nrm[1] = box_muller_fast(r.z, r.w);
            }
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int k = k0 + e0 + e;
                if (k < k_end && k >= k_in) {                        // k_end <= H
                    const float4 a = __ldg(R.air + o);
                    const float chi = type == 0 ? __ldg(R.chi + o) : 0.0f;
                    float2 w;
                    if constexpr (OwnWind) w = particle_wind_at<TP>(P, pw + (par * KB + e0 + e) * 16 * TP + j, x, y, z);
                    else w = wind_interp(wind_fetch(P, Wk, x, y, z));
                    w.x = fmaf(P.turb_sigma, nrm[e].x, w.x);
                    w.y = fmaf(P.turb_sigma, nrm[e].y, w.y);
                    const float vh = fabsf(a.y);
                    x = fmaf(P.dt, fmaf(vh, a.z, w.x), x);
                    y = fmaf(P.dt, fmaf(vh, a.w, w.y), y);
                    z = a.x;
                    const float th = atan2_poly(y, x);
                    if (type == 0) {
                        float r, ath;
                        const float beta = arc_glide(x, y, z, th, r, ath);
                        if constexpr (Log) log.polar[olog] = make_float2(th, beta);
                        // the landing sector of Eq. (TO_init); heading and speed in the record's sign
                        if (__float_as_int(a.y) < 0 && r <= P.P_runway && beta <= P.P_beta && x > 0.0f &&
                            ath <= P.P_chi) {
                            landed = true;
                            k_end = k + 1;
                        } else {
                            sA.add(angdist(chi - fmaf(2.0f, th, kPi)));
                            sB.add(fabsf(beta - target));
                        }
                    } else {
                        sA.add(angdist(th - target));
                    }
                    if (P.w_noise != 0.0f && !landed) {
                        const float za = z * P.Ac_inv;
                        const float hh = fmaxf(fmaf(-za, za, 1.0f), 0.0f);
                        if (hh > 0.0f) sN = fmaf(hh, popdense_at(P, x, y), sN);
                    }
                }
                // the published position: far away once landed (the masks leave out
                // the aircraft that are not flying for another reason)
                buf[(e0 + e) * B + t] = make_float2(landed ? 1e30f : x, y);
                if constexpr (Log)
                    if (k < H) log.xy[olog] = make_float2(x, y);
                if constexpr (Soft) zbuf[(e0 + e) * B + t] = z;
                o += B;
                if constexpr (Log) olog += B;
                Wk += P.P;
            }
        }
        // bounds of the chunk's flying positions: x, then y
        float4 lim = make_float4(1e30f, -1e30f, 1e30f, -1e30f);
#pragma unroll
        for (int e = 0; e < KB; ++e) {
            const float2 q = buf[e * B + t];
            if (q.x < 1e30f && k0 + e >= k_in && k0 + e < kd)
                lim = make_float4(fminf(lim.x, q.x), fmaxf(lim.y, q.x), fminf(lim.z, q.y), fmaxf(lim.w, q.y));
        }
        bx[t] = lim;
        uint4 m4 = make_uint4(0u, 0u, 0u, 0u);
        if (up) m4 = __ldg(R.mask + ((unsigned)tile * n_chunks(H) + (unsigned)(k0 / KB)) * B + t);
        if constexpr (OwnWind) {
            for (int k = k0 + KB; k < min(k0 + 2 * KB, H); ++k) own_wind_step(k);
        }
        __syncthreads();
        // Separation among the partners within vertical reach.  First the bounds of
        // the whole chunk: subtraction and product round monotonically, so boxes
        // whose gap is beyond reach hold no position within it.
        unsigned cand = 0u;
        for (unsigned mk = m4.x | m4.y | m4.z | m4.w; mk != 0u; mk &= mk - 1u) {
            const int b = __ffs(mk) - 1;
            const float4 q = bx[partner_of(i, b, n_own, N) * TP + j];
            const float gx = fmaxf(fmaxf(lim.x - q.y, q.x - lim.y), 0.0f);
            const float gy = fmaxf(fmaxf(lim.z - q.w, q.z - lim.w), 0.0f);
            if (fmaf(gx, gx, gy * gy) < far2) cand |= 1u << b;
        }
        unsigned hits = 0u;        // Log: steps of the chunk with a partner within reach
        if (cand != 0u) {
#pragma unroll 1
            for (int e = 0; e < KB; ++e) {
                unsigned mk = cand & (e < 2 ? (e == 0 ? m4.x : m4.y) : (e == 2 ? m4.z : m4.w));
                if (mk == 0u) continue;
                const float2 *prow = buf + e * B + j;
                const float *zrow = zbuf + e * B + j;
                const float2 me = prow[i * TP];
                if (me.x >= 1e30f) continue;                 // landed: no pair, not even with another landed one
                const float zme = Soft ? zrow[i * TP] : 0.0f;
                float3 d = make_float3(0.0f, 0.0f, 0.0f);
                bool hit = false;
                for (; mk != 0u; mk &= mk - 1u) {
                    const int i2 = partner_of(i, __ffs(mk) - 1, n_own, N);
                    const float2 q = prow[i2 * TP];
                    const float dx = me.x - q.x, dy = me.y - q.y;
                    const float dh2 = fmaf(dx, dx, dy * dy);
                    if (dh2 < far2) {
                        if constexpr (Soft) {
                            const float adz = fabsf(zme - zrow[i2 * TP]);
                            if (dh2 < P.Sh2 && adz < P.Sv) sepv = true;
                            if constexpr (Log) {
                                const float dz = zme - zrow[i2 * TP];
                                const float2 ps = pair_penalty(P, dx, dy, dz);
                                soft = __fadd_rn(soft, ps.x);
                                pair_grad(P, sep_c * ps.y, dx, dy, dz, d.x, d.y, d.z);
                                hit = true;
                            } else {
                                const float pen = softplus(fminf(fmaf(-sqrtf(dh2), P.Sh_inv, 1.0f),
                                                                 fmaf(-adz, P.Sv_inv, 1.0f)),
                                                           P.sp_beta, P.sp_inv_beta);
                                // rounded before it is added, as the one-sample tile passes it on
                                soft = __fadd_rn(soft, pen);
                            }
                        } else {
                            sepv = true;
                            vflag[i2 * TP + j] = 1;
                        }
                    }
                }
                if constexpr (Log)
                    if (hit) {
                        hits |= 1u << e;
                        log.sep[((unsigned)log_tile * H + (unsigned)(k0 + e)) * B + t] = make_float4(d.x, d.y, d.z, 0.0f);
                    }
            }
        }
        if constexpr (Log) log.near[((unsigned)log_tile * n_chunks(H) + (unsigned)(k0 / KB)) * B + t] = hits;
    }
    if constexpr (!Soft) {
        __syncthreads();                       // the partners' last marks
        sepv = sepv || vflag[t] != 0;
    }
    Flown r;
    r.sA = sA;
    r.sB = sB;
    r.sN = sN;
    r.soft = soft;
    r.k_end = k_end;
    r.landed = landed;
    r.sepv = sepv;
    return r;
}

// trajectory_kernel over the particles [l_begin, l_end) (rollout_traj.cu); soft:
// masks of every partner within reach of a penalty; states: R.state too (with soft).
int traj_tile(int N);
void launch_trajectories(const ProblemC &P, const DynState *dyn, const float *u, long long l_begin, long long l_end,
                         const TrajOut &R, bool soft, cudaStream_t st, bool states = false);
// The records' bytes for n particles (a multiple of the tile) and their places in a buffer.
size_t traj_slab_bytes(const ProblemC &P, size_t n);
TrajOut traj_records(const ProblemC &P, size_t n, void *ws);

}  // namespace tma
