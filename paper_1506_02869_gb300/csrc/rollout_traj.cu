// Rollout in two kernels (the inner loop of Algorithm 1, Sec. 3.3-3.6, Sec. 7.1):
// what does not depend on the wind is computed once per particle, the rest once
// per wind sample.
//
// Of an aircraft's state only the position (x, y) depends on the wind: the
// altitude, airspeed and heading follow the controls alone (Eq. (hor) with
// v sin(gamma) = hdot, dv/dt = a, dchi/dt = w), and the thrust, the fuel flow
// and so the mass follow from those.  So the control and state limits, and
// whether two aircraft are vertically near enough to matter to each other, are
// the same under every wind sample.
//
//   trajectory_kernel   one thread per (particle, aircraft) runs those equations
//                       over the horizon and writes, per step, the new altitude,
//                       the ground-speed factors (v cos(gamma), cos chi, sin chi),
//                       arrivals' heading and fuel, and a bit mask of the partners
//                       within vertical reach; at the end the step at which a
//                       limit stopped the aircraft, the fuel burned and the
//                       departure's altitude and speed sums.
//   wind_rollout_kernel one thread per (particle, aircraft) and wind sample: wind,
//                       turbulence, position, bearing, glide angle, landing, and
//                       the horizontal distance to the partners in the mask.
//
// Both use the step function's own pieces (rollout_tile.cuh) in its order, so
// that the costs are the one-sample tile's bits.
//
// Bound: the L1 data pipe (four 16-byte gathers of the wind cell a step) and
// instruction issue, 78 and 65 % busy on the 8-aircraft workload.  Against the
// one-sample tile this drops from every sample's step the limit arithmetic, drag,
// thrust, fuel, two compensated sums, the sine and cosine of the heading and the
// vertical test of every pair (437 -> 262 warp instructions a step of 32
// aircraft, counted with 8 samples); it adds coalesced loads of 24 bytes a step.
// Positions are exchanged once per four steps, nothing of the motion depends on
// the partners.  Late particles: 8 aircraft, L 65536, M 32: 13.3 -> 9.4 ms; 24
// aircraft, soft, L 8192, M 64: 35.4 -> 28.7 ms; 10 aircraft with own winds, 6
// steps, 63 samples: 0.90 -> 0.72 ms.  Two samples per thread were slower (80
// registers with spills 12.5 ms, 128 registers 13.6 ms on the 8-aircraft
// workload), and so was fetching the next step's wind cell ahead of this step's
// terms (11.0 ms).
#include "rollout_tile.cuh"

namespace tma {

namespace {

// Records of a slab of particles, in tiles of TP particles, B = N TP threads:
// element ((tile H + k) B + t), t = i TP + j, for every array.
struct TrajOut {
    float4 *air;       // z after step k, v cos(gamma) (its sign bit: heading and speed fit the landing sector), cos chi, sin chi
    float *chi;        // arrivals: heading after step k
    float *fuel;       // arrivals: fuel burned after step k
    uint4 *mask;       // partner masks of the steps of chunk c: element ((tile nc + c) B + t), nc = ceil(H / 4)
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

template <int TP, bool Soft>
__global__ void __launch_bounds__(256) trajectory_kernel(const ProblemC P, const DynState *__restrict__ dyn,
                                                             const float *__restrict__ u, long long l_begin,
                                                             long long l_end, const TrajOut R)
{
    extern __shared__ float zsh[];                   // [2][kStepsPerBarrier][N][TP]
    const int N = P.N, B = N * TP;
    const int t = threadIdx.x, i = t / TP, j = t % TP;
    const long long l = l_begin + (long long)blockIdx.x * TP + j;
    const bool exists = l < l_end;
    const AircraftC A = P.ac[i];
    const uint32_t mpc = dyn->mpc_step;
    bool out;
    const int k_in = entry_step(P, A.t_enter, dyn, i, mpc, out);
    AcState s;
    ac_init(s, dyn, i, exists && !out, P.S);
    const float m0 = dyn->x0[i][5];
    const float *ul = u + ((size_t)(exists ? l : 0) * N + i) * (size_t)(P.S * 3);
    const int n_own = ((N - 1) >> 1) + (((N & 1) == 0 && i < (N >> 1)) ? 1 : 0);
    const int n_mask = Soft ? N - 1 : n_own;          // the hard form marks the partner of a violation
    const float reach = Soft ? P.sp_far_v : P.Sv;
    Kahan dB, dC;
    int kd = s.dead ? 0 : P.H;
    size_t o = (size_t)blockIdx.x * P.H * B + t, om = (size_t)blockIdx.x * n_chunks(P.H) * B + t;
    constexpr int KB = kStepsPerBarrier;
    static_assert(KB == 4, "a chunk's masks are one uint4");
    for (int k0 = 0; k0 < P.H; k0 += KB) {
        float *buf = zsh + ((k0 / KB) & 1) * KB * B;
        float zz[KB];
#pragma unroll
        for (int e = 0; e < KB; ++e) {
            const int k = k0 + e;
            zz[e] = 1e30f;                            // a far-away altitude when not flying
            if (!s.dead && k >= k_in && k < P.H) {
                segment_advance(P, s, ul, k);
                float cg, T, sc, cc;
                bool ok = control_limits(P, A, s, m0, cg, T);
                if (ok) {
                    sincos_reduced(s.chi, &sc, &cc);
                    const float vh = s.v * cg;
                    ok = air_advance(P, A, s, m0, k, T);
                    const bool fits = angdist(s.chi - kPi) <= P.P_chi && s.v <= P.P_vs;
                    R.air[o + (size_t)e * B] = make_float4(s.z, fits ? -vh : vh, cc, sc);
                    if (A.type == 0) {
                        R.chi[o + (size_t)e * B] = s.chi;
                        R.fuel[o + (size_t)e * B] = s.F.s;
                    } else if (ok) {
                        dB.add(fabsf(A.Z - s.z));
                        dC.add(fabsf(s.v - A.vD));
                    }
                }
                if (ok) {
                    zz[e] = s.z;
                } else {
                    s.dead = true;
                    kd = k;
                }
            }
            buf[e * B + t] = zz[e];
        }
        __syncthreads();
        unsigned mask[KB] = {0u, 0u, 0u, 0u};
        for (int b = 0; b < n_mask; ++b) {
            const float *zp = buf + j + partner_of(i, b, n_own, N) * TP;
#pragma unroll
            for (int e = 0; e < KB; ++e)
                if (zz[e] < 1e30f && fabsf(zz[e] - zp[e * B]) < reach) mask[e] |= 1u << b;
        }
        R.mask[om] = make_uint4(mask[0], mask[1], mask[2], mask[3]);
        om += B;
        o += (size_t)KB * B;
    }
    R.fin[(size_t)blockIdx.x * B + t] = make_float4(dB.s, dC.s, s.F.s, __int_as_float(kd));
}

// Shared memory of a block (32-bit words): positions float2 [2 (chunk parity)]
// [kStepsPerBarrier][N][TP], their bounds over the chunk float4 [2][N][TP]; soft:
// the altitudes as the positions; hard: separation flags [N][TP]; wind mode 1: the
// particles' wind state [2][kStepsPerBarrier][16][TP].
__host__ __device__ constexpr int wind_rollout_words(int N, int tp, bool soft, bool own_wind)
{
    return (2 * kStepsPerBarrier * N * (soft ? 3 : 2) + 8 * N + (soft ? 0 : N) +
            (own_wind ? 2 * kStepsPerBarrier * 16 : 0)) * tp;
}

template <int kMinBlocks, int TP, bool OwnWind, bool Soft>
__global__ void __launch_bounds__(256, kMinBlocks)
    wind_rollout_kernel(const ProblemC P, const DynState *__restrict__ dyn, const float4 *__restrict__ W,
                        const TrajOut R, long long L, long long l_begin, long long l_end, int n_tiles, int J,
                        float *__restrict__ cost_ms, float *__restrict__ cost_ms_soft,
                        unsigned long long *__restrict__ live)
{
    extern __shared__ __align__(16) float sh[];
    constexpr int KB = kStepsPerBarrier;
    const int N = P.N, H = P.H, B = N * TP;
    const int t = threadIdx.x, i = t / TP, j = t % TP;
    const int m = blockIdx.x / n_tiles, tile = blockIdx.x - m * n_tiles;    // sample: block-uniform, slowest
    const long long l = l_begin + (long long)tile * TP + j;
    const bool exists = l < l_end;
    const uint32_t mpc = dyn->mpc_step;
    const int type = P.ac[i].type;
    const float target = type == 0 ? P.beta_f : P.ac[i].thF;
    bool out;
    const int k_in = entry_step(P, P.ac[i].t_enter, dyn, i, mpc, out);
    const int kd = __float_as_int(R.fin[(size_t)tile * B + t].w);
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

    const float4 *Wk = W + (size_t)m * H * P.P;
    unsigned o = (unsigned)tile * H * B + t;                   // the workspace bound keeps the records within 32 bits
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
                if constexpr (Soft) zbuf[(e0 + e) * B + t] = z;
                o += B;
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
                for (; mk != 0u; mk &= mk - 1u) {
                    const int i2 = partner_of(i, __ffs(mk) - 1, n_own, N);
                    const float2 q = prow[i2 * TP];
                    const float dx = me.x - q.x, dy = me.y - q.y;
                    const float dh2 = fmaf(dx, dx, dy * dy);
                    if (dh2 < far2) {
                        if constexpr (Soft) {
                            const float adz = fabsf(zme - zrow[i2 * TP]);
                            if (dh2 < P.Sh2 && adz < P.Sv) sepv = true;
                            const float pen = softplus(fminf(fmaf(-sqrtf(dh2), P.Sh_inv, 1.0f), fmaf(-adz, P.Sv_inv, 1.0f)),
                                                       P.sp_beta, P.sp_inv_beta);
                            // rounded before it is added, as the one-sample tile passes it on
                            soft = __fadd_rn(soft, pen);
                        } else {
                            sepv = true;
                            vflag[i2 * TP + j] = 1;
                        }
                    }
                }
            }
        }
    }
    if constexpr (!Soft) __syncthreads();      // the partners' last marks

    const AircraftC A = P.ac[i];
    const float4 fn = R.fin[(size_t)tile * B + t];
    const int Ha = H - k_in;
    const AltBounds ab = alt_bounds(P, A, dyn->x0[i][2], Ha);
    const bool dead = !landed && kd < H;
    if constexpr (!Soft) sepv = sepv || vflag[t] != 0;
    CostSums cs;
    cs.sA = sA;
    cs.sB = sB;
    if (type != 0) {
        cs.sB.s = fn.x;
        cs.sC.s = fn.y;
    }
    cs.sN = sN;
    const float Fs = landed ? __ldg(R.fuel + ((unsigned)tile * H + (unsigned)(k_end - 1)) * B + t) : fn.z;
    const float c = -logf(fmaxf(total_objective(P, A, cs, Fs, ab, Ha), 1e-30f));
    unsigned tot = 0;
    if (exists) {
        const float inf = __int_as_float(0x7f800000);
        const size_t o = ((size_t)m * N + i) * (size_t)L + l;
        cost_ms[o] = out ? 0.0f : (dead || sepv) ? inf : c;
        if constexpr (Soft) cost_ms_soft[o] = out ? 0.0f : dead ? inf : fmaf(P.mu_sep, soft, c);
        if (!out) tot = (unsigned)((landed ? k_end : min(kd + 1, H)) - k_in);
    }
    if (live != nullptr) {
        const int in_warp = B - (t & ~31);            // lanes of this warp (the last one may be partly filled)
        const unsigned w = __reduce_add_sync(in_warp >= 32 ? 0xffffffffu : (1u << in_warp) - 1u, tot);
        if ((threadIdx.x & 31) == 0 && w) atomicAdd(live, (unsigned long long)w);
    }
}

}  // namespace

// Variants: minimum resident blocks of 256 threads (64 or 48 registers a thread).
// Late particles, hard form, 8 aircraft at L 65536: 9.57 and 9.43 ms (one-sample
// tile 13.26); soft form, 24 aircraft at L 8192: 28.7 and 29.4 ms (35.4).
constexpr int kTrajMinBlocks[] = {4, 5};
constexpr int kNumTrajVariants = sizeof(kTrajMinBlocks) / sizeof(kTrajMinBlocks[0]);
static_assert(kTrajVariantBase + kNumTrajVariants <= kMaxRolloutVariants, "variant table");

// Particles per block: as many as 256 threads allow, so that several blocks of any
// aircraft count share an SM and one block's barrier overlaps the others' work
// (768-thread blocks of 32 particles were no faster on 24 aircraft).
static int traj_tile(int N) { return N <= 8 ? 32 : (N <= 16 ? 16 : 8); }

// workspace bytes of a slab of n particles (a multiple of the tile)
static size_t traj_slab_bytes(const ProblemC &P, size_t n)
{
    return n * (size_t)P.N * ((size_t)P.H * (sizeof(float4) + 2 * sizeof(float)) +
                              (size_t)(n_chunks(P.H) + 1) * sizeof(float4));
}

size_t traj_workspace(const ProblemC &P, int64_t L)
{
    // 24-256 MB slabs ran 10-2 % slower than 1 GB ones on 65536 particles of 8 aircraft
    const size_t most = (size_t)512 << 20;
    const size_t per32 = traj_slab_bytes(P, 32);
    const size_t want = ((size_t)L + 31) / 32, fit = most / per32;
    // a slab of few tiles would leave the chip idle: no workspace, one-sample kernels
    if (fit < want && fit < 32) return 0;
    return (want < fit ? want : fit) * per32;
}

int rollout_traj_variants(const ProblemC &P, size_t ws_bytes, int *out)
{
    if (P.M < 2 || ws_bytes < traj_slab_bytes(P, 32)) return 0;
    for (int v = 0; v < kNumTrajVariants; ++v) out[v] = v;
    return kNumTrajVariants;
}

template <int MB, int TP>
static void launch_slab(const ProblemC &P, const DynState *dyn, const float *u, const float4 *W, const TrajOut &R,
                        int64_t L, long long l0, long long l1, int J, float *cost_ms, float *cost_ms_soft,
                        unsigned long long *live, cudaStream_t st)
{
    const int n_tiles = (int)((l1 - l0 + TP - 1) / TP);
    const bool soft = cost_ms_soft != nullptr;
    size_t smem = (size_t)2 * kStepsPerBarrier * P.N * TP * sizeof(float);
    if (soft) trajectory_kernel<TP, true><<<n_tiles, P.N * TP, smem, st>>>(P, dyn, u, l0, l1, R);
    else trajectory_kernel<TP, false><<<n_tiles, P.N * TP, smem, st>>>(P, dyn, u, l0, l1, R);
    smem = (size_t)wind_rollout_words(P.N, TP, soft, P.wind_mode == 1) * sizeof(float);
    const auto launch = [&](auto kernel) {
        // above the default 48 KB of dynamic shared memory the kernel must opt in
        if (smem > 48 * 1024) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        kernel<<<(unsigned)n_tiles * (unsigned)P.M, P.N * TP, smem, st>>>(P, dyn, W, R, L, l0, l1, n_tiles, J, cost_ms,
                                                                          cost_ms_soft, live);
    };
    if (P.wind_mode == 1) {
        if (soft) launch(wind_rollout_kernel<MB, TP, true, true>);
        else launch(wind_rollout_kernel<MB, TP, true, false>);
    } else {
        if (soft) launch(wind_rollout_kernel<MB, TP, false, true>);
        else launch(wind_rollout_kernel<MB, TP, false, false>);
    }
    count_launch(2);
}

cudaError_t launch_rollout_traj(const ProblemC &P, const DynState *dyn, const float *u, const float *W, int64_t L,
                                int J, float *cost_ms, float *cost_ms_soft, unsigned long long *live,
                                cudaStream_t st, int variant, void *ws, size_t ws_bytes)
{
    if (L <= 0) return cudaSuccess;
    const size_t slab = ws_bytes / traj_slab_bytes(P, 32) * 32;
    if (variant < 0 || variant >= kNumTrajVariants || P.M < 1 || !ws || slab == 0) return cudaErrorInvalidValue;
    const size_t n = slab < ((size_t)L + 31) / 32 * 32 ? slab : ((size_t)L + 31) / 32 * 32;
    TrajOut R;
    R.air = static_cast<float4 *>(ws);
    R.fin = R.air + n * P.N * (size_t)P.H;
    R.mask = reinterpret_cast<uint4 *>(R.fin + n * P.N);
    R.chi = reinterpret_cast<float *>(R.mask + n * P.N * (size_t)n_chunks(P.H));
    R.fuel = R.chi + n * P.N * (size_t)P.H;
    const float4 *W4 = reinterpret_cast<const float4 *>(W);
    for (int64_t l0 = 0; l0 < L; l0 += (int64_t)n) {
        const long long l1 = l0 + (int64_t)n < L ? l0 + (int64_t)n : L;
#define TMA_SLAB(MB, TP) launch_slab<MB, TP>(P, dyn, u, W4, R, L, l0, l1, J, cost_ms, cost_ms_soft, live, st)
        switch (traj_tile(P.N)) {
        case 32: if (variant == 0) TMA_SLAB(4, 32); else TMA_SLAB(5, 32); break;
        case 16: if (variant == 0) TMA_SLAB(4, 16); else TMA_SLAB(5, 16); break;
        default: if (variant == 0) TMA_SLAB(4, 8); else TMA_SLAB(5, 8); break;
        }
#undef TMA_SLAB
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace tma
