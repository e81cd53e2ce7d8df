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
// instruction issue, 73-78 and 63-65 % busy on the 8-aircraft workload.  Against the
// one-sample tile this drops from every sample's step the limit arithmetic, drag,
// thrust, fuel, two compensated sums, the sine and cosine of the heading and the
// vertical test of every pair (437 -> 258 warp instructions a step of 32
// aircraft, counted with 8 samples); it adds coalesced loads of 24 bytes a step.
// Positions are exchanged once per four steps, nothing of the motion depends on
// the partners.  Late particles: 8 aircraft, L 65536, M 32: 13.3 -> 9.4 ms; 24
// aircraft, soft, L 8192, M 64: 35.4 -> 28.7 ms; 10 aircraft with own winds, 6
// steps, 63 samples: 0.90 -> 0.72 ms.  Two samples per thread were slower (80
// registers with spills 12.5 ms, 128 registers 13.6 ms on the 8-aircraft
// workload), and so was fetching the next step's wind cell ahead of this step's
// terms (11.0 ms).
#include "wind_rollout.cuh"

namespace tma {

namespace {

template <int TP, bool Soft, bool States>
__global__ void __launch_bounds__(256) trajectory_kernel(const ProblemC P, const DynState *__restrict__ dyn,
                                                             const float *__restrict__ u, long long l_begin,
                                                             long long l_end, const TrajOut R)
{
    extern __shared__ float zsh[];                   // [2][kStepsPerBarrier][N][TP]
    grid_begin();
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
    if constexpr (States)
        if (i == 0) R.bad[(size_t)blockIdx.x * TP + j] = exists ? 0u : 1u;
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
                    if constexpr (States) R.state[o + (size_t)e * B] = make_float4(s.z, s.v, s.F.s, s.chi);
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

template <int kMinBlocks, int TP, bool OwnWind, bool Soft>
__global__ void __launch_bounds__(256, kMinBlocks)
    wind_rollout_kernel(const ProblemC P, const DynState *__restrict__ dyn, const float4 *__restrict__ W,
                        const TrajOut R, long long L, long long l_begin, long long l_end, int n_tiles, int J,
                        float *__restrict__ cost_ms, float *__restrict__ cost_ms_soft,
                        unsigned long long *__restrict__ live)
{
    extern __shared__ __align__(16) float sh[];
    grid_begin();
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

    const Flown q = wind_forward<TP, OwnWind, Soft, false>(P, dyn, W + (size_t)m * H * P.P, R, sh, tile, t, l, m, J, mpc,
                                                           type, target, k_in, kd, FlightLog(), 0, 0.0f);

    const AircraftC A = P.ac[i];
    const float4 fn = R.fin[(size_t)tile * B + t];
    const int Ha = H - k_in;
    const AltBounds ab = alt_bounds(P, A, dyn->x0[i][2], Ha);
    const bool dead = !q.landed && kd < H;
    CostSums cs;
    cs.sA = q.sA;
    cs.sB = q.sB;
    if (type != 0) {
        cs.sB.s = fn.x;
        cs.sC.s = fn.y;
    }
    cs.sN = q.sN;
    const float Fs = q.landed ? __ldg(R.fuel + ((unsigned)tile * H + (unsigned)(q.k_end - 1)) * B + t) : fn.z;
    const float c = -logf(fmaxf(total_objective(P, A, cs, Fs, ab, Ha), 1e-30f));
    unsigned tot = 0;
    if (exists) {
        const float inf = __int_as_float(0x7f800000);
        const size_t o = ((size_t)m * N + i) * (size_t)L + l;
        cost_ms[o] = out ? 0.0f : (dead || q.sepv) ? inf : c;
        if constexpr (Soft) cost_ms_soft[o] = out ? 0.0f : dead ? inf : fmaf(P.mu_sep, q.soft, c);
        if (!out) tot = (unsigned)((q.landed ? q.k_end : min(kd + 1, H)) - k_in);
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
int traj_tile(int N) { return N <= 8 ? 32 : (N <= 16 ? 16 : 8); }

// workspace bytes of a slab of n particles (a multiple of the tile)
size_t traj_slab_bytes(const ProblemC &P, size_t n)
{
    return n * (size_t)P.N * ((size_t)P.H * (sizeof(float4) + 2 * sizeof(float)) +
                              (size_t)(n_chunks(P.H) + 1) * sizeof(float4));
}

TrajOut traj_records(const ProblemC &P, size_t n, void *ws)
{
    TrajOut R;
    R.air = static_cast<float4 *>(ws);
    R.state = nullptr;
    R.bad = nullptr;
    R.fin = R.air + n * P.N * (size_t)P.H;
    R.mask = reinterpret_cast<uint4 *>(R.fin + n * P.N);
    R.chi = reinterpret_cast<float *>(R.mask + n * P.N * (size_t)n_chunks(P.H));
    R.fuel = R.chi + n * P.N * (size_t)P.H;
    return R;
}

size_t traj_workspace(const ProblemC &P, int64_t L)
{
    // 65536 particles of 8 aircraft, 32 samples: slabs of 24 MB 11.7 ms, 64-256 MB 10.5,
    // 512 MB 10.32, 1 GB 10.24
    const size_t most = (size_t)512 << 20;
    const size_t per32 = traj_slab_bytes(P, 32);
    const size_t want = ((size_t)L + 31) / 32, fit = most / per32;
    // A slab of fewer than 1024 particles would leave the chip idle: no workspace,
    // one-sample kernels.  (Long horizons: 32 aircraft beyond 584 steps.  With slabs of
    // 1024 they ran 6.1 -> 4.6 ms, hard, but 6.4 -> 7.1 ms, soft, and 12.3 -> 12.9 ms of
    // 8192 particles: the tuner's short first-iteration flights favour the two-kernel form.)
    if (fit < want && fit < 32) return 0;
    return (want < fit ? want : fit) * per32;
}

int rollout_traj_variants(const ProblemC &P, size_t ws_bytes, int *out)
{
    if (P.M < 2 || ws_bytes < traj_slab_bytes(P, 32)) return 0;
    for (int v = 0; v < kNumTrajVariants; ++v) out[v] = v;
    return kNumTrajVariants;
}

template <int TP>
static void launch_trajectories_tp(const ProblemC &P, const DynState *dyn, const float *u, long long l0, long long l1,
                                   const TrajOut &R, bool soft, bool states, cudaStream_t st)
{
    const int n_tiles = (int)((l1 - l0 + TP - 1) / TP);
    const size_t smem = (size_t)2 * kStepsPerBarrier * P.N * TP * sizeof(float);
    if (states) launch_dependent(trajectory_kernel<TP, true, true>, n_tiles, P.N * TP, smem, st, P, dyn, u, l0, l1, R);
    else if (soft) launch_dependent(trajectory_kernel<TP, true, false>, n_tiles, P.N * TP, smem, st, P, dyn, u, l0, l1, R);
    else launch_dependent(trajectory_kernel<TP, false, false>, n_tiles, P.N * TP, smem, st, P, dyn, u, l0, l1, R);
    count_launch();
}

void launch_trajectories(const ProblemC &P, const DynState *dyn, const float *u, long long l_begin, long long l_end,
                         const TrajOut &R, bool soft, cudaStream_t st, bool states)
{
    switch (traj_tile(P.N)) {
    case 32: launch_trajectories_tp<32>(P, dyn, u, l_begin, l_end, R, soft, states, st); break;
    case 16: launch_trajectories_tp<16>(P, dyn, u, l_begin, l_end, R, soft, states, st); break;
    default: launch_trajectories_tp<8>(P, dyn, u, l_begin, l_end, R, soft, states, st); break;
    }
}

template <int MB, int TP>
static void launch_slab(const ProblemC &P, const DynState *dyn, const float *u, const float4 *W, const TrajOut &R,
                        int64_t L, long long l0, long long l1, int J, float *cost_ms, float *cost_ms_soft,
                        unsigned long long *live, cudaStream_t st)
{
    const int n_tiles = (int)((l1 - l0 + TP - 1) / TP);
    const bool soft = cost_ms_soft != nullptr;
    launch_trajectories(P, dyn, u, l0, l1, R, soft, st);
    const size_t smem = (size_t)wind_rollout_words(P.N, TP, soft, P.wind_mode == 1) * sizeof(float);
    const auto launch = [&](auto kernel) {
        // above the default 48 KB of dynamic shared memory the kernel must opt in
        if (smem > 48 * 1024) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        launch_dependent(kernel, (unsigned)n_tiles * (unsigned)P.M, P.N * TP, smem, st, P, dyn, W, R, L, l0, l1, n_tiles, J,
                         cost_ms, cost_ms_soft, live);
    };
    if (P.wind_mode == 1) {
        if (soft) launch(wind_rollout_kernel<MB, TP, true, true>);
        else launch(wind_rollout_kernel<MB, TP, true, false>);
    } else {
        if (soft) launch(wind_rollout_kernel<MB, TP, false, true>);
        else launch(wind_rollout_kernel<MB, TP, false, false>);
    }
    count_launch();
}

cudaError_t launch_rollout_traj(const ProblemC &P, const DynState *dyn, const float *u, const float *W, int64_t L,
                                int J, float *cost_ms, float *cost_ms_soft, unsigned long long *live,
                                cudaStream_t st, int variant, void *ws, size_t ws_bytes)
{
    if (L <= 0) return cudaSuccess;
    const size_t slab = ws_bytes / traj_slab_bytes(P, 32) * 32;
    if (variant < 0 || variant >= kNumTrajVariants || P.M < 1 || !ws || slab == 0) return cudaErrorInvalidValue;
    const size_t n = slab < ((size_t)L + 31) / 32 * 32 ? slab : ((size_t)L + 31) / 32 * 32;
    const TrajOut R = traj_records(P, n, ws);
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
