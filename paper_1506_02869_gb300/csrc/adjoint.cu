// Reverse-mode derivative of the soft cost with respect to the controls: the
// gradient of C_l = sum_i (1/M) sum_m c_soft[i][m] (the rollout of Sec. 3.3-3.6
// and Sec. 7.1 with the softplus separation penalty; unary and control limits
// stay hard) for every particle l, used by the Langevin move.
//
// The wind enters the position alone, so the adjoint splits as the rollout does
// (rollout_traj.cu).  The adjoints of x and y run backwards under each sample; those of
// altitude, airspeed, heading and fuel propagate through factors that no sample
// changes, and they are linear in what x and y feed them, so they run once on the
// sums over the samples:
//   trajectory_kernel     the wind-independent records, once per particle;
//   grad_samples_kernel   per sample: the forward pass of the rollout, keeping the
//                         positions and the penalties' derivatives; its J_T fixes the
//                         cost coefficients; then backwards with the adjoint (x, y),
//                         adding the step's x and y adjoints and what they and the
//                         cost terms feed the altitude and the heading to sums over
//                         the block's samples (a block takes 32, 16 or 8 particles and a
//                         range of the samples, one after the other: no atomics, a
//                         fixed order);
//   grad_sum_kernel       with few tiles or many ranges, their sums, a thread per element;
//   grad_controls_kernel  the costs' means over the samples; once per particle:
//                         backwards with the summed sources, the altitude, airspeed, heading
//                         and fuel adjoints, and each segment's control gradient.
// Limit, landing and interpolation-cell decisions keep their forward values.
//
// Bound: instruction issue (52 % busy, 750 warp instructions a step of 32 aircraft,
// forward and back together; 1400 with the whole adjoint per sample) and the latency
// of the wind gathers, here twice a step; DRAM 31 % for the sums and the flight log.
// Late particles, 12 aircraft, L 16384, M 16: 11.5 -> 7.4 ms; 24 aircraft, L 4096, M 8,
// 90 steps: 6.13 -> 3.64 ms; 6 aircraft, L 4096, M 8: 0.66 -> 0.52 ms.  Of the 7.4 ms
// the backward half is 3.2, the pairs 1.5, grad_controls_kernel 0.2.  With few particles
// the four chains of dependent steps are the time, and grad_controls_kernel must not add
// waits for memory to them: summing the ranges inside it, four steps at a time, took 8
// aircraft, 90 steps, L 200, M 40 from 457 us (one kernel, checkpoints) to 1250 us, the
// sums by a kernel of their own and the fetch ahead to 429 us.
#include "wind_rollout.cuh"

#include <algorithm>

namespace tma {

namespace {

// wrapped angle in [-pi, pi] (the signed counterpart of angdist)
__device__ __forceinline__ float wrapf(float a)
{
    const float twopi = 6.28318530717958647692f;
    return a - twopi * rintf(a * (1.0f / twopi));
}

// Trilinear wind and its derivative with respect to position; zero along an
// axis where the position lies outside the box (it is clamped there).
__device__ __forceinline__ void wind_grad(const ProblemC &P, const float4 *__restrict__ Wk, float x,
                                          float y, float z, float2 &dwx, float2 &dwy, float2 &dwz)
{
    const WindFetch f = wind_fetch(P, Wk, x, y, z);
    float2 c00, c01, c10, c11, e00, e01, e10, e11;
    // records hold (value, difference to the node one level up)
    c00.x = fmaf(f.tz, f.a00.z, f.a00.x); c00.y = fmaf(f.tz, f.a00.w, f.a00.y);
    c01.x = fmaf(f.tz, f.a01.z, f.a01.x); c01.y = fmaf(f.tz, f.a01.w, f.a01.y);
    c10.x = fmaf(f.tz, f.a10.z, f.a10.x); c10.y = fmaf(f.tz, f.a10.w, f.a10.y);
    c11.x = fmaf(f.tz, f.a11.z, f.a11.x); c11.y = fmaf(f.tz, f.a11.w, f.a11.y);
    e00 = make_float2(f.a00.z, f.a00.w);
    e01 = make_float2(f.a01.z, f.a01.w);
    e10 = make_float2(f.a10.z, f.a10.w);
    e11 = make_float2(f.a11.z, f.a11.w);
    float2 c0, c1, e0, e1;
    c0.x = fmaf(f.ty, c01.x - c00.x, c00.x); c0.y = fmaf(f.ty, c01.y - c00.y, c00.y);
    c1.x = fmaf(f.ty, c11.x - c10.x, c10.x); c1.y = fmaf(f.ty, c11.y - c10.y, c10.y);
    e0.x = fmaf(f.ty, e01.x - e00.x, e00.x); e0.y = fmaf(f.ty, e01.y - e00.y, e00.y);
    e1.x = fmaf(f.ty, e11.x - e10.x, e10.x); e1.y = fmaf(f.ty, e11.y - e10.y, e10.y);
    const bool ix = x > P.box_lo[0] && x < P.box_hi[0];
    const bool iy = y > P.box_lo[1] && y < P.box_hi[1];
    const bool iz = z > P.box_lo[2] && z < P.box_hi[2];
    // d/dx: difference across the x cell; d/dy: across y, bilinear in x; d/dz likewise
    dwx = ix ? make_float2((c1.x - c0.x) * P.inv_h[0], (c1.y - c0.y) * P.inv_h[0]) : make_float2(0.f, 0.f);
    const float2 dy0 = make_float2(c01.x - c00.x, c01.y - c00.y);
    const float2 dy1 = make_float2(c11.x - c10.x, c11.y - c10.y);
    dwy = iy ? make_float2(fmaf(f.tx, dy1.x - dy0.x, dy0.x) * P.inv_h[1],
                           fmaf(f.tx, dy1.y - dy0.y, dy0.y) * P.inv_h[1])
             : make_float2(0.f, 0.f);
    dwz = iz ? make_float2(fmaf(f.tx, e1.x - e0.x, e0.x) * P.inv_h[2],
                           fmaf(f.tx, e1.y - e0.y, e0.y) * P.inv_h[2])
             : make_float2(0.f, 0.f);
}

// Population density (Sec. 7.1) and its gradient; 0 outside the grid.
__device__ __forceinline__ float popdense_grad(const ProblemC &P, float x, float y, float &gx, float &gy)
{
    gx = gy = 0.0f;
    if (P.popcell == nullptr) return 0.0f;
    if (!(x >= P.pop_lo[0] && x <= P.pop_hi[0] && y >= P.pop_lo[1] && y <= P.pop_hi[1]))
        return 0.0f;
    const float f0 = (x - P.pop_lo[0]) * P.pop_inv_h[0];
    const float f1 = (y - P.pop_lo[1]) * P.pop_inv_h[1];
    const int i0 = min((int)f0, P.pop_n[0] - 2), i1 = min((int)f1, P.pop_n[1] - 2);
    const float t0 = f0 - (float)i0, t1 = f1 - (float)i1;
    const float4 g = __ldg(P.popcell + (size_t)i0 * (P.pop_n[1] - 1) + i1);
    const float g00 = g.x, g01 = g.y, g10 = g.z, g11 = g.w;
    gx = fmaf(t1, (g11 - g01) - (g10 - g00), g10 - g00) * P.pop_inv_h[0];
    gy = fmaf(t0, (g11 - g10) - (g01 - g00), g01 - g00) * P.pop_inv_h[1];
    const float a = fmaf(t1, g01 - g00, g00), b = fmaf(t1, g11 - g10, g10);
    return fmaf(t0, b - a, a);
}

// Coefficients d c / d (deviation sums, fuel) of one aircraft's per-sample cost
// c = -ln J_T, already divided by M.
struct CostGrad {
    float gA, gB, gC, gN, gF;
};

__device__ __forceinline__ CostGrad cost_grad(const ProblemC &P, const AircraftC &A, float JT,
                                              AltBounds ab, float invM)
{
    CostGrad g{0.f, 0.f, 0.f, 0.f, 0.f};
    if (!(JT > 1e-30f)) return g;            // the cost is clamped there
    const float invH = 1.0f / (float)P.H;
    const float s = -invM / JT;              // d c / d J_T, over M
    const float wj = (1.0f - P.w_noise) * s;
    if (A.type == 1) {
        g.gA = wj * (-P.a_dep[0] * invH / kPi);
        g.gB = wj * (-P.a_dep[2] * invH * ab.invSupInf);
        g.gC = wj * (-P.a_dep[3] * invH * A.invCmax);
        g.gF = wj * (-P.a_dep[1] * A.invFmax);
    } else {
        g.gA = wj * (-P.a_arr[0] * invH / kPi);
        g.gB = wj * (-P.a_arr[1] * invH * (2.0f / kPi));
        g.gF = wj * (-P.a_arr[2] * A.invFmax);
    }
    g.gN = s * (-P.w_noise * invH);
    return g;
}


// Derivative of a pair of deviation terms with respect to the position a sample
// reaches at a step: (x, y) go to the sample's own adjoint, z and chi to the sums.
struct Sources {
    float x = 0.f, y = 0.f, z = 0.f, chi = 0.f;
    __device__ __forceinline__ void bearing(float px, float py, float coef)
    {
        const float r2 = fmaf(px, px, py * py);
        const float ir2 = r2 > 0.0f ? 1.0f / r2 : 0.0f;
        x = fmaf(coef, -py * ir2, x);
        y = fmaf(coef, px * ir2, y);
    }
    // th, beta: the bearing and the glide angle there
    __device__ __forceinline__ void arrival(const ProblemC &P, const CostGrad &cg, float px, float py, float pz, float chi1,
                                            float th, float beta)
    {
        const float se = sgnf(wrapf(chi1 - fmaf(2.0f, th, kPi))) * cg.gA;
        chi += se;
        bearing(px, py, -2.0f * se);
        // glide angle beta = atan2(z, r ratio(theta)), ratio = |theta| / sin|theta|
        const float r = sqrtf(fmaf(px, px, py * py));
        const float ath = fabsf(th);
        float ratio, dratio;
        if (ath < 1e-3f) {
            ratio = fmaf(th * th, 1.0f / 6.0f, 1.0f);
            dratio = th * (1.0f / 3.0f);
        } else {
            float sn, cs;
            __sincosf(ath, &sn, &cs);                 // ath in [0, pi]: no range reduction needed
            if (sn >= 0.25f * ath) {
                ratio = ath / sn;
                dratio = sgnf(th) * (sn - ath * cs) / (sn * sn);
            } else {
                ratio = 4.0f;
                dratio = 0.0f;
            }
        }
        const float sa = r * ratio;
        const float den = fmaf(pz, pz, sa * sa);
        const float bb = cg.gB * sgnf(beta - P.beta_f);
        z = fmaf(bb, sa / den, z);
        // d(sa)/dx = ratio x / r + r ratio'(theta) dtheta/dx, likewise for y
        const float bsa = -bb * pz / den;
        const float ir = r > 0.0f ? 1.0f / r : 0.0f;
        x = fmaf(bsa, ratio * px * ir, x);
        y = fmaf(bsa, ratio * py * ir, y);
        bearing(px, py, bsa * r * dratio);
    }
    __device__ __forceinline__ void noise(const ProblemC &P, const CostGrad &cg, float px, float py, float pz)
    {
        const float za = pz * P.Ac_inv;
        const float h = fmaf(-za, za, 1.0f);
        if (h > 0.0f) {
            float gx, gy;
            const float pd = popdense_grad(P, px, py, gx, gy);
            x = fmaf(cg.gN * h, gx, x);
            y = fmaf(cg.gN * h, gy, y);
            z = fmaf(cg.gN * pd, -2.0f * pz * P.Ac_inv * P.Ac_inv, z);
        }
    }
};

// Scratch of a slab of n particles and nchunk ranges of samples, in the records' tiles;
// element ((g H + k) B + t) with g = range n_tiles + tile.
struct GradScratch {
    FlightLog log;     // the current sample's flight
    float4 *acc;       // sums over the range's samples: adjoints of x and y after step k; what feeds those of z and chi there
    float *land;       // fuel coefficients of the samples that landed at step k (arrivals)
    float4 *sums;      // [g][B]: sums of the samples' coefficients of altitude, speed and (not landed) fuel
};

template <int kMinBlocks, int TP>
__global__ void __launch_bounds__(256, kMinBlocks)
    grad_samples_kernel(const ProblemC P, const DynState *__restrict__ dyn, const float4 *__restrict__ W, const TrajOut R,
                        const GradScratch G, long long L, long long l_begin, long long l_end, int n_tiles, int m_per_block,
                        int J, float *__restrict__ cost_ms)
{
    extern __shared__ __align__(16) float sh[];
    grid_begin();
    const int N = P.N, H = P.H, B = N * TP;
    const int t = threadIdx.x, i = t / TP, j = t % TP;
    const int range = blockIdx.x / n_tiles, tile = blockIdx.x - range * n_tiles;
    const long long l = l_begin + (long long)tile * TP + j;
    const bool exists = l < l_end;
    const uint32_t mpc = dyn->mpc_step;
    const int type = P.ac[i].type;
    const float target = type == 0 ? P.beta_f : P.ac[i].thF;
    const int kd = __float_as_int(R.fin[(size_t)tile * B + t].w);
    const float invM = 1.0f / (float)P.M;
    const float sep_c = 2.0f * P.mu_sep * invM;        // each pair enters two aircraft's costs
    const unsigned g0 = (unsigned)blockIdx.x * H * B + t;         // the scratch bound keeps these within 32 bits
    const unsigned r0 = (unsigned)tile * H * B + t;
    float sB = 0.0f, sC = 0.0f, sF = 0.0f;
    float sinF, cosF;
    sincosf(P.ac[i].thF, &sinF, &cosF);
    if (type == 0)
        for (int k = 0; k < H; ++k) G.land[g0 + (unsigned)k * B] = 0.0f;
    const int mb = range * m_per_block, me = min(P.M, mb + m_per_block);
    for (int m = mb; m < me; ++m) {
        if (m > mb) __syncthreads();              // the previous sample's positions are read
        const float4 *Wm = W + (size_t)m * H * P.P;
        const Flown q = wind_forward<TP, false, true, true>(P, dyn, Wm, R, sh, tile, t, l, m, J, mpc, type, target, 0, kd,
                                                            G.log, (int)blockIdx.x, sep_c);
        const bool dead = !q.landed && kd < H;
        CostGrad cg;
        {
            const AircraftC A = P.ac[i];
            const float4 fn = R.fin[(size_t)tile * B + t];
            const AltBounds ab = alt_bounds(P, A, dyn->x0[i][2], H);
            CostSums cs;
            cs.sA = q.sA;
            cs.sB = q.sB;
            if (type != 0) {
                cs.sB.s = fn.x;
                cs.sC.s = fn.y;
            }
            cs.sN = q.sN;
            const float Fs = q.landed ? __ldg(R.fuel + r0 + (unsigned)(q.k_end - 1) * B) : fn.z;
            const float JT = total_objective(P, A, cs, Fs, ab, H);
            if (exists)
                cost_ms[((size_t)m * N + i) * (size_t)L + l] =
                    dead ? __int_as_float(0x7f800000) : fmaf(P.mu_sep, q.soft, -logf(fmaxf(JT, 1e-30f)));
            cg = cost_grad(P, A, JT, ab, invM);
        }
        if (dead || !exists) {                     // an infeasible particle's gradient is zero
            if (exists) R.bad[(size_t)tile * TP + j] = 1u;
            continue;
        }
        // the landing step itself has no terms, only the fuel burned up to it
        const int k_top = q.landed ? q.k_end - 1 : H;
        if (q.landed) {
            G.land[g0 + (unsigned)k_top * B] += cg.gF;
        } else {
            sF += cg.gF;
        }
        if (type != 0) {
            sB += cg.gB;
            sC += cg.gC;
        }
        if (m == mb)
            for (int k = k_top; k < H; ++k) G.acc[g0 + (unsigned)k * B] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (k_top == 0) continue;
        float X = 0.0f, Y = 0.0f, zc = 0.0f;       // adjoints of the position; what step k + 1 feeds the altitude's
        // positions after step k, before it, and before step k - 1, the last one in
        // flight while step k is worked on (its wind cell's address needs it)
        const float2 pi = make_float2(dyn->x0[i][0], dyn->x0[i][1]);
        const float zi = dyn->x0[i][2];
        unsigned o = (unsigned)(k_top - 1) * B;
        float2 p = G.log.xy[g0 + o], p0 = pi;
        float z = __ldg(R.air + r0 + o).x, z0 = zi;
        if (k_top > 1) {
            p0 = G.log.xy[g0 + o - B];
            z0 = __ldg(R.air + r0 + o - B).x;
        }
        for (int k = k_top - 1; k >= 0; --k) {
            float2 pn = pi;
            float zn = zi;
            if (k > 1) {
                pn = G.log.xy[g0 + o - 2 * B];
                zn = __ldg(R.air + r0 + o - 2 * B).x;
            }
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
            if (m > mb) a = G.acc[g0 + o];
            float2 pol = make_float2(0.f, 0.f);
            if (type == 0) pol = G.log.polar[g0 + o];
            const unsigned near = G.log.near[((unsigned)blockIdx.x * n_chunks(H) + (unsigned)(k / kStepsPerBarrier)) * B + t];
            float2 dwx, dwy, dwz;
            wind_grad(P, Wm + (size_t)k * P.P, p0.x, p0.y, z0, dwx, dwy, dwz);
            Sources s;
            // a departure's bearing error has the sign of the cross product of its
            // target direction and its position
            if (type == 0) s.arrival(P, cg, p.x, p.y, z, __ldg(R.chi + r0 + o), pol.x, pol.y);
            else s.bearing(p.x, p.y, sgnf(fmaf(cosF, p.y, -sinF * p.x)) * cg.gA);
            if (P.w_noise != 0.0f) s.noise(P, cg, p.x, p.y, z);
            if ((near >> (k % kStepsPerBarrier)) & 1u) {
                const float4 d = G.log.sep[g0 + o];
                s.x += d.x;
                s.y += d.y;
                s.z += d.z;
            }
            X += s.x;
            Y += s.y;
            G.acc[g0 + o] = make_float4(a.x + X, a.y + Y, a.z + (s.z + zc), a.w + s.chi);
            const float nX = X + P.dt * fmaf(X, dwx.x, Y * dwx.y);
            const float nY = Y + P.dt * fmaf(X, dwy.x, Y * dwy.y);
            zc = P.dt * fmaf(X, dwz.x, Y * dwz.y);
            X = nX;
            Y = nY;
            p = p0;
            z = z0;
            p0 = pn;
            z0 = zn;
            o -= B;
        }
    }
    G.sums[(size_t)blockIdx.x * B + t] = make_float4(sB, sC, sF, 0.0f);
}

// Derivatives of step k of one aircraft that no sample changes (Eq. (hor) with the
// drag of the coordinated turn in closed form, D = q CD0 + CD2 m^2 (g^2 cos^2(gamma)
// + w^2 v^2) / q, q = rho v^2 S / 2), times the step dt where they enter.
struct StepCoef {
    float cc, sc;              // heading
    float vP, cP, hP;          // along-track adjoint to V, cross-track to CH, along-track to the climb control
    float e;                   // fuel adjoint to the thrust: dt eta
    float zT, vT, mT;          // thrust (fuel) to Z, V (with eta's own share), and to FF
    float wT, hT, aT;          // thrust to the controls
};

__device__ __forceinline__ StepCoef step_coef(const ProblemC &P, const AircraftC &A, float z, float v, float chi,
                                              float mass, float uw, float uh, float ua)
{
    const float dt = P.dt;
    const float iv = 1.0f / v;
    const float sg = uh * iv;
    const float cg = sqrtf(fmaxf(1.0f - sg * sg, 1e-12f));
    const float icg = 1.0f / cg;
    const float dcg_dv = uh * uh * iv * iv * iv * icg;
    const float dcg_dh = -uh * iv * iv * icg;
    const float base = fmaxf(fmaf(-2.2558e-5f, z, 1.0f), 1e-30f);
    const float rho = 1.225f * ex2_approx(4.2559f * __log2f(base));   // as the forward step
    const float q = A.halfS * rho * v * v;
    const float iq = 1.0f / q;
    const float dq_dz = q * (4.2559f * -2.2558e-5f) / base;
    const float dq_dv = 2.0f * q * iv;
    const float g2 = kG0 * kG0;
    const float A2 = fmaf(g2, 1.0f - sg * sg, uw * uw * v * v);
    const float dA2_dv = 2.0f * g2 * uh * uh * iv * iv * iv + 2.0f * uw * uw * v;
    const float dA2_dh = -2.0f * g2 * uh * iv * iv;
    const float dA2_dw = 2.0f * uw * v * v;
    const float K2 = A.CD2 * mass * mass;
    const float D = fmaf(q, A.CD0, K2 * A2 * iq);
    const float T = fmaf(mass, fmaf(kG0, sg, ua), D);
    const float dD_dv = fmaf(A.CD0, dq_dv, K2 * (dA2_dv * iq - A2 * dq_dv * iq * iq));
    const float dD_dz = fmaf(A.CD0, dq_dz, -K2 * A2 * dq_dz * iq * iq);
    const float dD_dm = 2.0f * A.CD2 * mass * A2 * iq;
    const float dT_dv = fmaf(-mass * kG0 * uh, iv * iv, dD_dv);
    const float eta = A.Cf1 * fmaf(v, A.invCf2, 1.0f);
    const float deta_dv = A.Cf1 * A.invCf2;
    StepCoef c;
    sincos_reduced(chi, &c.sc, &c.cc);
    c.vP = dt * (cg + v * dcg_dv);
    c.cP = dt * v * cg;
    c.hP = dt * v * dcg_dh;
    c.e = dt * eta;
    c.zT = dD_dz;
    c.vT = dt * fmaf(deta_dv, T, eta * dT_dv);
    c.mT = ua + kG0 * sg + dD_dm;
    c.wT = K2 * dA2_dw * iq;
    c.hT = fmaf(mass * kG0, iv, K2 * dA2_dh * iq);
    c.aT = mass;
    return c;
}

// Sums over the ranges of samples, into the first range's place: one thread per KS steps
// of a (tile, thread t of B), the ranges in order; an infeasible particle's are left out.
// Four steps a thread where one would be more threads than the chip holds: a quarter of
// the blocks to start, and of those that find their particles infeasible.
template <int KS>
__global__ void __launch_bounds__(256) grad_sum_kernel(const ProblemC P, const GradScratch G,
                                                       const unsigned *__restrict__ bad, unsigned threads, int n_tiles,
                                                       int B, int tp, int n_ranges)
{
    grid_begin();
    const unsigned e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= threads) return;
    const unsigned row = e / (unsigned)B, t = e - row * (unsigned)B;
    const unsigned per = (unsigned)(P.H + KS - 1) / KS, tile = row / per, k0 = (row - tile * per) * KS;
    const unsigned ac = t / (unsigned)tp;
    if (bad[tile * (unsigned)tp + (t - ac * (unsigned)tp)] != 0u) return;
    const bool arrival = P.ac[ac].type == 0;
    const size_t range = (size_t)n_tiles * P.H * B;
    const size_t o = ((size_t)tile * P.H + k0) * B + t;
    const int steps = min(KS, P.H - (int)k0);
    float4 a[KS];
    float lf[KS];
#pragma unroll
    for (int q = 0; q < KS; ++q) {
        a[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        lf[q] = 0.0f;
    }
#pragma unroll(KS == 1 ? 8 : 2)
    for (int c = 0; c < n_ranges; ++c) {
#pragma unroll
        for (int q = 0; q < KS; ++q) {
            const size_t at = c * range + o + (size_t)min(q, steps - 1) * B;
            const float4 v = G.acc[at];
            a[q].x += v.x;
            a[q].y += v.y;
            a[q].z += v.z;
            a[q].w += v.w;
            if (arrival) lf[q] += G.land[at];
        }
    }
#pragma unroll
    for (int q = 0; q < KS; ++q) {
        if (q >= steps) break;
        G.acc[o + (size_t)q * B] = a[q];
        if (arrival) G.land[o + (size_t)q * B] = lf[q];
    }
    if (k0 == 0) {
        const unsigned so = tile * (unsigned)B + t;
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
        for (int c = 0; c < n_ranges; ++c) {
            const float4 q = G.sums[(size_t)c * n_tiles * B + so];
            s.x += q.x;
            s.y += q.y;
            s.z += q.z;
        }
        G.sums[so] = s;
    }
}

// Ahead: four steps are fetched while the four after them are worked on, from sums over
// all the samples (n_ranges 1): for grids that leave the chip idle, where waiting for each
// four is the kernel's time.  Else the ranges are summed here, with twice the blocks
// resident instead.
template <int TP, bool Ahead>
__global__ void __launch_bounds__(256, Ahead ? 1 : 2)
    grad_controls_kernel(const ProblemC P, const DynState *__restrict__ dyn, const float *__restrict__ u, const TrajOut R,
                         const GradScratch G, long long l_begin, long long l_end, int n_tiles, int n_ranges,
                         const float *__restrict__ cost_ms, long long L, float *__restrict__ cost,
                         float *__restrict__ grad, float *__restrict__ cbar)
{
    constexpr int KC = 4;
    __shared__ float means[256];
    grid_begin();
    const int N = P.N, H = P.H, B = N * TP, nS3 = P.S * 3;
    const int t = threadIdx.x, i = t / TP, j = t % TP;
    const int tile = blockIdx.x;
    const long long l = l_begin + (long long)tile * TP + j;
    // this aircraft's sample mean (as the rollout's: compensated, in sample order,
    // +inf when any sample was infeasible), then the particle's sum C_l
    float cb = __int_as_float(0x7f800000);
    if (l < l_end) {
        Kahan s;
        bool inf = false;
#pragma unroll 8
        for (int m = 0; m < P.M; ++m) {
            const float v = __ldg(cost_ms + ((size_t)m * N + i) * (size_t)L + l);
            if (isinf(v)) inf = true;
            else s.add(v);
        }
        if (!inf) cb = s.s / (float)P.M;
        if (cbar) cbar[(size_t)i * L + l] = cb;
    }
    means[t] = cb;
    __syncthreads();
    if (l >= l_end) return;
    bool infeasible = false;
    for (int q = 0; q < N; ++q) infeasible = infeasible || isinf(means[q * TP + j]);
    if (i == 0) {
        double tot = 0.0;
        for (int q = 0; q < N; ++q) tot += (double)means[q * TP + j];
        cost[l] = infeasible ? __int_as_float(0x7f800000) : (float)tot;
    }
    float *gout = grad + ((size_t)l * N + i) * (size_t)nS3;
    for (int n = 0; n < nS3; ++n) gout[n] = 0.0f;
    if (infeasible) return;
    const AircraftC A = P.ac[i];
    const float m0 = dyn->x0[i][5];
    const float *ul = u + ((size_t)l * N + i) * (size_t)nS3;
    const float4 *state = R.state + (size_t)tile * H * B + t;
    // every sample's flight has ended (in a landing) before a step beyond a limit
    const int k_stop = __float_as_int(R.fin[(size_t)tile * B + t].w);
    if (k_stop == 0) return;
    float gB = 0.0f, gC = 0.0f, FF = 0.0f;
    for (int c = 0; c < n_ranges; ++c) {
        const float4 q = G.sums[((size_t)c * n_tiles + tile) * B + t];
        gB += q.x;
        gC += q.y;
        FF += q.z;
    }
    float Z = 0.f, V = 0.f, CH = 0.f, gw = 0.f, gh = 0.f, ga = 0.f;
    int seg = (int)((long long)(k_stop - 1) * P.S / H);                 // the segment of step k
    int k_seg = (int)(((long long)seg * H + P.S - 1) / P.S);            // and its first step
    float4 post = state[(size_t)(k_stop - 1) * B];                      // the state after step k
    const float4 *acc = G.acc + (size_t)tile * H * B + t;
    const float *land = G.land + (size_t)tile * H * B + t;
    // four steps: the states before them and the sums over the ranges, all these
    // loads in flight together (one after the other they are the kernel's time)
    struct Steps {
        float4 pre[KC], a[KC];
        float lf[KC];
    };
    const auto fetch = [&](Steps &q, int kt) {
#pragma unroll
        for (int e = 0; e < KC; ++e) {
            const int k = kt - e;
            q.pre[e] = k > 0 ? state[(size_t)(k - 1) * B]
                             : make_float4(dyn->x0[i][2], dyn->x0[i][3], 0.0f, dyn->x0[i][4]);
            q.a[e] = make_float4(0.f, 0.f, 0.f, 0.f);
            q.lf[e] = 0.0f;
            if constexpr (Ahead) {
                q.a[e] = acc[(size_t)max(k, 0) * B];
                if (A.type == 0) q.lf[e] = land[(size_t)max(k, 0) * B];
            }
        }
        if constexpr (!Ahead) {
            const size_t range = (size_t)n_tiles * H * B;
#pragma unroll 2
            for (int c = 0; c < n_ranges; ++c)
#pragma unroll
                for (int e = 0; e < KC; ++e) {
                    const float4 v = acc[c * range + (size_t)max(kt - e, 0) * B];
                    q.a[e].x += v.x;
                    q.a[e].y += v.y;
                    q.a[e].z += v.z;
                    q.a[e].w += v.w;
                }
            if (A.type == 0) {
#pragma unroll 2
                for (int c = 0; c < n_ranges; ++c)
#pragma unroll
                    for (int e = 0; e < KC; ++e) q.lf[e] += land[c * range + (size_t)max(kt - e, 0) * B];
            }
        }
    };
    Steps now, next;
    if constexpr (Ahead) fetch(now, k_stop - 1);
    for (int kt = k_stop - 1; kt >= 0; kt -= KC) {
        if constexpr (Ahead) fetch(next, kt - KC);
        else fetch(now, kt);
#pragma unroll
        for (int e = 0; e < KC; ++e) {
            const int k = kt - e;
            if (k < 0) break;
            if (k < k_seg) {
                gout[3 * seg] = gw;
                gout[3 * seg + 1] = gh;
                gout[3 * seg + 2] = ga;
                gw = gh = ga = 0.0f;
                --seg;
                k_seg = (int)(((long long)seg * H + P.S - 1) / P.S);
            }
            const StepCoef c = step_coef(P, A, now.pre[e].x, now.pre[e].y, now.pre[e].w, m0 - now.pre[e].z,
                                         __ldg(ul + 3 * seg), __ldg(ul + 3 * seg + 1), __ldg(ul + 3 * seg + 2));
            Z += now.a[e].z;
            CH += now.a[e].w;
            FF += now.lf[e];
            if (A.type != 0) {
                Z = fmaf(gB, sgnf(post.x - A.Z), Z);
                V = fmaf(gC, sgnf(post.y - A.vD), V);
            }
            const float proj = fmaf(c.cc, now.a[e].x, c.sc * now.a[e].y);      // along-track adjoint
            const float fe = FF * c.e;                                  // fuel adjoint times d F'/d T
            gw += fmaf(P.dt, CH, fe * c.wT);
            gh += P.dt * Z + c.hP * proj + fe * c.hT;
            ga += fmaf(P.dt, V, fe * c.aT);
            V += c.vP * proj + FF * c.vT;
            CH += c.cP * fmaf(-c.sc, now.a[e].x, c.cc * now.a[e].y);
            Z += fe * c.zT;
            FF -= fe * c.mT;
            post = now.pre[e];
        }
        if constexpr (Ahead) now = next;
    }
    gout[3 * seg] = gw;
    gout[3 * seg + 1] = gh;
    gout[3 * seg + 2] = ga;
}

// bytes of the scratch of n particles (a multiple of the tile), and its places in a buffer
size_t grad_bytes(const ProblemC &P, size_t n, int n_ranges)
{
    const size_t steps = n * (size_t)P.N * (size_t)P.H;
    return traj_slab_bytes(P, n) + steps * sizeof(float4) + n * sizeof(unsigned) +
           (size_t)n_ranges * (steps * (2 * sizeof(float4) + 2 * sizeof(float2) + sizeof(float)) +
                               n * (size_t)P.N * ((size_t)n_chunks(P.H) * sizeof(unsigned) + sizeof(float4)));
}

GradScratch grad_places(const ProblemC &P, size_t n, int n_ranges, void *ws, TrajOut &R)
{
    const size_t ac = n * (size_t)P.N, steps = ac * (size_t)P.H;
    GradScratch G;
    R = traj_records(P, n, ws);
    R.state = reinterpret_cast<float4 *>(static_cast<char *>(ws) + traj_slab_bytes(P, n));
    G.acc = R.state + steps;
    G.log.sep = G.acc + steps * n_ranges;
    G.sums = G.log.sep + steps * n_ranges;
    G.log.xy = reinterpret_cast<float2 *>(G.sums + ac * n_ranges);
    G.log.polar = G.log.xy + steps * n_ranges;
    G.land = reinterpret_cast<float *>(G.log.polar + steps * n_ranges);
    G.log.near = reinterpret_cast<unsigned *>(G.land + steps * n_ranges);
    R.bad = G.log.near + ac * n_chunks(P.H) * n_ranges;
    return G;
}

// f(kernel) for the variant's instance of grad_samples_kernel at this aircraft count
template <class F>
auto with_samples_kernel(int N, int variant, F f)
{
    const int tp = traj_tile(N);
    if (variant == 0) {
        if (tp == 32) return f(grad_samples_kernel<3, 32>);
        return tp == 16 ? f(grad_samples_kernel<3, 16>) : f(grad_samples_kernel<3, 8>);
    }
    if (tp == 32) return f(grad_samples_kernel<4, 32>);
    return tp == 16 ? f(grad_samples_kernel<4, 16>) : f(grad_samples_kernel<4, 8>);
}

// Where grad_controls_kernel takes sums over all the samples and fetches ahead (with the
// sums inside it -> by grad_sum_kernel): below two tiles for each of 152 SMs, where nothing
// else hides its waits (6 aircraft, 30 steps, L 4096, M 8: 397 -> 262 us; 2 aircraft, 20
// steps, L 1024, M 8: 102 -> 51 us); with more tiles from four ranges on (12 aircraft, 60
// steps, L 6000, M 16, four ranges: 2850 -> 2833 us; L 9000, three: 4339 -> 4356 us, not
// taken).  Not for the shortest horizons: a range inside costs about 1 us per four steps,
// the launch 4 us (1 aircraft, 5 steps, L 200, M 2: 28 against 30 us).
constexpr int kFewTiles = 304;
constexpr size_t kManyThreads = 152 * 2048;    // grad_sum_kernel: those of a step a thread that the chip holds
constexpr int kInlineSums = 4;     // fours of steps, times ranges beyond the first

size_t samples_smem(int N) { return (size_t)wind_rollout_words(N, traj_tile(N), true, false) * sizeof(float); }

}  // namespace

// Launch-bound variants of grad_samples_kernel: minimum resident blocks of 256
// threads (80 and 64 registers a thread), chosen by timing.
int rollout_grad_variants(int N, int *out)
{
    (void)N;
    out[0] = 0;
    out[1] = 1;
    return 2;
}

cudaError_t rollout_grad_occupancy(int N, int variant, int *blocks_per_sm)
{
    return with_samples_kernel(N, variant, [&](auto kernel) {
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, kernel, N * traj_tile(N), samples_smem(N));
    });
}

int rollout_grad_tile(int N) { return traj_tile(N); }

GradPlan rollout_grad_plan(const ProblemC &P, int64_t L, int n_ranges, int slots, size_t budget, size_t wide)
{
    const size_t tp = traj_tile(P.N), tiles = ((size_t)L + tp - 1) / tp;
    const size_t base = grad_bytes(P, tp, 0), per = grad_bytes(P, tp, 1) - base;     // of a tile
    const auto ranges_in = [&](size_t n) { return budget / n > base ? (budget / n - base) / per : 0; };
    size_t r = (size_t)n_ranges, n = budget / (base + r * per);
    if (n < tiles && n * r < (size_t)slots) {
        // A slab with all the ranges would leave the chip idle (few particles, many
        // samples, a long horizon): wide, or else fewer ranges for more tiles, but a
        // resident wave of blocks if that fits.  32 aircraft, 320 steps, 512 samples:
        // L 32 6.5 ms with all the ranges (5.3 GB), 8.5 ms with those of 2 GB.
        if (tiles * (base + r * per) > wide) {
            const size_t wave = std::min(r, ((size_t)slots + tiles - 1) / tiles);
            r = std::max(std::min(r, ranges_in(tiles)), wave);
            r = std::max(std::min(r, ranges_in(1)), (size_t)1);
            n = budget / (base + r * per);
        } else {
            n = tiles;
        }
    }
    n = std::min(std::max(n, (size_t)1), tiles);
    return GradPlan{(int)r, n * (base + r * per)};
}

cudaError_t launch_rollout_grad(const ProblemC &P, const DynState *dyn, const float *u, const float *W, int64_t L,
                                int J, int n_ranges, float *cost_ms, void *ws, size_t ws_bytes, float *cost, float *grad,
                                float *cbar, cudaStream_t st, int variant)
{
    if (L <= 0) return cudaSuccess;
    const int m_per_block = (P.M + n_ranges - 1) / n_ranges;
    n_ranges = (P.M + m_per_block - 1) / m_per_block;
    const int tp = traj_tile(P.N), block = P.N * tp;
    const size_t slab = ws_bytes / grad_bytes(P, tp, n_ranges) * tp, all = ((size_t)L + tp - 1) / tp * tp;
    if (!ws || slab == 0) return cudaErrorInvalidValue;
    const size_t n = slab < all ? slab : all;
    TrajOut R;
    const GradScratch G = grad_places(P, n, n_ranges, ws, R);
    const float4 *W4 = reinterpret_cast<const float4 *>(W);
    const size_t smem = samples_smem(P.N);
    const auto slab_end = [&](int64_t l0) { return l0 + (int64_t)n < L ? l0 + (int64_t)n : L; };
    for (int64_t l0 = 0; l0 < L; l0 += (int64_t)n) {
        const long long l1 = slab_end(l0);
        const int n_tiles = (int)((l1 - l0 + tp - 1) / tp);
        launch_trajectories(P, dyn, u, l0, l1, R, true, st, true);
        with_samples_kernel(P.N, variant, [&](auto kernel) {
            // one-warp blocks let in beside the trajectories were placed crowded: 1 aircraft,
            // 30 steps, L 4096, M 12 106 us so, 82 us by an ordinary launch
            const unsigned grid = (unsigned)n_tiles * (unsigned)n_ranges;
            if (block > 32)
                launch_dependent(kernel, grid, block, smem, st, P, dyn, W4, R, G, L, l0, l1, n_tiles, m_per_block, J,
                                 cost_ms);
            else
                kernel<<<grid, block, smem, st>>>(P, dyn, W4, R, G, L, l0, l1, n_tiles, m_per_block, J, cost_ms);
            return 0;
        });
        count_launch();
        if (cost) {
            // few tiles, or many ranges: their sums by a kernel of its own
            const bool sum = n_ranges > 1 && n_chunks(P.H) * (n_ranges - 1) > kInlineSums &&
                             (n_tiles < kFewTiles || n_ranges > 3);
            const int left = sum ? 1 : n_ranges;
            if (sum) {
                const auto sums = [&](auto kernel, int ks) {
                    const unsigned threads = (unsigned)n_tiles * (unsigned)((P.H + ks - 1) / ks) * (unsigned)block;
                    launch_dependent(kernel, (threads + 255) / 256, 256, 0, st, P, G, R.bad, threads, n_tiles, block, tp,
                                     n_ranges);
                };
                if ((size_t)n_tiles * P.H * block <= kManyThreads) sums(grad_sum_kernel<1>, 1);
                else sums(grad_sum_kernel<4>, 4);
                count_launch();
            }
            const auto controls = [&](auto kernel) {
                launch_dependent(kernel, n_tiles, block, 0, st, P, dyn, u, R, G, l0, l1, n_tiles, left, cost_ms, L, cost,
                                 grad, cbar);
            };
            const bool ahead = left == 1 && n_tiles < kFewTiles;
            if (tp == 32) ahead ? controls(grad_controls_kernel<32, true>) : controls(grad_controls_kernel<32, false>);
            else if (tp == 16) ahead ? controls(grad_controls_kernel<16, true>) : controls(grad_controls_kernel<16, false>);
            else ahead ? controls(grad_controls_kernel<8, true>) : controls(grad_controls_kernel<8, false>);
            count_launch();
        }
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace tma
