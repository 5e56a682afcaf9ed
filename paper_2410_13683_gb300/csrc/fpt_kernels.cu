// fpt_kernels.cu -- sm_103a kernels of the first-passage sampler.
//
//   em_kernel      persistent Euler-Maruyama stepper: one trajectory per
//                  thread, Philox4x32-10 noise, phi-indexed noise table in
//                  shared memory, importance-sampling bias and Kahan-summed
//                  log-weight, warp-ballot refill of finished trajectories.
//   hist_*         weighted histogram of first-passage times (per-bin max,
//                  shifted FP64 sums over paths sorted by bin) and the FP64
//                  finalisation of P(delta N) and its errors.
//
// Method (arXiv:2410.13683): Euler-Maruyama steps, Eq. (4.1), of the 1-D-noise
// system, Eq. (4.6), with the bias of Eq. (4.7) along the noise vector
// (1, tan theta_n) (the direction for which the weights of Eq. (4.8) agree) and
// the diffusion-based amplitude of Eq. (4.10); weight increment
// dA = A (A dN/2 + xi sqrt(dN)) (Eq. 4.5 in one dimension), w = exp(-sum dA)
// (Eq. 4.4); first passage at the first step n >= 1 with phi_n <= phi_end,
// N = n dN (Sec. 4.1).
#include "fpt_internal.h"
#include "fpt_mlp.cuh"
#include "fpt_steps.h"

#include <cuda.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <mutex>

namespace fpt_dev {

// Device bounds checks of FPT_CHECKS builds: a failed check sets its bit
// (kCheck*) in the error word and redirects the access to a valid index; the
// kernel carries on (warp-synchronous code cannot leave early), and the host
// reads and clears the word after each run or histogram (checks_take) and
// turns it into FPT_E_STATE. Other builds compile the checks away.
#ifdef FPT_CHECKS
__device__ int g_check_word;
#define CHECK_INDEX(idx, n, bit)                        \
    do {                                                \
        if ((idx) < 0 || (idx) >= (n)) {                \
            atomicOr(&g_check_word, (bit));             \
            (idx) = 0;                                  \
        }                                               \
    } while (0)
#else
#define CHECK_INDEX(idx, n, bit) do {} while (0)
#endif

cudaError_t checks_take(int *word)
{
    *word = 0;
#ifdef FPT_CHECKS
    cudaError_t e = cudaMemcpyFromSymbol(word, g_check_word, sizeof(int));
    if (e != cudaSuccess) return e;
    const int zero = 0;
    return cudaMemcpyToSymbol(g_check_word, &zero, sizeof(int));
#else
    return cudaSuccess;
#endif
}

// ---------------------------------------------------------------------------
// Random numbers: Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11).
// ---------------------------------------------------------------------------
// The key schedule (k0 + r W0, k1 + r W1 for rounds r = 0..9) is the same for
// every call of a launch: it comes precomputed in the kernel parameters
// (rk[2r], rk[2r+1]), so each round is two wide multiplies and two
// three-input XORs with constant-bank operands. The counter of a draw is (block,
// trajectory, run id, 0): of the first round's products only the block's and of
// the second's only one depend on the block, so a lane keeps the others
// (PhiloxLane) from the time it loads its trajectory: 18 wide multiplies a draw
// instead of 20.
struct PhiloxLane {
    uint32_t a;      // lo(M1 run) ^ rk[2]
    uint32_t b, c;   // hi(M0 x1) ^ rk[3], lo(M0 x1), x1 = hi(M1 run) ^ trajectory ^ rk[0]
};

__device__ __forceinline__ PhiloxLane philox_lane(uint32_t traj, uint32_t run_id, const uint32_t (&rk)[20])
{
    const unsigned long long p1 = 0xCD9E8D57ull * (unsigned long long)run_id;
    const uint32_t x1 = (uint32_t)(p1 >> 32) ^ traj ^ rk[0];
    const unsigned long long p0 = 0xD2511F53ull * (unsigned long long)x1;
    return {(uint32_t)p1 ^ rk[2], (uint32_t)(p0 >> 32) ^ rk[3], (uint32_t)p0};
}

__device__ __forceinline__ uint4 philox4x32_10(uint32_t block, const PhiloxLane &L, const uint32_t (&rk)[20])
{
    const unsigned long long q0 = 0xD2511F53ull * (unsigned long long)block;
    const unsigned long long q1 = 0xCD9E8D57ull * (unsigned long long)((uint32_t)(q0 >> 32) ^ rk[1]);
    uint4 c = make_uint4((uint32_t)(q1 >> 32) ^ L.a, (uint32_t)q1, (uint32_t)q0 ^ L.b, L.c);
#pragma unroll
    for (int r = 2; r < 10; ++r) {
        const unsigned long long p0 = 0xD2511F53ull * (unsigned long long)c.x;
        const unsigned long long p1 = 0xCD9E8D57ull * (unsigned long long)c.z;
        const uint32_t hi0 = (uint32_t)(p0 >> 32), lo0 = (uint32_t)p0;
        const uint32_t hi1 = (uint32_t)(p1 >> 32), lo1 = (uint32_t)p1;
        c = make_uint4(hi1 ^ c.y ^ rk[2 * r], lo1, hi0 ^ c.w ^ rk[2 * r + 1], lo0);
    }
    return c;
}

__device__ __forceinline__ float rcp_approx(float v)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

__device__ __forceinline__ float sqrt_approx(float v)
{
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

// Two standard normals from two Philox words: 23-bit uniforms
// u = ((r >> 9) + 0.5) 2^-23, built from the mantissa bits (1 + (r >> 9) 2^-23
// minus (1 - 2^-24), exact by Sterbenz; one funnel shift puts the exponent of 1
// above the mantissa), then Box-Muller z0 = rho cos(2 pi u1),
// z1 = rho sin(2 pi u1), rho = sqrt(-2 ln u0); the angle is evaluated as
// 2 pi u1 - pi, inside the accurate range of the hardware sine/cosine, and the
// signs restored. u0 lies in [2^-24, 1 - 2^-24] and the angle's magnitude above
// 2^-22: neither is ever subnormal, so the flushing forms of the hardware
// functions give the same bits without their subnormal handling, and -2 ln u0
// is positive (all of this compared bit for bit over the 2^23 uniforms).
// Executed instructions per step of direct sampling: 51.0 (52.5 before the chained
// passage test); with the lane's Philox products 38.1 -> 37.2 ms on 2^22 paths, noise
// window 26.1 -> 24.6 ms and bump 10.6 -> 10.2 ms on 10^6.
__device__ __forceinline__ float uniform23(uint32_t r)
{
    return __uint_as_float(__funnelshift_r(r, 0x7fu, 9)) - 0.99999994039535522f;   // 1 - 2^-24
}

__device__ __forceinline__ float lg2_approx(float v)
{
    float r;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

__device__ __forceinline__ float sin_approx(float v)
{
    float r;
    asm("sin.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

__device__ __forceinline__ float cos_approx(float v)
{
    float r;
    asm("cos.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

// The normals are products (rho cos, rho sin): the record mode's sums of
// normals are explicit __fadd_rn, which the compiler never fuses with the
// product into an FMA. A contracted sum would round differently wherever the
// compiler chose to fuse, and the speculative and guarded paths (and the
// recomputation of a group's normals after a passage) would no longer give the
// same sums.
__device__ __forceinline__ void box_muller(uint32_t r0, uint32_t r1, float &z0, float &z1)
{
    const float u0 = uniform23(r0);
    const float u1 = uniform23(r1);
    const float rho = sqrt_approx(-1.38629436111989061f * lg2_approx(u0));   // -2 ln u0
    const float th = fmaf(u1, 6.28318530717958648f, -3.14159265358979324f);
    z0 = -rho * cos_approx(th);
    z1 = -rho * sin_approx(th);
}

// Compensated (Kahan) accumulation of v into the pair (hi, lo), whose value
// is hi - lo: lo holds the amount by which hi overshoots the exact sum.
__device__ __forceinline__ void kahan_add(float &hi, float &lo, float v)
{
    const float y = __fsub_rn(v, lo);
    const float t = __fadd_rn(hi, y);
    lo = __fsub_rn(__fsub_rn(t, hi), y);
    hi = t;
}

// ---------------------------------------------------------------------------
// K1: persistent Euler-Maruyama stepper
// ---------------------------------------------------------------------------
struct RunSm {               // per-run constants staged in shared memory
    long long unit_begin;
    long long traj_offset;
    float cb, half_cb2, cb_b;
    uint32_t run_id;
    int32_t model;
    int32_t is_mlp;
    float sqrt_dN, dN;
};

struct Lane {                // per-thread trajectory state and its constants
    float x, x_c;            // shifted field phi - phi_end as a Kahan pair: x - x_c
    float p, p_c;            // momentum; p_c compensates it (Kahan) in the variants with pi-noise
    float lw_hi, lw_lo;      // ln w as a Kahan pair
    int grp;                 // steps taken / 4 (a live lane's count is a multiple of 4 between groups)
    int nmax;
    PhiloxLane rng;
    float cb, half_cb2, dN, sqrt_dN;
    float cb_b;              // 2-D noise: beta_2 sqrt(dN) (cb = beta_1 sqrt(dN))
    union {                  // drift constants of the lane's potential
        struct { float x_star, x_star_lo, inv_a_plus, inv_a_minus, c; } pw;   // piecewise-linear / exponential
        struct { float scale, umax; int dtab, model; } bump;              // Gaussian bump: cubic V'/V table
    } dc;
    float u_scale, u_shift, u_max;
    int tbase;
    int M;                   // noise-table points of the lane's model (bounds checks)
    bool mlp;
    bool nidx;               // noise table indexed by the step count
    int win_lo, win_hi;      // noise window in steps (nidx)
    int run;                 // index of the lane's run in the launch
    uint32_t unit;           // launch unit (a launch has at most 2^32)
};

struct SegRec {              // open segment of the record variant
    float in0, in1, in2, tan_t, raw, sum_xi;
    float sum_xi2;           // 2-D noise: sum of xi_2 (sum_xi holds xi_1)
    int n0;
    bool open;
};

__device__ __forceinline__ void lane_load(Lane &L, long long unit, const RunSm *s_run,
                                          const ModelDev *s_model, int n_runs, const uint32_t (&rk)[20])
{
    // last run whose first unit is <= unit (runs are contiguous in unit order)
    int lo = 0, hi = n_runs - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (s_run[mid].unit_begin <= unit) lo = mid; else hi = mid - 1;
    }
    const RunSm &r = s_run[lo];
    const ModelDev &m = s_model[r.model];
    L.run = lo;
    L.unit = (uint32_t)unit;
    L.rng = philox_lane((uint32_t)(r.traj_offset + (unit - r.unit_begin)), r.run_id, rk);
    L.cb = r.cb;
    L.half_cb2 = r.half_cb2;
    L.cb_b = r.cb_b;
    L.mlp = r.is_mlp != 0;
    L.dN = m.dN;
    L.sqrt_dN = r.sqrt_dN;
    if (m.dtab >= 0) {
        L.dc.bump.scale = m.d_scale;
        L.dc.bump.umax = m.d_umax;
        L.dc.bump.dtab = m.dtab;
        L.dc.bump.model = r.model;
    } else {
        L.dc.pw.x_star = m.x_star;
        L.dc.pw.x_star_lo = m.x_star_lo;
        L.dc.pw.inv_a_plus = m.inv_a_plus;
        L.dc.pw.inv_a_minus = m.inv_a_minus;
        L.dc.pw.c = m.drift_c;
    }
    L.u_scale = m.u_scale;
    L.u_shift = m.u_shift;
    L.u_max = m.u_umax;
    L.tbase = m.table_offset;
    L.M = m.M;
    L.nidx = m.nidx != 0;
    L.win_lo = m.win_lo;
    L.win_hi = m.win_hi;
    L.nmax = m.max_steps;
    L.x = m.x_in;
    L.x_c = 0.0f;
    L.p = m.pi_in;
    L.p_c = 0.0f;
    L.lw_hi = 0.0f;
    L.lw_lo = 0.0f;
    L.grp = 0;
}

// Table entry and interpolation weight at the lane's field. The 1-D tables
// hold, per interval k, the midpoint values (v_k + v_{k+1})/2 and the slopes
// v_{k+1} - v_k of (S', T') (times sqrt(dN)); with u' = (phi - phi_lo)/h - 1/2
// clamped to [-1/2, M - 3/2], k = round(u') comes from adding 1.5 2^23 (round
// to nearest in the mantissa, no float/int conversion) and f' = u' - k lies in
// [-1/2, 1/2]: v(u) = mid_k + f' slope_k. The last entry repeats v_{M-1} with
// zero slope, so every reachable k (0 .. M-1) is a valid entry.
template <bool SMEM, bool NIDX = false>
__device__ __forceinline__ float4 table_at(const Lane &L, const float4 *__restrict__ tab, float &f,
                                           const ModelDev &M0, int n = 0)
{
    const float kMagic = 12582912.0f;                        // 1.5 * 2^23
    // N-indexed tables: coordinate from the exact step count (n < 2^24 is exact in FP32)
    const float coord = (NIDX && L.nidx) ? __int2float_rn(n) : L.x;
    float u = fmaf(coord, SMEM ? M0.u_scale : L.u_scale, SMEM ? M0.u_shift : L.u_shift);
    u = fminf(fmaxf(u, -0.5f), SMEM ? M0.u_umax : L.u_max);
    const float t = u + kMagic;
    int i = __float_as_int(t) - 0x4b400000;
    f = u - (t - kMagic);
    CHECK_INDEX(i, SMEM ? M0.M : L.M, kCheckTable);
    return SMEM ? tab[i] : __ldg(tab + L.tbase + i);
}

// V'/V at the lane's field. Piecewise-linear (relative slopes) and
// exponential potentials: a / (1 + b (x - x_star)), branch by side.
// Gaussian bump (DTAB): near its inflection point V'/V is the small
// difference of two terms of size ~0.05, which FP32 cannot resolve, so it is
// read from a cubic (Hermite) table of the FP64 values on a uniform x grid
// (coefficients c0..c3 of s in [0, 1] per interval; one padding entry), and
// evaluated from the closed form in FP32 only above the table.
template <bool DTAB, bool SMEM>
__device__ __forceinline__ float drift_vpv(const Lane &L, const float4 *__restrict__ tab,
                                           const ModelDev *s_model, const ModelDev &M0)
{
    if (!DTAB) {
        // side of the kink from the compensated field and kink position:
        // x - x_c >= x_star + x_star_lo (x - x_star is exact near the kink), so
        // the branch follows the field itself, not the rounding of its FP32 head.
        // V'/V = a / (1 + a d) = 1 / (1/a + d) on each side (c = 1; the
        // exponential potential has c = 0 and V'/V = 1/(1/mu)).
        const float d = L.x - (SMEM ? M0.x_star : L.dc.pw.x_star);
        const bool up = d >= L.x_c + (SMEM ? M0.x_star_lo : L.dc.pw.x_star_lo);
        const float ia = up ? (SMEM ? M0.inv_a_plus : L.dc.pw.inv_a_plus)
                            : (SMEM ? M0.inv_a_minus : L.dc.pw.inv_a_minus);
        return rcp_approx(fmaf(SMEM ? M0.drift_c : L.dc.pw.c, d, ia));
    }
    const float u = fmaxf(L.x * (SMEM ? M0.d_scale : L.dc.bump.scale), 0.0f);
    if (u <= (SMEM ? M0.d_umax : L.dc.bump.umax)) {
        const float kMagic = 12582912.0f;                    // 1.5 * 2^23
        const float t = (u - 0.5f) + kMagic;
        int i = __float_as_int(t) - 0x4b400000;
        const float sv = u - (t - kMagic);
        CHECK_INDEX(i, (int)(SMEM ? M0.d_umax : L.dc.bump.umax) + 1, kCheckDriftTable);
        const float4 c = SMEM ? tab[M0.dtab + i] : __ldg(tab + L.tbase + L.dc.bump.dtab + i);
        return fmaf(sv, fmaf(sv, fmaf(sv, c.w, c.z), c.y), c.x);
    }
    const ModelDev &md = SMEM ? M0 : s_model[L.dc.bump.model];
    const float phi = L.x + md.bump_phi_end;
    const float d = L.x + md.bump_dphi0;                     // phi - phi0
    const float g = md.bump_K * __expf(-0.5f * d * d * md.bump_inv_w2);
    return __fdividef(2.0f * md.bump_m2, phi * fmaf(phi, phi, md.bump_m2)) -
           __fdividef(g * d * md.bump_inv_w2, 1.0f + g);
}

// Passage test on the compensated field: the pair's value x - x_c is <= 0
// exactly when x <= x_c (without flush-to-zero the rounded difference of two
// floats is zero or negative only when the exact one is), so the test needs
// no subtraction.
__device__ __forceinline__ bool passed(const Lane &L)
{
    return L.x <= L.x_c;
}

// Steps outside the noise window of an N-indexed table (step count below
// win_lo or above win_hi) are classical.
template <bool NIDX>
__device__ __forceinline__ bool outside_window(const Lane &L, int n)
{
    return NIDX && L.nidx && (n < L.win_lo || n > L.win_hi);
}

// (pi^2/2 - 3) dN, the momentum drift's factor, as (0.5 dN pi) pi - 3 dN with
// the FP32 constants 0.5 dN and -3 dN (single-model launches read them from
// the model descriptor, the others form the same products from dN).
template <bool SMEM>
__device__ __forceinline__ float hh_dN(const Lane &L, const ModelDev &M0)
{
    const float h = SMEM ? M0.half_dN : 0.5f * L.dN;
    const float m3 = SMEM ? M0.m3dN : -3.0f * L.dN;
    return fmaf(h * L.p, L.p, m3);
}

// One Euler-Maruyama step of Eq. (4.7) with bias amplitude L.cb / sqrt(dN),
// step number n. The field increment (drift + bias + noise) is formed first and
// added to the compensated field pair: a plain FP32 field would add the same
// drift increment to a value on its own grid every step, a rounding error with
// a fixed sign. lw: ln w increments of the current group.
template <bool WEIGHTED, bool SMEM, bool NIDX = false, bool DTAB = false>
__device__ __forceinline__ void em_step(Lane &L, int n, float z, float &lw, const float4 *__restrict__ tab,
                                        const ModelDev *s_model, const ModelDev &M0)
{
    // noise table: linear interpolation in x (or in time), end values held outside
    float f;
    const float4 e = table_at<SMEM, NIDX>(L, tab, f, M0, n);
    const float dN = SMEM ? M0.dN : L.dN;
    float S = fmaf(f, e.y, e.x);               // S_phiphi sqrt(dN)
    float T = fmaf(f, e.w, e.z);               // tan(theta_n) S_phiphi sqrt(dN)
    float cb = L.cb, half_cb2 = L.half_cb2;
    if (outside_window<NIDX>(L, n)) {
        // outside the noise window the step is classical: no noise, no bias, no weight
        S = 0.0f;
        T = 0.0f;
        cb = 0.0f;
        half_cb2 = 0.0f;
    }
    const float vpv = drift_vpv<DTAB, SMEM>(L, tab, s_model, M0);
    const float hdN = hh_dN<SMEM>(L, M0);               // (pi^2/2 - 3) dN
    const float zb = z + cb;                             // xi + alpha sqrt(dN)
    const float dx = fmaf(S, zb, L.p * dN);             // (pi + alpha S) dN + S xi sqrt(dN)
    if (DTAB) {
        // correlated pi-noise (tan theta_n ~ 0.3): the momentum is a compensated
        // pair, or its rounding performs a random walk that the field integrates
        kahan_add(L.p, L.p_c, fmaf(T, zb, hdN * (L.p + vpv)));
    } else {
        L.p = fmaf(T, zb, fmaf(hdN, L.p + vpv, L.p));
    }
    if (WEIGHTED) lw -= fmaf(cb, z, half_cb2);          // the step's ln w increment (see group_lw)
    kahan_add(L.x, L.x_c, dx);
}

// ln w increments of the first k + 1 steps of a group that starts at step
// n0, summed as the steps sum them (same operands, same order).
template <bool NIDX, bool RANK2>
__device__ __forceinline__ float group_lw(const Lane &L, const float *z, int n0, int k)
{
    float lw = 0.0f;
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        if (s > k) break;
        const bool off = outside_window<NIDX>(L, n0 + s);
        const float cb = off ? 0.0f : L.cb, half_cb2 = off ? 0.0f : L.half_cb2;
        lw -= RANK2 ? fmaf(cb, z[2 * s], fmaf(L.cb_b, z[2 * s + 1], half_cb2)) : fmaf(cb, z[s], half_cb2);
    }
    return lw;
}

__device__ __forceinline__ unsigned long long globaltimer()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Learned proposal at a segment start: alpha from the warp's MLP evaluation
// at the current state; every lane of the warp takes part.
template <bool SMEM, bool REC>
__device__ __forceinline__ void mlp_segment_start(Lane &L, bool live, SegRec &sg, const float4 *tab,
                                                  const uint2 *tiles, const float *bias, const RunDev &pr,
                                                  const ModelDev &M0)
{
    const float dN = SMEM ? M0.dN : L.dN, sqrt_dN = SMEM ? M0.sqrt_dN : L.sqrt_dN;
    float in0 = 0.0f, in1 = 0.0f, in2 = 0.0f, tan_t = 0.0f;
    if (live) {
        const float xv = __fsub_rn(L.x, L.x_c);
        in0 = ((pr.mlp_flags & FPT_MLP_LOG_X) ? __logf(fmaxf(xv, pr.x_floor)) : xv);
        in0 = (in0 - pr.shift[0]) * pr.scale[0];
        in1 = (L.p - pr.shift[1]) * pr.scale[1];
        in2 = ((float)steps_of(L.grp) * dN - pr.shift[2]) * pr.scale[2];
        float f;
        const float4 e = table_at<SMEM>(L, tab, f, M0);
        const float S = fmaf(f, e.y, e.x), T = fmaf(f, e.w, e.z);
        tan_t = S > 0.0f ? __fdividef(T, S) : 0.0f;
    }
    float o1, o2;
    mlp_forward_warp(tiles, bias, in0, in1, in2, __ballot_sync(0xffffffffu, live), o1, o2);
    if (live) {
        float raw;
        const float al = mlp_alpha_of(o1, o2, tan_t, pr.alpha_max, raw);
        L.cb = al * sqrt_dN;
        L.half_cb2 = 0.5f * al * al * dN;
        if (REC) {
            sg.in0 = in0; sg.in1 = in1; sg.in2 = in2; sg.tan_t = tan_t; sg.raw = raw;
            sg.sum_xi = 0.0f;
            sg.n0 = steps_of(L.grp);
            sg.open = true;
        }
    }
}

// Learned proposal with one network per run (the runs of a launch may carry
// different networks, input normalisations and clamps; they share the
// segment length): the warp evaluates the network of each run among its live
// lanes in turn -- runs are contiguous in unit order, so a warp mostly holds
// one run -- reading that run's packed weights through L1.
template <bool SMEM, bool REC>
__device__ __forceinline__ void mlp_segment_start_multi(Lane &L, bool live, SegRec &sg, const float4 *tab,
                                                        const RunDev *runs, const ModelDev &M0)
{
    const unsigned FULL = 0xffffffffu;
    const float dN = SMEM ? M0.dN : L.dN, sqrt_dN = SMEM ? M0.sqrt_dN : L.sqrt_dN;
    unsigned pend = __ballot_sync(FULL, live);
    while (pend) {
        const int run = __shfl_sync(FULL, L.run, __ffs(pend) - 1);
        const bool mine = live && L.run == run;
        pend &= ~__ballot_sync(FULL, mine);
        const RunDev &pr = runs[run];
        float in0 = 0.0f, in1 = 0.0f, in2 = 0.0f, tan_t = 0.0f;
        if (mine) {
            const float xv = __fsub_rn(L.x, L.x_c);
            in0 = ((pr.mlp_flags & FPT_MLP_LOG_X) ? __logf(fmaxf(xv, pr.x_floor)) : xv);
            in0 = (in0 - pr.shift[0]) * pr.scale[0];
            in1 = (L.p - pr.shift[1]) * pr.scale[1];
            in2 = ((float)steps_of(L.grp) * dN - pr.shift[2]) * pr.scale[2];
            float f;
            const float4 e = table_at<SMEM>(L, tab, f, M0);
            const float S = fmaf(f, e.y, e.x), T = fmaf(f, e.w, e.z);
            tan_t = S > 0.0f ? __fdividef(T, S) : 0.0f;
        }
        const uint2 *tiles = reinterpret_cast<const uint2 *>(pr.mlp);
        const float *bias = reinterpret_cast<const float *>(tiles + kMlpTiles * 32);
        float o1, o2;
        mlp_forward_warp(tiles, bias, in0, in1, in2, __ballot_sync(FULL, mine), o1, o2);
        if (mine) {
            float raw;
            const float al = mlp_alpha_of(o1, o2, tan_t, pr.alpha_max, raw);
            L.cb = al * sqrt_dN;
            L.half_cb2 = 0.5f * al * al * dN;
            if (REC) {
                sg.in0 = in0; sg.in1 = in1; sg.in2 = in2; sg.tan_t = tan_t; sg.raw = raw;
                sg.sum_xi = 0.0f;
                sg.n0 = steps_of(L.grp);
                sg.open = true;
            }
        }
    }
}

// Shared memory of the launch's tail (see tail_meeting).
constexpr int kPoolLanes = 128;          // lanes one compaction can move (4 KB of shared memory)
constexpr int kMaxWarps = 16;
constexpr int kMaxPairs = 4;             // warps of a block that can have a helper
constexpr int kSlotVecs = 4 * 32;        // float4 of a ring slot: four Philox blocks of 32 lanes

struct PairSm {
    float4 ring[2 * kSlotVecs];
    uint4 lane[32];                      // generator state of the consumer's lanes, next group
};

struct TailSm {
    float4 pool[2 * kPoolLanes];
    int count[2][kMaxWarps];             // live lanes per warp, double-buffered by round
    int dry;
};

// Dynamic shared memory of a stepper launch: the table (SMEM variants), the
// staged proposal blob (single-network learned variants), then the launch's
// run constants and model descriptors, each as many as the launch has, and the
// rings of the tail's helper warps.
__device__ __forceinline__ RunSm *smem_runs(float4 *s_dyn, int table_entries, bool staged_blob)
{
    unsigned char *p = reinterpret_cast<unsigned char *>(s_dyn + table_entries);
    return reinterpret_cast<RunSm *>(p + (staged_blob ? kMlpBlobBytes : 0));
}

__device__ __forceinline__ ModelDev *smem_models(RunSm *s_run, int n_runs)
{
    const size_t b = ((sizeof(RunSm) * (size_t)n_runs + 15) / 16) * 16;
    return reinterpret_cast<ModelDev *>(reinterpret_cast<unsigned char *>(s_run) + b);
}


__device__ __forceinline__ PairSm *smem_pairs(ModelDev *s_model, int n_models)
{
    const size_t b = ((sizeof(ModelDev) * (size_t)n_models + 15) / 16) * 16;
    return reinterpret_cast<PairSm *>(reinterpret_cast<unsigned char *>(s_model) + b);
}

// Launch prologue shared by the steppers: clock origin, per-run and per-model
// constants, the table (SMEM variants) and the proposal blob (MLP variants)
// staged in shared memory. `table_entries` float4 entries are staged.
template <bool SMEM, bool MLP>
__device__ __forceinline__ void stage_launch(const EmParams &P, float4 *s_tab, RunSm *s_run,
                                             ModelDev *s_model, unsigned long long &s_t0,
                                             uint2 *s_tiles)
{
    if (P.budget_ns && threadIdx.x == 0) {
        // the launch's clock origin: the first block to start sets it
        const unsigned long long now = globaltimer();
        const unsigned long long prev = atomicCAS(P.t0, 0ull, now);
        s_t0 = prev ? prev : now;
    }
    for (int i = threadIdx.x; i < P.n_runs; i += blockDim.x) {
        const RunDev &r = P.runs[i];
        s_run[i].unit_begin = r.unit_begin;
        s_run[i].traj_offset = r.traj_offset;
        s_run[i].cb = r.cb;
        s_run[i].half_cb2 = r.half_cb2;
        s_run[i].cb_b = r.cb_b;
        s_run[i].run_id = r.run_id;
        s_run[i].model = r.model;
        s_run[i].is_mlp = r.bias_kind == FPT_BIAS_MLP;
        s_run[i].sqrt_dN = r.sqrt_dN;
        s_run[i].dN = r.dN;
    }
    for (int i = threadIdx.x; i < P.n_models; i += blockDim.x) s_model[i] = P.models[i];
    if (SMEM) {
        const float4 *src = P.tables + P.smem_table_offset;
        for (int i = threadIdx.x; i < P.smem_table_points; i += blockDim.x) s_tab[i] = src[i];
    }
    if (MLP) {
        const float4 *src = reinterpret_cast<const float4 *>(P.runs[P.mlp_run].mlp);
        float4 *dst = reinterpret_cast<float4 *>(s_tiles);
        for (int i = threadIdx.x; i < kMlpBlobBytes / 16; i += blockDim.x) dst[i] = src[i];
    }
    __syncthreads();
}

// A trajectory that has ended after n steps: its results, written once.
__device__ __forceinline__ void finish(const EmParams &P, const Lane &L, int n, bool pas)
{
    long long u = L.unit;
    CHECK_INDEX(u, P.total_units, kCheckUnit);
    P.nsteps[u] = n;
    P.logw[u] = (double)L.lw_hi - (double)L.lw_lo;     // the pair holds hi - lo
    P.status[u] = pas ? (uint8_t)FPT_TRAJ_PASSED : (uint8_t)FPT_TRAJ_CAPPED;
    if (!pas) atomicAdd(P.flags + kFlagCapped, 1);
}

// First units of a warp: chunk c of 32 units goes to block c mod grid, so that a
// launch with fewer chunks than resident warps loads every SM alike (taken from
// the cursor instead, the first blocks to start took 16 chunks each: 16,384
// paths ran on a quarter of the SMs, 2.26 ms a launch against 0.60 ms; eight
// runs of 20,011 paths, most of them capped at 2^18 steps, 125 -> 74 ms). Within a
// block the chunks go to warps in the order of warp_at(), rotated for the
// blocks that share an SM, so that their first warps sit on different
// sub-partitions.
__device__ __forceinline__ int block_rotation(const EmParams &P)
{
    return (int)(2 * (blockIdx.x / (unsigned)P.sm_count) % (blockDim.x >> 5));
}

__device__ __forceinline__ bool first_units(const EmParams &P, Lane &L, const RunSm *s_run,
                                            const ModelDev *s_model)
{
    const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int pos = (warp + nw - block_rotation(P)) % nw;
    const long long unit = ((long long)pos * gridDim.x + blockIdx.x) * 32 + (threadIdx.x & 31u);
    // lanes without a trajectory step along harmlessly on zeros: every table index is clamped
    L = Lane{};
    L.M = 1;
    if (unit >= P.total_units) return false;
    lane_load(L, unit, s_run, s_model, P.n_runs, P.rk);
    return true;
}

// Refill point: lanes without a trajectory fetch new units with one
// warp-aggregated atomic on the work cursor (units past the launch's first
// ones). Returns true when a lane was loaded; s_dry is set once the cursor has
// run past the last unit.
__device__ __forceinline__ bool refill_point(const EmParams &P, Lane &L, bool &live, const RunSm *s_run,
                                             const ModelDev *s_model, int *s_dry)
{
    const unsigned FULL = 0xffffffffu;
    const unsigned lane = threadIdx.x & 31u;
    const unsigned idle = __ballot_sync(FULL, !live);
    if (!idle) return false;
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(P.cursor, (unsigned long long)__popc(idle));
    base = __shfl_sync(FULL, base, 0) + (unsigned long long)gridDim.x * blockDim.x;
    if ((long long)base + __popc(idle) > P.total_units && lane == 0) *(volatile int *)s_dry = 1;
    bool got = false;
    if (!live) {
        const long long unit = (long long)(base + __popc(idle & ((1u << lane) - 1u)));
        if (unit < P.total_units) {
            lane_load(L, unit, s_run, s_model, P.n_runs, P.rk);
            live = got = true;
        }
    }
    return __any_sync(FULL, got);
}

// ---------------------------------------------------------------------------
// The launch's tail: compaction of the block's live lanes
// ---------------------------------------------------------------------------
// Path lengths are heavy-tailed, so once the work cursor is dry the warps keep
// one or two live lanes each for most of a launch, at the price of full ones.
// From then on (tail mode) the warps of a block meet every tail_intervals
// intervals (about 512 steps) and the live lanes of the last warps move into free
// lanes of the first ones, through a small pool in shared memory, whenever that
// empties a warp. A lane's state is eight words; everything else is loaded
// from its run and model again. A lane moves between intervals, where no group
// and no held-alpha segment is open, so results do not depend on it. Measured
// with the straight-line groups below: 2^18 learned paths (median 8,902 steps,
// longest 262,144) 78 -> 34 ms, where the longest path's step took 324 ns
// among 24 sparse warps per SM; 64 models x 8,192 paths 76 -> 32 ms.
//
// When few warps are left, each gets an idle warp of its block as a helper that
// draws its normals: a lone warp takes ~150 cycles a step, of which its own
// chain (field -> table -> field) is about 85 and a third of the instructions
// are the generator's. The helper keeps one slot ahead in a ring of two slots
// in shared memory; the two warps meet at a named barrier per slot.
struct TailRole {
    int pair;                            // index of the warp's ring, -1: none
    bool helper;
};

__device__ __forceinline__ int warp_at(int pos, int rot, int nw)
{
    const int w = pos + rot;
    return w >= nw ? w - nw : w;
}

__device__ __forceinline__ int scan_incl(int v)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < kMaxWarps; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    return v;
}

// One meeting of the block's warps. Returns false when the block has no live
// lane left or must stop. COMPACT: lanes move to as few warps as hold them; a step
// costs a warp the same for one lane and for 32 (2^18 learned paths: 30.3 ms, with
// four warps kept busy 33.2, with eight 47.7). Not in the steppers with one network
// per run: a warp evaluates the networks of its lanes in turn, so lanes stay where
// they are and only the helpers are handed out (training round of 64 networks,
// 1,024 paths each, in blocks of eight warps: 18.8 ms; compacted to six warps 19.5,
// four 19.9, two 21.5, one 22.8; 16 networks or 200 paths each: no difference).
// Lane j of every warp holds the count of the warp at position j, so all warps come
// to the same decision.
template <bool COMPACT>
__device__ __forceinline__ bool tail_meeting(const EmParams &P, Lane &L, bool &live, bool stop, int round,
                                             TailSm &T, PairSm *pairs, const RunSm *s_run,
                                             const ModelDev *s_model, TailRole &role)
{
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int rot = block_rotation(P), pos = warp_at(warp, nw - rot, nw);
    const unsigned mask = __ballot_sync(FULL, live);
    int *cnt = T.count[round & 1];
    if (lane == 0) cnt[warp] = __popc(mask);
    if (__syncthreads_or(stop)) return false;
    const int c = lane < nw ? cnt[warp_at(lane, rot, nw)] : 0;
    const int total = __reduce_add_sync(FULL, c);
    if (!total) return false;
    unsigned busy = __ballot_sync(FULL, c > 0);
    const int need = (total + 31) >> 5;
    if (COMPACT && need < __popc(busy)) {
        // keep the first positions; the lanes of the later ones must fit the pool
        const int excl = scan_incl(c) - c;
        const unsigned fits = __ballot_sync(FULL, lane >= need && lane < nw && total - excl <= kPoolLanes);
        const int keep = fits ? __ffs(fits) - 1 : nw;
        const int moved = fits ? total - __shfl_sync(FULL, excl, keep & 31) : 0;
        if (moved) {
            // donors in order of position fill the pool, free lanes in the same order empty it
            const int room = lane < keep ? max(0, (total + keep - 1) / keep - c) : 0;
            const int room_excl = scan_incl(room) - room;
            const bool donor = pos >= keep;
            const int from = __shfl_sync(FULL, excl, pos) - (total - moved), to = __shfl_sync(FULL, room_excl, pos);
            busy = __ballot_sync(FULL, lane < keep && (c > 0 || (room > 0 && room_excl < moved)));
            const unsigned below = (1u << lane) - 1u;
            if (donor && live) {
                const int e = from + __popc(mask & below);
                T.pool[2 * e] = make_float4(L.x, L.x_c, L.p, L.p_c);
                T.pool[2 * e + 1] = make_float4(L.lw_hi, L.lw_lo, __int_as_float(L.grp), __uint_as_float(L.unit));
                live = false;
            }
            __syncthreads();
            const int free = __popc(~mask & below), mine = __shfl_sync(FULL, room, pos), e = to + free;
            const bool take = !donor && !live && free < mine && e < moved;
            if (take) {
                const float4 u = T.pool[2 * e], v = T.pool[2 * e + 1];
                lane_load(L, (long long)__float_as_uint(v.w), s_run, s_model, P.n_runs, P.rk);
                L.x = u.x; L.x_c = u.y; L.p = u.z; L.p_c = u.w;
                L.lw_hi = v.x; L.lw_lo = v.y;
                L.grp = __float_as_int(v.z);
                live = true;
            }
        }
    }
    // helpers for the busy warps, if there are few enough
    const int n_busy = __popc(busy);
    role.pair = -1;
    if (n_busy <= P.pairs && 2 * n_busy <= nw) {
        const unsigned below = (1u << pos) - 1u;
        role.helper = !((busy >> pos) & 1u);
        const int rank = __popc((role.helper ? ~busy : busy) & below);
        if (rank < n_busy) role.pair = rank;
        if (!role.helper) pairs[rank].lane[lane] = make_uint4(L.rng.a, L.rng.b, L.rng.c, (uint32_t)L.grp);
        __syncthreads();
    }
    return true;
}

// bar.sync is the aligned form: all lanes of a warp must reach it together, and the
// consumer comes to it from the divergent end of a group in which a lane passed.
__device__ __forceinline__ void pair_barrier(int pair)
{
    __syncwarp();
    asm volatile("bar.sync %0, 64;" ::"r"(pair + 1) : "memory");
}

// Deadline: true when the launch should stop (lane 0 reads the device clock).
__device__ __forceinline__ bool past_deadline(const EmParams &P, unsigned long long t0)
{
    int stop = 0;
    if ((threadIdx.x & 31u) == 0) {
        if (globaltimer() - t0 > P.budget_ns) atomicExch(P.flags, 1);
        stop = *(volatile int *)P.flags;
    }
    return __shfl_sync(0xffffffffu, stop, 0) != 0;
}

// Segment record idx: q0 = (inputs, tan theta_n), q1 = (raw alpha, sum xi, unit,
// first step); full-rank noise: q0 = (inputs, sum xi_2), q1 = (0, sum xi_1, unit,
// first step). Records past the buffer raise a flag instead of being written.
template <bool RANK2>
__device__ __forceinline__ void put_record(const EmParams &P, const Lane &L, const SegRec &sg, long long idx)
{
    if (idx < P.rec_cap) {
        float4 *q = reinterpret_cast<float4 *>(P.records + 8 * idx);
        q[0] = make_float4(sg.in0, sg.in1, sg.in2, RANK2 ? sg.sum_xi2 : sg.tan_t);
        q[1] = make_float4(RANK2 ? 0.0f : sg.raw, sg.sum_xi, __uint_as_float(L.unit), __int_as_float(sg.n0));
    } else {
        atomicExch(P.flags + kFlagRecOverflow, 1);
    }
}

// Close the warp's open segments at a refill point, appended with one
// warp-aggregated atomic on the record cursor.
template <bool RANK2>
__device__ __forceinline__ void write_records(const EmParams &P, const Lane &L, SegRec &sg)
{
    const unsigned FULL = 0xffffffffu;
    const unsigned lane = threadIdx.x & 31u;
    const unsigned m = __ballot_sync(FULL, sg.open);
    if (m) {
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd(P.rec_cursor, (unsigned long long)__popc(m));
        base = __shfl_sync(FULL, base, 0);
        if (sg.open) put_record<RANK2>(P, L, sg, (long long)(base + __popc(m & ((1u << lane) - 1u))));
    }
    sg.open = false;
}

// ---------------------------------------------------------------------------
// K1b: full-rank (2-D) noise stepper
// ---------------------------------------------------------------------------
// Euler-Maruyama of Eq. (2.24) with the symmetric noise matrix S = sqrt(Xi)
// (Eq. 3.9): two normals per step, step n using normals 2(n & 1), 2(n & 1) + 1
// of Philox block n >> 1. Bias in standardised form B = S beta, so that
// Eq. (4.5) reduces to dA = beta . (beta dN/2 + xi sqrt(dN)) (S^T Xi^-1 S = 1).
// Table: M + 1 float4 entries (S_phiphi, S_phipi, S_pipi, 0) sqrt(dN) at the
// grid points, entry M repeating entry M - 1; linear interpolation reads
// entries k and k + 1.
template <bool SMEM>
__device__ __forceinline__ void table2_at(const Lane &L, const float4 *__restrict__ tab, float &a,
                                          float &b, float &c, const ModelDev &M0)
{
    const float kMagic = 12582912.0f;                        // 1.5 * 2^23
    float u = fmaf(L.x, SMEM ? M0.u_scale : L.u_scale, SMEM ? M0.u_shift : L.u_shift);
    u = fminf(fmaxf(u, 0.0f), SMEM ? M0.u_umax : L.u_max);
    const float t = (u - 0.5f) + kMagic;
    int i = __float_as_int(t) - 0x4b400000;
    const float f = u - (t - kMagic);
    CHECK_INDEX(i, SMEM ? M0.M : L.M, kCheckTable);          // entries i, i + 1 of M + 1
    const float4 e0 = SMEM ? tab[i] : __ldg(tab + L.tbase + i);
    const float4 e1 = SMEM ? tab[i + 1] : __ldg(tab + L.tbase + i + 1);
    a = fmaf(f, e1.x - e0.x, e0.x);
    b = fmaf(f, e1.y - e0.y, e0.y);
    c = fmaf(f, e1.z - e0.z, e0.z);
}

template <bool WEIGHTED, bool SMEM, bool DTAB>
__device__ __forceinline__ void em2_step(Lane &L, float z1, float z2, float &lw, const float4 *__restrict__ tab,
                                         const ModelDev *s_model, const ModelDev &M0)
{
    float a, b, c;                                       // S sqrt(dN), interpolated in x
    table2_at<SMEM>(L, tab, a, b, c, M0);
    const float vpv = drift_vpv<DTAB, SMEM>(L, tab, s_model, M0);
    const float dN = SMEM ? M0.dN : L.dN;
    const float hdN = hh_dN<SMEM>(L, M0);               // (pi^2/2 - 3) dN
    const float e1 = z1 + L.cb, e2 = z2 + L.cb_b;       // xi + beta sqrt(dN)
    // (phi, pi) += D dN + S beta dN + S xi sqrt(dN) = D dN + (S sqrt(dN)) e
    const float dx = fmaf(a, e1, fmaf(b, e2, L.p * dN));
    // full-rank noise drives pi directly: compensated momentum (see em_step)
    kahan_add(L.p, L.p_c, fmaf(b, e1, fmaf(c, e2, hdN * (L.p + vpv))));
    if (WEIGHTED) lw -= fmaf(L.cb, z1, fmaf(L.cb_b, z2, L.half_cb2));
    kahan_add(L.x, L.x_c, dx);
}

// Learned proposal in 2-D: beta = (clamp(o1), clamp(o2)) at the segment start.
template <bool SMEM, bool REC>
__device__ __forceinline__ void mlp2_segment_start(Lane &L, bool live, SegRec &sg, const uint2 *tiles,
                                                   const float *bias, const RunDev &pr, const ModelDev &M0)
{
    const float dN = SMEM ? M0.dN : L.dN, sqrt_dN = SMEM ? M0.sqrt_dN : L.sqrt_dN;
    float in0 = 0.0f, in1 = 0.0f, in2 = 0.0f;
    if (live) {
        const float xv = __fsub_rn(L.x, L.x_c);
        in0 = ((pr.mlp_flags & FPT_MLP_LOG_X) ? __logf(fmaxf(xv, pr.x_floor)) : xv);
        in0 = (in0 - pr.shift[0]) * pr.scale[0];
        in1 = (L.p - pr.shift[1]) * pr.scale[1];
        in2 = ((float)steps_of(L.grp) * dN - pr.shift[2]) * pr.scale[2];
    }
    float o1, o2;
    mlp_forward_warp(tiles, bias, in0, in1, in2, __ballot_sync(0xffffffffu, live), o1, o2);
    if (live) {
        const float b1 = fminf(fmaxf(o1, -pr.alpha_max), pr.alpha_max);
        const float b2 = fminf(fmaxf(o2, -pr.alpha_max), pr.alpha_max);
        L.cb = b1 * sqrt_dN;
        L.cb_b = b2 * sqrt_dN;
        L.half_cb2 = 0.5f * fmaf(b1, b1, b2 * b2) * dN;
        if (REC) {
            sg.in0 = in0; sg.in1 = in1; sg.in2 = in2;
            sg.sum_xi = 0.0f;
            sg.sum_xi2 = 0.0f;
            sg.n0 = steps_of(L.grp);
            sg.open = true;
        }
    }
}

// ---------------------------------------------------------------------------
// The interval between two refill points
// ---------------------------------------------------------------------------
// One group of four steps of every lane, in either noise rank.
template <bool WEIGHTED, bool SMEM, bool NIDX, bool DTAB, bool RANK2>
__device__ __forceinline__ void any_step(Lane &L, int n, int s, const float *z, float &lw,
                                         const float4 *__restrict__ tab, const ModelDev *s_model,
                                         const ModelDev &M0)
{
    if (RANK2) em2_step<WEIGHTED, SMEM, DTAB>(L, z[2 * s], z[2 * s + 1], lw, tab, s_model, M0);
    else em_step<WEIGHTED, SMEM, NIDX, DTAB>(L, n, z[s], lw, tab, s_model, M0);
}

// Normals of group grp: Philox block grp (1-D noise: one normal per step), blocks
// 2 grp and 2 grp + 1 (full-rank noise: two per step).
template <bool RANK2>
__device__ __forceinline__ void group_normals(const EmParams &P, const PhiloxLane &rng, int grp, float *z)
{
#pragma unroll
    for (int h = 0; h < (RANK2 ? 2 : 1); ++h) {
        const uint4 r = philox4x32_10((RANK2 ? 2u : 1u) * (uint32_t)grp + h, rng, P.rk);
        box_muller(r.x, r.y, z[4 * h], z[4 * h + 1]);
        box_muller(r.z, r.w, z[4 * h + 2], z[4 * h + 3]);
    }
}

// Ring of normals between a helper warp and its consumer: slots of four Philox
// blocks. The helper passes the slot's barrier when it has filled the slot, the
// consumer when it starts on it (and has read the one before).
template <bool RANK2>
struct Ring {
    static constexpr int kGroups = RANK2 ? 2 : 4;
    PairSm *pair;
    int index, g;                        // pair index, groups consumed

    __device__ __forceinline__ void skip()
    {
        if (g % kGroups == 0) pair_barrier(index);
        ++g;
    }
    __device__ __forceinline__ void take(float *z)
    {
        const float4 *q = pair->ring + (g & (2 * kGroups - 1)) * (RANK2 ? 64 : 32) + (threadIdx.x & 31);
        skip();
#pragma unroll
        for (int h = 0; h < (RANK2 ? 2 : 1); ++h) {
            const float4 v = q[32 * h];
            z[4 * h] = v.x; z[4 * h + 1] = v.y; z[4 * h + 2] = v.z; z[4 * h + 3] = v.w;
        }
    }
};

// The helper's part: normals of `groups` groups of the consumer's lanes.
template <bool RANK2>
__device__ __forceinline__ void help(const EmParams &P, PairSm &pair, int index, int groups)
{
    constexpr int kGroups = Ring<RANK2>::kGroups;
    const int lane = threadIdx.x & 31;
    const uint4 q = pair.lane[lane];
    const PhiloxLane rng = {q.x, q.y, q.z};
    for (int g = 0; g < groups; g += kGroups) {
        float4 *slot = pair.ring + (g & (2 * kGroups - 1)) * (RANK2 ? 64 : 32) + lane;
#pragma unroll
        for (int k = 0; k < kGroups; ++k) {
            float z[RANK2 ? 8 : 4];
            group_normals<RANK2>(P, rng, (int)q.w + g + k, z);
#pragma unroll
            for (int h = 0; h < (RANK2 ? 2 : 1); ++h)
                slot[32 * ((RANK2 ? 2 : 1) * k + h)] = make_float4(z[4 * h], z[4 * h + 1], z[4 * h + 2], z[4 * h + 3]);
        }
        pair_barrier(index);
    }
}

// Sums of normals over the first k + 1 steps of a group (record mode).
template <bool RANK2>
__device__ __forceinline__ void add_xi(SegRec &sg, const float *z, int k)
{
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        if (s > k) break;
        sg.sum_xi = __fadd_rn(sg.sum_xi, z[RANK2 ? 2 * s : s]);
        if (RANK2) sg.sum_xi2 = __fadd_rn(sg.sum_xi2, z[2 * s + 1]);
    }
}

// Every lane of the warp steps through the group, without a branch per step; a
// lane notes after which steps its field was at or below the end surface. A
// live lane that passed at step k ends there: its step count is 4 grp + k + 1,
// its ln w and noise sums are formed from the increments of those k + 1 steps,
// in the same order as the running sums, and its results are written at once.
// What the lane computes after that (until it is refilled) is never read, and
// every table index is clamped, so it stays in bounds. A warp with idle lanes
// thus runs the same straight code as a full one.
template <bool WEIGHTED, bool SMEM, bool REC, bool NIDX, bool DTAB, bool RANK2>
__device__ __forceinline__ void run_group(const EmParams &P, Lane &L, bool &live, SegRec &sg, const float *z,
                                          const float4 *__restrict__ tab, const ModelDev *s_model)
{
    const int n0 = steps_of(L.grp);
    float lw = 0.0f;
    // the fields after each step are kept for the lane that passed, the others have
    // one chained comparison a step (four flags instead: 64 models 32.0 ms
    // against 29.6, eight biases 73.2 against 72.3, 2,048 paths 430 us against 419)
    float xs[4], cs[4];
    bool hit = false;
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        any_step<WEIGHTED, SMEM, NIDX, DTAB, RANK2>(L, n0 + s, s, z, lw, tab, s_model, P.m0);
        xs[s] = L.x;
        cs[s] = L.x_c;
        hit |= passed(L);
    }
    if (live && hit) {
        bool h[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) h[s] = xs[s] <= cs[s];
        const int k = h[0] ? 0 : h[1] ? 1 : h[2] ? 2 : 3;
        if (WEIGHTED) {
            const float lk = group_lw<NIDX, RANK2>(L, z, n0, k);
            if (lk != 0.0f) kahan_add(L.lw_hi, L.lw_lo, lk);
        }
        finish(P, L, n0 + k + 1, true);
        live = false;
        if (REC && sg.open) {
            add_xi<RANK2>(sg, z, k);
            put_record<RANK2>(P, L, sg, (long long)atomicAdd(P.rec_cursor, 1ull));
            sg.open = false;
        }
    }
    if (REC) add_xi<RANK2>(sg, z, 3);
    // the group's weight increments (at most 4, so a plain FP32 sum) into the pair;
    // adding a zero sum would re-round the pair
    if (WEIGHTED && lw != 0.0f) kahan_add(L.lw_hi, L.lw_lo, lw);
    ++L.grp;
}

// A group of an interval that is tried without looking for passages: the steps, the
// weights and the noise sums only. Returns whether the lane's field was at or
// below the end surface after one of the steps.
template <bool WEIGHTED, bool SMEM, bool REC, bool NIDX, bool DTAB, bool RANK2>
__device__ __forceinline__ bool try_group(const EmParams &P, Lane &L, SegRec &sg, const float *z,
                                          const float4 *__restrict__ tab, const ModelDev *s_model)
{
    const int n0 = steps_of(L.grp);
    float lw = 0.0f;
    bool hit = false;
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        any_step<WEIGHTED, SMEM, NIDX, DTAB, RANK2>(L, n0 + s, s, z, lw, tab, s_model, P.m0);
        hit |= passed(L);
    }
    if (REC) add_xi<RANK2>(sg, z, 3);
    if (WEIGHTED && lw != 0.0f) kahan_add(L.lw_hi, L.lw_lo, lw);
    ++L.grp;
    return hit;
}

// The same as run_group with a branch per step, for the interval in which a lane of
// the warp reaches the step cap inside a group.
template <bool WEIGHTED, bool SMEM, bool REC, bool NIDX, bool DTAB, bool RANK2>
__device__ __forceinline__ void run_group_guarded(const EmParams &P, Lane &L, bool &live, SegRec &sg,
                                                  const float *z, const float4 *__restrict__ tab,
                                                  const ModelDev *s_model)
{
    const int nmax = SMEM ? P.m0.max_steps : L.nmax;
    int n = steps_of(L.grp);
    float lw = 0.0f;
    bool done = !live;
#pragma unroll
    for (int s = 0; s < 4; ++s)
        if (!done) {
            if (REC) {
                sg.sum_xi = __fadd_rn(sg.sum_xi, z[RANK2 ? 2 * s : s]);
                if (RANK2) sg.sum_xi2 = __fadd_rn(sg.sum_xi2, z[2 * s + 1]);
            }
            any_step<WEIGHTED, SMEM, NIDX, DTAB, RANK2>(L, n, s, z, lw, tab, s_model, P.m0);
            ++n;
            done = passed(L) | (n >= nmax);
        }
    if (WEIGHTED && lw != 0.0f) kahan_add(L.lw_hi, L.lw_lo, lw);
    if (live && done) {
        finish(P, L, n, passed(L));
        live = false;
    }
    ++L.grp;
}

// ---------------------------------------------------------------------------
// Past the noise window
// ---------------------------------------------------------------------------
// After the last step of its noise window a path is classical: no normals, no
// table, no weight. Left among noisy lanes it would take their full steps (65
// instructions for 16), and more than half of a path's steps lie there (window of
// 4.9 e-folds, paths of 11.5). So a lane is parked when its window has ended --
// state into a buffer, the lane free for the next path -- and classical_kernel
// finishes the parked paths after the stepper, all lanes alike. 10^6 paths:
// 25.2 -> 15.9 ms. A lane that finds the buffer full goes on in the stepper.
// Parked path: (x, x_c, pi, unit), (ln w pair, steps / 4, -).
__device__ __forceinline__ void park(const EmParams &P, Lane &L, bool &live)
{
    const bool ended = live && L.nidx && steps_of(L.grp) > L.win_hi;
    const unsigned m = __ballot_sync(0xffffffffu, ended);
    if (!m || !P.park_cap) return;
    const unsigned lane = threadIdx.x & 31u;
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(P.cursor + 1, (unsigned long long)__popc(m));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (!ended) return;
    const unsigned long long i = base + __popc(m & ((1u << lane) - 1u));
    if (i < (unsigned long long)P.park_cap) {
        P.parked[2 * i] = make_float4(L.x, L.x_c, L.p, __uint_as_float(L.unit));
        P.parked[2 * i + 1] = make_float4(L.lw_hi, L.lw_lo, __int_as_float(L.grp), 0.0f);
        live = false;
    } else {
        L.win_hi = 0x7fffffff;           // every later step stays classical: the window has
        L.win_lo = 0x7fffffff;           // not begun for it
    }
}

// One classical step: em_step with S = T = 0 and no bias.
__device__ __forceinline__ void classical_step(Lane &L, const ModelDev *s_model)
{
    const float vpv = drift_vpv<false, false>(L, nullptr, s_model, s_model[0]);
    const float hdN = hh_dN<false>(L, s_model[0]);
    const float dx = L.p * L.dN;
    L.p = fmaf(hdN, L.p + vpv, L.p);
    kahan_add(L.x, L.x_c, dx);
}

constexpr int kClassicalBlock = 256;

__device__ __forceinline__ bool load_parked(const EmParams &P, Lane &L, unsigned long long i, unsigned long long count,
                                            const RunSm *s_run, const ModelDev *s_model, unsigned &slot)
{
    if (i >= count) return false;
    const float4 a = P.parked[2 * i];
    lane_load(L, (long long)__float_as_uint(a.w), s_run, s_model, P.n_runs, P.rk);
    L.x = a.x; L.x_c = a.y; L.p = a.z;
    L.grp = __float_as_int(P.parked[2 * i + 1].z);
    slot = (unsigned)i;
    return true;
}

__global__ void __launch_bounds__(kClassicalBlock, 5) classical_kernel(const EmParams P)
{
    extern __shared__ __align__(16) float4 s_tab[];
    __shared__ unsigned long long s_t0;
    RunSm *s_run = smem_runs(s_tab, 0, false);
    ModelDev *s_model = smem_models(s_run, P.n_runs);
    const unsigned long long count = min(P.cursor[1], (unsigned long long)P.park_cap);
    if (!count) return;
    stage_launch<false, false>(P, s_tab, s_run, s_model, s_t0, nullptr);
    const unsigned FULL = 0xffffffffu, lane = threadIdx.x & 31u;
    Lane L{};
    unsigned slot = 0;
    const unsigned long long first = ((unsigned long long)(threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32 + lane;
    bool live = load_parked(P, L, first, count, s_run, s_model, slot);
    const unsigned long long dealt = (unsigned long long)gridDim.x * blockDim.x;

    auto end = [&](int n, bool pas) {
        const float4 w = P.parked[2 * (size_t)slot + 1];
        L.lw_hi = w.x;
        L.lw_lo = w.y;
        finish(P, L, n, pas);
        live = false;
    };
    while (__any_sync(FULL, live)) {
        for (int g = 0; g < P.groups_per_check; ++g) {
            bool h[4];
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                classical_step(L, s_model);
                h[s] = passed(L);
            }
            const int n0 = steps_of(L.grp);
            if (live && ((h[0] | h[1] | h[2] | h[3]) || cap_in_group(L.grp, L.nmax))) {
                const int k = h[0] ? 0 : h[1] ? 1 : h[2] ? 2 : h[3] ? 3 : 4;
                if (k < 4 && step_within(L.grp, k, L.nmax)) end(n0 + k + 1, true);
                else end(L.nmax, false);
            }
            ++L.grp;
        }
        const unsigned idle = __ballot_sync(FULL, !live);
        if (idle) {
            unsigned long long base = 0;
            if (lane == 0) base = atomicAdd(P.cursor + 2, (unsigned long long)__popc(idle));
            base = __shfl_sync(FULL, base, 0) + dealt;
            if (!live) live = load_parked(P, L, base + __popc(idle & ((1u << lane) - 1u)), count, s_run, s_model, slot);
        }
        if (P.budget_ns && past_deadline(P, s_t0)) break;
    }
}

cudaError_t classical_launch(const EmParams &p, int sm_count, cudaStream_t s)
{
    const size_t smem = em_smem_bytes(EmVariant{}, 0, p.n_runs, p.n_models, 0);
    classical_kernel<<<5 * sm_count, kClassicalBlock, smem, s>>>(p);
    return cudaGetLastError();
}

// One interval of the warp: the proposal's evaluation, the groups, the records.
template <bool WEIGHTED, bool SMEM, bool MLP, bool REC, bool NIDX, bool DTAB, bool MNET, bool RANK2, bool RING>
__device__ __forceinline__ void run_interval(const EmParams &P, Lane &L, bool &live, SegRec &sg, Ring<RANK2> &ring,
                                             const float4 *__restrict__ tab, const RunSm *s_run,
                                             const ModelDev *s_model, const uint2 *s_tiles, const float *s_bias,
                                             const RunDev &prun)
{
    const unsigned FULL = 0xffffffffu;
    if (!__any_sync(FULL, live)) {
        if (RING)
            for (int g = 0; g < P.groups_per_check; ++g) ring.skip();
        return;
    }
    if (MLP && __any_sync(FULL, live && L.mlp)) {
        if (RANK2) mlp2_segment_start<SMEM, REC>(L, live && L.mlp, sg, s_tiles, s_bias, prun, P.m0);
        else if (MNET) mlp_segment_start_multi<SMEM, REC>(L, live && L.mlp, sg, tab, P.runs, P.m0);
        else mlp_segment_start<SMEM, REC>(L, live && L.mlp, sg, tab, s_tiles, s_bias, prun, P.m0);
    }
    const int nmax = SMEM ? P.m0.max_steps : L.nmax;
    const bool capped_inside = __any_sync(FULL, live && cap_inside(L.grp, P.groups_per_check, nmax));
    constexpr int kZ = RANK2 ? 8 : 4;
    float z[kZ];
    if (!capped_inside) {
        bool again = true;
        if (RING && MLP) {
            // A lone warp waits for every group's passage test and branch. On the long
            // paths of a learned proposal it tries the whole segment without them, and only
            // if a live lane passed in it does it go back and take the segment again:
            // training round of 2^15 paths 24.5 -> 22.7 ms, 2^18 learned paths 29.5 ->
            // 28.6 ms. Where many short paths end in the tail the second attempts cost
            // more than they give (16,384 linear paths 0.46 -> 0.50 ms), so the others
            // look after every group.
            const float x = L.x, x_c = L.x_c, p = L.p, p_c = L.p_c, lw_hi = L.lw_hi, lw_lo = L.lw_lo;
            const float sx = sg.sum_xi, sy = sg.sum_xi2;
            const int grp = L.grp;
            bool hit = false;
            float zn[kZ];
            ring.take(zn);
            for (int g = 1; g < P.groups_per_check; ++g) {
#pragma unroll
                for (int i = 0; i < kZ; ++i) z[i] = zn[i];
                ring.take(zn);
                hit |= try_group<WEIGHTED, SMEM, REC, NIDX, DTAB, RANK2>(P, L, sg, z, tab, s_model);
            }
            hit |= try_group<WEIGHTED, SMEM, REC, NIDX, DTAB, RANK2>(P, L, sg, zn, tab, s_model);
            again = __any_sync(FULL, live && hit);
            if (again) {
                L.x = x; L.x_c = x_c; L.p = p; L.p_c = p_c; L.lw_hi = lw_hi; L.lw_lo = lw_lo;
                sg.sum_xi = sx; sg.sum_xi2 = sy;
                L.grp = grp;
            }
        }
        for (int g = 0; again && g < P.groups_per_check; ++g) {
            if (RING && !MLP) ring.take(z);
            else group_normals<RANK2>(P, L.rng, L.grp, z);
            run_group<WEIGHTED, SMEM, REC, NIDX, DTAB, RANK2>(P, L, live, sg, z, tab, s_model);
        }
        if (live && cap_reached(L.grp, nmax)) {        // the cap falls on the interval's end
            finish(P, L, steps_of(L.grp), false);
            live = false;
        }
    } else {
        for (int g = 0; g < P.groups_per_check; ++g) {
            if (RING) ring.skip();
            group_normals<RANK2>(P, L.rng, L.grp, z);
            run_group_guarded<WEIGHTED, SMEM, REC, NIDX, DTAB, RANK2>(P, L, live, sg, z, tab, s_model);
        }
    }
    if (NIDX) park(P, L, live);
    if (REC) write_records<RANK2>(P, L, sg);
}

// Register budgets: two 512-thread blocks per SM (32 warps, at most 64
// registers; three blocks of 40 registers: direct sampling of 2^22 paths 37.6 ms
// against 36.0, eight biases 87.2 against 73.3); spilled: nothing with the table in
// shared memory, 12 bytes at most without. The learned-proposal steppers take at
// most 384 threads per block and two blocks, 80 registers (a 64-register build ran
// 512-thread blocks but executed ~7% more instructions per step); with the tail's
// second copy of the interval they spill 20-82 bytes, with several models 76-226.
// The steppers with one network per run keep each run's constants per lane and
// take 256-thread blocks of 128 registers: they spill 68-94 bytes, of 80 registers
// 280-430 (training round of 64 networks x 1,024 paths 18.8 -> 18.3 ms, 64 x 8,192
// paths to a cap of 2^14 steps 15.7 -> 15.0 ms); the others gained nothing from it.
template <bool WEIGHTED, bool SMEM, bool MLP, bool REC, bool NIDX, bool DTAB, bool MNET, bool RANK2>
__device__ __forceinline__ void stepper(const EmParams &P)
{
    extern __shared__ __align__(16) float4 s_tab[];
    __shared__ unsigned long long s_t0;
    __shared__ TailSm s_tail;

    // single-network MLP variants: the proposal's fragment blob follows the
    // table in shared memory; then the run constants and model descriptors
    const int tab_entries = SMEM ? P.smem_table_points : 0;
    uint2 *s_tiles = reinterpret_cast<uint2 *>(s_tab + tab_entries);
    float *s_bias = reinterpret_cast<float *>(s_tiles + kMlpTiles * 32);
    RunSm *s_run = smem_runs(s_tab, tab_entries, MLP && !MNET);
    ModelDev *s_model = smem_models(s_run, P.n_runs);
    PairSm *s_pairs = smem_pairs(s_model, P.n_models);
    const RunDev &prun = P.runs[MLP ? P.mlp_run : 0];
    // units of the first chunks cover the launch: the tail starts at once
    if (threadIdx.x == 0) s_tail.dry = (long long)gridDim.x * blockDim.x >= P.total_units;
    stage_launch<SMEM, MLP && !MNET>(P, s_tab, s_run, s_model, s_t0, s_tiles);

    const float4 *tab = SMEM ? s_tab : P.tables;

    Lane L;
    SegRec sg;
    sg.open = false;
    bool live = first_units(P, L, s_run, s_model);
    Ring<RANK2> ring{};
    // until the work is dealt out: an interval, then new trajectories for the idle lanes
    bool stop = false;
    // (a vote: another warp may set dry between two lanes' reads, and all lanes must
    // take part in the interval's warp-wide calls, or none)
    while (!__any_sync(0xffffffffu, *(volatile int *)&s_tail.dry)) {
        run_interval<WEIGHTED, SMEM, MLP, REC, NIDX, DTAB, MNET, RANK2, false>(P, L, live, sg, ring, tab, s_run,
                                                                              s_model, s_tiles, s_bias, prun);
        refill_point(P, L, live, s_run, s_model, &s_tail.dry);
        // trajectories in flight keep the ABORTED status set before launch
        stop = P.budget_ns && past_deadline(P, s_t0);
        if (stop && (threadIdx.x & 31u) == 0) *(volatile int *)&s_tail.dry = 1;   // the others come to the meeting
        __syncwarp();
    }
    // the tail
    TailRole role;
    for (int round = 0;
         tail_meeting<!MNET>(P, L, live, stop, round, s_tail, s_pairs, s_run, s_model, role); ++round) {
        if (role.pair < 0) {
            for (int k = 0; k < P.tail_intervals; ++k)
                run_interval<WEIGHTED, SMEM, MLP, REC, NIDX, DTAB, MNET, RANK2, false>(
                    P, L, live, sg, ring, tab, s_run, s_model, s_tiles, s_bias, prun);
        } else if (role.helper) {
            help<RANK2>(P, s_pairs[role.pair], role.pair, P.tail_intervals * P.groups_per_check);
        } else {
            ring = Ring<RANK2>{s_pairs + role.pair, role.pair, 0};
            for (int k = 0; k < P.tail_intervals; ++k)
                run_interval<WEIGHTED, SMEM, MLP, REC, NIDX, DTAB, MNET, RANK2, true>(
                    P, L, live, sg, ring, tab, s_run, s_model, s_tiles, s_bias, prun);
        }
        stop = P.budget_ns && past_deadline(P, s_t0);
    }
}

template <bool WEIGHTED, bool SMEM, bool MLP, bool REC, bool NIDX, bool DTAB, bool MNET = false>
__global__ void __launch_bounds__(MNET ? kMnetMaxBlock : MLP ? kMlpMaxBlock : 512, 2) em_kernel(const EmParams P)
{
    stepper<WEIGHTED, SMEM, MLP, REC, NIDX, DTAB, MNET, false>(P);
}

template <bool WEIGHTED, bool SMEM, bool MLP, bool DTAB, bool REC = false>
__global__ void __launch_bounds__(MLP ? kMlpMaxBlock : 512, 2) em2_kernel(const EmParams P)
{
    stepper<WEIGHTED, SMEM, MLP, REC, false, DTAB, false, true>(P);
}

template <bool DTAB>
static const void *em_fn_t(EmVariant v)
{
    if (v.rank2) {
        if (v.rec) return v.smem ? (const void *)em2_kernel<true, true, true, DTAB, true>
                                 : (const void *)em2_kernel<true, false, true, DTAB, true>;
        if (v.mlp) return v.smem ? (const void *)em2_kernel<true, true, true, DTAB>
                                 : (const void *)em2_kernel<true, false, true, DTAB>;
        if (v.weighted) return v.smem ? (const void *)em2_kernel<true, true, false, DTAB>
                                      : (const void *)em2_kernel<true, false, false, DTAB>;
        return v.smem ? (const void *)em2_kernel<false, true, false, DTAB>
                      : (const void *)em2_kernel<false, false, false, DTAB>;
    }
    if (v.rec) return v.smem ? (const void *)em_kernel<true, true, true, true, false, DTAB>
                             : (const void *)em_kernel<true, false, true, true, false, DTAB>;
    if (v.mlp) return v.smem ? (const void *)em_kernel<true, true, true, false, false, DTAB>
                             : (const void *)em_kernel<true, false, true, false, false, DTAB>;
    if (v.weighted) return v.smem ? (const void *)em_kernel<true, true, false, false, false, DTAB>
                                  : (const void *)em_kernel<true, false, false, false, false, DTAB>;
    return v.smem ? (const void *)em_kernel<false, true, false, false, false, DTAB>
                  : (const void *)em_kernel<false, false, false, false, false, DTAB>;
}

static const void *em_fn(EmVariant v)
{
    if (v.mnet) {   // one network per run: 1-D, phi-indexed tables
        if (v.rec) return v.smem ? (const void *)em_kernel<true, true, true, true, false, false, true>
                                 : (const void *)em_kernel<true, false, true, true, false, false, true>;
        return v.smem ? (const void *)em_kernel<true, true, true, false, false, false, true>
                      : (const void *)em_kernel<true, false, true, false, false, false, true>;
    }
    if (v.dtab) return em_fn_t<true>(v);
    if (v.nidx && !v.rank2 && !v.mlp) {
        if (v.weighted) return v.smem ? (const void *)em_kernel<true, true, false, false, true, false>
                                      : (const void *)em_kernel<true, false, false, false, true, false>;
        return v.smem ? (const void *)em_kernel<false, true, false, false, true, false>
                      : (const void *)em_kernel<false, false, false, false, true, false>;
    }
    return em_fn_t<false>(v);
}

size_t em_smem_bytes(EmVariant v, int table_entries, int n_runs, int n_models, int pairs)
{
    return sizeof(float4) * (size_t)table_entries + ((v.mlp && !v.mnet) ? (size_t)kMlpBlobBytes : 0) +
           ((sizeof(RunSm) * (size_t)n_runs + 15) / 16) * 16 + ((sizeof(ModelDev) * (size_t)n_models + 15) / 16) * 16 +
           sizeof(PairSm) * (size_t)pairs;
}

int em_max_pairs() { return kMaxPairs; }

// Opt in to dynamic shared memory, outside any stream capture. The opt-in is state
// of the kernel on the device, shared by every thread of the process, and a launch
// above it is refused: it is always the most the kernel can have (*most), so that
// contexts on other threads, which need other sizes, set the same value.
cudaError_t em_opt_in(EmVariant v, size_t *most)
{
    const void *f = em_fn(v);
    cudaFuncAttributes a;
    cudaError_t e = cudaFuncGetAttributes(&a, f);
    int dev = 0, bytes = 0;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&bytes, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    bytes -= (int)a.sharedSizeBytes;
    *most = (size_t)bytes;
    return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

// Resident blocks per SM for this shape (0: it does not fit); most: from em_opt_in().
int em_occupancy(EmVariant v, int block, size_t smem_bytes, size_t most)
{
    int nb = 0;
    if (smem_bytes > most ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, em_fn(v), block, smem_bytes) != cudaSuccess)
        return 0;
    return nb;
}

// Launch only (safe inside stream capture): em_opt_in() must have been called for
// this variant first.
cudaError_t em_launch(const EmParams &p, EmVariant v, int grid, int block, size_t smem_bytes, cudaStream_t s)
{
    void *args[] = {const_cast<EmParams *>(&p)};
    return cudaLaunchKernel(em_fn(v), dim3(grid), dim3(block), args, smem_bytes, s);
}

// ---------------------------------------------------------------------------
// K2: weighted histogram
// ---------------------------------------------------------------------------
// The FP64 units are the scarce resource here: they take two operations per SM
// and clock (64 cycles per warp instruction and sub-partition, measured), a
// DRAM pass over the 13 bytes of a path hardly counts. So the kernels do per
// path what needs FP64 and nothing else:
//   - the bin of a path follows from its step count by integer comparisons: the
//     first step count of each bin, in the FP64 arithmetic of the definition, is
//     found once per call (hist_prep_kernel) instead of a product, a difference
//     and a division per path;
//   - one exponential per path, e = exp(ln w - M_bin), in nine FP64 operations,
//     and none where ln w = M_bin (direct sampling); the sums over all weights
//     and over the tail are formed from the bins' sums, exp(M_bin - M) each;
//   - paths are sorted by bin inside a tile, so that a thread sums a stretch of
//     one bin in registers and touches the shared accumulators once per stretch.
// Measured, 10^7 weighted paths, 512 bins: 2.24 -> 0.77 ms (direct sampling,
// equal weights, 2.23 -> 0.38 ms); 16,384 paths, 512 bins: 300 -> 118 us a call.
//
// Classes of paths: bins 0 .. nb-1, nb: below N_lo, nb + 1: at or above N_hi,
// nb + 2: the tail part (N >= N_tail) of the class that N_tail cuts.
struct HistHead {
    unsigned long long capped, sum_n;    // capped paths; sum of the passed paths' step counts (two's complement)
    long long n_tail;                    // first step count with N >= N_tail (2^31: none)
    unsigned blocks_done;
    float step, off;                     // bins per step, bin coordinate at the first step count of bin 0
};

struct HistScratch {
    HistHead *head;
    unsigned long long *key;             // [nc] order-preserving keys of the classes' largest ln w (0: empty)
    long long *thr;                      // [nb + 1] first step counts
    double *tab;                         // [256] 2^(j/256)
    double *swn;                         // [nc] sum of e n
    double *tot;                         // [nc][5] count; shares of the sums of w, w n and the tail's w, w^2
    double *mom;                         // [kJackknife][nc][5]: count, sums of e, e^2, d, d^2 (d = ln w - M)
};

__host__ __device__ __forceinline__ int hist_classes(int nb) { return nb + 3; }

__host__ __device__ __forceinline__ HistScratch hist_scratch(unsigned char *base, int nb)
{
    const size_t nc = (size_t)hist_classes(nb);
    HistScratch s;
    s.head = reinterpret_cast<HistHead *>(base);
    s.key = reinterpret_cast<unsigned long long *>(base + 64);
    s.thr = reinterpret_cast<long long *>(s.key + nc);
    s.tab = reinterpret_cast<double *>(s.thr + nb + 1);
    s.swn = s.tab + 256;
    s.tot = s.swn + nc;
    s.mom = s.tot + 5 * nc;
    return s;
}

size_t hist_scratch_bytes(int nb)
{
    const size_t nc = (size_t)hist_classes(nb);
    return 64 + 8 * (nc + (size_t)nb + 1 + 256 + nc + 5 * nc + (size_t)kJackknife * nc * 5);
}

// Order-preserving map of doubles onto unsigned 64-bit keys (0 = empty).
__device__ __forceinline__ unsigned long long dkey(double v)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__device__ __forceinline__ double dkey_inv(unsigned long long k)
{
    const unsigned long long b = (k >> 63) ? (k & 0x7fffffffffffffffull) : ~k;
    return __longlong_as_double((long long)b);
}

// Reference of a class's deviations d = ln w - ref: its largest ln w, or 0 where that
// is infinite (a class of zero weights, an infinite weight), so that the sums of d
// are those of ln w itself. The sums of e = exp(ln w - M) of such a class mean
// nothing; their values follow from M alone (hist_finalize_kernel).
__device__ __forceinline__ double hist_ref(double M) { return isinf(M) ? 0.0 : M; }

// Jackknife block g covers trajectories [ceil(g n / G), ceil((g+1) n / G)).
__device__ __forceinline__ long long jk_begin(long long g, long long n)
{
    return (g * n + kJackknife - 1) / kJackknife;
}

// Smallest step count n in [-2^31, 2^31] that has reached a bound (2^31: none),
// `reached` being false below it and true from it on: bisection from a bracket
// around the guess g.
template <class F>
__device__ __forceinline__ long long first_n(double g, F reached)
{
    const long long kMin = -2147483648LL, kEnd = 2147483648LL;
    long long lo = kMin - 1, hi = kEnd;
    const long long c = g >= (double)kEnd ? kEnd : (g > (double)kMin ? (long long)g : kMin);
    const long long p = max(c - 2, kMin), q = min(c + 2, kEnd - 1);
    if (p < kEnd) {
        if (reached(p)) hi = p; else lo = p;
    }
    if (q > lo && q < hi) {
        if (reached(q)) hi = q; else lo = q;
    }
    while (hi - lo > 1) {
        const long long m = lo + ((hi - lo) >> 1);
        if (reached(m)) hi = m; else lo = m;
    }
    return hi;
}

// Clears the scratch, finds the bins' first step counts and tabulates 2^(j/256).
// The bin coordinate is q = (n dN - N_lo)/db in IEEE double without contraction,
// the same operations as the FP64 definition; it does not decrease with n.
__global__ void __launch_bounds__(256) hist_prep_kernel(const HistParams P)
{
    const int nb = P.n_bins, nc = hist_classes(nb);
    const HistScratch S = hist_scratch(P.scratch, nb);
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x, nt = (long long)gridDim.x * blockDim.x;
    for (long long i = t; i < nc; i += nt) {
        S.key[i] = 0ull;
        S.swn[i] = 0.0;
    }
    for (long long i = t; i < (long long)kJackknife * nc * 5; i += nt) S.mom[i] = 0.0;
    if (t == 0) {
        S.head->capped = 0ull;
        S.head->sum_n = 0ull;
        S.head->blocks_done = 0u;
    }
    auto N_of = [&](long long n) { return __dmul_rn((double)n, P.dN); };
    auto q_of = [&](long long n) { return __ddiv_rn(__dsub_rn(N_of(n), P.N_lo), P.db); };
    // FP64 tasks spread over the blocks
    for (int j = (int)(threadIdx.x * gridDim.x + blockIdx.x); j < nb + 2 + 256; j += (int)nt) {
        if (j <= nb) {
            // q >= j: the division only where the product cannot tell (within 2^-48 of
            // the bound; the quotient's own rounding is 2^-53), FP64 latency being what
            // this kernel is made of
            const double b = (double)j, at = b * P.db, sure = at * 3.6e-15;
            const long long n = first_n((P.N_lo + at) * P.inv_dN, [&](long long m) {
                const double x = __dsub_rn(N_of(m), P.N_lo), d = x - at;
                if (j > 0 && d > sure) return true;
                if (j > 0 && d < -sure) return false;
                return __ddiv_rn(x, P.db) >= b;
            });
            S.thr[j] = n;
            if (j == 0) {
                // bins far narrower than a step: only the first step count can lie in range
                const double step = P.dN / P.db;
                S.head->step = step < 2.0 * kMaxBins ? (float)step : 0.0f;
                S.head->off = n < 2147483648LL ? (float)q_of(n) : 0.0f;
            }
        } else if (j == nb + 1) {
            S.head->n_tail = isnan(P.N_tail) ? 2147483648LL : first_n(P.N_tail * P.inv_dN, [&](long long m) { return N_of(m) >= P.N_tail; });
        } else {
            S.tab[j - nb - 2] = exp2((double)(j - nb - 2) * (1.0 / 256.0));
        }
    }
}

// The class of a step count: bin by a float estimate (its error is below 4096
// 2^-21 bins, so it is at most one bin off), corrected by the bins' first step
// counts without a branch.
struct HistClasses {
    const long long *thr;
    long long t0, t1, n_tail;            // first step counts of bin 0, above N_hi, in the tail
    float step, off;
    int nb, cut;                         // class that n_tail lies in

    __device__ __forceinline__ int plain(long long n) const
    {
        if (n < t0) return nb;
        if (n >= t1) return nb + 1;
        int b = (int)fmaf((float)(uint32_t)(n - t0), step, off);
        b = min(max(b, 0), nb - 1);
        b += (int)(n >= thr[b + 1]) - (int)(n < thr[b]);
        CHECK_INDEX(b, nb, kCheckBin);
        return b;
    }
    __device__ __forceinline__ int of(long long n) const
    {
        const int c = plain(n);
        return (c == cut && n >= n_tail) ? nb + 2 : c;
    }
};

// Whether class c lies wholly in the tail (order: below, bins, above).
__device__ __forceinline__ bool tail_class(int c, int cut, int nb, bool any)
{
    if (!any) return false;
    if (c == nb + 2) return true;
    const int a = c == nb ? -1 : c == nb + 1 ? nb : c, b = cut == nb ? -1 : cut == nb + 1 ? nb : cut;
    return a > b;
}

__device__ __forceinline__ HistClasses hist_stage(const HistScratch &S, int nb, long long *s_thr)
{
    for (int i = threadIdx.x; i <= nb; i += blockDim.x) s_thr[i] = S.thr[i];
    __syncthreads();
    HistClasses C{s_thr, s_thr[0], s_thr[nb], S.head->n_tail, S.head->step, S.head->off, nb, 0};
    C.cut = C.n_tail < 2147483648LL ? C.plain(C.n_tail) : nb + 1;
    return C;
}

// Largest ln w per class; capped paths; sum of step counts. An atomic only where
// the value raises the block's maximum.
__global__ void __launch_bounds__(256) hist_max_kernel(const HistParams P)
{
    extern __shared__ unsigned long long s_dyn64[];
    const int nb = P.n_bins, nc = hist_classes(nb);
    const HistScratch S = hist_scratch(P.scratch, nb);
    unsigned long long *s_max = s_dyn64;
    long long *s_thr = reinterpret_cast<long long *>(s_dyn64 + nc);
    for (int i = threadIdx.x; i < nc; i += blockDim.x) s_max[i] = 0ull;
    const HistClasses C = hist_stage(S, nb, s_thr);
    long long sum_n = 0;
    unsigned capped = 0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < P.n;
         i += (long long)gridDim.x * blockDim.x) {
        const long long u = P.unit_begin + i;
        const uint8_t st = P.status[u];
        capped += st == FPT_TRAJ_CAPPED;
        if (st != FPT_TRAJ_PASSED) continue;
        const int n = P.nsteps[u];
        const unsigned long long k = dkey(P.logw[u]);
        sum_n += n;
        const int c = C.of(n);
        if (k > *(volatile unsigned long long *)&s_max[c]) atomicMax(&s_max[c], k);
    }
    for (int o = 16; o > 0; o >>= 1) {
        sum_n += __shfl_xor_sync(0xffffffffu, sum_n, o);
        capped += __shfl_xor_sync(0xffffffffu, capped, o);
    }
    if ((threadIdx.x & 31) == 0) {
        if (sum_n) atomicAdd(&S.head->sum_n, (unsigned long long)sum_n);
        if (capped) atomicAdd(&S.head->capped, (unsigned long long)capped);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nc; i += blockDim.x)
        if (s_max[i] && s_max[i] > *(volatile unsigned long long *)&S.key[i]) atomicMax(&S.key[i], s_max[i]);
}

// exp(d) for d <= 0 (0 below -708, where the result leaves the normal range), by
// Tang's table-driven method (ACM TOMS 15, 1989): d = k ln2/256 + r, |r| < 0.00136, exp(d) = 2^(k >> 8) 2^((k & 255)/256) exp(r)
// with exp(r) to r^4/24 (next term 4e-17) and ln2/256 in two parts.
__device__ __forceinline__ double exp_neg(double d, const double *__restrict__ tab)
{
    const double kMagic = 6755399441055744.0;                    // 1.5 2^52
    const double t = fma(d, 369.32993046757463, kMagic);         // 256 / ln 2
    const int k = __double2loint(t);
    const double kd = t - kMagic;
    double r = fma(kd, -0x1.62e42fefa0000p-9, d);                // ln2/256 to 41 bits
    r = fma(kd, -0x1.cf79abc9e3b3ap-48, r);                      // the rest
    const double q = fma(r, fma(r, 1.0 / 24.0, 1.0 / 6.0), 0.5);
    const double p = fma(r * r, q, r);
    const double T = tab[k & 255];
    const double e = fma(T, p, T);
    const double s = __hiloint2double(__double2hiint(e) + (int)((unsigned)(k >> 8) << 20), __double2loint(e));
    const unsigned a = (unsigned)__double2hiint(d) & 0x7fffffffu;
    return a > 0x7ff00000u ? d : a > 0x40862000u ? 0.0 : s;      // NaN; |d| > 708
}

constexpr int kHistTile = 4096, kHistThreads = 256, kHistPer = kHistTile / kHistThreads;
constexpr int kHistSmemClasses = 1027;   // classes whose sums stay in shared memory over a block's tiles

size_t hist_sum_smem(int nb)
{
    const size_t nc = (size_t)hist_classes(nb);
    return 8 * (256 + nc + (size_t)nb + 1) + (size_t)kHistTile * 14 + 4 * ((nc + 1) & ~(size_t)1) +
           (nc <= kHistSmemClasses ? 56 * nc : 0);
}

struct Stretch {                         // sums over a stretch of one class
    int c;
    unsigned cnt, ones;                  // paths; paths with ln w = M (e = 1, d = 0)
    long long ones_n;                    // their step counts
    double s1, s2, d1, d2, wn;
};

// grid = (CTAs, kJackknife): CTA (c, g) takes chunk c of jackknife block g.
__global__ void __launch_bounds__(kHistThreads) hist_sum_kernel(const HistParams P)
{
    extern __shared__ double s_dynd[];
    __shared__ unsigned s_warp[kHistThreads / 32];
    const int nb = P.n_bins, nc = hist_classes(nb);
    const HistScratch S = hist_scratch(P.scratch, nb);
    const bool smom = nc <= kHistSmemClasses && P.chunk > kHistTile;   // a single tile adds to the totals at once
    double *s_tab = s_dynd, *s_M = s_tab + 256;
    long long *s_thr = reinterpret_cast<long long *>(s_M + nc);
    double *s_lw = reinterpret_cast<double *>(s_thr + nb + 1);
    // smom only: sums of e, e^2, d, d^2, e n; step counts of the e = 1 paths; counts of all and of those
    double *s_mom = s_lw + kHistTile;                                            // [nc][5]
    unsigned long long *s_onen = reinterpret_cast<unsigned long long *>(s_mom + (smom ? 5 * nc : 0));
    unsigned *s_cnt = reinterpret_cast<unsigned *>(s_onen + (smom ? nc : 0));    // [nc][2]
    int *s_n = reinterpret_cast<int *>(s_cnt + (smom ? 2 * nc : 0));
    unsigned *s_off = reinterpret_cast<unsigned *>(s_n + kHistTile);             // [nc]
    uint16_t *s_c = reinterpret_cast<uint16_t *>(s_off + ((nc + 1) & ~1));
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned FULL = 0xffffffffu;

    for (int i = tid; i < 256; i += kHistThreads) s_tab[i] = S.tab[i];
    for (int i = tid; i < nc; i += kHistThreads) s_M[i] = S.key[i] ? hist_ref(dkey_inv(S.key[i])) : 0.0;
    if (smom)
        for (int i = tid; i < nc; i += kHistThreads) {
            for (int k = 0; k < 5; ++k) s_mom[5 * i + k] = 0.0;
            s_onen[i] = 0ull;
            s_cnt[2 * i] = s_cnt[2 * i + 1] = 0u;
        }
    const HistClasses C = hist_stage(S, nb, s_thr);
    const long long g = blockIdx.y;
    const long long b0 = jk_begin(g, P.n), b1 = jk_begin(g + 1, P.n);
    const long long c0 = b0 + (long long)blockIdx.x * P.chunk, c1 = min(b1, c0 + (long long)P.chunk);
    double *gm = S.mom + (size_t)g * nc * 5;

    // counts go by integer atomics; the FP64 sums, which a stretch of e = 1 paths
    // does not have, by compare-and-swap
    auto add = [&](const Stretch &q) {
        const double v[5] = {q.s1, q.s2, q.d1, q.d2, q.wn};
        if (smom) {
            atomicAdd(&s_cnt[2 * q.c], q.cnt);
            if (q.ones) {
                atomicAdd(&s_cnt[2 * q.c + 1], q.ones);
                atomicAdd(&s_onen[q.c], (unsigned long long)q.ones_n);
            }
            if (q.cnt != q.ones)
#pragma unroll
                for (int k = 0; k < 5; ++k) atomicAdd(&s_mom[5 * q.c + k], v[k]);
        } else {
            const double one = (double)q.ones;
            atomicAdd(&gm[5 * q.c], (double)q.cnt);
            atomicAdd(&gm[5 * q.c + 1], v[0] + one);
            atomicAdd(&gm[5 * q.c + 2], v[1] + one);
            if (q.cnt != q.ones) {
                atomicAdd(&gm[5 * q.c + 3], v[2]);
                atomicAdd(&gm[5 * q.c + 4], v[3]);
            }
            atomicAdd(&S.swn[q.c], v[4] + (double)q.ones_n);
        }
    };

    for (long long base = c0; base < c1; base += kHistTile) {
        for (int i = tid; i < nc; i += kHistThreads) s_off[i] = 0u;
        __syncthreads();
        // class and rank of the tile's paths
        double lw[kHistPer];
        int n[kHistPer];
        unsigned where[kHistPer];        // class << 16 | rank, all ones: not passed
#pragma unroll
        for (int k = 0; k < kHistPer; ++k) {
            const long long i = base + k * kHistThreads + tid;
            where[k] = 0xffffffffu;
            if (i < c1 && P.status[P.unit_begin + i] == FPT_TRAJ_PASSED) {
                n[k] = P.nsteps[P.unit_begin + i];
                lw[k] = P.logw[P.unit_begin + i];
                const int c = C.of(n[k]);
                where[k] = ((unsigned)c << 16) | atomicAdd(&s_off[c], 1u);
            }
        }
        __syncthreads();
        // exclusive scan of the classes' counts
        const int per = (nc + kHistThreads - 1) / kHistThreads, f = min(tid * per, nc), l = min(f + per, nc);
        unsigned mine = 0;
        for (int i = f; i < l; ++i) mine += s_off[i];
        unsigned incl = mine;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned v = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane == 31) s_warp[warp] = incl;
        __syncthreads();
        unsigned at = incl - mine, m = 0;
        for (int w = 0; w < kHistThreads / 32; ++w) {
            if (w < warp) at += s_warp[w];
            m += s_warp[w];
        }
        for (int i = f; i < l; ++i) {
            const unsigned v = s_off[i];
            s_off[i] = at;
            at += v;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kHistPer; ++k) {
            if (where[k] == 0xffffffffu) continue;
            const unsigned c = where[k] >> 16, p = s_off[c] + (where[k] & 0xffffu);
            s_lw[p] = lw[k];
            s_n[p] = n[k];
            s_c[p] = (uint16_t)c;
        }
        __syncthreads();
        // a stretch of sorted paths per thread, of odd length (distinct banks)
        const unsigned len = ((m + kHistThreads - 1) / kHistThreads) | 1u;
        const unsigned p0 = min((unsigned)tid * len, m), p1 = min(p0 + len, m);
        Stretch q{-1, 0u, 0u, 0, 0.0, 0.0, 0.0, 0.0, 0.0};
        for (unsigned p = p0; p < p1; ++p) {
            const int c = s_c[p];
            if (c != q.c) {
                if (q.c >= 0) add(q);
                q = Stretch{c, 0u, 0u, 0, 0.0, 0.0, 0.0, 0.0, 0.0};
            }
            const double v = s_lw[p], M = s_M[c];
            const int nn = s_n[p];
            ++q.cnt;
            if (__double_as_longlong(v) == __double_as_longlong(M) && isfinite(v)) {
                ++q.ones;
                q.ones_n += nn;
            } else {
                const double d = v - M, e = exp_neg(d, s_tab);
                // the step count as a double: exponent bits around a biased integer
                const double dn = __hiloint2double(0x43300000, nn ^ (int)0x80000000) - 4503601774854144.0;
                q.s1 += e;
                q.s2 = fma(e, e, q.s2);
                q.d1 += d;
                q.d2 = fma(d, d, q.d2);
                q.wn = fma(e, dn, q.wn);
            }
        }
        // where the whole warp ends in one class (few bins), one lane adds for all
        const int head = __shfl_sync(FULL, q.c, 0);
        if (__all_sync(FULL, q.c == head)) {
            const bool all_ones = __all_sync(FULL, q.cnt == q.ones);
            for (int o = 16; o > 0; o >>= 1) {
                q.cnt += __shfl_xor_sync(FULL, q.cnt, o);
                q.ones += __shfl_xor_sync(FULL, q.ones, o);
                q.ones_n += __shfl_xor_sync(FULL, q.ones_n, o);
                if (all_ones) continue;
                q.s1 += __shfl_xor_sync(FULL, q.s1, o);
                q.s2 += __shfl_xor_sync(FULL, q.s2, o);
                q.d1 += __shfl_xor_sync(FULL, q.d1, o);
                q.d2 += __shfl_xor_sync(FULL, q.d2, o);
                q.wn += __shfl_xor_sync(FULL, q.wn, o);
            }
            if (lane == 0 && q.c >= 0) add(q);
        } else if (q.c >= 0) {
            add(q);
        }
        __syncthreads();
    }
    if (smom) {
        __syncthreads();
        for (int i = tid; i < nc; i += kHistThreads) {
            if (!s_cnt[2 * i]) continue;
            const double one = (double)s_cnt[2 * i + 1], *v = s_mom + 5 * i;
            atomicAdd(&gm[5 * i], (double)s_cnt[2 * i]);
            atomicAdd(&gm[5 * i + 1], v[0] + one);
            atomicAdd(&gm[5 * i + 2], v[1] + one);
            atomicAdd(&gm[5 * i + 3], v[2]);
            atomicAdd(&gm[5 * i + 4], v[3]);
            atomicAdd(&S.swn[i], v[4] + (double)(long long)s_onen[i]);
        }
    }
}

__device__ __forceinline__ double warp_sum(double v)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// a on lane 0, b on lane 1, c on lane 2, d on the others: the logarithms,
// exponentials, quotients and roots of a bin are taken side by side in one call
// (one after the other they made this kernel 35-45 us long, all FP64 latency).
__device__ __forceinline__ double on_lanes(double a, double b, double c = 1.0, double d = 1.0)
{
    const int lane = threadIdx.x & 31;
    return lane == 0 ? a : lane == 1 ? b : lane == 2 ? c : d;
}
__device__ __forceinline__ double from_lane(double v, int lane) { return __shfl_sync(0xffffffffu, v, lane); }

// Largest keys over all classes and over the tail's, by the whole warp.
__device__ __forceinline__ void hist_max_keys(const HistScratch &S, int nb, int cut, bool any_tail,
                                              unsigned long long &kg, unsigned long long &kt)
{
    kg = kt = 0ull;
    for (int c = threadIdx.x & 31; c < hist_classes(nb); c += 32) {
        const unsigned long long k = S.key[c];
        kg = max(kg, k);
        if (tail_class(c, cut, nb, any_tail)) kt = max(kt, k);
    }
    for (int o = 16; o > 0; o >>= 1) {
        kg = max(kg, __shfl_xor_sync(0xffffffffu, kg, o));
        kt = max(kt, __shfl_xor_sync(0xffffffffu, kt, o));
    }
}

// Output layout (doubles): 10 arrays of n_bins (count, log_sum_w, log_sum_w2,
// sum_lw, sum_lw2, pdf, se_w, pdf_ln, se_ln, se_jk) then 16 scalars. One warp per
// class, a lane per jackknife block (32 of them); the last block to finish adds
// the classes' shares of the scalars.
__global__ void __launch_bounds__(128) hist_finalize_kernel(const HistParams P, double *out)
{
    __shared__ bool s_last;
    __shared__ double s_sum[4][6];
    const int nb = P.n_bins, nc = hist_classes(nb);
    const HistScratch S = hist_scratch(P.scratch, nb);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, b = blockIdx.x * 4 + warp;
    const double n = (double)P.n;
    // the class that n_tail lies in, from the bins' first step counts
    const long long n_tail = S.head->n_tail;
    const HistClasses C{S.thr, S.thr[0], S.thr[nb], n_tail, S.head->step, S.head->off, nb, 0};
    const bool any_tail = n_tail < 2147483648LL;
    const int cut = any_tail ? C.plain(n_tail) : nb + 1;
    if (b < nc) {
        const double *m = S.mom + ((size_t)lane * nc + b) * 5;
        double cg = m[0], s1 = m[1], s2 = m[2], d1 = m[3], d2 = m[4];
        const unsigned long long key = S.key[b];
        double M = key ? dkey_inv(key) : 0.0;
        if (isinf(M)) s1 = s2 = NAN;     // exp(M - M)
        unsigned long long kg, kt;
        hist_max_keys(S, nb, cut, any_tail, kg, kt);
        const double tc = warp_sum(cg), t1 = warp_sum(s1), t2 = warp_sum(s2);
        // shares of this class in the sums over all weights and over the tail's: none
        // where every weight is zero (a sum of ln w that is not a number has a weight
        // that is none either)
        const bool some = key && (M != -INFINITY || isnan(warp_sum(d1)));
        const bool in_tail = some && tail_class(b, cut, nb, any_tail);
        {
            const double x = on_lanes(some ? M - dkey_inv(kg) : 0.0, in_tail ? M - dkey_inv(kt) : 0.0, 0.0, 0.0);
            const double ex = exp(x), f = from_lane(ex, 0), h = from_lane(ex, 1);
            if (lane == 0) {
                S.tot[5 * b] = tc;
                S.tot[5 * b + 1] = some ? f * t1 : 0.0;
                S.tot[5 * b + 2] = some ? f * S.swn[b] : 0.0;
                S.tot[5 * b + 3] = in_tail ? h * t1 : 0.0;
                S.tot[5 * b + 4] = in_tail ? h * h * t2 : 0.0;
            }
        }
        if (b < nb) {
            double cnt = tc, S1 = t1, S2 = t2;
            if (b == cut && S.key[nb + 2]) {
                // the bin that the tail cuts: both parts about the larger of their maxima
                const double *w = S.mom + ((size_t)lane * nc + nb + 2) * 5;
                const double Mt = dkey_inv(S.key[nb + 2]), Ma = key ? M : Mt;
                M = dkey_inv(max(key, S.key[nb + 2]));
                auto scale = [&](double Mp) { return Mp == M ? 1.0 : exp(Mp - M); };
                auto part = [&](double Mp, double f, double v, double u) {
                    return Mp == -INFINITY && Mp != M && !isnan(u) ? 0.0 : v * f;
                };
                const double fa = scale(Ma), ft = scale(Mt), none = isinf(Mt) ? NAN : 0.0;
                s1 = part(Ma, fa, s1, d1) + part(Mt, ft, w[1] + none, w[3]);
                s2 = part(Ma, fa * fa, s2, d1) + part(Mt, ft * ft, w[2] + none, w[3]);
                // deviations about the common reference
                const double da = hist_ref(Ma) - hist_ref(M), dt = hist_ref(Mt) - hist_ref(M);
                auto shift2 = [](double c, double u, double u2, double h) { return isinf(u2) ? u2 : u2 + h * (2.0 * u + c * h); };
                d2 = shift2(cg, d1, d2, da) + shift2(w[0], w[3], w[4], dt);
                d1 = (d1 + cg * da) + (w[3] + w[0] * dt);
                cg += w[0];
                cnt = warp_sum(cg);
                S1 = warp_sum(s1);
                S2 = warp_sum(s2);
            }
            const double D1 = warp_sum(d1), D2 = warp_sum(d2), R = hist_ref(M);
            // delete-one-block jackknife of the weighted estimator
            const double ng = (double)(jk_begin(lane + 1, P.n) - jk_begin(lane, P.n));
            const double q = (S1 - s1) / (n - ng);
            const double qm = warp_sum(q) / kJackknife;
            const double ss = warp_sum((q - qm) * (q - qm));
            if (!(cnt > 0)) {
                if (lane < 10)
                    out[lane * nb + b] = (lane == 1 || lane == 2) ? -INFINITY : (lane == 7 || lane == 8) ? NAN : 0.0;
            } else {
                // lognormal-mean estimator (n_b >= 2): mean, variance about it, Cox's error
                const double r1 = on_lanes(D1, S1 * S1, cnt) / on_lanes(cnt, n, n);
                const double mean = from_lane(r1, 0), share = from_lane(r1, 2);
                const double r2 = on_lanes(D2 - cnt * mean * mean, fmax(S2 - from_lane(r1, 1), 0.0),
                                           fmax(1.0 - share, 0.0)) / on_lanes(cnt - 1.0, (n - 1.0) * n, cnt);
                const double v = fmax(from_lane(r2, 0), 0.0);
                const double r3 = on_lanes(v, v * v) / on_lanes(cnt, 2.0 * (cnt - 1.0));
                const double cox2 = from_lane(r3, 0) + from_lane(r3, 1);
                const double rt = sqrt(on_lanes(cox2 + from_lane(r2, 2), from_lane(r2, 1),
                                                (kJackknife - 1.0) / kJackknife * ss));
                const double lg = log(on_lanes(S1, S2, n * P.db));
                const double lsw = M + from_lane(lg, 0);
                const double ex = exp(on_lanes(lsw - from_lane(lg, 2), M, R + mean + 0.5 * v));
                const double eM = from_lane(ex, 1);
                // per bin width: lognormal mean, errors of the weighted mean
                const double r4 = on_lanes(share * from_lane(ex, 2), eM * from_lane(rt, 1), eM * from_lane(rt, 2)) / P.db;
                const double pl = from_lane(r4, 0);
                const bool two = cnt >= 2.0;
                const double o[10] = {cnt, lsw, 2.0 * M + from_lane(lg, 1), D1 + cnt * R,
                                      isinf(D2) ? D2 : D2 + R * (2.0 * D1 + cnt * R), from_lane(ex, 0),
                                      from_lane(r4, 1), two ? pl : NAN, two ? pl * from_lane(rt, 0) : NAN,
                                      from_lane(r4, 2)};
                if (lane == 0)
#pragma unroll
                    for (int k = 0; k < 10; ++k) out[k * nb + b] = o[k];
            }
        }
    }
    // scalars
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&S.head->blocks_done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const volatile double *tot = S.tot;
    double v[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};   // passed, sum w, sum w n, tail: sum w, sum w^2, count
    for (int c = threadIdx.x; c < nc; c += 128) {
        for (int k = 0; k < 5; ++k) v[k] += tot[5 * c + k];
        if (tail_class(c, cut, nb, any_tail)) v[5] += tot[5 * c];
    }
    for (int k = 0; k < 6; ++k) v[k] = warp_sum(v[k]);
    if (lane == 0)
        for (int k = 0; k < 6; ++k) s_sum[warp][k] = v[k];
    __syncthreads();
    if (warp) return;
    for (int k = 0; k < 6; ++k) v[k] = (s_sum[0][k] + s_sum[1][k]) + (s_sum[2][k] + s_sum[3][k]);
    unsigned long long kg, kt;
    hist_max_keys(S, nb, cut, any_tail, kg, kt);
    const double r = on_lanes((double)(long long)S.head->sum_n * P.dN, v[2] * P.dN, v[3] * v[3]) /
                     on_lanes(v[0], v[1], v[4]);
    const double lg = log(on_lanes(v[3], n));
    const double p_tail = exp((kt ? dkey_inv(kt) : 0.0) + from_lane(lg, 0) - from_lane(lg, 1));
    const double mean = from_lane(r, 0), mean_w = from_lane(r, 1), ess = from_lane(r, 2);
    if (lane == 0) {
        const double cut_part = tot[5 * (nb + 2)];
        double *o = out + 10 * nb;
        o[0] = n;
        o[1] = v[0];
        o[2] = tot[5 * nb] + (cut == nb ? cut_part : 0.0);
        o[3] = tot[5 * (nb + 1)] + (cut == nb + 1 ? cut_part : 0.0);
        o[4] = (double)S.head->capped;
        o[5] = v[5];
        o[6] = v[0] > 0 ? mean : NAN;
        o[7] = v[1] > 0 ? mean_w : NAN;
        o[8] = v[4] > 0 ? ess : 0.0;
        o[9] = v[3] > 0 ? p_tail : 0.0;
        o[10] = kg ? dkey_inv(kg) : -INFINITY;
        for (int k = 11; k < 16; ++k) o[k] = 0.0;     // reserved
    }
}

cudaError_t hist_launch(const HistParams &params, double *out, cudaStream_t s)
{
    HistParams p = params;
    const int nb = p.n_bins, nc = hist_classes(nb);
    cudaError_t e;
    hist_prep_kernel<<<64, 256, 0, s>>>(p);
    if ((e = cudaGetLastError())) return e;
    // short calls are latency: a block per 256 paths up to four per SM. The opt-in to
    // more than 48 KB is shared by the threads of the process: every call sets the
    // value of the largest histogram (see em_opt_in)
    auto max_smem = [](int n) { return 8 * ((size_t)hist_classes(n) + n + 1); };
    const size_t smax = max_smem(nb);
    if (smax > 48 * 1024 &&
        (e = cudaFuncSetAttribute(hist_max_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)max_smem(kMaxBins))))
        return e;
    hist_max_kernel<<<(int)min(608LL, max(1LL, (p.n + 255) / 256)), 256, smax, s>>>(p);
    if ((e = cudaGetLastError())) return e;
    // per jackknife block: CTAs of at least a tile
    const size_t ssum = hist_sum_smem(nb);
    const size_t ssum_most = std::max(hist_sum_smem(kMaxBins), hist_sum_smem(kHistSmemClasses - 3));
    if (ssum > 48 * 1024 &&
        (e = cudaFuncSetAttribute(hist_sum_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ssum_most)))
        return e;
    const long long per_block = (p.n + kJackknife - 1) / kJackknife;
    const long long most = ssum > 113 * 1024 ? 4 : 9;             // one or two CTAs per SM: a single wave
    const int ctas = (int)min(most, max(1LL, (per_block + kHistTile - 1) / kHistTile));
    p.chunk = (per_block + ctas - 1) / ctas;
    hist_sum_kernel<<<dim3(ctas, kJackknife), kHistThreads, ssum, s>>>(p);
    if ((e = cudaGetLastError())) return e;
    hist_finalize_kernel<<<(nc + 3) / 4, 128, 0, s>>>(p, out);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Histogram without allocation: the scratch lives in a file-scope device array
// ---------------------------------------------------------------------------
constexpr size_t kNoAllocBytes =
    64 + 8 * ((size_t)8 * (kNoAllocMaxBins + 3) + 1 + 256 + (size_t)kJackknife * (kNoAllocMaxBins + 3) * 5);

// Every GPU that loads the library holds this array until the process exits.
static __device__ __align__(256) unsigned char g_hist_scratch[kNoAllocBytes];

size_t hist_noalloc_scratch_bytes() { return kNoAllocBytes; }

// Device address of the array. A device address is valid only in the context
// it was looked up in, so the cache is keyed by the id of the calling thread's
// current context (cuCtxGetId: unique for the life of the process, so a
// context created after cudaDeviceReset, or a non-primary context pushed by
// another library, looks the address up again). The first call in a context
// does the lookup; host code must not use the symbol itself as an address.
typedef CUresult (*CtxGetCurrentFn)(CUcontext *);
typedef CUresult (*CtxGetIdFn)(CUcontext, unsigned long long *);
struct NoAllocEntry {
    unsigned long long ctx_id;
    unsigned char *ptr;
};
static std::mutex g_noalloc_mu;
static NoAllocEntry g_noalloc_cache[64];
static int g_noalloc_n = 0;
static CtxGetCurrentFn g_ctx_get_current = nullptr;
static CtxGetIdFn g_ctx_get_id = nullptr;

// Id of the current context; 0 when no context is current.
static cudaError_t current_ctx_id(unsigned long long *id)
{
    *id = 0;
    if (!g_ctx_get_current || !g_ctx_get_id) {
        void *f1 = nullptr, *f2 = nullptr;
        cudaDriverEntryPointQueryResult q1, q2;
        cudaError_t e = cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f1, 12000, cudaEnableDefault, &q1);
        if (e != cudaSuccess) return e;
        e = cudaGetDriverEntryPointByVersion("cuCtxGetId", &f2, 12000, cudaEnableDefault, &q2);
        if (e != cudaSuccess) return e;
        if (q1 != cudaDriverEntryPointSuccess || q2 != cudaDriverEntryPointSuccess || !f1 || !f2)
            return cudaErrorNotSupported;
        g_ctx_get_current = reinterpret_cast<CtxGetCurrentFn>(f1);
        g_ctx_get_id = reinterpret_cast<CtxGetIdFn>(f2);
    }
    CUcontext c = nullptr;
    if (g_ctx_get_current(&c) != CUDA_SUCCESS) return cudaErrorContextIsDestroyed;
    if (!c) return cudaSuccess;
    if (g_ctx_get_id(c, id) != CUDA_SUCCESS) return cudaErrorContextIsDestroyed;
    return cudaSuccess;
}

static cudaError_t noalloc_scratch(unsigned char **out)
{
    std::lock_guard<std::mutex> g(g_noalloc_mu);
    unsigned long long id = 0;
    cudaError_t e = current_ctx_id(&id);
    if (e != cudaSuccess) return e;
    for (int i = 0; id && i < g_noalloc_n; ++i)
        if (g_noalloc_cache[i].ctx_id == id) {
            *out = g_noalloc_cache[i].ptr;
            return cudaSuccess;
        }
    // no cached address for this context: look it up (with no context
    // current, this initialises the current device's primary context first)
    void *p = nullptr;
    e = cudaGetSymbolAddress(&p, g_hist_scratch);
    if (e != cudaSuccess) return e;
    if (!id && (e = current_ctx_id(&id)) != cudaSuccess) return e;
    if (id && g_noalloc_n < 64) g_noalloc_cache[g_noalloc_n++] = NoAllocEntry{id, static_cast<unsigned char *>(p)};
    *out = static_cast<unsigned char *>(p);
    return cudaSuccess;
}

cudaError_t hist_noalloc_launch(HistParams p, double *out, cudaStream_t s)
{
    if (p.n_bins < 1 || p.n_bins > kNoAllocMaxBins) return cudaErrorInvalidValue;
    unsigned char *base = nullptr;
    cudaError_t e = noalloc_scratch(&base);
    if (e != cudaSuccess) return e;
    p.scratch = base;
    // hist_launch clears the scratch before it bins
    return hist_launch(p, out, s);
}

__global__ void n_of_steps_kernel(const int32_t *nsteps, long long n, double dN, double *N)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        N[i] = __dmul_rn((double)nsteps[i], dN);
}

cudaError_t n_of_steps_launch(const int32_t *nsteps, long long n, double dN, double *N,
                              cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    const int grid = (int)min(4096LL, (n + 255) / 256);
    n_of_steps_kernel<<<grid, 256, 0, s>>>(nsteps, n, dN, N);
    return cudaGetLastError();
}

}  // namespace fpt_dev
