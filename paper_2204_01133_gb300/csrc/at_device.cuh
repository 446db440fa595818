// at_device.cuh -- device-side pieces of the AT stage kernels (sm_103a, FP64).
//
// Everything a stage kernel needs that is not the kernel itself: the launch
// argument block, the Philox4x32-10 delay draw, the temporal extrapolation of
// halo values from the history ring, and the per-PDE derived quantities.
#pragma once
#include <cuda/atomic>

#include <cstdint>

#include "at_fixed.cuh"
#include "exp_table.h"

#define AT_KMAX_LIMIT 15
#define AT_QMAX 3
#define AT_HMAX 3
#define AT_NDER 8

namespace atk {

enum { ADVDIFF = 0, RNS = 1, EULER = 2, ADV_WENO = 3, BURGERS = 4, RNS_CHAIN = 5 };
enum { RK2 = 0, RK3TVD = 1, RK4 = 2 };
enum { SYNC = 0, AS = 1, AT = 2 };

// Everything one stage launch needs, passed by value (well under the
// kernel-parameter limit).
struct StageArgs {
    const double* X;   // stencil source: the stage argument U^{n,(s)}   [nvar][N]
    const double* u;   // u^n (read pointwise)                            [nvar][N]
    double* acc;       // RK accumulator (RK2, RK4)                       [nvar][N]
    double* Y;         // output: next stage argument, or u^{n+1} in place [nvar][N]
    double* ring;      // edge windows of stage arguments [R][S][P][2][H][nvar]
    uint8_t* dlog;     // delays of this step [S][P][2]
    int* status;       // bit 0: a non-finite value was written
    int64_t N, P;
    int64_t level;     // n: the step being computed
    int B, Tw, wpp;    // PE size, window length, windows per PE
    int wpc, win_smem; // per-stage central kernels: windows per CTA, shared doubles per window
    int stage, S, R, H, q, nvar;
    int mode, kmax, per_stage, rk;
    uint32_t instance, key0, key1;
    double dt, hdt, dt6;                      // dt, dt/2, dt/6 (formed once on the host)
    uint64_t thr[AT_KMAX_LIMIT];              // Philox word-0 thresholds
    double w[AT_KMAX_LIMIT + 1][AT_QMAX + 1]; // extrapolation weights by delay
    uint8_t wnz[AT_KMAX_LIMIT + 1];           // bit l: level l enters at delay k (weight != 0)
    double s1;                                // -1 / (D1 dx): scales fx_d1 (central first derivative, negated)
    double s2;                                // 1 / (D2 dx^2): scales fx_d2
    double cm[2 * AT_HMAX + 1];               // merged advection-diffusion taps
    double prm[16];                           // physics constants (see at.h)
    double k0;                                // derived physics constants (WENO: k0 = 1/dx, 3 eps)
    union {
        struct {
            double k1, k2, k3;
        };
        FxU eps3;
    };
    // reacting flow: the diffusion rows are u, the energy term over lambda and
    // Y, with the constants in the scale: s2v[v-1] = s2 times (4/3) mu,
    // lambda, lambda / (cp Le) for v = 1, 2, 3; kd1 = k1 / k2, kd3 = qc k3 / k2
    double s2v[3];
    double kd1, kd3;
    // persistent path only
    int64_t* done;       // per PE: stages completed, as the index n*S + s + 1 [P]
    double* gring;       // derived quantities of the edge windows [R][S][P][2][H][ND]
    int* abort_flag;     // set by the first wait that runs out
    int* place;          // per CTA: the SM it runs on, for the PE placement [P]
    int* place_count;    // CTAs that have written their SM
    int64_t wait_limit;  // polls before a wait gives up (bounded spin)
    int64_t withhold_pe; // fault injection: this PE never publishes (-1: none)
    int slack;           // ring levels beyond k_max + q + 1
    int arrival;         // 1: a delay is the age of the freshest neighbour data that has arrived
    int hist_recompute;  // 1: the ring holds stage values recomputed from u^m (reading A); the
                         //    stage kernels then push nothing into it
    int weno_interp;     // WENO PDEs: 1 the interpolation form (edge values, halo 4)
    // a PE range of a larger domain (split over ranks)
    int open_ends;       // 1: the range's outer buffer points read ext, not the ring
    double* ext;         // windows beyond the range's ends [R][S][2][H][nvar]
    int64_t pe_base, pe_total;  // global index of PE 0 and the domain's PE count (0: P)
    // delay trace (optional): the delay of every (step, stage, PE, side) of
    // levels trace_n0 .. trace_n0 + trace_steps - 1, [steps][S][P][2]
    uint8_t* trace;
    int64_t trace_n0, trace_steps;
    // batched path: the solve's own buffers (the stage kernels get X/Y/u per launch)
    double* bufA;
    double* bufB;
    double* state;
};

// The answer of a capacity query that ended with an error: 0, the kernel does not
// fit, where the launch shape itself is refused; -1, unknown, otherwise.
inline int64_t fit_error(cudaError_t e)
{
    cudaGetLastError();
    return e == cudaErrorInvalidValue ? 0 : -1;
}

// what a solve's reset takes besides its StageArgs
struct ResetArgs {
    int64_t ring_elems, ext_elems;
    unsigned char* ws;    // canary zones of 256 bytes at ws + guard[i]
    size_t guard[10];
    int nguard;
    uint32_t guard_word;
    StageArgs* slot_args; // a batch slot's table entries (null: none)
    int64_t *slot_level, *slot_left, nsteps;
};

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon et al., SC'11): ten rounds of two 32x32->64 products
// with a Weyl key schedule; only output word 0 is used.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t philox_w0(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                              uint32_t k0, uint32_t k1)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t hi0 = __umulhi(0xD2511F53u, c0), lo0 = 0xD2511F53u * c0;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c2), lo1 = 0xCD9E8D57u * c2;
        const uint32_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
        c0 = n0;
        c1 = lo1;
        c2 = n2;
        c3 = lo0;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return c0;
}

// Delay seen by PE `pe` at its `side` (0 left, 1 right) at (level, stage),
// clamped so that no level below 0 is ever read.
__device__ __forceinline__ int keff_at(const StageArgs& a, int64_t level, int stage, int64_t pe, int side)
{
    if (a.mode == SYNC) return 0;
    const uint32_t sc = a.per_stage ? (uint32_t)stage : 0u;
    int64_t gpe = pe;  // the global PE index (a range of a larger domain draws the domain's delays)
    if (a.pe_total > 0) {
        gpe += a.pe_base;
        if (gpe >= a.pe_total) gpe -= a.pe_total;
    }
    const uint32_t x = philox_w0((uint32_t)level, (uint32_t)gpe, sc | ((uint32_t)side << 8), a.instance,
                                 a.key0, a.key1);
    int k = 0;
    for (int i = 0; i < a.kmax; ++i) k += ((uint64_t)x >= a.thr[i]) ? 1 : 0;
    const int qq = (a.mode == AT) ? a.q : 0;
    int64_t avail = level - qq;
    if (avail < 0) avail = 0;
    return (int64_t)k < avail ? k : (int)avail;
}

// largest delay the start-up clamp allows at `level` (no level below 0 is read)
__device__ __forceinline__ int kcap_at(const StageArgs& a, int64_t level)
{
    if (a.mode == SYNC) return 0;
    int64_t avail = level - ((a.mode == AT) ? a.q : 0);
    if (avail < 0) avail = 0;
    return avail < a.kmax ? (int)avail : a.kmax;
}

// record the delay used at (level, stage, PE, side): the per-step log and,
// when one is attached, the trace
__device__ __forceinline__ void log_delay(const StageArgs& a, int64_t level, int stage, int64_t pe, int side, int k)
{
    a.dlog[((int64_t)stage * a.P + pe) * 2 + side] = (uint8_t)k;
    if (a.trace) {
        const int64_t t = level - a.trace_n0;
        if (t >= 0 && t < a.trace_steps) a.trace[((t * a.S + stage) * a.P + pe) * 2 + side] = (uint8_t)k;
    }
}

__device__ __forceinline__ int keff(const StageArgs& a, int64_t pe, int side)
{
    return keff_at(a, a.level, a.stage, pe, side);
}

// exp(x) by Tang's table-driven method (P. T. P. Tang, ACM TOMS 15(2), 1989)
// with 256 table entries: x = (256 M + j) ln2/256 + r, |r| <= ln2/512, and
// exp(x) = 2^M 2^(j/256) (1 + expm1(r)), expm1(r) by its Taylor polynomial of
// degree 4 (the first omitted term, r^5/120, is below 4e-17).  The product
// with 2^M is an integer add to the exponent field, exact while the result is
// normal, which the fast path |x| < 512 guarantees (tested on the high word
// with integer instructions); every other x (and Inf, NaN) goes to exp().
// What needs no more than FP32's 24 bits is done there (1 cycle against 64): the
// nearest multiple (a slip by one next to a tie leaves |r| a hair larger) and
// the factor 1/6 + r/24 of r^3, whose 2^-23 relative error is 5e-17 of the
// result.  Six FP64 instructions; within 2 ulp of the correctly rounded value.
__device__ __forceinline__ double at_exp(double x)
{
    static_assert(AT_EXP_N == 256, "the table has 256 entries");
    const uint32_t hi = fx_hi(x), ah = hi & 0x7fffffffu;
    if (ah >= 0x40800000u) return exp(x);
    const float t = fmaf(fx_float(x), (float)AT_EXP_INV_L, 12582912.0f);  // 1.5 2^23: the integer lands in the low bits
    const int n = __float_as_int(t) - 0x4b400000;                         // 256 M + j
    const uint32_t nb = __float_as_uint(t - 12582912.0f);
    // -n as a double (at most 18 bits: its low word is zero)
    const double nd = fx_double(n == 0 ? 0u : (((nb & 0x7fffffffu) >> 3) + 0x38000000u) | (~nb & 0x80000000u), 0u);
    double r = fma(nd, AT_EXP_L_HI, x);
    r = fma(nd, AT_EXP_L_LO, r);
    const uint32_t cb = __float_as_uint(fmaf(fx_float(r), 1.0f / 24.0f, 1.0f / 6.0f));
    const double c = fma(fx_double((cb >> 3) + 0x38000000u, cb << 29), r, 0.5);
    const double em1 = fma(c, r * r, r);            // expm1(r)
    const double tj = __ldg(&at_exp_tab[n & 255]);  // 2^(j/256)
    const double e = fma(tj, em1, tj);
    return fx_double(fx_hi(e) + ((uint32_t)(n >> 8) << 20), fx_lo(e));
}

// 1/x by two Newton-Raphson steps r <- r + r (1 - x r) from the hardware's
// approximate reciprocal (rcp.approx.ftz.f64): each step squares the
// relative error, leaving the result within about an ulp of 1/x for the
// normal, finite, nonzero x the kernels divide by (densities, pressures,
// temperatures, WENO weight sums).  Zero, Inf or subnormal x give Inf or
// NaN, which the non-finite check reports.  Five FP64-pipe instructions, about
// half of an IEEE division (at_rcp3 below: one fewer).  Exported by the probe
// library beside the others for the reciprocal tests.
__device__ __forceinline__ double at_rcp(double x)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    double e = fma(-x, r, 1.0);
    r = fma(r, e, r);
    e = fma(-x, r, 1.0);
    return fma(r, e, r);
}

// 1/x by one cubic Newton step from the hardware's approximate reciprocal:
// with e = 1 - x r, 1/x = r (1 + e + e^2 + ...), so r + r (e + e^2) cubes the
// relative error of r (Householder's method of order 3, e.g. Householder,
// "The Numerical Treatment of a Single Nonlinear Equation", 1970), one FP64
// instruction fewer than at_rcp's two quadratic steps, within about an ulp
// of 1/x for normal, finite, nonzero x (both are tested against 1/x).  The
// kernels' reciprocals are integer ones (at_rcpi) and come here only outside the
// normal range.
__device__ __forceinline__ double at_rcp3(double x)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double e = fma(-x, r, 1.0);
    return fma(r, fma(e, e, e), r);
}

// 1/x in integers (fx_rcp, at_fixed.cuh: correctly rounded up to 2^-60), the
// kernels' reciprocals of densities, temperatures and pressures: about 75 issue
// cycles beside the FP64 unit instead of three FP64 instructions, 192 cycles
// of it.  Zero, Inf, NaN and the ends of the range go to at_rcp3.
__device__ __forceinline__ double at_rcpi(double x)
{
    bool ok;
    double r = fx_rcp(x, &ok);
    if (!ok) r = at_rcp3(x);
    return r;
}

// sqrt(x) in integers (fx_sqrt), about 105 issue cycles against some ten FP64
// instructions; everything but positive normal numbers goes to sqrt().
__device__ __forceinline__ double at_sqrt(double x)
{
    bool ok;
    double r = fx_sqrt(x, &ok);
    if (!ok) r = sqrt(x);
    return r;
}

// Inf or NaN: exponent field all ones, tested on the high word with integer
// instructions (the FP64 pipe is the scarce one on this chip)
__device__ __forceinline__ bool nonfinite(double v)
{
    return (__double2hiint(v) & 0x7ff00000) == 0x7ff00000;
}

// Ring element of (level, stage, PE, side, point h of the edge window,
// variable v).  Levels read or written are never negative (start-up clamp)
// and stay below 2^31 (the library refuses longer runs), so the slot comes
// from a 32-bit remainder: a 64-bit one is a long software sequence that
// occupies the FP64 pipe.
__device__ __forceinline__ int64_t ring_index(const StageArgs& a, int64_t level, int stage, int64_t pe, int side,
                                              int h, int v)
{
    const int64_t r = (int64_t)((uint32_t)level % (uint32_t)a.R);
    return ((((r * a.S + stage) * a.P + pe) * 2 + side) * a.H + h) * a.nvar + v;
}

// The nvar values buffer point h beyond PE pe's `side` edge reads at level m,
// stage s: the neighbour's edge window in the ring (the neighbour's side
// 1 - side), or, at the outer edges of a range with open ends, the window
// supplied from outside the range.
__device__ __forceinline__ const double* halo_window(const StageArgs& a, int64_t m, int s, int64_t pe, int side, int h)
{
    if (a.open_ends && (side == 0 ? pe == 0 : pe == a.P - 1)) {
        const int64_t r = (int64_t)((uint32_t)m % (uint32_t)a.R);
        return a.ext + (((r * a.S + s) * 2 + side) * a.H + h) * a.nvar;
    }
    const int64_t nbr = side == 0 ? (pe == 0 ? a.P - 1 : pe - 1) : (pe == a.P - 1 ? 0 : pe + 1);
    return a.ring + ring_index(a, m, s, nbr, 1 - side, h, 0);
}

// the same slot in the ring of derived quantities (nd per point)
__device__ __forceinline__ int64_t gring_index(const StageArgs& a, int64_t level, int stage, int64_t pe, int side,
                                               int h, int nd)
{
    const int64_t r = (int64_t)((uint32_t)level % (uint32_t)a.R);
    return ((((r * a.S + stage) * a.P + pe) * 2 + side) * a.H + h) * nd;
}

// ---------------------------------------------------------------------------
// Physics: derived quantities of one state vector.  Coefficients that only
// scale a derived quantity are folded in here (they commute with the
// temporal extrapolation, which is linear).
// ---------------------------------------------------------------------------
template <int PDE>
struct Phys;

// u_t + c u_x = a u_xx: the only derived quantity is u itself.
template <>
struct Phys<ADVDIFF> {
    static constexpr int NV = 1, ND = 1, SPLIT = 0;
    __device__ static void derive(const StageArgs&, const double* Q, double* g) { g[0] = Q[0]; }
};

// Reacting Navier-Stokes: g = [rho u, rho u^2 + p, u (rho E + p), rho u Y,
// u, ((2/3) mu u^2 + lam T + q_c rhoD Y) / lam, Y, T]; the diffusion rows
// 4..6 are differentiated with the scales s2v, which carry their constants
// (4/3) mu, lam and rhoD.  k0 = (4/3) mu, k1 = (2/3) mu, k2 = lam, k3 = rhoD.
template <>
struct Phys<RNS> {
    static constexpr int NV = 4, ND = 8, SPLIT = 7;  // SPLIT rows are differentiated, the last is T
    __device__ static void derive(const StageArgs& a, const double* Q, double* g)
    {
        const double gm1 = a.prm[0] - 1.0, qc = a.prm[6];
        const double rinv = at_rcpi(Q[0]);
        const double u = Q[1] * rinv;
        const double p = gm1 * (Q[2] - fma(fx_half(Q[1]), u, qc * Q[3]));
        const double T = p * rinv;
        const double Y = Q[3] * rinv;
        g[0] = Q[1];
        g[1] = fma(Q[1], u, p);
        g[2] = u * (Q[2] + p);
        g[3] = Q[3] * u;
        g[4] = u;                                      // times (4/3) mu in the scale
        g[5] = fma(a.kd1 * u, u, fma(a.kd3, Y, T));    // (k1 u^2 + k2 T + qc k3 Y) / k2; times k2 in the scale
        g[6] = Y;                                      // times k3 in the scale
        g[7] = T;
    }
    // the temperature exactly as derive() forms it (same operations, same rounding)
    __device__ static double temperature(const StageArgs& a, const double* Q)
    {
        const double gm1 = a.prm[0] - 1.0, qc = a.prm[6];
        const double rinv = at_rcpi(Q[0]);
        const double u = Q[1] * rinv;
        const double p = gm1 * (Q[2] - fma(fx_half(Q[1]), u, qc * Q[3]));
        return p * rinv;
    }
};

// Reacting Navier-Stokes in chain-rule form (Sec. 4): the product
// derivatives are expanded, so only the primitives g = [rho, u, p, rho E, Y,
// T] are differentiated (and extrapolated at buffer points).
template <>
struct Phys<RNS_CHAIN> {
    static constexpr int NV = 4, ND = 6, SPLIT = 6;
    __device__ static void derive(const StageArgs& a, const double* Q, double* g)
    {
        const double gm1 = a.prm[0] - 1.0, qc = a.prm[6];
        const double rinv = at_rcpi(Q[0]);
        const double u = Q[1] * rinv;
        const double p = gm1 * (Q[2] - fma(fx_half(Q[1]), u, qc * Q[3]));
        g[0] = Q[0];
        g[1] = u;
        g[2] = p;
        g[3] = Q[2];
        g[4] = Q[3] * rinv;
        g[5] = p * rinv;
    }
};

// Reactive Euler, WENO form: g = [C/2 (4), Q (4)], C = (rho u, rho u^2 + p,
// u (rho E + p), rho u Y); the split fluxes are C/2 +- (lam/2) Q.
template <>
struct Phys<EULER> {
    static constexpr int NV = 4, ND = 8, SPLIT = 0;
    __device__ static double pressure(const StageArgs& a, const double* Q, double u)
    {
        return (a.prm[0] - 1.0) * (Q[2] - fma(fx_half(Q[1]), u, a.prm[3] * Q[3]));
    }
    __device__ static void derive(const StageArgs& a, const double* Q, double* g)
    {
        const double u = Q[1] * at_rcpi(Q[0]);
        const double uh = fx_half(u);
        const double p = pressure(a, Q, u);
        g[0] = fx_half(Q[1]);
        g[1] = fx_half(fma(Q[1], u, p));
        g[2] = uh * (Q[2] + p);  // = (u (E + p)) / 2 exactly
        g[3] = Q[3] * uh;
        g[4] = Q[0];
        g[5] = Q[1];
        g[6] = Q[2];
        g[7] = Q[3];
    }
    // derive() and half the wave speed, (|u| + c) / 2, of one point at once
    // (1/rho, u and p formed once, by the same operations), and with ARR the
    // Arrhenius factor exp(-Ea rho / p) of the point's reaction source.
    // Halving is exact, so g[2] = (u/2)(E + p), g[3] = rho Y (u/2) and the half
    // speed |u/2| + sqrt(gamma p / (4 rho)) equal the halved products and the
    // halved speed up to the root's rounding.
    template <bool ARR>
    __device__ static void derive_weno(const StageArgs& a, const double* Q, double* g, double& sph, double& arr)
    {
        const double rinv = at_rcpi(Q[0]);
        const double u = Q[1] * rinv;
        const double uh = fx_half(u);
        const double p = pressure(a, Q, u);
        g[0] = fx_half(Q[1]);
        g[1] = fx_half(fma(Q[1], u, p));
        g[2] = uh * (Q[2] + p);
        g[3] = Q[3] * uh;
        g[4] = Q[0];
        g[5] = Q[1];
        g[6] = Q[2];
        g[7] = Q[3];
        sph = fabs(uh) + at_sqrt((0.25 * a.prm[0]) * p * rinv);
        if constexpr (ARR) arr = at_exp(-a.prm[2] * Q[0] * at_rcpi(p));
    }
};

// Scalar linear advection, WENO form: g = [c u / 2, u].
template <>
struct Phys<ADV_WENO> {
    static constexpr int NV = 1, ND = 2, SPLIT = 0;
    __device__ static void derive(const StageArgs& a, const double* Q, double* g)
    {
        g[0] = 0.5 * a.prm[0] * Q[0];
        g[1] = Q[0];
    }
    template <bool ARR>
    __device__ static void derive_weno(const StageArgs& a, const double* Q, double* g, double& sph, double&)
    {
        derive(a, Q, g);
        sph = 0.5 * fabs(a.prm[0]);  // half the wave speed
    }
};

// Inviscid Burgers, WENO form: g = [u^2 / 4, u] (C/2 with C = u^2/2); wave speed |u|.
template <>
struct Phys<BURGERS> {
    static constexpr int NV = 1, ND = 2, SPLIT = 0;
    __device__ static void derive(const StageArgs&, const double* Q, double* g)
    {
        g[0] = 0.5 * (0.5 * Q[0] * Q[0]);
        g[1] = Q[0];
    }
    template <bool ARR>
    __device__ static void derive_weno(const StageArgs& a, const double* Q, double* g, double& sph, double&)
    {
        derive(a, Q, g);
        sph = 0.5 * fabs(Q[0]);  // half the wave speed |u|
    }
};

// the SM this thread runs on
__device__ __forceinline__ int sm_id()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(r));
    return (int)r;
}

// The position of this CTA in a cooperative launch whose CTAs hand data to
// their neighbours (the persistent kernel: one PE per CTA; the multi-step
// fused kernel: a range of PEs per CTA).  A hand-off between SMs far apart
// (GB300's two dies) costs more than one between SMs that share a GPC, and
// the blocks of a launch are spread over the SMs in an order the program
// does not choose, so positions are dealt out by the SMs the CTAs landed on:
// every CTA records its SM, meets the others at a one-time bounded barrier
// (the launch is cooperative, so all CTAs are resident), and takes as its
// position its rank in (SM, block) order.  Consecutive positions then sit on
// the same or neighbouring SMs.  The arithmetic does not depend on where it
// runs, so results are the same bit for bit; a barrier that runs out keeps
// position = block (status bit 2 and the abort flag stop the run).  The
// caller resets *a.place_count before the launch.
__device__ __forceinline__ int64_t place_rank(const StageArgs& a)
{
    __shared__ int s_pe;
    if (threadIdx.x == 0) {
        int rank = (int)blockIdx.x;
        if (a.place && a.place_count) {
            const int me = sm_id();
            a.place[blockIdx.x] = me;
            cuda::atomic_ref<int, cuda::thread_scope_device> cnt(*a.place_count);
            cnt.fetch_add(1, cuda::memory_order_release);
            bool ok = cnt.load(cuda::memory_order_acquire) >= (int)gridDim.x;
            for (int64_t it = 0; !ok && it < a.wait_limit; ++it) {
                __nanosleep(128);
                ok = cnt.load(cuda::memory_order_acquire) >= (int)gridDim.x;
                if (!ok && (it & 63) == 0 && *(volatile int*)a.abort_flag) break;
            }
            if (ok) {
                rank = 0;
                for (int j = 0; j < (int)gridDim.x; ++j) {
                    const int sj = __ldcg(a.place + j);
                    rank += (sj < me) || (sj == me && j < (int)blockIdx.x);
                }
            } else {
                atomicOr(a.status, 2);
                atomicExch(a.abort_flag, 1);
            }
        }
        s_pe = rank;
    }
    __syncthreads();
    return s_pe;
}

// ---------------------------------------------------------------------------
// The LLF-split WENO5-JS flux at the edge left of column c of a row: the
// reconstruction of f+ = C + hl Q from columns c-3..c+1 plus that of
// f- = C - hl Q from columns c+2..c-2 (mirrored), hl half the edge's wave
// speed (Eq. Csplit).  One reconstruction, at the right edge of f[2] from
// f[0..4] (candidates of Eq. atRecon at k = 0, ideal weights {1/10, 3/5, 3/10},
// indicators of Eq. betaS, weights of Eq. omg with power 2), is taken from
// the first differences a_k = f[k] - f[k-1] (k = 1..4):
//  * with the second differences s_i (centred on f[i+1]) s_0 = a_2 - a_1,
//    s_1 = a_3 - a_2, s_2 = a_4 - a_3 and the first-difference terms
//    r_0 = f0 - 4 f1 + 3 f2 = s_0 + 2 a_2, r_1 = f1 - f3 = -(s_1 + 2 a_2),
//    r_2 = 3 f2 - 4 f3 + f4 = s_2 - 2 a_3 the indicators
//    beta_i = (13 s_i^2 + 3 r_i^2) / 12 give
//      D_0 = eps + beta_0 = s_0 ((4/3) s_0 + a_2) + a_2^2 + eps,
//      D_1 = eps + beta_1 = s_1 ((4/3) s_1 + a_2) + a_2^2 + eps,
//      D_2 = eps + beta_2 = s_2 ((4/3) s_2 - a_3) + a_3^2 + eps;
//  * the middle candidate p_1 = (-f1 + 5 f2 + 2 f3) / 6 = f2 + a_2/6 + a_3/3,
//    and the others differ from it by third differences,
//    p_0 - p_1 = (s_0 - s_1) / 3 and p_2 - p_1 = (s_1 - s_2) / 6, so
//    sum omega_i p_i = p_1 + omega_0 (p_0 - p_1) + omega_2 (p_2 - p_1);
//  * alpha_i ~ gamma_i / D_i^2 times the common factor D_0^2 D_1^2 D_2^2, and
//    numerator and denominator scaled by 10 (ideal weights 1 : 6 : 3); with
//    E_i = D_i^2 and A = 3 E_0, den = E_1 (A + E_2) + 2 A E_2,
//      p = p_1 + (2 E_1 E_2 / den (s_0 - s_1) + E_1 A / den (s_1 - s_2)) / 6.
// The split fluxes' first differences are those of C and Q combined,
// P(j) = hl dQ(j) + dC(j) and M(j) = hl dQ(j) - dC(j) with
// dC(j) = C[j] - C[j-1], so they come from the rows' own first differences,
// formed once per column and shared by every edge and both signs; dC(j),
// dQ(j) are callables returning them.  The two middle candidates add up to a
// centred value: p+ = f+(c-1) + P(c-1)/6 + P(c)/3 and p- = f-(c) + M(c+1)/6 +
// M(c)/3, and with f+(c-1) + f-(c) = C[c-1] + C[c] - hl dQ(c) and
// P(c) + M(c) = 2 hl dQ(c),
//   p+ + p- = C[c-1] + C[c] + (P(c-1) - P(c) + M(c+1) - M(c)) / 6
//           = C[c-1] + C[c] - (s1+ + s1-) / 6,
// s1+ = P(c) - P(c-1) and s1- = M(c) - M(c+1) being the two
// reconstructions' middle second differences.
//
// What bounds it: an FP64 warp instruction holds a sub-partition's FP64 unit
// for 64 cycles, and the whole flux took 66 of them.  Seven are left: the
// products hl dQ and the last sum.  Everything between is integer arithmetic
// on the aligned differences (fx_weno_sum, at_fixed.cuh).
// ---------------------------------------------------------------------------
template <class DC, class DQ>
__device__ __forceinline__ double weno_flux(const StageArgs& a, const double* C, DC dC, DQ dQ, int c, double hl)
{
    double d[5], q[5];
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        d[j] = dC(c - 2 + j);
        q[j] = hl * dQ(c - 2 + j);
    }
    return fma(1.0 / 6.0, fx_weno_sum(d, q, a.eps3), C[c - 1] + C[c]);
}

// ---------------------------------------------------------------------------
// -dF_v/dx plus the diffusion term of variable v of the reacting flow at
// column c of the derived rows G (row stride ld): the differences in integers
// (at_fixed.cuh), one FP64 instruction each to scale and add them.
// ---------------------------------------------------------------------------
template <int H, class ROWS>
__device__ __forceinline__ double rns_flux_terms(const StageArgs& a, const ROWS& G, int v, int c)
{
    double K = a.s1 * fx_d1<H>(G.row(v, c));
    if (v > 0) K = fma(a.s2v[v - 1], fx_d2<H>(G.row(3 + v, c)), K);
    return K;
}

// Rows of derived quantities in shared memory, row stride ld: as doubles, or
// (the reacting flow) split for the integer differences where they are written
struct DoubleRows {
    double* g;
    int ld;
    __device__ __forceinline__ void put(int d, int c, double x) const { g[d * ld + c] = x; }
    __device__ __forceinline__ FxDoubles row(int d, int c) const { return FxDoubles{g + d * ld + c}; }
};
struct SplitRows {
    int64_t* m;
    uint32_t* e;
    int ld;
    __device__ __forceinline__ void put(int d, int c, double x) const
    {
        const FxV v = fx_split(x);
        m[d * ld + c] = v.m;
        e[d * ld + c] = v.e;
    }
    __device__ __forceinline__ FxRow row(int d, int c) const { return FxRow{m + d * ld + c, e + d * ld + c}; }
};
// 8-byte words of `rows` split rows of ld columns
__host__ __device__ constexpr int split_words(int rows, int ld) { return rows * ld + (rows * ld + 1) / 2; }

// ---------------------------------------------------------------------------
// The RK update of the step-fused kernels, stage by stage: the next stage
// argument (u^{n+1} after the last stage) from K, the stage argument x and
// u^n, with the formulas and operation order of the per-stage kernels'
// update; the accumulator (RK2, RK4) is carried by the caller.
// ---------------------------------------------------------------------------
template <int RK>
struct RkS {
    static constexpr int S = RK == RK4 ? 4 : (RK == RK3TVD ? 3 : 2);
};

// the update of the per-stage kernels (rk_update), stage by stage: y from K,
// the stage argument x and u^n; the accumulator is carried by the caller
template <int RK>
__device__ __forceinline__ double fused_update(const StageArgs& a, int s, double K, double x, double un, double& acc)
{
    if (RK == RK4) {
        if (s == 0) {
            acc = K;
            return fma(a.hdt, K, un);
        }
        if (s < 3) {
            acc = fma(2.0, K, acc);
            return fma(s == 1 ? a.hdt : a.dt, K, un);
        }
        return fma(a.dt6, acc + K, un);
    }
    if (RK == RK3TVD) {
        if (s == 0) return fma(a.dt, K, x);
        if (s == 1) return fma(0.75, un, 0.25 * fma(a.dt, K, x));
        return fma(1.0 / 3.0, un, (2.0 / 3.0) * fma(a.dt, K, x));
    }
    if (s == 0) {
        acc = K;
        return fma(a.dt, K, un);
    }
    return fma(a.hdt, acc + K, un);
}

} // namespace atk
