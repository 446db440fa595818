// at_persist.cu -- persistent, neighbour-synchronised AT kernel (central PDEs).
//
// One CTA owns one virtual PE for a whole run of steps.  The PE's u^n, RK
// accumulator and stage argument live in shared memory between stages and
// steps; only the edge windows go through the history ring in global memory
// (L2), exactly as in the per-stage path, so the arithmetic and its order are
// identical and the results agree bit for bit.
//
// The CTAs synchronise only pairwise, through per-PE progress counters
// done[p] = n*S + s + 1 after stage s of step n.  Before stage s of step n,
// PE p needs its neighbour's stage-s argument at level n-k: it waits for
// done[nbr] >= (n-k)*S + s.  With a drawn delay k >= 1 that is usually
// already true, so the asynchrony the AT scheme tolerates (Sec. 2.1-2.3)
// becomes slack in the GPU's own synchronisation: no grid barrier, no launch
// per stage.  Before overwriting a ring slot a PE waits until both
// neighbours are past every stage that can still read the slot's old level
// (the ring keeps `slack` spare levels, so this rarely binds).  Results do
// not depend on timing: what is read is fixed by the Philox draws.
//
// Every wait is bounded (wait_limit polls with a short sleep).  A wait that
// runs out sets status bit 1 and a global abort flag; every other wait sees
// the flag and returns, and the kernel ends: the host reports AT_ETIMEOUT.
// The launch is cooperative, so all CTAs are resident at once.
#include <cuda/atomic>
#include <cuda_runtime.h>

#include "at_device.cuh"

namespace atk {

__device__ __forceinline__ int64_t load_acquire(int64_t* p)
{
    cuda::atomic_ref<int64_t, cuda::thread_scope_device> r(*p);
    return r.load(cuda::memory_order_acquire);
}

__device__ __forceinline__ void store_release(int64_t* p, int64_t v)
{
    cuda::atomic_ref<int64_t, cuda::thread_scope_device> r(*p);
    r.store(v, cuda::memory_order_release);
}

// bounded wait for *ctr >= target; false if it ran out or another wait did
__device__ bool wait_ge(const StageArgs& a, int64_t* ctr, int64_t target)
{
    if (load_acquire(ctr) >= target) return true;
    for (int64_t it = 0; it < a.wait_limit; ++it) {
        __nanosleep(128);
        if (load_acquire(ctr) >= target) return true;
        if ((it & 63) == 0 && *(volatile int*)a.abort_flag) return false;
    }
    atomicOr(a.status, 2);
    atomicExch(a.abort_flag, 1);
    return false;
}

// stencil, source and RK update of own point (v, jl) for stage s, in shared
// memory: the same arithmetic, in the same order, as the per-stage kernels
// (the Arrhenius factor exp(-Ea/T) arrives precomputed in E)
template <int PDE, int H, class ROWS>
__device__ __forceinline__ double point_update(const StageArgs& a, int s, int v, int jl, const ROWS& G,
                                               const double* E, double* X, double* U, double* ACC, int B,
                                               bool last)
{
    const int it = v * B + jl;
    const int c = jl + H;
    double K = 0.0;
    const double x = X[it];
    if constexpr (PDE == ADVDIFF) {
#pragma unroll
        for (int o = -H; o <= H; ++o) K = fma(a.cm[o + H], G.g[c + o], K);
    } else {
        K = rns_flux_terms<H>(a, G, v, c);
        if (v == 3) K = fma(-a.prm[4] * x, E[jl], K);
    }
    const double dt = a.dt;
    const double un = U[it];
    double y;
    if (a.rk == RK4) {
        if (s == 0) {
            ACC[it] = K;
            y = fma(a.hdt, K, un);
        } else if (s < 3) {
            ACC[it] = fma(2.0, K, ACC[it]);
            y = fma(s == 1 ? a.hdt : dt, K, un);
        } else {
            y = fma(a.dt6, ACC[it] + K, un);
        }
    } else if (a.rk == RK3TVD) {
        const double xs = fma(dt, K, x);
        if (s == 0) y = xs;
        else if (s == 1) y = fma(0.75, un, 0.25 * xs);
        else y = fma(1.0 / 3.0, un, (2.0 / 3.0) * xs);
    } else {
        if (s == 0) {
            ACC[it] = K;
            y = fma(dt, K, un);
        } else {
            y = fma(a.hdt, ACC[it] + K, un);
        }
    }
    X[it] = y;  // next stage argument (u^{n+1} after the last stage)
    if (last) U[it] = y;
    return y;
}

// named barriers (ids 1..5; 0 is __syncthreads): bar.sync waits until
// `count` threads have arrived, bar.arrive counts this warp without waiting
template <int ID>
__device__ __forceinline__ void bar_sync(int count)
{
    asm volatile("bar.sync %0, %1;" ::"n"(ID), "r"(count) : "memory");
}
template <int ID>
__device__ __forceinline__ void bar_arrive(int count)
{
    asm volatile("bar.arrive %0, %1;" ::"n"(ID), "r"(count) : "memory");
}
// the barrier of parity p among a pair (ids B0, B0 + 1), with immediate ids
template <int B0>
__device__ __forceinline__ void bar_sync_p(int p, int count)
{
    if (p) bar_sync<B0 + 1>(count);
    else bar_sync<B0>(count);
}
template <int B0>
__device__ __forceinline__ void bar_arrive_p(int p, int count)
{
    if (p) bar_arrive<B0 + 1>(count);
    else bar_arrive<B0>(count);
}

// GB300's FP64 unit spends the same time on a warp instruction whatever the
// number of active lanes, so the work is laid out in whole, uniform warps
// with fixed roles.  Stage t (= step n, stage s) of a PE:
//   (A) derive warps: own-point derived quantities into G[t % 2] (the reacting
//       flow's split for its integer differences); beside them, where there are
//       enough, warps for the Arrhenius factor exp(-Ea/T);
//   (C) all worker warps: stencil, source and RK update of every (point,
//       variable), one variable per warp, the edge points straight into the
//       ring; then the progress counter is published.
// After a stage, warp 0 derives the new stage argument at the PE's 2H edge
// points into a ring of derived quantities and publishes the stage.  The
// halo warp runs one stage ahead of the workers: while they do stage t it
// takes the delays of stage t + 1, reads the neighbours' derived quantities of
// the delayed levels and writes the weighted buffer values into the halo
// columns of G[(t + 1) % 2], a side with delay 0 last, after a bounded wait, so
// that its latency hides behind the workers' arithmetic (a drawn delay of 0
// then costs the neighbour's edge derivation, not a derivation under the
// contention of the receiving SM).  What bounds it: the loop update (2,500
// cycles) - edge derivation and release (2,800) - the neighbour's read and copy
// (about 1,500) where delays of 0 chain; second differences on warps of their
// own shortened the update but not the stage.  Named barriers, by
// the parity p of the stage:
//   1 + p  halo of stage t ready      (halo warp arrives, workers sync)
//   3 + p  G[p] no longer read        (workers arrive after stage t, the
//                                      halo warp syncs before filling G[p]
//                                      for stage t + 2)
//   5      workers' phase C done      (workers only, before publishing)
// A failed wait records the stage in s_abort_at before the halo warp
// arrives; the workers stop at that stage and the halo warp matches the one
// arrival it would otherwise have consumed, so every barrier completes.
//
// How many PEs fit the chip is registers and shared memory.  CTAS = 2 of 288
// threads an SM leaves the registers the code wants (86 at order 6); CTAS = 3 holds
// it to 72 for more PEs (none spilt, 3 to 6 % slower where both fit; 456 PEs of 64
// points 23.6 us per step, one launch per stage 30.0).  CTAS = 1 has sixteen worker
// warps instead of eight, for some PE sizes where every PE has an SM to itself
// (persist_wide).  DENSE has the reacting flow's rows as doubles, split where they
// are read, in 27 words a point instead of 34, for large PEs that no other holds
// (456 of 300 points 69.8 us; per stage 75.7).
template <int PDE, int H, int CTAS, bool DENSE>
__global__ void __launch_bounds__(CTAS == 1 ? 544 : 288, CTAS) persist_central(const StageArgs a, int64_t level0, int64_t nsteps)
{
    using P = Phys<PDE>;
    constexpr int NV = P::NV, ND = P::ND;
    constexpr bool SPLITROWS = P::SPLIT > 0 && !DENSE;
    const int B = a.B, W2 = B + 2 * H, S = a.S;
    const int64_t pe = place_rank(a);
    const int64_t nbr[2] = {pe == 0 ? a.P - 1 : pe - 1, pe == a.P - 1 ? 0 : pe + 1};
    extern __shared__ double sm[];
    double* U = sm;                // u^n                 [NV][B]
    double* ACC = U + NV * B;      // RK accumulator      [NV][B]
    double* X = ACC + NV * B;      // stage argument      [NV][B]
    double* E = X + NV * B;        // exp(-Ea/T) of own points [B]
    double* G2 = E + B;            // derived rows by stage parity: [2][W2] doubles, or the
                                   // reacting flow's split rows
    constexpr int NG = P::SPLIT > 0 ? P::SPLIT : ND;
    const int gwords = SPLITROWS ? split_words(NG, W2) : NG * W2;
    auto rows = [&](int p) {
        if constexpr (SPLITROWS) {
            int64_t* m = (int64_t*)(G2 + p * gwords);
            return SplitRows{m, (uint32_t*)(m + NG * W2), W2};
        } else {
            return DoubleRows{G2 + p * gwords, W2};
        }
    };
    __shared__ long long s_abort_at;  // first stage whose halo could not be formed
    const int nw = (a.mode == AT) ? a.q + 1 : 1;
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int hwarp = (int)(blockDim.x >> 5) - 1;  // the halo warp
    const int nwork = hwarp * 32;                    // threads of the worker warps
    const int nall = nwork + 32;
    // warps per role in phase A: enough for one point per lane
    int bw = (B + 31) / 32;
    if (bw > hwarp) bw = hwarp;
    if (bw < 1) bw = 1;
    // Roles of the worker warps in phase A.  Warp w runs on SM sub-partition
    // w % 4 and the halo warp on hwarp % 4 (sub-partition 0 with 8 workers).
    // The derive warps start at warp 1, so that two of them (a 64-point PE)
    // take sub-partitions 1 and 2, away from the halo warp.
    int derive_rank = -1, arr_rank = -1;
    if (warp < hwarp) {
        const int r = (warp + hwarp - 1) % hwarp;  // warp 1 -> rank 0, warp 2 -> rank 1, ...
        if (r < bw) derive_rank = r;
    }
    // The Arrhenius factor exp(-Ea/T) on warps of its own where there are enough
    // (the last ones; for two derive warps of eight, warps 3 and 7 on
    // sub-partition 3, which has no other work in phase A): derivation and factor
    // took 2,600 cycles one after the other, 1,300 and 2,000 side by side
    const bool arr_apart = PDE == RNS && hwarp > 2 * bw;
    if (arr_apart && warp < hwarp) {
        if (bw == 2 && hwarp == 8) arr_rank = warp == 3 ? 0 : (warp == 7 ? 1 : -1);
        else if (warp >= hwarp - bw) arr_rank = warp - (hwarp - bw);
    }

    for (int i = threadIdx.x; i < NV * B; i += blockDim.x) {
        const int v = i / B, j = i - v * B;
        const double x = a.u[v * a.N + pe * B + j];
        U[i] = x;
        X[i] = x;
    }
    if (threadIdx.x == 0) s_abort_at = 0x7fffffffffffffffLL;
    int bad = 0;
    // this PE's ring of derived quantities of its edge windows, from its ring
    // of stage arguments (steps before this launch may have run elsewhere);
    // the neighbours read it only after the release below
    for (int i = threadIdx.x; i < a.R * S * 2 * H; i += blockDim.x) {
        const int h = i % H, side = (i / H) % 2, st = (i / (2 * H)) % S, r = i / (2 * H * S);
        double Q[NV], g[ND];
#pragma unroll
        for (int v = 0; v < NV; ++v) Q[v] = a.ring[ring_index(a, r, st, pe, side, h, v)];
        P::derive(a, Q, g);
        const int64_t gi = gring_index(a, r, st, pe, side, h, ND);
#pragma unroll
        for (int d = 0; d < ND; ++d) a.gring[gi + d] = g[d];
    }
    __syncthreads();
    if (threadIdx.x == 0 && pe != a.withhold_pe) store_release(a.done + pe, level0 * S);
    const int64_t T = nsteps * S;

    if (warp == hwarp) {
        // ---- the halo warp: stage t's buffer values, one stage ahead ----
        // Lane items: (buffer point, derived quantity), NP a lane, read straight
        // from the neighbours' rings of derived quantities, all levels in flight
        // at once.  A side with delay k >= 1 reads what the neighbour published
        // a step ago, which the last progress counter seen usually covers: its
        // values are formed first, and only a side with delay 0 waits for the
        // stage just finished, with nothing but one copy left to do.
        constexpr int NI = 2 * H * NG, NP = (NI + 31) / 32;
        int64_t n = level0;
        int64_t seen = -0x7fffffffffffffffLL;  // lanes 0, 1: the neighbour's counter as last read
        int s = 0;
        int r0 = (int)((uint32_t)level0 % (uint32_t)a.R);  // ring slot of level n
        for (int64_t t = 0; t < T; ++t) {
            const int p = (int)(t & 1);
            const auto G = rows(p);
            const bool last = (s == S - 1);
            const int64_t Ln = last ? n + 1 : n;  // the stage argument stage t produces: (Ln, sn)
            const int sn = last ? 0 : s + 1;
            // the ring slot of (Ln, sn) this stage writes is no longer read by the neighbour
            const int64_t free_at = (Ln - a.slack - 1) * S + sn + 1;
            int k = 0;
            if (lane < 2 && !a.arrival) {
                k = keff_at(a, n, s, pe, lane);
                if (a.trace || n == level0 + nsteps - 1) log_delay(a, n, s, pe, lane, k);  // the log keeps the last step
            }
            if (t >= 2) bar_sync_p<3>(p, nall);  // the workers are done with G[p] (stage t - 2)
            bool ok = true;
            // with delays by arrival: the freshest stage-s argument of the
            // neighbour that has arrived, once one recent enough for the clamp is there
            if (lane < 2 && a.arrival) {
                const int kc = kcap_at(a, n);
                const int64_t need = (n - kc) * S + s;
                const int64_t target = need > free_at ? need : free_at;
                seen = load_acquire(a.done + nbr[lane]);
                if (seen < target) {
                    ok = wait_ge(a, a.done + nbr[lane], target);
                    seen = load_acquire(a.done + nbr[lane]);
                }
                const int64_t m = (seen - s) / S;
                k = m >= n ? 0 : (int)(n - m);
                if (k > kc) k = kc;  // only if the wait gave up
                log_delay(a, n, s, pe, lane, k);
            }
            const int k0 = __shfl_sync(0xffffffffu, k, 0), k1 = __shfl_sync(0xffffffffu, k, 1);
            // both passes wait for "published" and "slot free" on the neighbour's counter
            auto wait_for = [&](bool mine) {
                if (mine && !a.arrival) {
                    const int64_t need = (n - k) * S + s, target = need > free_at ? need : free_at;
                    if (seen < target) {
                        ok = wait_ge(a, a.done + nbr[lane], target);
                        seen = load_acquire(a.done + nbr[lane]);
                    }
                }
            };
            // A side with delay 0 has weights (1, +-0, ...), exact integer ratios:
            // its buffer values are the neighbour's level-n quantities themselves,
            // up to the sign of a zero, which no stencil sum sees.  which: 1 the
            // sides with delays, 2 those without, 3 both.
            auto fill = [&](int which) {
                double v[NP][AT_QMAX + 1];
#pragma unroll
                for (int i = 0; i < NP; ++i) {
                    const int c = lane + 32 * i, hp = c / NG, d = c - hp * NG;
                    const int side = hp < H ? 0 : 1, h = side == 0 ? hp : hp - H;
                    const int kk = side == 0 ? k0 : k1;
                    const bool in = c < NI && (which & (kk == 0 ? 2 : 1)) != 0;
                    const int levels = kk == 0 ? 1 : nw, used = kk == 0 ? 1 : a.wnz[kk];
#pragma unroll
                    for (int l = 0; l <= AT_QMAX; ++l) {
                        v[i][l] = 0.0;  // a level with weight 0 is not part of the scheme
                        if (in && l < levels && ((used >> l) & 1)) {
                            int r = r0 - kk - l;
                            if (r < 0) r += a.R;
                            v[i][l] = __ldcg(a.gring + ((((int64_t)(r * S + s) * a.P + nbr[side]) * 2 + 1 - side) * H + h) * ND + d);
                        }
                    }
                }
#pragma unroll
                for (int i = 0; i < NP; ++i) {
                    const int c = lane + 32 * i, hp = c / NG, d = c - hp * NG;
                    const int kk = hp < H ? k0 : k1;
                    if (c < NI && (which & (kk == 0 ? 2 : 1)) != 0) {
                        double acc = v[i][0];
                        if (kk != 0) {
                            acc = ((a.mode == AT) ? a.w[kk][0] : 1.0) * v[i][0];
#pragma unroll
                            for (int l = 1; l <= AT_QMAX; ++l)
                                if (l < nw) acc = fma(a.w[kk][l], v[i][l], acc);
                        }
                        G.put(d, hp < H ? hp : B + hp, acc);
                    }
                }
            };
            // drawn delays: the sides with delays before the wait for the others;
            // by arrival both counters have been seen, and both sides are one round
            // trip to L2 (advection-diffusion in 100 PEs of 48 points, AT6, RK3-TVD:
            // 5.1 us per step, 6.7 with two)
            bool failed = false;
            for (int which = a.arrival ? 3 : (k0 >= 1 || k1 >= 1 ? 1 : 2);; which = 2) {
                wait_for(lane < 2 && which == (k == 0 ? 2 : 1));
                failed = __any_sync(0xffffffffu, !ok);
                __syncwarp();  // orders the other lanes' reads after lanes 0 and 1 saw the counters
                if (failed) break;
                fill(which);
                if (which != 1 || (k0 != 0 && k1 != 0)) break;
            }
            if (failed && lane == 0) s_abort_at = t;
            __syncwarp();
            bar_arrive_p<1>(p, nall);  // stage t's halo is ready (or the run stops at t)
            if (failed) {
                // the workers arrive on 3 + parity after stage t - 1 and stop at t:
                // consume that arrival so the barrier completes
                if (t >= 1 && t + 1 < T) bar_sync_p<3>((int)((t - 1) & 1), nall);
                break;
            }
            if (++s == S) {
                s = 0;
                ++n;
                if (++r0 == a.R) r0 = 0;
            }
        }
    } else {
        // ---- the worker warps ----
        int64_t n = level0;
        int s = 0;
        int r0 = (int)((uint32_t)level0 % (uint32_t)a.R);  // ring slot of level n
        for (int64_t t = 0; t < T; ++t) {
            const int p = (int)(t & 1);
            const auto G = rows(p);
            const bool last = (s == S - 1);
            const int sn = last ? 0 : s + 1;
            const int rn = last ? (r0 + 1 == a.R ? 0 : r0 + 1) : r0;
            // this PE's windows of the stage argument stage t produces, in points
            const int64_t win = ((int64_t)(rn * S + sn) * a.P + pe) * 2 * H;
            // (A)
            if (derive_rank >= 0) {
                for (int it = derive_rank * 32 + lane; it < B; it += bw * 32) {
                    double g[ND];
                    double Q[NV];
#pragma unroll
                    for (int v = 0; v < NV; ++v) Q[v] = X[v * B + it];
                    P::derive(a, Q, g);
#pragma unroll
                    for (int d = 0; d < NG; ++d) G.put(d, H + it, g[d]);
                    if constexpr (PDE == RNS)
                        if (!arr_apart) E[it] = at_exp(-a.prm[5] * at_rcpi(g[7]));  // g[7] = T
                }
            }
            if constexpr (PDE == RNS) {
                if (arr_rank >= 0) {
                    for (int it = arr_rank * 32 + lane; it < B; it += bw * 32) {
                        double Q[NV];
#pragma unroll
                        for (int v = 0; v < NV; ++v) Q[v] = X[v * B + it];
                        E[it] = at_exp(-a.prm[5] * at_rcpi(P::temperature(a, Q)));
                    }
                }
            }
            bar_sync_p<1>(p, nall);  // own derived quantities and stage t's halo in G[p]
            if (t >= *(volatile long long*)&s_abort_at) break;
            // (C) item (v, jl).  With one warp per 32 points of a variable, warp w
            // takes variable w % NV: the two warps of the density equation (first
            // derivatives only, the lightest) then share sub-partition 0 with the
            // halo warp, which is on the critical path when a drawn delay is 0.
            const bool by_warp = (nwork == NV * B) && (B % 32 == 0);
            for (int it = threadIdx.x; it < NV * B; it += nwork) {
                const int v = by_warp ? warp % NV : it / B;
                const int jl = by_warp ? (warp / NV) * 32 + lane : it - v * B;
                const double y = point_update<PDE, H>(a, s, v, jl, G, E, X, U, ACC, B, last);
                if (nonfinite(y)) bad = 1;
                int side = -1, h = 0;
                if (jl < H) {
                    side = 0;
                    h = jl;
                } else if (jl >= B - H) {
                    side = 1;
                    h = jl - (B - H);
                }
                if (side >= 0) __stcg(a.ring + (win + side * H + h) * NV + v, y);
            }
            bar_sync<5>(nwork);
            // the derived quantities of the new stage argument at the edge
            // points, for the neighbours' halos; then publish: the barriers
            // order every worker's ring writes before lane 0's device-scope
            // release store, which is cumulative
            if (warp == 0) {
                if (lane < 2 * H) {
                    const int side = lane < H ? 0 : 1;
                    const int h = lane - side * H;
                    const int jl = side == 0 ? h : B - H + h;
                    double Q[NV], g[ND];
#pragma unroll
                    for (int v = 0; v < NV; ++v) Q[v] = X[v * B + jl];
                    P::derive(a, Q, g);
                    const int64_t gi = (win + lane) * ND;  // lane = side H + h
#pragma unroll
                    for (int d = 0; d < NG; ++d) __stcg(a.gring + gi + d, g[d]);
                }
                __syncwarp();
                if (lane == 0 && pe != a.withhold_pe) store_release(a.done + pe, n * S + s + 1);
            }
            if (t + 2 < T) bar_arrive_p<3>(p, nall);  // G[p] may be refilled for stage t + 2
            if (++s == S) {
                s = 0;
                ++n;
                r0 = rn;
            }
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < NV * B; i += blockDim.x) {
        const int v = i / B, j = i - v * B;
        a.Y[v * a.N + pe * B + j] = U[i];
    }
    if (bad) atomicOr(a.status, 1);
}

__global__ void counters_set(int64_t* done, int64_t P, int64_t value, int* abort_flag, int* place_count)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < P; i += (int64_t)gridDim.x * blockDim.x)
        done[i] = value;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *abort_flag = 0;
        *place_count = 0;
    }
}

} // namespace atk

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
namespace {
// the variants of the kernel, in the order in which they are preferred
constexpr int kVariants = 4;

template <int H>
void* persist_fn(int pde, int variant)
{
    if (pde == atk::ADVDIFF) return variant == 1 ? (void*)atk::persist_central<atk::ADVDIFF, H, 2, false> : nullptr;
    if (pde != atk::RNS) return nullptr;
    return variant == 0   ? (void*)atk::persist_central<atk::RNS, H, 1, false>
           : variant == 1 ? (void*)atk::persist_central<atk::RNS, H, 2, false>
           : variant == 2 ? (void*)atk::persist_central<atk::RNS, H, 3, false>
                          : (void*)atk::persist_central<atk::RNS, H, 3, true>;
}

void* persist_kernel(int pde, int order, int variant)
{
    return order == 2 ? persist_fn<1>(pde, variant) : order == 4 ? persist_fn<2>(pde, variant) : persist_fn<3>(pde, variant);
}

size_t persist_smem_bytes(int pde, int B, int H, int variant)
{
    const int W2 = B + 2 * H, nv = pde == atk::RNS ? 4 : 1, rows = pde == atk::RNS ? atk::Phys<atk::RNS>::SPLIT : 1;
    const size_t words = pde == atk::RNS && variant < 3 ? atk::split_words(rows, W2) : rows * W2;
    return sizeof(double) * ((size_t)3 * nv * B + 2 * words + (size_t)B);
}

// The PE sizes the path takes: u, argument and accumulator, eight (one) rows of
// derived quantities by stage parity, their halo levels and a factor for each
// point within 200 KB (the reacting flow at order 6: up to 872 points).
bool persist_takes(int pde, int B, int H)
{
    const int nv = pde == atk::RNS ? 4 : 1, nd = pde == atk::RNS ? 8 : 1;
    return sizeof(double) * ((size_t)3 * nv * B + (size_t)2 * nd * (B + 2 * H) + (size_t)2 * H * (AT_QMAX + 1) * nd +
                             (size_t)B) <= 200 * 1024;
}
// Whether the variant with sixteen worker warps is the faster one for PEs of B
// points, each with an SM to itself: from 65 points on eight warps have a second
// round of (point, variable) items, mostly empty up to 96, and from 224 on half as
// many rounds are left; between, waiting for twice the warps costs more than it saves
// (order 6, whose items are longer, gains up to 128).  us per step with eight and
// sixteen, order 6: 72 points 17.8 and 16.3, 96 18.2 and 16.3, 128 21.3 and 20.2 (by
// arrival 20.6 and 17.9, FP64 throughout 17.7), 150 21.9 and 22.4, 192 25.2 and 26.1,
// 256 37.8 and 27.9 (FP64 36.3), 600 59.5 and 50.8; order 4: 96 16.7 and 15.6, 128 17.9
// and 18.0, 150 19.4 and 21.0, 224 24.0 and 24.1, 256 32.8 and 26.0 (FP64 31.4)
bool persist_wide(int pde, int B, int H)
{
    return pde == atk::RNS && ((B > 64 && B <= (H == 3 ? 128 : 96)) || B >= 224);
}

// worker warps for the PE's points (at least two roles' worth for phase A)
// plus one halo warp
int persist_block(int pde, int B, int variant)
{
    const int nv = pde == atk::RNS ? 4 : 1, most = variant == 0 ? 512 : 256;
    const int bw = (B + 31) / 32;
    int want = ((nv * B + 31) / 32) * 32;
    if (want > most) want = most;
    if (want < 64 * bw) want = 64 * bw;
    if (want > most) want = most;
    return want + 32;
}
} // namespace

// how many PEs one cooperative launch of a variant can hold (0: not available, -1: the query failed)
int64_t atk_persist_capacity(int pde, int order, int B, int variant, int device)
{
    void* fn = variant < kVariants ? persist_kernel(pde, order, variant) : nullptr;
    const int H = order / 2;
    if (!fn || !persist_takes(pde, B, H) || (variant == 0 && !persist_wide(pde, B, H))) return 0;
    const size_t smem = persist_smem_bytes(pde, B, H, variant);
    if (smem > 227 * 1024 - 64) return 0;  // (64 for the kernel's own shared variables)
    int per_sm = 0, sms = 0, coop = 0;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, persist_block(pde, B, variant), smem);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, device);
    if (e != cudaSuccess) return atk::fit_error(e);
    return coop ? (int64_t)per_sm * sms : 0;
}

cudaError_t atk_launch_persist(const atk::StageArgs& a, int pde, int order, int variant, int64_t level0, int64_t nsteps,
                               cudaStream_t st)
{
    void* fn = persist_kernel(pde, order, variant);
    if (!fn) return cudaErrorInvalidValue;
    atk::counters_set<<<(unsigned)((a.P + 255) / 256 < 1024 ? (a.P + 255) / 256 : 1024), 256, 0, st>>>(
        a.done, a.P, (level0 - a.R) * a.S, a.abort_flag, a.place_count);  // raised to level0 S by each PE's prologue
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const size_t smem = persist_smem_bytes(pde, a.B, order / 2, variant);
    // the attribute is per kernel, not per context: set it for this launch
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    atk::StageArgs args = a;
    void* params[] = {(void*)&args, (void*)&level0, (void*)&nsteps};
    return cudaLaunchCooperativeKernel(fn, dim3((unsigned)a.P), dim3(persist_block(pde, a.B, variant)), params, smem, st);
}
