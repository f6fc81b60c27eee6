// plain.cu -- every trajectory of one problem to its escape, without an engine (Alg. 1 / Alg. 3;
// FP32: one trajectory per thread), the exact reduction of escape steps into sums and histograms,
// and random-number hooks.
//
// FP64 kernel: the arithmetic of every step is spelled out with round-to-nearest intrinsics
// (__dadd_rn, __dmul_rn, ...) so that no multiply-add is fused, in the operation order of the
// algorithm as written:
//   gamma_k = gamma0 + (nu dt) k
//   underdamped  phi_k = phi + v dt ;  v_k = (v + ((-alpha v - A sin phi) + gamma_k) dt) + sigma z
//   overdamped   phi_k = (phi + (gamma_k - A sin phi) dt) + sigma z
// and for the stochastic Heun integrator (gamma_{k-1}, gamma_k at the two ends of the step)
//   underdamped  a0 = ((-alpha v) - A sin phi) + gamma_{k-1};  p = phi + v dt;
//                q = (v + a0 dt) + sigma z;  a1 = ((-alpha q) - A sin p) + gamma_k
//                phi_k = phi + ((v + q) 0.5) dt;  v_k = (v + ((a0 + a1) 0.5) dt) + sigma z
//   overdamped   f0 = gamma_{k-1} - A sin phi;  p = (phi + f0 dt) + sigma z;  f1 = gamma_k - A sin p
//                phi_k = (phi + ((f0 + f1) 0.5) dt) + sigma z
// with an unwrapped phase.  FP32: the engine's single-precision step on a wrapped phase.
#include <cstdint>
#include <cstring>
#include <string>

#include "fpt_device.cuh"
#include "internal.h"

namespace fpt {

namespace {

__device__ __forceinline__ uint32_t lo32(uint64_t x) { return static_cast<uint32_t>(x); }
__device__ __forceinline__ uint32_t hi32(uint64_t x) { return static_cast<uint32_t>(x >> 32); }

// One FP64 instruction of a warp holds the FP64 unit of its scheduler for 64 cycles on this GPU
// (measured: 67-80 cycles per DFMA / DADD / DMUL, with 32 or with 8 active lanes, and each of an
// SM's four schedulers has its own unit).  Everything else in these kernels hides behind it, so
// what a run costs is the FP64 instructions of the busiest scheduler, and the time of one
// trajectory is the chain of its own steps.  A step splits into the noise increment (log, sqrt,
// sincos: ~40 FP64 instructions, independent of the state) and the state update (sin and 4-8
// more, a serial chain).  So the kernel keeps at most 32 trajectories per scheduler in flight,
// as up to four groups of 32 lanes per SM; in rounds of kF64Blocks Philox blocks the first warps
// advance one group each with increments from shared memory while the warps on the schedulers
// that hold no group fill the other half of the buffer for the next round (and the group warps
// join them when their steps are done).  Between rounds one warp drops the finished lanes, closes
// the gaps and starts the next trajectories of the CTA's id range, so no warp integrates for the
// sake of one slow lane and a CTA's last trajectories have a scheduler to themselves.
// Measured, against one trajectory per thread in 128-thread CTAs with noise and update in one
// chain: 4096 underdamped trajectories of <= 20 000 steps 56.4 -> 21.1 ms (2.8 -> 1.05 us per
// step; 17.5 ms with F64Pair), 65 536 overdamped ones of 19 000 steps on average 755 -> 239 ms (1.6 -> 5.2 Gstep/s; the
// longest of them decides: 228-262 ms over six sets).
constexpr int kF64Warps = 8;
constexpr int kF64Blocks = 16;                  // Philox blocks per round (fewer for a smaller step budget)
constexpr int kF64Steps = 4 * kF64Blocks;       // steps per round
constexpr int kF64Groups = 4;                   // groups of 32 lanes, one per scheduler

// Doubles ordered as integers, so that the escape test costs no FP64 instruction: the key grows
// with the value; a NaN phase compares as not reached, as IEEE phi >= th does, and th = +-0 takes
// the key of -0, which both zeros reach.
__device__ __forceinline__ long long order_key(double x) {
    const long long b = __double_as_longlong(x);
    return b ^ ((b >> 63) & 0x7FFFFFFFFFFFFFFFll);
}
__device__ __forceinline__ bool reached(double phi, long long th_key) {
    const long long k = order_key(phi);
    return k >= th_key && k <= 0x7FF0000000000000ll;
}

// Shared memory of a CTA of `cols` lanes: noise increments of two rounds, then the lanes.
struct F64Lanes {
    double *nz;                 // [2][kF64Steps][cols] sigma z
    double *phi, *v;
    unsigned long long *blk;    // Philox blocks consumed
    unsigned *idx;              // trajectory of the CTA's range
    int *col;                   // column of this round's increments; -1: none yet
    int *alive;
};
size_t f64_shared_bytes(int cols) {
    return static_cast<size_t>(cols) * (2 * kF64Steps * 8 + 3 * 8 + 3 * 4);
}

// The underdamped chain has room for a second warp: phi_{k+1} = phi_k + v_k dt does not wait for
// sin phi_k, so one warp's sine of the new phase runs beside another's new velocity (Euler: 24
// operations per step instead of 30), and Heun's two sines, of phi and of phi + v dt, run beside
// each other (40 instead of 64).  With at most two groups in the CTA, group g's second warp is warp
// groups + g, on a scheduler of its own; the two meet at a named barrier once per step and
// exchange values through shared memory by the parity of the step.  Lanes that are done go on to the
// round's end without effect.  4096 trajectories of <= 20 000 steps: 21.0 -> 17.5 ms.
struct F64Pair {
    double x[2][32], y[2][32];   // by parity: Euler sin phi and v; Heun's first warp q and a0 ...
    double p[2][32];             // ... and its second sin p
};
__device__ __forceinline__ void pair_barrier(int group) {
    asm volatile("bar.sync %0, 64;" ::"r"(group + 1) : "memory");
}

// One round of a group by its two warps (`second`: which of them); returns the step of the round at
// whose end the phase reached th, or kF64Steps.  phi and v are the lane's at the start and the end;
// Euler's first warp ends with phi, its second with v, Heun's with both.
template <int H, int R, int A1>
__device__ __forceinline__ int f64_pair_round(const PlainArgs &a, F64Pair &x, int group, bool second, const double *nz,
                                              int cols, double &phi, double &v, double kd, double g_const,
                                              long long th_key, int steps, int lim) {
    const int lane = threadIdx.x & 31;
    int hit = kF64Steps;
    const auto sine = [&](double p) { return A1 ? sin(p) : __dmul_rn(a.amp, sin(p)); };
    if constexpr (H == kEuler) {
        if (second) x.y[0][lane] = v;
        else x.x[0][lane] = sine(phi);
        pair_barrier(group);
    }
    for (int t = 0; t < steps; ++t) {
        double g = g_const, g0 = g_const;
        if constexpr (R) {
            if constexpr (H == kHeun) g0 = __dadd_rn(a.gamma0, __dmul_rn(a.nudt, kd));
            if (H == kHeun || second) {
                kd = __dadd_rn(kd, 1.0);
                g = __dadd_rn(a.gamma0, __dmul_rn(a.nudt, kd));
            }
        }
        const int now = t & 1, next = now ^ 1;
        if constexpr (H == kEuler) {
            if (second) {
                const double acc = __dadd_rn(__dsub_rn(__dmul_rn(-a.alpha, v), x.x[now][lane]), g);
                v = __dadd_rn(__dadd_rn(v, __dmul_rn(acc, a.dt)), nz[t * cols]);
                x.y[next][lane] = v;
            } else {
                phi = __dadd_rn(phi, __dmul_rn(x.y[now][lane], a.dt));
                if (hit == kF64Steps && t < lim && reached(phi, th_key)) hit = t;
                x.x[next][lane] = sine(phi);
            }
            pair_barrier(group);
        } else {
            const double z = nz[t * cols];
            double a0, q, sp;
            if (second) {
                sp = sine(__dadd_rn(phi, __dmul_rn(v, a.dt)));
                x.p[now][lane] = sp;
                pair_barrier(group);
                q = x.x[now][lane];
                a0 = x.y[now][lane];
            } else {
                a0 = __dadd_rn(__dsub_rn(__dmul_rn(-a.alpha, v), sine(phi)), g0);
                q = __dadd_rn(__dadd_rn(v, __dmul_rn(a0, a.dt)), z);
                x.x[now][lane] = q;
                x.y[now][lane] = a0;
                pair_barrier(group);
                sp = x.p[now][lane];
            }
            const double a1 = __dadd_rn(__dsub_rn(__dmul_rn(-a.alpha, q), sp), g);
            phi = __dadd_rn(phi, __dmul_rn(__dmul_rn(__dadd_rn(v, q), 0.5), a.dt));
            v = __dadd_rn(__dadd_rn(v, __dmul_rn(__dmul_rn(__dadd_rn(a0, a1), 0.5), a.dt)), z);
            if (hit == kF64Steps && t < lim && reached(phi, th_key)) hit = t;
        }
    }
    return hit;
}

// R: ramped bias (0: gamma0 throughout, the value gamma0 + 0 k has); A1: the sin term's amplitude
// is 1 (its product is exact and left out).
template <int M, int H, int R, int A1>
__global__ void __launch_bounds__(32 * kF64Warps, 1) plain_f64_kernel(PlainArgs a, int cols) {
    extern __shared__ double f64_shared[];
    __shared__ unsigned long long sh_next, sh_end;   // the CTA's ids not yet started
    __shared__ int sh_cnt, sh_ticket;
    __shared__ F64Pair pairs[M == kUnder ? 2 : 1];
    F64Lanes L;
    L.nz = f64_shared;
    L.phi = L.nz + 2 * kF64Steps * cols;
    L.v = L.phi + cols;
    L.blk = reinterpret_cast<unsigned long long *>(L.v + cols);
    L.idx = reinterpret_cast<unsigned *>(L.blk + cols);
    L.col = reinterpret_cast<int *>(L.idx + cols);
    L.alive = L.col + cols;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint64_t first = a.n * blockIdx.x / gridDim.x;   // n <= 2^32: no overflow
    if (threadIdx.x == 0) {
        sh_next = 0;
        sh_end = a.n * (blockIdx.x + 1ull) / gridDim.x - first;
        sh_cnt = 0;
    }
    const long long th_key = a.th == 0.0 ? -1ll : order_key(a.th);
    const int blocks = a.max_steps < static_cast<uint64_t>(kF64Steps) ? static_cast<int>(a.max_steps + 3) / 4 : kF64Blocks;
    const int steps = 4 * blocks;                    // of a round
    const double g_const = __dadd_rn(a.gamma0, __dmul_rn(a.nudt, 1.0));   // R = 0: nudt = 0
    __syncthreads();
    for (int buf = 0;; buf ^= 1) {
        if (warp == 0) {   // drop finished lanes, close the gaps, start new trajectories
            int kept = 0;
            const int cnt = sh_cnt;
            for (int p0 = 0; p0 < cnt; p0 += 32) {
                const int p = p0 + lane;
                const bool live = p < cnt && L.alive[p];
                double phi = 0.0, v = 0.0;
                unsigned long long blk = 0;
                unsigned idx = 0;
                if (live) {
                    phi = L.phi[p];
                    v = L.v[p];
                    blk = L.blk[p] + (L.col[p] >= 0 ? blocks : 0);
                    idx = L.idx[p];
                }
                const unsigned m = __ballot_sync(0xFFFFFFFFu, live);
                if (live) {   // positions only move down, below the entries still to be read
                    const int q = kept + __popc(m & ((1u << lane) - 1u));
                    L.phi[q] = phi;
                    L.v[q] = v;
                    L.blk[q] = blk;
                    L.idx[q] = idx;
                    L.col[q] = p;
                    L.alive[q] = 1;
                }
                kept += __popc(m);
                __syncwarp();
            }
            const unsigned long long next = sh_next, left = sh_end - next;
            const int add = left < static_cast<unsigned long long>(cols - kept) ? static_cast<int>(left) : cols - kept;
            for (int q = kept + lane; q < kept + add; q += 32) {
                L.phi[q] = a.phi0;
                L.v[q] = a.v0;
                L.blk[q] = 0;
                L.idx[q] = static_cast<unsigned>(next + static_cast<unsigned>(q - kept));
                L.col[q] = -1;
                L.alive[q] = 1;
            }
            __syncwarp();
            if (lane == 0) {
                sh_cnt = kept + add;
                sh_next = next + static_cast<unsigned>(add);
                sh_ticket = 0;
            }
        }
        __syncthreads();
        const int cnt = sh_cnt;
        if (cnt == 0) break;
        const int groups = (cnt + 31) >> 5;
        const bool paired = M == kUnder && groups <= 2;
        if (M == kUnder && paired && warp < 2 * groups) {
            // both warps of a group take part in every step; lanes without noise yet idle
            const int group = warp % groups, p = 32 * group + lane;
            const bool second = warp >= groups, runs = p < cnt && L.col[p] >= 0;
            double phi = runs ? L.phi[p] : 0.0, v = runs ? L.v[p] : 0.0;
            const uint64_t k0 = runs ? 4ull * L.blk[p] : 0ull;
            const uint64_t left = a.max_steps - k0;
            const int lim = !runs ? 0 : left < static_cast<uint64_t>(steps) ? static_cast<int>(left) : steps;
            const double *nz = L.nz + static_cast<size_t>(buf) * kF64Steps * cols + (runs ? L.col[p] : 0);
            if (__any_sync(0xFFFFFFFFu, runs)) {   // the same for both warps
                const int hit = f64_pair_round<H, R, A1>(a, pairs[group], group, second, nz, cols, phi, v,
                                                         static_cast<double>(k0), g_const, th_key, steps, lim);
                if (runs) {
                    const bool esc = hit < kF64Steps;
                    if (second) {
                        L.v[p] = v;
                    } else {
                        L.phi[p] = phi;
                        if (esc || k0 + static_cast<uint64_t>(lim) >= a.max_steps) {
                            a.steps[first + L.idx[p]] = esc ? static_cast<int64_t>(k0 + static_cast<uint64_t>(hit) + 1ull) : -1;
                            L.alive[p] = 0;
                        }
                    }
                }
            }
        }
        const int p = 32 * warp + lane;
        if (!paired && warp < groups && p < cnt && L.col[p] >= 0) {
            double phi = L.phi[p], v = L.v[p];
            const uint64_t k0 = 4ull * L.blk[p];
            const uint64_t left = a.max_steps - k0;
            const int lim = left < static_cast<uint64_t>(steps) ? static_cast<int>(left) : steps;
            const double *nz = L.nz + static_cast<size_t>(buf) * kF64Steps * cols + L.col[p];
            double kd = static_cast<double>(k0);   // exact below 2^53
            bool esc = false;
            int t = 0;
#pragma unroll 4
            for (; t < lim; ++t) {
                const double z = nz[t * cols];
                double g = g_const, g0 = g_const;
                if constexpr (R) {
                    if constexpr (H == kHeun) g0 = __dadd_rn(a.gamma0, __dmul_rn(a.nudt, kd));
                    kd = __dadd_rn(kd, 1.0);
                    g = __dadd_rn(a.gamma0, __dmul_rn(a.nudt, kd));
                }
                const double sn = A1 ? sin(phi) : __dmul_rn(a.amp, sin(phi));
                if constexpr (H == kHeun) {
                    if constexpr (M == kUnder) {
                        const double a0 = __dadd_rn(__dsub_rn(__dmul_rn(-a.alpha, v), sn), g0);
                        const double pp = __dadd_rn(phi, __dmul_rn(v, a.dt));
                        const double q = __dadd_rn(__dadd_rn(v, __dmul_rn(a0, a.dt)), z);
                        const double sp = A1 ? sin(pp) : __dmul_rn(a.amp, sin(pp));
                        const double a1 = __dadd_rn(__dsub_rn(__dmul_rn(-a.alpha, q), sp), g);
                        phi = __dadd_rn(phi, __dmul_rn(__dmul_rn(__dadd_rn(v, q), 0.5), a.dt));
                        v = __dadd_rn(__dadd_rn(v, __dmul_rn(__dmul_rn(__dadd_rn(a0, a1), 0.5), a.dt)), z);
                    } else {
                        const double f0 = __dsub_rn(g0, sn);
                        const double pp = __dadd_rn(__dadd_rn(phi, __dmul_rn(f0, a.dt)), z);
                        const double f1 = __dsub_rn(g, A1 ? sin(pp) : __dmul_rn(a.amp, sin(pp)));
                        phi = __dadd_rn(__dadd_rn(phi, __dmul_rn(__dmul_rn(__dadd_rn(f0, f1), 0.5), a.dt)), z);
                    }
                } else if constexpr (M == kUnder) {
                    const double phin = __dadd_rn(phi, __dmul_rn(v, a.dt));
                    const double acc = __dadd_rn(__dsub_rn(__dmul_rn(-a.alpha, v), sn), g);
                    v = __dadd_rn(__dadd_rn(v, __dmul_rn(acc, a.dt)), z);
                    phi = phin;
                } else {
                    phi = __dadd_rn(__dadd_rn(phi, __dmul_rn(__dsub_rn(g, sn), a.dt)), z);
                }
                if (reached(phi, th_key)) {
                    esc = true;
                    break;
                }
            }
            if (esc || k0 + static_cast<uint64_t>(lim) >= a.max_steps) {
                a.steps[first + L.idx[p]] = esc ? static_cast<int64_t>(k0 + static_cast<uint64_t>(t) + 1ull) : -1;
                L.alive[p] = 0;
            } else {
                L.phi[p] = phi;
                L.v[p] = v;
            }
        }
        // The next round's increments, one Philox block of one group at a time.  With fewer
        // groups than schedulers the warps beside a group's leave its scheduler's FP64 unit to it.
        const int busy = paired ? 2 * groups : groups;   // schedulers with an integrating warp
        if (warp < busy || groups == kF64Groups || busy >= kF64Groups || (warp & 3) >= busy) {
            double *out = L.nz + static_cast<size_t>(buf ^ 1) * kF64Steps * cols;
            __syncwarp();
            for (;;) {
                int item = 0;
                if (lane == 0) item = atomicAdd(&sh_ticket, 1);
                item = __shfl_sync(0xFFFFFFFFu, item, 0);
                if (item >= groups * blocks) break;
                const int q = 32 * (item % groups) + lane, b = item / groups;
                if (q < cnt) {
                    const uint64_t blk = L.blk[q] + (L.col[q] >= 0 ? blocks : 0) + b;
                    const uint64_t gid = a.traj0 + first + L.idx[q];
                    const uint4 x = philox4x32_10(make_uint4(lo32(blk), hi32(blk), lo32(gid), hi32(gid)),
                                                  a.key0, a.key1);
                    double z[4];
                    bm_pair_f64(x.x, x.y, z[0], z[1]);
                    bm_pair_f64(x.z, x.w, z[2], z[3]);
#pragma unroll
                    for (int s = 0; s < 4; ++s) out[(4 * b + s) * cols + q] = __dmul_rn(a.sigma, z[s]);
                }
            }
        }
        __syncthreads();
    }
}

// FP32: wrapped phase r in [-pi, pi) with winding w; escape when r >= eb = phi* - 2 pi w, the
// threshold in the current cell's coordinates; hb = min(eb, pi) is the one bound tested.  One
// trajectory per thread, its warp waiting for the slowest of 32 (App. A's loss): the plain
// counterpart of the engine's kernel, which shares only the step and the generator with it.  A block of kBlockSteps
// steps runs without a branch and tracks its largest phase; the rare block that reached hb is
// replayed with the test after every step, as in the engine, so wraps and the escape step are those
// of a step-by-step test.  2^18 overdamped trajectories of 52 000 steps on average, against a test
// per step and a full Philox per call: 73 -> 55 ms; 1024 of 19 000 steps: 5.8 -> 2.9 ms.
template <int M, int H, int R>
__global__ void __launch_bounds__(64, 12) plain_f32_kernel(PlainArgs a) {
    const uint64_t i = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= a.n) return;
    const uint64_t gid = a.traj0 + i;
    float r = a.r0_f, v = a.v0_f;
    int w = a.w0;
    float hb = fminf(a.eb0_f, kPiF);
    const uint64_t nblocks = (a.max_steps + 3) / 4;
    int64_t result = -1;
    uint64_t blk = 0;
    while (blk < nblocks) {
        // re-base the single-precision bias every 2^20 blocks of the trajectory:
        // gamma_k = (gb + nudt Jf) + nudt (s + 1), Jf = 4 x blocks since the base
        const uint64_t seg_end = blk + (1ull << 20) < nblocks ? blk + (1ull << 20) : nblocks;
        const float gb = static_cast<float>(a.gamma0 + a.nudt * static_cast<double>(4 * blk));
        float Jf = 0.0f;
        PhiloxLane P;   // the high counter word changes only between segments
        philox_lane_init(P, a.key0, a.key1, hi32(blk), lo32(gid), hi32(gid));
        float gs, gsl;
        bias_line(fmaf(a.nudt_f, Jf, gb), a.nudt_f, a.dt_f, gs, gsl);
        for (; blk < seg_end; blk += kBlockPhilox) {
            float rr[2 * kBlockPhilox], tg[kBlockSteps];
            uint4 x[kBlockPhilox];
#pragma unroll
            for (int h = 0; h < kBlockPhilox; ++h) x[h] = philox_lane_block(P, lo32(blk), static_cast<uint32_t>(h));
#pragma unroll
            for (int h = 0; h < kBlockPhilox; ++h) {
                bm_pair_f32(x[h].x, x[h].y, a.bmc_f, rr[2 * h], tg[4 * h], tg[4 * h + 1]);
                bm_pair_f32(x[h].z, x[h].w, a.bmc_f, rr[2 * h + 1], tg[4 * h + 2], tg[4 * h + 3]);
            }
            if constexpr (R) bias_line(fmaf(a.nudt_f, Jf, gb), a.nudt_f, a.dt_f, gs, gsl);
            const float r0 = r, v0 = v;
            float mx = -INFINITY;
#pragma unroll
            for (int s = 0; s < kBlockSteps; ++s) {
                step_f32<M, H>(r, v, rr[s >> 1], tg[s], bias_b0<H, R>(gs, gsl, s),
                               bias_b1<H, R>(gs, gsl, s), a.dt_f, a.A_f, a.amp_f);
                mx = fmaxf(mx, r);
            }
            if (mx >= hb) {
                r = r0;
                v = v0;
#pragma unroll
                for (int s = 0; s < kBlockSteps; ++s) {
                    step_f32<M, H>(r, v, rr[s >> 1], tg[s], bias_b0<H, R>(gs, gsl, s),
                                   bias_b1<H, R>(gs, gsl, s), a.dt_f, a.A_f, a.amp_f);
                    if (r >= hb) {
                        // threshold in the current cell: eb = phi* - 2 pi w (same rounding as the engine)
                        const float eb = fmaf(-kTwoPiF, static_cast<float>(w - a.w0), a.eb0_f);
                        if (r >= eb) {
                            const uint64_t k = 4 * blk + s + 1;
                            if (k <= a.max_steps) result = static_cast<int64_t>(k);
                            goto done;
                        }
                        r -= kTwoPiF;
                        w += 1;
                        hb = fminf(fmaf(-kTwoPiF, static_cast<float>(w - a.w0), a.eb0_f), kPiF);
                    }
                }
            }
            if (r < -kPiF) {   // lower wrap at the block end, as in the engine
                r += kTwoPiF;
                w -= 1;
                hb = fminf(fmaf(-kTwoPiF, static_cast<float>(w - a.w0), a.eb0_f), kPiF);
            }
            Jf += static_cast<float>(kBlockSteps);
        }
    }
done:
    a.steps[i] = result;
}

__device__ __forceinline__ void add128(uint64_t &lo, uint64_t &hi, uint64_t alo, uint64_t ahi) {
    lo += alo;
    hi += ahi + (lo < alo ? 1 : 0);
}

__device__ __forceinline__ void atomic_add128(uint64_t *lo_p, uint64_t *hi_p, uint64_t alo,
                                              uint64_t ahi) {
    unsigned long long *lp = reinterpret_cast<unsigned long long *>(lo_p);
    const unsigned long long old = atomicAdd(lp, static_cast<unsigned long long>(alo));
    const uint64_t carry = (old + alo < old) ? 1 : 0;
    if (ahi + carry) atomicAdd(reinterpret_cast<unsigned long long *>(hi_p),
                               static_cast<unsigned long long>(ahi + carry));
}

// The reduction reads 8 bytes per escape step and should run at the memory's rate; what holds it
// back is arithmetic.  The bin of a step takes five FP64 operations, 64 cycles of a scheduler each,
// which alone held the kernel to an eighth of that rate; so bins come from integers (BinMap, formed
// on the host) and only a step that the map leaves open takes the FP64 formula.  Steps below 2^32
// take two wide multiplies for the bin and one for the square, sums of 64 and 96 bits, ~25
// instructions in all.  Each of a few copies of the histogram in shared memory serves some of the
// CTA's warps (low bins are hit by many lanes at once), and a CTA adds its sums once.
// 2^24 exponential escape times, 100 bins: 300 -> 37 us (3.6 TB/s).
constexpr int kSharedBins = 8192;
constexpr int kReduceBlock = 512;
constexpr int kReduceUnroll = 4;      // 16-byte loads in flight per thread

// Bin of x(k): -1 below the range, nbins above it.
__device__ __forceinline__ int exact_bin(const ReduceArgs &a, uint64_t k) {
    const double x = a.output == FPT_OUT_TIME
                         ? __dmul_rn(a.out_b, static_cast<double>(k))
                         : __dadd_rn(a.out_a, __dmul_rn(a.out_b, static_cast<double>(k)));
    if (x < a.lo) return -1;
    if (x >= a.hi) return a.nbins;
    const int b = static_cast<int>(floor(__dmul_rn(__dsub_rn(x, a.lo), a.inv_w)));
    return b >= a.nbins ? a.nbins - 1 : b;
}

struct ReduceThread {
    uint64_t s1lo = 0, s1hi = 0, s2lo = 0, s2hi = 0;
    unsigned esc = 0, under = 0, over = 0;
    // steps of 2^32 and more, apart from the others' short sums
    uint64_t b1lo = 0, b1hi = 0, b2lo = 0, b2hi = 0;
    __device__ __forceinline__ void big(uint64_t k) {
        esc += 1;
        add128(b1lo, b1hi, k, 0);
        add128(b2lo, b2hi, k * k, __umul64hi(k, k));
    }
};

enum : int { kNoHist = 0, kSharedHist = 1, kGlobalHist = 2 };

// Hist: where the counts go.
template <int Hist>
__device__ __forceinline__ void reduce_one(const ReduceArgs &a, unsigned *bins, int64_t k, ReduceThread &t) {
    int b = -2;
    if (hi32(static_cast<uint64_t>(k)) == 0) {   // a thread has fewer than 2^32 entries: s1 < 2^64
        const uint32_t v = lo32(static_cast<uint64_t>(k));
        t.esc += 1;
        t.s1lo += v;
        const uint64_t q = static_cast<uint64_t>(v) * v;
        uint32_t top = static_cast<uint32_t>(t.s2hi);   // s2 < 2^96
        asm("{\n\t.reg .u32 l, h, ql, qh;\n\t"
            "mov.b64 {l, h}, %0;\n\tmov.b64 {ql, qh}, %2;\n\t"
            "add.cc.u32 l, l, ql;\n\taddc.cc.u32 h, h, qh;\n\taddc.u32 %1, %1, 0;\n\t"
            "mov.b64 %0, {l, h};\n\t}"
            : "+l"(t.s2lo), "+r"(top)
            : "l"(q));
        t.s2hi = top;
        if constexpr (Hist == kNoHist) return;
        b = mapped_bin(a.map, v);
        if constexpr (Hist == kSharedHist) {
            if (b >= 0) {
                atomicAdd(&bins[b], 1u);
                return;
            }
        }
    } else {
        if (k < 0) return;
        t.big(static_cast<uint64_t>(k));
        if constexpr (Hist == kNoHist) return;
    }
    const uint64_t uk = static_cast<uint64_t>(k);
    if (b == -2) b = uk >= a.map.k_over ? a.nbins : (uk < a.map.k_under ? -1 : exact_bin(a, uk));
    if (b < 0) t.under += 1;
    else if (b >= a.nbins) t.over += 1;
    else if constexpr (Hist == kSharedHist) atomicAdd(&bins[b], 1u);
    else atomicAdd(&a.hist[b], 1ull);
}

template <int Hist>
__global__ void __launch_bounds__(kReduceBlock) reduce_kernel(ReduceArgs a, int copies) {
    extern __shared__ unsigned int sh_hist[];
    __shared__ uint64_t sh_s[kReduceBlock / 32][4];
    __shared__ unsigned sh_c[kReduceBlock / 32][3];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int b = threadIdx.x; b < copies * a.nbins; b += blockDim.x) sh_hist[b] = 0;
    __syncthreads();
    unsigned *bins = copies ? sh_hist + (warp % copies) * a.nbins : nullptr;
    ReduceThread t;
    // 16-byte loads from the first aligned entry on; the odd entries at the ends one by one
    const uint64_t head = (reinterpret_cast<uintptr_t>(a.steps) & 8) && a.n ? 1 : 0;
    const uint64_t pairs = (a.n - head) / 2;
    const longlong2 *p = reinterpret_cast<const longlong2 *>(a.steps + head);
    const uint64_t span = static_cast<uint64_t>(kReduceBlock) * kReduceUnroll;
    for (uint64_t base = blockIdx.x * span; base < pairs; base += gridDim.x * span) {
        longlong2 k[kReduceUnroll];
#pragma unroll
        for (int u = 0; u < kReduceUnroll; ++u) {
            const uint64_t i = base + static_cast<uint64_t>(u) * kReduceBlock + threadIdx.x;
            k[u] = i < pairs ? __ldcs(p + i) : make_longlong2(-1, -1);
        }
#pragma unroll
        for (int u = 0; u < kReduceUnroll; ++u) {
            reduce_one<Hist>(a, bins, k[u].x, t);
            reduce_one<Hist>(a, bins, k[u].y, t);
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (head) reduce_one<Hist>(a, bins, a.steps[0], t);
        if (head + 2 * pairs < a.n) reduce_one<Hist>(a, bins, a.steps[a.n - 1], t);
    }
    add128(t.s1lo, t.s1hi, t.b1lo, t.b1hi);
    add128(t.s2lo, t.s2hi, t.b2lo, t.b2hi);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        t.esc += __shfl_down_sync(0xFFFFFFFFu, t.esc, off);
        t.under += __shfl_down_sync(0xFFFFFFFFu, t.under, off);
        t.over += __shfl_down_sync(0xFFFFFFFFu, t.over, off);
        const uint64_t a1 = __shfl_down_sync(0xFFFFFFFFu, t.s1lo, off);
        const uint64_t b1 = __shfl_down_sync(0xFFFFFFFFu, t.s1hi, off);
        const uint64_t a2 = __shfl_down_sync(0xFFFFFFFFu, t.s2lo, off);
        const uint64_t b2 = __shfl_down_sync(0xFFFFFFFFu, t.s2hi, off);
        add128(t.s1lo, t.s1hi, a1, b1);
        add128(t.s2lo, t.s2hi, a2, b2);
    }
    if (lane == 0) {
        sh_s[warp][0] = t.s1lo;
        sh_s[warp][1] = t.s1hi;
        sh_s[warp][2] = t.s2lo;
        sh_s[warp][3] = t.s2hi;
        sh_c[warp][0] = t.esc;
        sh_c[warp][1] = t.under;
        sh_c[warp][2] = t.over;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        uint64_t s1lo = 0, s1hi = 0, s2lo = 0, s2hi = 0, c[3] = {0, 0, 0};
        for (int w = 0; w < kReduceBlock / 32; ++w) {
            add128(s1lo, s1hi, sh_s[w][0], sh_s[w][1]);
            add128(s2lo, s2hi, sh_s[w][2], sh_s[w][3]);
            for (int j = 0; j < 3; ++j) c[j] += sh_c[w][j];
        }
        if (blockIdx.x == 0) atomicAdd(reinterpret_cast<unsigned long long *>(&a.sums->n_done), a.n);
        if (c[0]) {
            atomicAdd(reinterpret_cast<unsigned long long *>(&a.sums->n_escaped), c[0]);
            atomic_add128(&a.sums->s1_lo, &a.sums->s1_hi, s1lo, s1hi);
            atomic_add128(&a.sums->s2_lo, &a.sums->s2_hi, s2lo, s2hi);
        }
        if (c[1]) atomicAdd(reinterpret_cast<unsigned long long *>(&a.sums->under), c[1]);
        if (c[2]) atomicAdd(reinterpret_cast<unsigned long long *>(&a.sums->over), c[2]);
    }
    if (copies)
        for (int b = threadIdx.x; b < a.nbins; b += blockDim.x) {
            unsigned long long sum = 0;
            for (int q = 0; q < copies; ++q) sum += sh_hist[q * a.nbins + b];
            if (sum) atomicAdd(&a.hist[b], sum);
        }
}

__global__ void philox_fill_kernel(uint32_t k0, uint32_t k1, uint64_t traj, uint64_t block0,
                                   uint64_t nblocks, uint32_t *out) {
    const uint64_t j = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (j >= nblocks) return;
    const uint64_t b = block0 + j;
    const uint4 x = philox4x32_10(make_uint4(lo32(b), hi32(b), lo32(traj), hi32(traj)), k0, k1);
    out[4 * j + 0] = x.x;
    out[4 * j + 1] = x.y;
    out[4 * j + 2] = x.z;
    out[4 * j + 3] = x.w;
}

__global__ void normals_fill_kernel(int precision, uint32_t k0, uint32_t k1, uint64_t traj,
                                    uint64_t n0, uint64_t n, double *out) {
    const uint64_t j = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const uint64_t idx = n0 + j, b = idx / 4;
    const int slot = static_cast<int>(idx % 4);
    const uint4 x = philox4x32_10(make_uint4(lo32(b), hi32(b), lo32(traj), hi32(traj)), k0, k1);
    const uint32_t w0 = slot < 2 ? x.x : x.z, w1 = slot < 2 ? x.y : x.w;
    if (precision == FPT_FP64) {
        double z0, z1;
        bm_pair_f64(w0, w1, z0, z1);
        out[j] = (slot & 1) ? z1 : z0;
    } else {
        float rr, cs, sn;
        bm_pair_f32(w0, w1, -1.3862943611198906f /* -2 ln 2: unit variance */, rr, cs, sn);
        out[j] = static_cast<double>(__fmul_rn(rr, (slot & 1) ? sn : cs));
    }
}

unsigned grid_for(uint64_t n, unsigned block) {
    return static_cast<unsigned>((n + block - 1) / block);
}

}  // namespace

// One CTA per SM, at most one per 32 trajectories; each takes a contiguous range of ids (no
// queue in global memory, so launches on several streams share nothing) and as many lanes as its
// range fills, up to kF64Groups x 32.
cudaError_t launch_plain_f64(const PlainArgs &a, cudaStream_t s) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const uint64_t warps = (a.n + 31) / 32;
    const unsigned grid = static_cast<unsigned>(warps < static_cast<uint64_t>(sms) ? warps : sms);
    const uint64_t groups = ((a.n + grid - 1) / grid + 31) / 32;
    const int cols = 32 * static_cast<int>(groups < kF64Groups ? groups : kF64Groups);
    void (*kernel)(PlainArgs, int) = nullptr;
    const int ramp = a.nudt != 0.0, one = a.amp == 1.0;
    switch (a.model + 2 * a.integrator + 4 * ramp + 8 * one) {
#define FPT_F64_CASE(M_, H_, R_, A_) \
    case M_ + 2 * H_ + 4 * R_ + 8 * A_: kernel = plain_f64_kernel<M_, H_, R_, A_>; break;
#define FPT_F64_MODELS(R_, A_)          \
    FPT_F64_CASE(kUnder, kEuler, R_, A_) \
    FPT_F64_CASE(kOver, kEuler, R_, A_)  \
    FPT_F64_CASE(kUnder, kHeun, R_, A_)  \
    FPT_F64_CASE(kOver, kHeun, R_, A_)
    FPT_F64_MODELS(0, 0)
    FPT_F64_MODELS(1, 0)
    FPT_F64_MODELS(0, 1)
    FPT_F64_MODELS(1, 1)
#undef FPT_F64_MODELS
#undef FPT_F64_CASE
    }
    const size_t shared = f64_shared_bytes(cols);
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(f64_shared_bytes(32 * kF64Groups)));
    if (e != cudaSuccess) return e;
    kernel<<<grid, 32 * kF64Warps, shared, s>>>(a, cols);
    return cudaGetLastError();
}

cudaError_t launch_plain_f32(const PlainArgs &a, cudaStream_t s) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    // CTAs of one warp while every warp can have a scheduler to itself (four per SM), so that few
    // trajectories spread over all of them; then of two, so that a CTA waits for 64 trajectories
    // rather than 256 before its place is free (2^18 trajectories: 56 -> 55 ms).
    const unsigned block = a.n <= 32ull * 4 * static_cast<unsigned>(sms) ? 32 : 64;
    const unsigned grid = grid_for(a.n, block);
    switch (a.kind) {
#define FPT_KIND_CASE(M_, H_, R_) \
    case kind_of(M_, H_, R_): plain_f32_kernel<M_, H_, R_><<<grid, block, 0, s>>>(a); break;
    FPT_KIND_CASE(kUnder, kEuler, kConstBias)
    FPT_KIND_CASE(kOver, kEuler, kConstBias)
    FPT_KIND_CASE(kUnder, kHeun, kConstBias)
    FPT_KIND_CASE(kOver, kHeun, kConstBias)
    FPT_KIND_CASE(kUnder, kEuler, kRamp)
    FPT_KIND_CASE(kOver, kEuler, kRamp)
    FPT_KIND_CASE(kUnder, kHeun, kRamp)
#undef FPT_KIND_CASE
    default: plain_f32_kernel<kOver, kHeun, kRamp><<<grid, block, 0, s>>>(a); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_reduce(const ReduceArgs &a, cudaStream_t s) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const uint64_t span = 2ull * kReduceBlock * kReduceUnroll;
    uint64_t g = (a.n + span - 1) / span;
    const uint64_t gmax = static_cast<uint64_t>(sms > 0 ? sms : 1) * 4;
    if (g > gmax) g = gmax;
    if (g == 0) g = 1;
    // copies of the histogram in shared memory: up to eight in 32 KB, none beyond kSharedBins
    int copies = 0;
    if (a.hist && a.nbins <= kSharedBins) copies = kSharedBins / a.nbins < 8 ? kSharedBins / a.nbins : 8;
    const size_t shmem = static_cast<size_t>(copies) * a.nbins * sizeof(unsigned int);
    const unsigned grid = static_cast<unsigned>(g);
    if (!a.hist) reduce_kernel<kNoHist><<<grid, kReduceBlock, 0, s>>>(a, 0);
    else if (copies) reduce_kernel<kSharedHist><<<grid, kReduceBlock, shmem, s>>>(a, copies);
    else reduce_kernel<kGlobalHist><<<grid, kReduceBlock, 0, s>>>(a, 0);
    return cudaGetLastError();
}

cudaError_t launch_philox_fill(uint64_t seed, uint64_t traj, uint64_t block0, uint64_t nblocks,
                               uint32_t *out, cudaStream_t s) {
    philox_fill_kernel<<<grid_for(nblocks, 256), 256, 0, s>>>(
        static_cast<uint32_t>(seed), static_cast<uint32_t>(seed >> 32), traj, block0, nblocks, out);
    return cudaGetLastError();
}

cudaError_t launch_normals_fill(int precision, uint64_t seed, uint64_t traj, uint64_t n0,
                                uint64_t n, double *out, cudaStream_t s) {
    normals_fill_kernel<<<grid_for(n, 256), 256, 0, s>>>(
        precision, static_cast<uint32_t>(seed), static_cast<uint32_t>(seed >> 32), traj, n0, n, out);
    return cudaGetLastError();
}

}  // namespace fpt

using namespace fpt;

static fpt_status cuda_fail(cudaError_t e, const char *what) {
    set_error(std::string(what) + ": " + cudaGetErrorString(e));
    return FPT_ECUDA;
}

extern "C" fpt_status fpt_plain_launch(const fpt_params *params, uint64_t seed, uint64_t traj0,
                                       uint64_t n, int64_t *d_steps, void *stream) {
    Decoded d;
    std::string err;
    if (!decode(params, &d, &err)) {
        set_error(err);
        return FPT_EINVAL;
    }
    if (params->precision != FPT_FP32 && params->precision != FPT_FP64) {
        set_error("unknown precision");
        return FPT_EINVAL;
    }
    if (n > (1ull << 32)) {
        set_error("n must be <= 2^32");
        return FPT_EINVAL;
    }
    if (n == 0) return FPT_OK;
    if (!d_steps) {
        set_error("d_steps is NULL");
        return FPT_EINVAL;
    }
    PlainArgs a;
    std::memset(&a, 0, sizeof(a));
    a.model = d.model;
    a.integrator = d.integrator;
    a.kind = d.kind;
    a.key0 = static_cast<uint32_t>(seed);
    a.key1 = static_cast<uint32_t>(seed >> 32);
    a.traj0 = traj0;
    a.n = n;
    a.steps = d_steps;
    a.max_steps = d.max_steps;
    a.alpha = d.alpha;
    a.amp = d.amp;
    a.dt = d.dt;
    a.sigma = d.sigma;
    a.gamma0 = d.gamma0;
    a.nudt = d.nudt;
    a.phi0 = d.phi0;
    a.v0 = d.v0;
    a.th = d.th;
    a.dt_f = d.dt_f;
    a.A_f = d.A_f;
    a.amp_f = d.amp_f;
    a.bmc_f = d.bmc_f;
    a.nudt_f = d.nudt_f;
    a.v0_f = d.v0_f;
    a.r0_f = d.r0_f;
    a.eb0_f = d.eb0_f;
    a.w0 = d.w0;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const cudaError_t e =
        params->precision == FPT_FP64 ? launch_plain_f64(a, s) : launch_plain_f32(a, s);
    if (e != cudaSuccess) return cuda_fail(e, "plain kernel launch");
    return FPT_OK;
}

extern "C" fpt_status fpt_reduce_steps(const fpt_params *params, const int64_t *d_steps,
                                       uint64_t n, fpt_sums *d_sums, uint64_t *d_hist,
                                       void *stream) {
    Decoded d;
    std::string err;
    if (!decode(params, &d, &err)) {
        set_error(err);
        return FPT_EINVAL;
    }
    if (!d_sums || (n && !d_steps)) {
        set_error("NULL device pointer");
        return FPT_EINVAL;
    }
    if (n == 0) return FPT_OK;
    ReduceArgs a;
    a.steps = d_steps;
    a.n = n;
    a.output = d.output;
    a.out_a = d.out_a;
    a.out_b = d.out_b;
    a.lo = d.hist_lo;
    a.hi = d.hist_hi;
    a.inv_w = d.hist_inv_w;
    a.nbins = d.hist_bins;
    a.sums = d_sums;
    a.hist = reinterpret_cast<unsigned long long *>(d_hist);
    a.map = bin_map(d);
    const cudaError_t e = launch_reduce(a, static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return cuda_fail(e, "reduce kernel launch");
    return FPT_OK;
}

extern "C" fpt_status fpt_philox_fill(uint64_t seed, uint64_t traj, uint64_t block0,
                                      uint64_t nblocks, uint32_t *d_out, void *stream) {
    if (nblocks == 0) return FPT_OK;
    if (!d_out || nblocks > (1ull << 31)) {
        set_error("bad output buffer or size");
        return FPT_EINVAL;
    }
    const cudaError_t e =
        launch_philox_fill(seed, traj, block0, nblocks, d_out, static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return cuda_fail(e, "philox fill");
    return FPT_OK;
}

extern "C" fpt_status fpt_normals_fill(int precision, uint64_t seed, uint64_t traj, uint64_t n0,
                                       uint64_t n, double *d_out, void *stream) {
    if (n == 0) return FPT_OK;
    if (!d_out || n > (1ull << 31) || (precision != FPT_FP32 && precision != FPT_FP64)) {
        set_error("bad output buffer, size or precision");
        return FPT_EINVAL;
    }
    const cudaError_t e = launch_normals_fill(precision, seed, traj, n0, n, d_out,
                                              static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return cuda_fail(e, "normals fill");
    return FPT_OK;
}
