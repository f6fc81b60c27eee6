// engine_kernels.cu -- the persistent batched FPT kernel, the completion scan, and one request's
// kernel without an engine.
//
// One launch ("chunk") advances the resident lanes by the launch's blocks of kBlockSteps steps
// per warp on average (chunk_blocks, or fewer while a small request is new; Euler-Maruyama or
// stochastic Heun; the last quarter of the blocks is a per-CTA pool, so the warps of an SM
// finish together).  A lane integrates one trajectory:
// Philox4x32-10 -> Box-Muller -> step (Alg. 1 / 3) on a phase wrapped to [-pi, pi) with an
// integer winding count.  Escape and upper-wrap events are caught by one running maximum per
// block (exact replay of the rare block that reached a bound); the lower wrap (r < -pi) is
// applied at the end of each block.  At the block end the warp votes, finished lanes publish
// their exact result (grouped in the warp, additions nobody waits for) and the warp refills them
// -- with suspended trajectories, then ids of its reservoir, then new ids from the requests'
// work queues (one atomic per claim) -- so lanes never wait for the slowest trajectory of a
// batch (the dynamic job assignment of Sec. III.B, Fig. 6).
//
// Preemption: at the end of a launch, lanes of requests above their fair share may suspend
// their trajectory into the request's ring (state r, v, w, step count, id); a later refill
// resumes it exactly.  The ramped bias is formed from the trajectory's own step count, so a
// trajectory's arithmetic never depends on which lane, launch or schedule ran it.
//
// A warp integrates one kind at a time (model x integrator x constant or ramped bias: eight
// code paths); the request of each lane is free, so requests of the same kind share warps.
// Refill is round-robin over the claimable requests; while some request is starved, each is
// kept within a fair-share cap on the lanes it holds, otherwise no lane idles while any request
// has work.
#include <cstdint>

#include "engine_dev.h"
#include "fpt_device.cuh"
#include "internal.h"

namespace fpt {

namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;

struct Lane {
    float r, v, hb;
    int w, slot, esc;
    unsigned c_lo, c_hi, gid_lo, gid_hi;
    unsigned budget;      // blocks to the next event: step budget end, bias re-base, carry
    float gb, Jf;         // bias base and 4 x blocks since the base (exact)
    float dt, A, amp, bmc, nudt;
    PhiloxLane P;         // the trajectory's Philox stream (round keys, fixed words of rounds 0-2)
};

__device__ __forceinline__ float qnan_f() { return __int_as_float(0x7FFFFFFF); }

// Bounds checks of the FPT_CHECK build: a violated one sets its bit in the global check word
// (counters[kCntCheck], read back with the engine counters) and the access is skipped; nothing
// traps.  In the regular build every check is `true`.
enum : unsigned {
    kChkSlot = 0,      // request slot outside [0, max_requests)
    kChkLane = 1,      // lane-state index outside [0, n_lanes)
    kChkIdBlock = 2,   // id block outside [0, n_idblocks)
    kChkHistRow = 3,   // histogram row outside [0, hist_rows)
    kChkBin = 4,       // histogram bin outside [0, hist_bins)
    kChkTraj = 5,      // trajectory index outside [0, n_traj)
    kChkPark = 6,      // suspended-trajectory ring index outside [0, park_cap)
    kChkKind = 7,      // kind outside [0, kNumKinds)
    kChkReservoir = 8,   // a warp goes on to the packed last trajectories with ids in its reservoir
    kChkDry = 9,       // a warp skips its blocks for a meeting that is not called
};
#ifdef FPT_CHECK
__device__ __forceinline__ bool checked(const EngineDev &E, bool ok, unsigned bit) {
    if (!ok) atomicOr(&E.counters[kCntCheck], 1ull << bit);
    return ok;
}
#else
__device__ __forceinline__ constexpr bool checked(const EngineDev &, bool, unsigned) { return true; }
#endif

template <typename V>
__device__ __forceinline__ V vload(const V &x) {
    return *const_cast<const volatile V *>(&x);
}

__device__ __forceinline__ void set_idle(Lane &L) {
    L.slot = -1;
    L.r = qnan_f();
    L.v = 0.0f;
    L.hb = 0.0f;
    L.esc = -1;
    L.budget = 0xFFFFFFFFu;
    L.dt = L.A = L.amp = L.bmc = L.nudt = L.gb = L.Jf = 0.0f;
}

// Request constants and the trajectory's Philox stream; gid and the block count c are set.
__device__ __forceinline__ void load_consts(Lane &L, const SlotDev *S) {
    L.dt = S->dt;
    L.A = S->A;
    L.amp = S->amp;
    L.bmc = S->bmc;
    L.nudt = S->nudt;
    philox_lane_init(L.P, S->key0, S->key1, L.c_hi, L.gid_lo, L.gid_hi);
}

__device__ __forceinline__ unsigned long long lane_c(const Lane &L) {
    return (static_cast<unsigned long long>(L.c_hi) << 32) | L.c_lo;
}

// Bias base and event countdown from the trajectory's Philox block count c (4 steps each; c is
// a multiple of kBlockPhilox at block boundaries):
// gb = gamma0 + nu dt 4 c_base (FP64, rounded once), Jf = 4 (c - c_base),
// budget = kernel blocks until the step budget ends, the next re-base or the next carry of the
// low 32-bit word of c, whichever is first (the high word is only updated at that event).
__device__ __forceinline__ void set_progress(Lane &L, const SlotDev *S) {
    const unsigned long long c = lane_c(L);
    const unsigned long long cb = c - (c % kRebaseBlocks);
    L.gb = static_cast<float>(S->gamma0 + S->nudt_d * static_cast<double>(4ull * cb));
    L.Jf = static_cast<float>(4ull * (c - cb));
    const unsigned long long to_end = S->nblocks > c ? S->nblocks - c : 0ull;
    const unsigned long long to_base = kRebaseBlocks - (c - cb);
    const unsigned long long to_carry = 0x100000000ull - (c & 0xFFFFFFFFull);
    unsigned long long m = to_end < to_base ? to_end : to_base;
    m = m < to_carry ? m : to_carry;
    L.budget = static_cast<unsigned>((m + kBlockPhilox - 1) / kBlockPhilox);
}

// Start trajectory `idx` of request slot s.
__device__ __forceinline__ void init_lane(Lane &L, const EngineDev &E, int s, unsigned long long idx) {
    const SlotDev *S = E.slots + s;
    const unsigned long long gid = S->traj_offset + idx;
    L.slot = s;
    L.gid_lo = static_cast<unsigned>(gid);
    L.gid_hi = static_cast<unsigned>(gid >> 32);
    L.c_lo = L.c_hi = 0;
    L.r = S->r0;
    L.v = S->v0;
    L.w = S->w0;
    L.hb = fminf(S->eb0, kPiF);
    L.esc = -1;
    load_consts(L, S);
    L.gb = S->gb0;       // set_progress at c = 0, formed on the host
    L.Jf = 0.0f;
    L.budget = S->budget0;
}

// Continue a trajectory exactly where it stopped (a suspended one, or one that changes warps).
template <typename State>
__device__ __forceinline__ void resume_from(Lane &L, const EngineDev &E, int s, const State &P) {
    const SlotDev *S = E.slots + s;
    L.slot = s;
    L.r = P.r;
    L.v = P.v;
    L.w = P.w;
    L.c_lo = P.c_lo;
    L.c_hi = P.c_hi;
    L.gid_lo = P.gid_lo;
    L.gid_hi = P.gid_hi;
    L.hb = fminf(fmaf(-kTwoPiF, static_cast<float>(P.w - S->w0), S->eb0), kPiF);
    L.esc = -1;
    load_consts(L, S);
    set_progress(L, S);
}

// Histogram bin of x = out_a + out_b k (IEEE double, separately rounded): -1 below the range,
// hist_bins above it.  From the request's integer map where that names it: the formula's FP64
// operations hold a scheduler's unit for 64 cycles each.
__device__ __forceinline__ int hist_bin(const SlotDev *S, unsigned long long k) {
    if (k >> 32 == 0) {
        const int b = mapped_bin(S->map, static_cast<uint32_t>(k));
        if (b >= 0) return b;
    }
    if (k >= S->map.k_over) return S->hist_bins;
    if (k < S->map.k_under) return -1;
    const double kd = static_cast<double>(k);
    const double x = S->output == FPT_OUT_TIME ? __dmul_rn(S->out_b, kd)
                                               : __dadd_rn(S->out_a, __dmul_rn(S->out_b, kd));
    if (x < S->hist_lo) return -1;
    if (x >= S->hist_hi) return S->hist_bins;
    const int bin = static_cast<int>(floor(__dmul_rn(__dsub_rn(x, S->hist_lo), S->hist_inv_w)));
    return bin < S->hist_bins ? bin : S->hist_bins - 1;
}

// Per-CTA view of the requests during one launch (shared memory), set up at kernel start:
//   ok[s]   bit 0: request s has ids left to claim, bit 1: it has suspended trajectories to
//           resume (both as of the launch start; cleared when a warp finds them exhausted),
//   held[s] lanes of this CTA that hold a trajectory of s (the CTA's share of the fair-share
//           cap is checked against it, so claims need no global read),
//   budget[s] reservoir ids this CTA may hold for s: its share of the room the request's ring
//           had at launch start beyond one slot per lane (kept for suspensions), so that the
//           reservoirs returned to the ring at the end of the launch always fit.
struct CtaView {
    unsigned *ok;
    int *held;
    int *budget;                 // ids this CTA's warps may still hold in reservoirs, per request
    int *res_slot, *res_cnt;     // per warp of the CTA: reservoir request and count ...
    unsigned long long *res_base;   // ... and first id (ids res_base .. res_base + res_cnt - 1)
    int *started;                // per warp: trajectories it started in this launch
    int *pool;                   // blocks of this launch not yet taken by a warp of the CTA
    int *warp_act, *warp_knd;    // per warp: lanes with a trajectory, and their kind
    unsigned *share;             // blocks of the launch every warp runs before it takes from the pool
    int *tail;                   // 1: the CTA's warps meet to run its last trajectories together
    // Groups of 32 lanes the CTA can run that way (0: it never does).  In shared memory like the rest: a
    // register held through run_blocks costs its loop 1 % (1188 -> 1199 Gstep/s over the 12-point sweep).
    const int *tail_groups;
    const int *act_count;        // the launch's lists and flags, read once: claimable slots per kind,
    const int *flags;            // {strict caps, warps of the CTA that claim}
};

// Publish the trajectories finishing in this warp at this block end (warp-collective: every lane
// calls it, `fin` says whether its trajectory finished).  Lanes are grouped by (request slot, id
// block) with a match; each group's counts and the 32-bit limbs of k and k^2 are gathered by
// shuffles, and its first lane adds them into the id block with atomic additions whose result
// it does not wait for, and gives back the group's in-flight places.  Histogram counts are
// grouped by (slot, id block, bin) the same way.  The scan kernel reads the id blocks only
// after the launch, so the order of the additions is free.
__device__ __forceinline__ void emit_warp(const EngineDev &E, int *held, bool fin, int slot,
                                          unsigned long long gid, bool escaped, unsigned long long k) {
    const int lane = threadIdx.x & 31;
    // an index out of range (checked build only) drops the trajectory's result
    if (fin) fin = checked(E, slot >= 0 && slot < E.max_requests, kChkSlot);
    if (!__any_sync(kFull, fin)) return;   // an event block without a finished trajectory
    const SlotDev *S = E.slots + (fin ? slot : 0);
    unsigned long long idx = 0;
    unsigned ib = 0, row = 0;
    int bin = -2;
    if (fin) {
        idx = gid - S->traj_offset;
        ib = static_cast<unsigned>(id_block_quot(idx, S->ib_magic, S->ib_shift));
        row = S->hist_per_block ? ib : static_cast<unsigned>(idx / kHistRowIds);
        if (escaped && S->hist) bin = hist_bin(S, k);
        fin = checked(E, idx < S->n_traj, kChkTraj) && checked(E, ib < S->n_idblocks, kChkIdBlock) &&
              checked(E, row < S->hist_rows, kChkHistRow) &&
              checked(E, bin == -2 || (bin >= -1 && bin <= S->hist_bins), kChkBin);
        if (fin && S->per_traj) S->per_traj[idx] = escaped ? static_cast<long long>(k) : -1ll;
    }
    // slot < 2^10, id block and row < 2^32, bin < 2^21: distinct keys for distinct groups
    const unsigned long long gkey = fin ? (static_cast<unsigned long long>(slot) << 32) | ib : ~0ull;
    const unsigned grp = __match_any_sync(kFull, gkey);
    const unsigned long long bkey =
        fin && bin >= 0 && bin < S->hist_bins
            ? (static_cast<unsigned long long>(slot) << 53) | (static_cast<unsigned long long>(row) << 21) |
                  static_cast<unsigned long long>(bin)
            : ~0ull;
    const unsigned bgrp = __match_any_sync(kFull, bkey);
    if (!fin) return;
    IdBlockAcc *A = S->acc + ib;
    if (bkey != ~0ull && lane == __ffs(bgrp) - 1)
        atomicAdd(S->hist + static_cast<size_t>(row) * S->hist_bins + bin, static_cast<unsigned>(__popc(bgrp)));
    // limbs: k = k0 + 2^32 k1, k^2 = q0 + 2^32 q1 + 2^64 q2 (each < 2^32)
    const unsigned long long kk_lo = escaped ? k * k : 0ull, kk_hi = escaped ? __umul64hi(k, k) : 0ull;
    const unsigned long long ke = escaped ? k : 0ull;
    unsigned long long l[5] = {ke & 0xFFFFFFFFull, ke >> 32, kk_lo & 0xFFFFFFFFull, kk_lo >> 32, kk_hi};
    unsigned cnt = (escaped ? 1u : 0u) | (bin == -1 ? 2u : 0u) | (escaped && bin == S->hist_bins ? 4u : 0u);
    unsigned n_e = cnt & 1u, n_u = (cnt >> 1) & 1u, n_o = cnt >> 2;
    const int leader = __ffs(grp) - 1;
    unsigned rest = grp & ~(1u << leader);
    while (rest) {   // every lane of the group runs the same sequence of shuffles
        const int src = __ffs(rest) - 1;
        rest &= rest - 1u;
        const unsigned c = __shfl_sync(grp, cnt, src);
        unsigned long long m[5];
#pragma unroll
        for (int j = 0; j < 5; ++j) m[j] = __shfl_sync(grp, l[j], src);   // src's l is unchanged
        if (lane == leader) {
            n_e += c & 1u;
            n_u += (c >> 1) & 1u;
            n_o += c >> 2;
#pragma unroll
            for (int j = 0; j < 5; ++j) l[j] += m[j];
        }
    }
    if (lane != leader) return;
    if (n_e) {
        atomicAdd(&A->escaped, n_e);
        atomicAdd(&A->s1[0], l[0]);
        if (l[1]) atomicAdd(&A->s1[1], l[1]);
        atomicAdd(&A->s2[0], l[2]);
        if (l[3]) atomicAdd(&A->s2[1], l[3]);
        if (l[4]) atomicAdd(&A->s2[2], l[4]);
    }
    if (n_u) atomicAdd(&A->under, n_u);
    if (n_o) atomicAdd(&A->over, n_o);
    const int n = __popc(grp);
    atomicAdd(&A->done, static_cast<unsigned>(n));
    atomicSub(&E.ctl[slot].inflight, n);
    atomicSub(&held[slot], n);
}

// Escapes wait for their publication and the lane's refill, whose cost (~550 instructions of a warp)
// hardly depends on how many lanes it serves: a warp that starts a trajectory at least every eight
// blocks takes the escapes of up to kDeferBlocks further blocks together.  Lane::esc holds the step
// in its block and that block's number modulo kDeferMask + 1.  (Trajectories of 950 steps, 60
// blocks: 8.4 -> 6.8 ms for 2^22, with the integer bins of hist_bin.  Kinds whose trajectories last 10^4
// steps never wait, but their loop holds the test: ramped Euler at seven warps per SM 40.8 -> 42.6 ns per
// step, a switching histogram of 30 000 trajectories 43.1 -> 45.)
constexpr unsigned kDeferBlocks = 5, kDeferMask = 15u;
constexpr int kDeferShift = 8;

// Rare per-lane path: the phase reached hb = min(eb, pi), where eb = phi* - 2 pi w is the
// threshold in the current cell's coordinates.  Escape freezes the lane (NaN phase: no further
// events) and records the step within the block; otherwise wrap upwards and count a winding.
__device__ __forceinline__ void phase_event(Lane &L, const EngineDev &E, int s, unsigned b = 0) {
    const SlotDev *S = E.slots + L.slot;
    const float eb0 = S->eb0;
    const int w0 = S->w0;
    const float eb = fmaf(-kTwoPiF, static_cast<float>(L.w - w0), eb0);
    if (L.r >= eb) {
        L.esc = s | static_cast<int>((b & kDeferMask) << kDeferShift);
        L.r = qnan_f();
        return;
    }
    L.r -= kTwoPiF;
    L.w += 1;
    L.hb = fminf(fmaf(-kTwoPiF, static_cast<float>(L.w - w0), eb0), kPiF);
}

// Lower wrap, applied at block ends (sin is accurate a little below -pi in between).
__device__ __forceinline__ void wrap_down(Lane &L, const EngineDev &E) {
    const SlotDev *S = E.slots + L.slot;
    L.r += kTwoPiF;
    L.w -= 1;
    L.hb = fminf(fmaf(-kTwoPiF, static_cast<float>(L.w - S->w0), S->eb0), kPiF);
}

// At the end of block `b` (its number after the increment): lane L has escaped in it or in one of the
// blocks before, or its countdown ran out: true when the trajectory is finished, with its step in
// `k` if it escaped within its budget; otherwise the bias is re-based.  `useful` (the caller counted
// whole blocks) loses the steps past the end.
__device__ __forceinline__ bool finished(Lane &L, const EngineDev &E, unsigned b, bool &escaped,
                                         unsigned long long &k, unsigned long long &useful) {
    const SlotDev *S = E.slots + L.slot;
    const unsigned long long c = lane_c(L);
    const unsigned long long max_steps = S->max_steps;
    if (L.esc < 0 && c < S->nblocks) {   // re-base of the bias, not the end of the budget
        set_progress(L, S);
        return false;
    }
    const unsigned step = static_cast<unsigned>(L.esc) & (kBlockSteps - 1);
    const unsigned since = (b - (static_cast<unsigned>(L.esc) >> kDeferShift)) & kDeferMask;   // blocks
    if (L.esc >= 0) {
        k = 4ull * (c - kBlockPhilox) - kBlockSteps * since + step + 1ull;
        escaped = k <= max_steps;
    }
    if (escaped) useful -= kBlockSteps - 1u - step + kBlockSteps * since;
    else useful -= 4ull * c - max_steps;
    return true;
}

// Finish lanes that escaped up to block `b` or reached the step budget (warp-collective).
template <int T>
__device__ __forceinline__ void finish_lanes(Lane (&L)[T], const EngineDev &E, int *held, unsigned b,
                                             unsigned long long &useful, int &n_active, unsigned &n_esc,
                                             unsigned &n_cens) {
#pragma unroll
    for (int t = 0; t < T; ++t) {
        bool fin = false, escaped = false;
        unsigned long long k = 0;
        if (L[t].slot < 0) {
            L[t].budget = 0xFFFFFFFFu;
        } else if (L[t].esc >= 0 || L[t].budget == 0) {
            fin = finished(L[t], E, b, escaped, k, useful);
        }
        const unsigned long long gid = (static_cast<unsigned long long>(L[t].gid_hi) << 32) | L[t].gid_lo;
        emit_warp(E, held, fin, L[t].slot, gid, escaped, k);
        if (fin) {
            if (escaped) ++n_esc;
            else ++n_cens;
            set_idle(L[t]);
            --n_active;
        }
    }
}

// Warp-collective refill of idle lanes with trajectories of requests of kind `kind`.  Lane 0
// takes, per request in round-robin order, suspended trajectories first, then ids from the
// warp's reservoir, then new ids from the request's queue head: one atomic addition on the head
// per claim, claiming up to kReserveIds more for the reservoir when it is empty and the CTA's
// budget allows, and the in-flight count raised by what was actually started (an addition
// nobody waits for).  While some request is
// starved (strict caps, set by the host with preemption orders) each request is kept within
// this CTA's share of its fair-share cap, counted in shared memory; otherwise lanes take work
// from the first request that has some, so no lane idles while any request has work.  Returns the
// lanes that stay idle.
template <int T>
__device__ __forceinline__ int refill(Lane (&L)[T], const EngineDev &E, const CtaView &V, int kind,
                                      int &n_active, unsigned &cursor, unsigned b) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    unsigned idle[T];
    int total = 0;
#pragma unroll
    for (int t = 0; t < T; ++t) {
        idle[t] = __ballot_sync(kFull, L[t].slot < 0);
        total += __popc(idle[t]);
    }
    if (total == 0) return 0;
    if (static_cast<int>(threadIdx.x >> 5) >= V.flags[1]) return total;   // spread scarce work
    if (!checked(E, kind >= 0 && kind < kNumKinds, kChkKind)) return total;
    const int cnt = V.act_count[kind];
    if (cnt <= 0) return total;
    const int *list = E.act_list + kind * E.max_requests;
    const bool capped = V.flags[0] != 0;
    const int wl = static_cast<int>(threadIdx.x >> 5);
    // A warp that holds a reservoir serves its request first, so the reservoir drains.
    __syncwarp();
    const int rs = V.res_slot[wl];
    const bool res_first = V.res_cnt[wl] > 0 && rs >= 0 && rs < E.max_requests && E.slots[rs].kind == kind;
    {
        for (int scanned = res_first ? -1 : 0; scanned < cnt && total > 0; ++scanned) {
            const int s = scanned < 0 ? rs : list[cursor % static_cast<unsigned>(cnt)];
            if (scanned >= 0) ++cursor;
            if (!checked(E, s >= 0 && s < E.max_requests, kChkSlot)) continue;
            unsigned long long base = 0, rb = 0;
            int got = 0, gp = 0, rt = 0;
            unsigned p0 = 0;
            if (lane == 0 && ((V.ok[s] & 3u) || V.res_slot[wl] == s)) {
                SlotCtl *C = E.ctl + s;
                const unsigned long long n_traj = E.slots[s].n_traj;
                int want = total;
                if (capped) {
                    const int cap = (E.caps[s] + static_cast<int>(gridDim.x) - 1) / static_cast<int>(gridDim.x);
                    const int room = cap - V.held[s];
                    want = room < 0 ? 0 : (room < want ? room : want);
                }
                // 1. suspended trajectories
                if (want > 0 && (V.ok[s] & 2u)) {
                    const int pv = atomicSub(&C->park_avail, want);
                    if (pv <= 0) {
                        atomicAdd(&C->park_avail, want);
                        atomicAnd(&V.ok[s], ~2u);
                    } else {
                        gp = pv < want ? pv : want;
                        if (gp < want) atomicAdd(&C->park_avail, want - gp);
                        p0 = atomicAdd(&C->park_head, static_cast<unsigned>(gp));
                        atomicSub(&C->park_used, gp);
                    }
                }
                got = gp;
                // 2. this warp's reservoir of ids claimed earlier
                if (want > got && V.res_slot[wl] == s && V.res_cnt[wl] > 0) {
                    rt = want - got < V.res_cnt[wl] ? want - got : V.res_cnt[wl];
                    rb = V.res_base[wl];
                    V.res_base[wl] += static_cast<unsigned long long>(rt);
                    V.res_cnt[wl] -= rt;
                    atomicAdd(&V.budget[s], rt);
                    got += rt;
                }
                // 3. the queue head, with more for the reservoir when it is free: as many as this
                //    warp is expected to start in the rest of a full launch at its rate so far
                //    (at most kReserveIds, none while caps are enforced), within the CTA's budget;
                //    in a shorter launch the surplus goes back to the ring at its end.
                //    Only warps that start a trajectory at least every 8 blocks keep one: for
                //    long trajectories the ids would mostly return to the ring unused.
                if (want > got && (V.ok[s] & 1u)) {
                    const unsigned long long end = claim_end(n_traj, E.slots[s].stop_block, C->claim_blocks);
                    // a limited request: look before claiming (warps that look at once go past it)
                    if (end < n_traj && vload(C->head) >= end) atomicAnd(&V.ok[s], ~1u);
                }
                if (want > got && (V.ok[s] & 1u)) {
                    const int wn = want - got;
                    int extra = 0;
                    if (V.res_cnt[wl] == 0 && !capped && b > 0 && 8u * static_cast<unsigned>(V.started[wl]) >= b) {
                        const unsigned long long expect =
                            static_cast<unsigned long long>(V.started[wl]) * (E.chunk_blocks > b ? E.chunk_blocks - b : 0u) / b;
                        const int want_extra = expect < static_cast<unsigned long long>(kReserveIds)
                                                   ? static_cast<int>(expect) : kReserveIds;
                        if (want_extra > 0) {
                            if (atomicSub(&V.budget[s], want_extra) >= want_extra) extra = want_extra;
                            else atomicAdd(&V.budget[s], want_extra);
                        }
                    }
                    const int cl = wn + extra;
                    base = atomicAdd(&C->head, static_cast<unsigned long long>(cl));
                    int keep = 0;
                    if (base < n_traj) {
                        const unsigned long long left = n_traj - base;
                        const int avail = left < static_cast<unsigned long long>(cl) ? static_cast<int>(left) : cl;
                        const int use = avail < wn ? avail : wn;
                        got += use;
                        keep = avail - use;
                        if (keep > 0) {
                            V.res_slot[wl] = s;
                            V.res_base[wl] = base + static_cast<unsigned long long>(use);
                            V.res_cnt[wl] = keep;
                        }
                    }
                    if (extra > keep) atomicAdd(&V.budget[s], extra - keep);
                    if (base + static_cast<unsigned long long>(cl) >= claim_end(n_traj, E.slots[s].stop_block, C->claim_blocks))
                        atomicAnd(&V.ok[s], ~1u);
                }
                if (got) {
                    atomicAdd(&C->inflight, got);
                    atomicAdd(&V.held[s], got);
                    V.started[wl] += got;
                }
            }
            got = __shfl_sync(kFull, got, 0);
            if (got == 0) continue;
            gp = __shfl_sync(kFull, gp, 0);
            p0 = __shfl_sync(kFull, p0, 0);
            rt = __shfl_sync(kFull, rt, 0);
            rb = __shfl_sync(kFull, rb, 0);
            base = __shfl_sync(kFull, base, 0);
            const SlotDev *S = E.slots + s;
            int before = 0;
#pragma unroll
            for (int t = 0; t < T; ++t) {
                const unsigned m = idle[t];
                const int rank = before + __popc(m & lt);
                if (((m >> lane) & 1u) && rank < got) {
                    if (rank < gp) {
                        const unsigned pi = (p0 + static_cast<unsigned>(rank)) % S->park_cap;
                        if (checked(E, pi < S->park_cap, kChkPark)) resume_from(L[t], E, s, S->park[pi]);
                    } else if (rank < gp + rt) {
                        init_lane(L[t], E, s, rb + static_cast<unsigned long long>(rank - gp));
                    } else {
                        init_lane(L[t], E, s, base + static_cast<unsigned long long>(rank - gp - rt));
                    }
                    ++n_active;
                }
                before += __popc(m);
                idle[t] = __ballot_sync(kFull, L[t].slot < 0);
            }
            total -= got;
            if (total == 0 && lane == 0) V.warp_act[wl] = 32;
        }
    }
    return total;
}

// A launch's blocks: each warp first runs (1 - 1/kPoolDiv) of the launch's block count, then
// takes kGrant blocks at a time from its CTA's pool of the rest, so warps whose lanes had more
// events (replays, refills) do fewer blocks and the warps of an SM finish together instead of
// leaving the SM to a few late ones (+3.7 % at 4096-step launches, +0.8 % at 65 536).
constexpr unsigned kPoolDiv = 4;
constexpr int kGrant = 4;

// More blocks for this warp from its CTA's pool (warp-collective); false when the pool is empty.
__device__ __forceinline__ bool grant(const CtaView &V, unsigned &limit) {
    int g = 0;
    if ((threadIdx.x & 31) == 0) {
        const int p = atomicSub(V.pool, kGrant);
        g = p >= kGrant ? kGrant : (p > 0 ? p : 0);
    }
    g = __shfl_sync(kFull, g, 0);
    limit += static_cast<unsigned>(g);
    return g > 0;
}

// Whether the trajectories the CTA's warps have published fit its groups, or three quarters of the
// warps that hold them (warp-collective; the same for every warp between two publications).  (Twelve
// full warps take 52 ns per step, twenty sparse ones 82.)
__device__ __forceinline__ bool thinned_out(const CtaView &V) {
    const int lane = threadIdx.x & 31, warps = static_cast<int>(blockDim.x >> 5);
    const int a = lane < warps ? vload(V.warp_act[lane]) : 0;
    const int total = __reduce_add_sync(kFull, a);
    const int kinds = __popc(__reduce_or_sync(kFull, a > 0 ? 1u << (vload(V.warp_knd[lane]) & 31) : 0u));
    // warps they need: ceil(lanes / 32) of one kind, at most (lanes + 31 kinds) / 32 of several
    const int need = (total + 31 * kinds) >> 5, holding = __popc(__ballot_sync(kFull, a > 0));
    return total > 0 && (need <= *V.tail_groups || 4 * need <= 3 * holding);
}

// This warp's lanes after an event, for the CTA's view, and whether the CTA has run dry
// (warp-collective): nothing left to claim or resume in any listed request, no reservoir, and
// trajectories thinned out.  Then the warps are called together (V.tail); the exact counts are taken
// when they have met.  Flags before reservoirs: refill fills a warp's reservoir before it clears the
// flag.  A claim can still be under way here whose ids nobody sees yet, so a warp gives back what its
// reservoir holds on its way to the meeting.
template <int T>
__device__ __forceinline__ void look_dry(Lane (&L)[T], const EngineDev &E, const CtaView &V, int kind) {
    if constexpr (T == 1) {
        if (*V.tail_groups == 0) return;
        const int lane = threadIdx.x & 31, warps = static_cast<int>(blockDim.x >> 5);
        const int act = __popc(__ballot_sync(kFull, L[0].slot >= 0));
        if (lane == 0) {
            V.warp_act[threadIdx.x >> 5] = act;
            V.warp_knd[threadIdx.x >> 5] = kind;
        }
        __syncwarp();
        if (!thinned_out(V)) return;
        bool work = false;
        for (int k = 0; k < kNumKinds; ++k)
            for (int j = lane; j < V.act_count[k]; j += 32)
                work |= (vload(V.ok[E.act_list[k * E.max_requests + j]]) & 3u) != 0u;
        work |= lane < warps && vload(V.res_cnt[lane]) > 0;
        if (!__any_sync(kFull, work) && lane == 0) *V.tail = 1;
    }
}

// Blocks this warp may run before it looks again whether the CTA's warps are called together (a
// look per block costs 2 % of a full CTA's rate).
constexpr unsigned kLookBlocks = 8;

// More blocks for this warp (warp-collective): its own share kLookBlocks at a time, then the
// CTA's pool; false when there are none or the warps are called together.
__device__ __forceinline__ bool more(const CtaView &V, unsigned &limit) {
    if (vload(*V.tail) != 0) return false;
    const unsigned share = *V.share;
    if (limit < share) {
        limit = limit + kLookBlocks < share ? limit + kLookBlocks : share;
        return true;
    }
    return grant(V, limit);
}

// Integrate blocks of kBlockSteps steps with model M, integrator H and bias kind R (constant or
// ramped) until the warp's share of the launch's blocks is done (`limit`, extended from the
// CTA's pool), the whole warp has run out of work, or some of its lanes find no more: then the caller
// looks whether the CTA has run dry.  Returns the next block index.  (With that look in here the loop of
// a full CTA took 1 % more time: 1176 -> 1188 Gstep/s over the 12-point sweep.)
template <int M, int H, int R, int T>
__device__ __forceinline__ unsigned run_blocks(Lane (&L)[T], const EngineDev &E, const CtaView &V, unsigned b,
                                               int &n_active,
                               unsigned &cursor, unsigned long long &useful, unsigned &n_esc,
                               unsigned &n_cens, unsigned &limit) {
    // Steps are counted when the number of active lanes changes (at events) and at the end:
    // useful += kBlockSteps x active lanes x blocks since the last count.
    unsigned b_count = b;
    // Constant bias (R = 0): the bias line is the same in every block until an event changes the
    // lane (re-base, refill); it is formed here and after each event.
    float gs[T], gsl[T];
#pragma unroll
    for (int t = 0; t < T; ++t)
        if constexpr (!R) bias_line(fmaf(L[t].nudt, L[t].Jf, L[t].gb), L[t].nudt, L[t].dt, gs[t], gsl[t]);
    while (b < limit || more(V, limit)) {
        // the block's normals: Philox blocks c .. c + kBlockPhilox - 1 (c is a multiple of
        // kBlockPhilox, so c_lo + h never carries into c_hi)
        float rr[T][2 * kBlockPhilox], tg[T][kBlockSteps];
#pragma unroll
        for (int t = 0; t < T; ++t) {
            // the block's Philox words first, then their Box-Muller pairs (measured +0.4 % over
            // interleaving them per call: the MUFU work of the pairs comes in one stretch)
            uint4 xs[kBlockPhilox];
#pragma unroll
            for (int h = 0; h < kBlockPhilox; ++h) xs[h] = philox_lane_block(L[t].P, L[t].c_lo, static_cast<unsigned>(h));
#pragma unroll
            for (int h = 0; h < kBlockPhilox; ++h) {
                bm_pair_f32(xs[h].x, xs[h].y, L[t].bmc, rr[t][2 * h], tg[t][4 * h], tg[t][4 * h + 1]);
                bm_pair_f32(xs[h].z, xs[h].w, L[t].bmc, rr[t][2 * h + 1], tg[t][4 * h + 2], tg[t][4 * h + 3]);
            }
            if constexpr (R) bias_line(fmaf(L[t].nudt, L[t].Jf, L[t].gb), L[t].nudt, L[t].dt, gs[t], gsl[t]);
        }
        // The block's steps without a branch: each lane only tracks the largest phase of the block.
        // In the rare block where it reached the lane's bound hb, the lane's block is replayed
        // (in the warp's event path below) from the saved start state with the event test after
        // every step, so wraps and the escape step are exactly those of a step-by-step test.
        float r0s[T], v0s[T], mx[T];
#pragma unroll
        for (int t = 0; t < T; ++t) {
            r0s[t] = L[t].r;
            v0s[t] = L[t].v;
            mx[t] = -INFINITY;
        }
#pragma unroll
        for (int s = 0; s < kBlockSteps; ++s) {
#pragma unroll
            for (int t = 0; t < T; ++t) {
                step_f32<M, H>(L[t].r, L[t].v, rr[t][s >> 1], tg[t][s], bias_b0<H, R>(gs[t], gsl[t], s),
                               bias_b1<H, R>(gs[t], gsl[t], s), L[t].dt, L[t].A, L[t].amp);
                mx[t] = fmaxf(mx[t], L[t].r);
            }
        }
        bool ev = false;
#pragma unroll
        for (int t = 0; t < T; ++t) {
            L[t].c_lo += kBlockPhilox;
            if constexpr (R) L[t].Jf += static_cast<float>(kBlockSteps);
            L[t].budget -= 1u;
            // one vote covers every rare case: a bound reached (escape or upper wrap), the
            // countdown (step budget, bias re-base, low-word carry) and the lower wrap
            ev |= (mx[t] >= L[t].hb) || (L[t].budget == 0u) || (L[t].r < -kPiF);
        }
        ++b;
        if (__any_sync(kFull, ev)) {
            useful += static_cast<unsigned long long>(kBlockSteps) * static_cast<unsigned>(n_active) * (b - b_count);
            b_count = b;
#pragma unroll
            for (int t = 0; t < T; ++t) {
                if (mx[t] >= L[t].hb) {
                    L[t].r = r0s[t];
                    L[t].v = v0s[t];
#pragma unroll
                    for (int s = 0; s < kBlockSteps; ++s) {
                        step_f32<M, H>(L[t].r, L[t].v, rr[t][s >> 1], tg[t][s],
                                       bias_b0<H, R>(gs[t], gsl[t], s), bias_b1<H, R>(gs[t], gsl[t], s),
                                       L[t].dt, L[t].A, L[t].amp);
                        if (L[t].r >= L[t].hb) phase_event(L[t], E, s, b);
                    }
                }
                if (L[t].r < -kPiF) wrap_down(L[t], E);
                if (L[t].slot >= 0 && L[t].c_lo == 0u) {   // 2^32-block carry: new fixed words
                    L[t].c_hi += 1u;
                    const SlotDev *S = E.slots + L[t].slot;
                    philox_lane_init(L[t].P, S->key0, S->key1, L[t].c_hi, L[t].gid_lo, L[t].gid_hi);
                }
            }
            // an escape that is to wait counts down its lane's budget: the first one to reach 0 takes
            // all that wait with it
            const unsigned wait = 8u * static_cast<unsigned>(vload(V.started[threadIdx.x >> 5])) >= b ? kDeferBlocks : 0u;
            bool out = false;
#pragma unroll
            for (int t = 0; t < T; ++t) {
                if (L[t].esc >= 0 && L[t].budget > wait) L[t].budget = wait;
                out |= L[t].slot >= 0 && L[t].budget == 0u;
            }
            if (__any_sync(kFull, out)) {
                finish_lanes(L, E, V.held, b, useful, n_active, n_esc, n_cens);
                const int idle = refill(L, E, V, kind_of(M, H, R), n_active, cursor, b);
                if (!__any_sync(kFull, n_active > 0) || (idle > 0 && *V.tail_groups > 0)) break;
            }
            if constexpr (!R) {
#pragma unroll
                for (int t = 0; t < T; ++t)
                    bias_line(fmaf(L[t].nudt, L[t].Jf, L[t].gb), L[t].nudt, L[t].dt, gs[t], gsl[t]);
            }
        }
    }
    useful += static_cast<unsigned long long>(kBlockSteps) * static_cast<unsigned>(n_active) * (b - b_count);
    bool waits = false;
#pragma unroll
    for (int t = 0; t < T; ++t) waits |= L[t].esc >= 0;
    if (__any_sync(kFull, waits)) finish_lanes(L, E, V.held, b, useful, n_active, n_esc, n_cens);
    return b;
}

// An idle warp looks for work of any kind, starting from a warp-dependent one; returns the kind
// it took work of, or -1.
template <int T>
__device__ __forceinline__ int seek_work(Lane (&L)[T], const EngineDev &E, const CtaView &V, int &n_active,
                                         unsigned &cursor, unsigned b) {
    const unsigned warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int first = static_cast<int>(warp % kNumKinds);
    for (int q = 0; q < kNumKinds; ++q) {
        const int m = (first + q) % kNumKinds;
        refill(L, E, V, m, n_active, cursor, b);
        if (__any_sync(kFull, n_active > 0)) return m;
    }
    return -1;
}

// ---- the CTA's last trajectories -----------------------------------------------------------
// When a CTA has nothing left to claim, its lanes thin out while its warps keep their issue
// slots: a warp with one lane costs what a full one does, and a full CTA takes 82 ns per step.
// One warp alone on a scheduler still takes 31 ns per step, of which the chain phase -> sin ->
// phase is 14 ns and the rest the noise made in front of it.  So the CTA's warps meet, the
// remaining trajectories are packed into the fewest groups of 32 lanes of one kind, and each group
// gets one warp that only integrates and three that only make its noise: chunks of blocks of 16
// steps through a ring of three chunks in shared memory, one named barrier of the group per chunk
// (the noise is two chunks ahead, so the next block's loads never wait).  Integrating takes ~8
// cycles of a scheduler per step and noise ~27, so the integrating warps sit on one scheduler (warp
// index mod 4) and the noise on the other three: beside a noise warp the chain waits for the MUFU
// and multiply pipes (measured in a loop of these parts alone, four groups with two noise warps:
// 26 ns per step mixed).  After each round of kRoundBlocks blocks or more the groups
// are packed again if that makes them fewer.  The arithmetic of a trajectory is that of
// run_blocks, bit for bit.  ns per step at 1 / 2 / 3 / 4 full warps per SM, the plain loop -> this:
// overdamped Euler 31.5 / 31.5 / 31.5 / 31.5 -> 17.5 / 18.5 / 21.2 / 22.8, underdamped ramped Euler
// 30.4 / 30.5 / 30.5 / 30.5 -> 12.8 / 17.5 / 21.4 / 23.0, underdamped Heun 40 -> 24 / 25 / 29 / 33;
// a request of 1024 trajectories of 19 000 steps 3.7 -> 2.0 ms.
constexpr int kTailGroupsMax = 5;       // a quarter of the warps: one scheduler's
constexpr int kTailMakers = 3;          // noise warps per group
constexpr int kTailChunk = 3;           // blocks per chunk, one for each of them
constexpr int kTailRing = 3 * kTailChunk;                     // blocks in a group's ring
// Floats of one block of a group.  Euler: the 16 addends of the steps (noise and bias, formed by
// the noise warps: an operation and half a load per step less in the chain's warp); Heun: 8 radii
// and 16 cosines / sines, as its two stages take different biases.
template <int H>
constexpr int kNoiseBlock = 32 * (H == kEuler ? 16 : 24);
constexpr int kNoiseBlockMax = 32 * 24;
constexpr int kTailMinWarps = 8;

// A request that runs without an engine (solo_kernel).
constexpr int kSoloThreads = 640;
struct SoloArgs {
    SlotDev slot;                  // n_traj, acc and hist are each CTA's own
    unsigned long long n;
    fpt_sums *sums;                // accumulated into, may be null
    unsigned long long *hist;      // accumulated into: nbins counts, 0 without
    int nbins;
};

struct TailLane {      // a trajectory while it changes warps, or its result
    float r, v;
    int w, slot;
    unsigned c_lo, c_hi, gid_lo, gid_hi;   // result: c is the escape step
    int fin;                               // kTailRuns, kTailEscaped or kTailCensored
};
enum : int { kTailRuns = 0, kTailEscaped = 1, kTailCensored = 2 };

// Groups a CTA of `warps` warps takes on; CTAs below kTailMinWarps warps do without.
__host__ __device__ constexpr int tail_groups_of(int T, int warps) {
    return T != 1 || warps < kTailMinWarps ? 0 : (warps / 4 < kTailGroupsMax ? warps / 4 : kTailGroupsMax);
}
__host__ __device__ constexpr size_t tail_shared_bytes(int warps) {
    return tail_groups_of(1, warps) == 0 ? 0 : static_cast<size_t>(tail_groups_of(1, warps)) * kTailRing * kNoiseBlockMax * 4 +
                                               kTailGroupsMax * 32 * sizeof(TailLane);
}

__device__ __forceinline__ void group_barrier(int group) {
    asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "n"(32 * (1 + kTailMakers)) : "memory");
}

// The noise of one call (steps 4 h .. 4 h + 3 of a block) of one lane, in shared memory as a float4
// and, for Heun, a float2 behind the block's float4s.
template <int H>
struct TailCall {
    float4 t;      // Euler: addends; Heun: cos, sin, cos, sin
    float2 rr;     // Heun: the two radii
    __device__ __forceinline__ void store(float *block, int lane, int h) const {
        reinterpret_cast<float4 *>(block)[32 * h + lane] = t;
        if constexpr (H == kHeun) reinterpret_cast<float2 *>(block + 16 * 32)[32 * h + lane] = rr;
    }
    __device__ __forceinline__ void load(const float *block, int lane, int h) {
        t = reinterpret_cast<const float4 *>(block)[32 * h + lane];
        if constexpr (H == kHeun) rr = reinterpret_cast<const float2 *>(block + 16 * 32)[32 * h + lane];
    }
};

// Steps of call h of a block.
template <int M, int H, int R, typename F>
__device__ __forceinline__ void four_steps(Lane &L, int h, const TailCall<H> &n, float gs, float gsl, F after) {
    const float t[4] = {n.t.x, n.t.y, n.t.z, n.t.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int s = 4 * h + q;
        if constexpr (H == kEuler)
            step_euler<M>(L.r, L.v, t[q], L.dt, L.A, __fmul_rn(-L.amp, L.dt));
        else
            step_f32<M, H>(L.r, L.v, q < 2 ? n.rr.x : n.rr.y, t[q], bias_b0<H, R>(gs, gsl, s),
                           bias_b1<H, R>(gs, gsl, s), L.dt, L.A, L.amp);
        after(s);
    }
}

static_assert(kTailGroupsMax <= kNumKinds, "the packing keeps the groups' kinds in count[]");
// The packed lanes and, behind them, the noise of the groups (a CTA's dynamic shared memory).
extern __shared__ __align__(16) unsigned char tail_mem[];
__device__ __forceinline__ TailLane *tail_lanes() { return reinterpret_cast<TailLane *>(tail_mem); }
__device__ __forceinline__ float *tail_group_noise(int group) {
    return reinterpret_cast<float *>(tail_mem + kTailGroupsMax * 32 * sizeof(TailLane)) +
           group * kTailRing * kNoiseBlockMax;
}
struct TailShared {
    int count[kNumKinds];                   // lanes per kind (of the packing that is under way)
    int kind[32];                           // of each group (a CTA has at most 32 warps)
    int alive[kTailGroupsMax];              // its lanes with a trajectory, after a round
    int stop[2][kTailGroupsMax];            // group done, by parity of the chunk
};
__shared__ TailShared tail_sh;

// Groups of 32 lanes of one kind that the CTA's trajectories make (CTA-collective); `base` gets
// the place of this warp's first lane among the lanes of its kind, `at` its kind's first group.
__device__ __forceinline__ int tail_count(Lane (&L)[1], int (&count)[kNumKinds], int kind, int &base, int &at) {
    __syncthreads();
    if (threadIdx.x < kNumKinds) count[threadIdx.x] = 0;
    __syncthreads();
    const unsigned held = __ballot_sync(kFull, L[0].slot >= 0);
    base = 0;
    if (held) {
        if ((threadIdx.x & 31) == 0) base = atomicAdd(&count[kind], __popc(held));
        base = __shfl_sync(kFull, base, 0);
    }
    __syncthreads();
    int groups = 0;
    at = 0;
    for (int k = 0; k < kNumKinds; ++k) {
        if (k == kind) at = groups;
        groups += (count[k] + 31) >> 5;
    }
    return groups;
}

// Packs the CTA's trajectories into groups of 32 of one kind in shared memory (CTA-collective) and
// returns how many there are.  No more than the CTA has warps: each warp's trajectories are of one
// kind, so packing never takes more groups than the warps that held them.
__device__ __forceinline__ int tail_pack(Lane (&L)[1], int kind) {
    const int lane = threadIdx.x & 31;
    int base, at;
    const int groups = tail_count(L, tail_sh.count, kind, base, at);
    TailLane *lanes = tail_lanes();
    for (int i = threadIdx.x; i < 32 * groups; i += blockDim.x) lanes[i].slot = -1;
    __syncthreads();
    const unsigned have = __ballot_sync(kFull, L[0].slot >= 0);
    if (L[0].slot >= 0) {
        TailLane &P = lanes[32 * at + base + __popc(have & ((1u << lane) - 1u))];
        P.r = L[0].r;
        P.v = L[0].v;
        P.w = L[0].w;
        P.slot = L[0].slot;
        P.c_lo = L[0].c_lo;
        P.c_hi = L[0].c_hi;
        P.gid_lo = L[0].gid_lo;
        P.gid_hi = L[0].gid_hi;
        P.fin = kTailRuns;
    }
    if (threadIdx.x == 0)
        for (int k = 0, g = 0; k < kNumKinds; ++k)
            for (int n = tail_sh.count[k]; n > 0; n -= 32) tail_sh.kind[g++] = k;
    __syncthreads();
    return groups;
}

// More groups than tail_run takes: they go on in as many full warps (CTA-collective).
__device__ __forceinline__ void tail_spread(Lane (&L)[1], const EngineDev &E, const CtaView &V, int groups, int &kind,
                                            int &n_active) {
    const int warp = static_cast<int>(threadIdx.x >> 5), lane = threadIdx.x & 31;
    set_idle(L[0]);
    n_active = 0;
    kind = -1;
    int act = 0;
    if (warp < groups) {
        kind = tail_sh.kind[warp];
        const TailLane T = tail_lanes()[32 * warp + lane];
        if (T.slot >= 0) {
            resume_from(L[0], E, T.slot, T);
            n_active = 1;
        }
        act = __popc(__ballot_sync(kFull, n_active > 0));
    }
    if (lane == 0) {
        V.warp_act[warp] = act;
        V.warp_knd[warp] = kind < 0 ? 0 : kind;
    }
    if (threadIdx.x == 0) *V.tail = 0;
    __syncthreads();
}

// Lane state between launches.
template <typename State>
__device__ __forceinline__ void store_lane(const EngineDev &E, unsigned i, const State &L) {
    if (!checked(E, i < E.n_lanes, kChkLane)) return;
    E.lanes.slot[i] = L.slot;
    if (L.slot < 0) return;
    E.lanes.r[i] = L.r;
    E.lanes.v[i] = L.v;
    E.lanes.w[i] = L.w;
    E.lanes.c_lo[i] = L.c_lo;
    E.lanes.c_hi[i] = L.c_hi;
    E.lanes.gid_lo[i] = L.gid_lo;
    E.lanes.gid_hi[i] = L.gid_hi;
}
__device__ __forceinline__ void load_lane(Lane &L, const EngineDev &E, unsigned i, int s) {
    TailLane T;
    T.r = E.lanes.r[i];
    T.v = E.lanes.v[i];
    T.w = E.lanes.w[i];
    T.c_lo = E.lanes.c_lo[i];
    T.c_hi = E.lanes.c_hi[i];
    T.gid_lo = E.lanes.gid_lo[i];
    T.gid_hi = E.lanes.gid_hi[i];
    resume_from(L, E, s, T);
}

// A warp's share of the launch's counters (warp-collective).
__device__ __forceinline__ void add_counters(const EngineDev &E, unsigned long long useful, unsigned n_esc, unsigned n_cens) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        useful += __shfl_down_sync(kFull, useful, off);
        n_esc += __shfl_down_sync(kFull, n_esc, off);
        n_cens += __shfl_down_sync(kFull, n_cens, off);
    }
    if ((threadIdx.x & 31) == 0) {
        if (useful) atomicAdd(&E.counters[kCntUseful], useful);
        if (n_esc) atomicAdd(&E.counters[kCntEscapes], static_cast<unsigned long long>(n_esc));
        if (n_cens) atomicAdd(&E.counters[kCntCensored], static_cast<unsigned long long>(n_cens));
    }
}

// One round of a group's integrating warp: its lanes from shared memory and back, results left
// there.  A call's registers are loaded with the next block's noise
// as soon as its steps are done, so the loads are off the chain; the rare replay reads its block
// again.
template <int M, int H, int R>
__device__ __forceinline__ void tail_integrate(const EngineDev &E, int group, int round) {
    const int lane = threadIdx.x & 31;
    const float *noise = tail_group_noise(group);
    TailShared &sh = tail_sh;
    unsigned long long useful = 0;
    unsigned n_esc = 0, n_cens = 0;
    Lane L;
    TailLane &T = tail_lanes()[32 * group + lane];
    set_idle(L);
    L.c_lo = 0u;
    if (T.slot >= 0) resume_from(L, E, T.slot, T);
    float gs, gsl;   // Heun's bias line; an Euler step finds its bias in the noise
    bias_line(fmaf(L.nudt, L.Jf, L.gb), L.nudt, L.dt, gs, gsl);
    const float *end = noise + kTailRing * kNoiseBlock<H>, *cur = noise;   // this block's noise
    TailCall<H> calls[kBlockPhilox];
    group_barrier(group);
#pragma unroll
    for (int h = 0; h < kBlockPhilox; ++h) calls[h].load(cur, lane, h);
    int b = 0, left = kTailChunk;   // blocks done, blocks left of the chunk
    for (int parity = 0;;) {
        if constexpr (R && H == kHeun) bias_line(fmaf(L.nudt, L.Jf, L.gb), L.nudt, L.dt, gs, gsl);
        const float *next = cur + kNoiseBlock<H> == end ? noise : cur + kNoiseBlock<H>;
        const float r0 = L.r, v0 = L.v;
        float mx = -INFINITY;
#pragma unroll
        for (int h = 0; h < kBlockPhilox; ++h) {
            four_steps<M, H, R>(L, h, calls[h], gs, gsl, [&](int) { mx = fmaxf(mx, L.r); });
            calls[h].load(next, lane, h);
        }
        L.c_lo += kBlockPhilox;
        if constexpr (R) L.Jf += static_cast<float>(kBlockSteps);
        L.budget -= 1u;
        ++b;
        // Each lane sees to its own event: nothing in here needs the warp, and the vote that
        // run_blocks takes would hold up the chain at every block.
        if (mx >= L.hb || L.budget == 0u || L.r < -kPiF) {
            if (mx >= L.hb) {
                L.r = r0;
                L.v = v0;
#pragma unroll
                for (int h = 0; h < kBlockPhilox; ++h) {
                    TailCall<H> again;
                    again.load(cur, lane, h);
                    four_steps<M, H, R>(L, h, again, gs, gsl, [&](int s) {
                        if (L.r >= L.hb) phase_event(L, E, s);
                    });
                }
            }
            if (L.r < -kPiF) wrap_down(L, E);
            if (L.c_lo == 0u) L.c_hi += 1u;   // 2^32-block carry
            if (L.slot >= 0 && (L.esc >= 0 || L.budget == 0u)) {
                bool escaped = false;
                unsigned long long k = 0ull;
                if (finished(L, E, 0u, escaped, k, useful)) {
                    useful += static_cast<unsigned long long>(kBlockSteps) * static_cast<unsigned>(b);
                    T.fin = escaped ? kTailEscaped : kTailCensored;
                    T.c_lo = static_cast<unsigned>(k);
                    T.c_hi = static_cast<unsigned>(k >> 32);
                    if (escaped) ++n_esc;
                    else ++n_cens;
                    set_idle(L);
                }
            }
            if constexpr (!R && H == kHeun) bias_line(fmaf(L.nudt, L.Jf, L.gb), L.nudt, L.dt, gs, gsl);
        }
        cur = next;
        if (--left == 0 || b == round) {
            // Every warp of the group passes the same barriers: the verdict on a chunk lies in the
            // slot of its parity, written again only after the barrier that follows.
            const bool over = !__any_sync(kFull, L.slot >= 0);
            if (lane == 0) sh.stop[parity][group] = over ? 1 : 0;
            group_barrier(group);
            if (over || b == round) break;
            parity ^= 1;
            left = kTailChunk;
        }
    }
    if (L.slot >= 0) useful += static_cast<unsigned long long>(kBlockSteps) * static_cast<unsigned>(b);
    if (L.slot >= 0) {
        T.r = L.r;
        T.v = L.v;
        T.w = L.w;
        T.c_lo = L.c_lo;
        T.c_hi = L.c_hi;
    }
    const int alive = __popc(__ballot_sync(kFull, L.slot >= 0));
    if (lane == 0) sh.alive[group] = alive;
    add_counters(E, useful, n_esc, n_cens);
}

// One round of one of a group's noise warps: block `rank` of every chunk, two chunks ahead of the
// integrating warp.  Euler's addends take the bias line of set_progress and run_blocks: the base is
// formed anew when the block count reaches a multiple of kRebaseBlocks.
template <int H, int R>
__device__ __forceinline__ void tail_noise(const EngineDev &E, int group, int rank, int round) {
    const int lane = threadIdx.x & 31;
    float *ring = tail_group_noise(group);
    const TailLane &T = tail_lanes()[32 * group + lane];
    const SlotDev *S = E.slots + (T.slot >= 0 ? T.slot : 0);
    unsigned key0 = 0u, key1 = 0u, gid_lo = 0u, gid_hi = 0u, lo = 0u, hi = 0u;
    float bmc = 0.0f, dt = 0.0f, nudt = 0.0f;
    if (T.slot >= 0) {
        key0 = S->key0;
        key1 = S->key1;
        bmc = S->bmc;
        dt = S->dt;
        nudt = S->nudt;
        gid_lo = T.gid_lo;
        gid_hi = T.gid_hi;
        const unsigned long long c = ((static_cast<unsigned long long>(T.c_hi) << 32) | T.c_lo) +
                                     static_cast<unsigned>(kBlockPhilox * rank);
        lo = static_cast<unsigned>(c);
        hi = static_cast<unsigned>(c >> 32);
    }
    PhiloxLane P;
    philox_lane_init(P, key0, key1, hi, gid_lo, gid_hi);
    // keep the round keys in registers: formed again at each use they cost four instructions per step
#pragma unroll
    for (int r = 0; r < 8; ++r) asm volatile("" : "+r"(P.ka[r]));
#pragma unroll
    for (int r = 0; r < 7; ++r) asm volatile("" : "+r"(P.kb[r]));
    constexpr unsigned step = kBlockPhilox * kTailMakers;
    float gb = 0.0f, Jf = 0.0f, gs = 0.0f, gsl = 0.0f;
    const auto rebase = [&]() {   // bias base and steps since it at block count (hi : lo)
        const unsigned long long c = (static_cast<unsigned long long>(hi) << 32) | lo, cb = c - c % kRebaseBlocks;
        gb = static_cast<float>(S->gamma0 + S->nudt_d * static_cast<double>(4ull * cb));
        Jf = static_cast<float>(4ull * (c - cb));
        bias_line(fmaf(nudt, Jf, gb), nudt, dt, gs, gsl);
    };
    if constexpr (H == kEuler) rebase();
    const float *end = ring + kTailRing * kNoiseBlock<H>;
    float *block = ring + rank * kNoiseBlock<H>;
    int to_go = round - rank;                        // blocks from this one to the round's end
    for (int i = -2; kTailChunk * i < round; ++i) {   // makes chunk i + 2 while chunk i is used
        if (to_go > 0) {
            if constexpr (H == kEuler && R) bias_line(fmaf(nudt, Jf, gb), nudt, dt, gs, gsl);
#pragma unroll
            for (int h = 0; h < kBlockPhilox; ++h) {
                const uint4 x = philox_lane_block(P, lo, static_cast<unsigned>(h));
                TailCall<H> n;
                bm_pair_f32(x.x, x.y, bmc, n.rr.x, n.t.x, n.t.y);
                bm_pair_f32(x.z, x.w, bmc, n.rr.y, n.t.z, n.t.w);
                if constexpr (H == kEuler) {
                    n.t.x = fmaf(n.rr.x, n.t.x, bias_b1<H, R>(gs, gsl, 4 * h));
                    n.t.y = fmaf(n.rr.x, n.t.y, bias_b1<H, R>(gs, gsl, 4 * h + 1));
                    n.t.z = fmaf(n.rr.y, n.t.z, bias_b1<H, R>(gs, gsl, 4 * h + 2));
                    n.t.w = fmaf(n.rr.y, n.t.w, bias_b1<H, R>(gs, gsl, 4 * h + 3));
                }
                n.store(block, lane, h);
            }
        }
        to_go -= kTailMakers;
        block += kTailChunk * kNoiseBlock<H>;
        if (block >= end) block -= kTailRing * kNoiseBlock<H>;
        lo += step;
        Jf += static_cast<float>(4u * step);
        // past a multiple of kRebaseBlocks: another bias base; past 2^32: new fixed words
        if (__any_sync(kFull, (lo & (kRebaseBlocks - 1u)) < step)) {
            if (lo < step) {
                ++hi;
                PhiloxLane Q;
                philox_lane_init(Q, key0, key1, hi, gid_lo, gid_hi);
                P.m0 = Q.m0;
                P.x1m = Q.x1m;
                P.z1m = Q.z1m;
                P.z2m = Q.z2m;
            }
            if constexpr (H == kEuler) rebase();
        }
        if (i == -2) continue;   // the first barrier follows the second chunk
        group_barrier(group);
        if (i >= 0 && tail_sh.stop[i & 1][group]) break;
    }
}
static_assert((kRebaseBlocks & (kRebaseBlocks - 1u)) == 0u, "re-bases are found by a mask");
static_assert(kTailChunk == kTailMakers, "a noise warp makes one block of each chunk");

// Runs the CTA's trajectories, `groups` packed groups of them, at most `blocks` blocks of each, to
// the end of the launch (CTA-collective), and leaves the rest in the lane state if there is one.
// K: the kind of every group, or -1.
template <int K>
__device__ __noinline__ void tail_run(const EngineDev &E, int *held, int groups, unsigned long long blocks) {
    TailShared &sh = tail_sh;
    TailLane *lanes = tail_lanes();
    const int warp = static_cast<int>(threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int warps = static_cast<int>(blockDim.x >> 5);
    const unsigned gtid = blockIdx.x * blockDim.x + threadIdx.x;
    unsigned most = kRoundBlocks;
    while (blocks > 0 && groups > 0) {
        // Roles.  Euler: warp 4 g integrates group g (scheduler 0), the warps of the other
        // schedulers make noise, the m-th of them for group m mod groups.  A Heun step's two sines
        // take ~17 cycles of a scheduler: warp 2 g integrates (schedulers 0 and 2), the odd warps
        // make noise and then the even ones that are left (four groups: 44 -> 33 ns per step).
        bool heun = false;
        for (int g = 0; g < groups; ++g) heun |= (sh.kind[g] & 2) != 0;
        const int spread = heun ? 2 : 4;
        const bool integrates = warp % spread == 0 && warp / spread < groups;
        int m;
        if (!heun) m = (warp & 3) == 0 ? 3 * kTailGroupsMax : (warp >> 2) * 3 + (warp & 3) - 1;
        else m = (warp & 1) ? warp >> 1 : (warps >> 1) + (warp >> 1) - groups;
        const int group = integrates ? warp / spread : m % groups;
        const int rank = m / groups;
        const int round = round_blocks(blocks, most);
        if (integrates) {
            if constexpr (K >= 0) tail_integrate<(K & 1), ((K >> 1) & 1), (K >> 2)>(E, group, round);
            else switch (sh.kind[group]) {
#define FPT_KIND_CASE(M_, H_, R_) \
    case kind_of(M_, H_, R_): tail_integrate<M_, H_, R_>(E, group, round); break;
            FPT_KIND_CASE(kUnder, kEuler, kConstBias)
            FPT_KIND_CASE(kOver, kEuler, kConstBias)
            FPT_KIND_CASE(kUnder, kHeun, kConstBias)
            FPT_KIND_CASE(kOver, kHeun, kConstBias)
            FPT_KIND_CASE(kUnder, kEuler, kRamp)
            FPT_KIND_CASE(kOver, kEuler, kRamp)
            FPT_KIND_CASE(kUnder, kHeun, kRamp)
#undef FPT_KIND_CASE
            default: tail_integrate<kOver, kHeun, kRamp>(E, group, round); break;
            }
        } else if (rank < kTailMakers) {
            const int k = K >= 0 ? K : sh.kind[group];
            if (k & 2) tail_noise<kHeun, kConstBias>(E, group, rank, round);
            else if (k & 4) tail_noise<kEuler, kRamp>(E, group, rank, round);
            else tail_noise<kEuler, kConstBias>(E, group, rank, round);
        }
        blocks -= static_cast<unsigned>(round);
        __syncthreads();
        if (warp < groups) {   // publish the round's results
            TailLane &T = lanes[32 * warp + lane];
            const bool fin = T.slot >= 0 && T.fin != kTailRuns;
            emit_warp(E, held, fin, T.slot, (static_cast<unsigned long long>(T.gid_hi) << 32) | T.gid_lo,
                      T.fin == kTailEscaped, (static_cast<unsigned long long>(T.c_hi) << 32) | T.c_lo);
            if (fin) T.slot = -1;
        }
        int fewer = 0;
        for (int g = 0, n = 0; g < groups; ++g) {
            n += sh.alive[g];
            if (g + 1 == groups || sh.kind[g + 1] != sh.kind[g]) {
                fewer += (n + 31) >> 5;
                n = 0;
            }
        }
        __syncthreads();
        if (fewer == groups) {
            most = longer_round(most);
            continue;
        }
        most = kRoundBlocks;
        if (warp == 0) {   // close the gaps: entries only move down, past what has been read
            int to = 0;    // next place
            for (int g = 0; g < groups; ++g) {
                const int k = sh.kind[g];
                if (g > 0 && k != sh.kind[g - 1]) {   // a new kind starts a new group
                    const int pad = (32 - (to & 31)) & 31;
                    if (lane < pad) lanes[to + lane].slot = -1;
                    to += pad;
                }
                const TailLane T = lanes[32 * g + lane];
                const unsigned m = __ballot_sync(kFull, T.slot >= 0);
                __syncwarp();
                if (T.slot >= 0) lanes[to + __popc(m & ((1u << lane) - 1u))] = T;
                __syncwarp();
                const int first = (to + 31) >> 5, last = (to + __popc(m) + 31) >> 5;   // groups this one begins
                if (lane == 0)
                    for (int q = first; q < last; ++q) sh.count[q] = k;   // kinds of the new groups
                to += __popc(m);
            }
            const int pad = (32 - (to & 31)) & 31;
            if (lane < pad) lanes[to + lane].slot = -1;
            __syncwarp();
            if (lane < fewer) sh.kind[lane] = sh.count[lane];
        }
        groups = fewer;
        __syncthreads();
    }
    if (!E.lanes.slot) return;
    // back into the lane state: group g in warp g
    TailLane T{};
    T.slot = -1;
    if (warp < groups) T = lanes[32 * warp + lane];
    store_lane(E, gtid, T);
    if (lane == 0) E.warp_kind[gtid >> 5] = warp < groups ? sh.kind[warp] : -1;
}

// One trajectory per thread runs best as one CTA of 640 threads per SM: 20 warps, five per
// scheduler, at 96 registers (measured against 512, 576, 672 and 768); two per thread as CTAs
// of up to 256.
// kTail: with the packed last trajectories.  Their named barriers count as all 16 of a CTA, which an SM
// has for four CTAs: small CTAs, which run no groups, get the kernel without (one to four warps: 16, 10,
// 6 and 5 CTAs per SM; the sweep at 32 / 64 / 128 threads with four: 493 / 821 / 1012 Gstep/s, so:
// 986 / 1034 / 1039).
template <int T, bool kTail>
__global__ void __launch_bounds__(T == 1 ? 640 : 256, 1) engine_chunk_kernel(const __grid_constant__ EngineDev E) {
    const unsigned nthreads = gridDim.x * blockDim.x;
    const unsigned gtid = blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned warp = gtid >> 5;
    const int lane = threadIdx.x & 31;
    // This CTA's view of the requests for the launch: which listed requests have ids or suspended
    // trajectories to hand out, and how many of its lanes hold each.
    __shared__ unsigned sh_ok[kMaxRequests];
    __shared__ int sh_held[kMaxRequests], sh_budget[kMaxRequests];
    __shared__ int sh_res_slot[32], sh_res_cnt[32], sh_started[32];   // a CTA has at most 32 warps
    __shared__ unsigned long long sh_res_base[32];
    __shared__ int sh_pool;
    __shared__ unsigned sh_chunk, sh_share;
    __shared__ int sh_warp_act[32], sh_warp_knd[32], sh_tail, sh_done, sh_act_count[kNumKinds], sh_flags[2], sh_tail_groups;
    // while caps are enforced the lanes that idle are meant to
    const int tail_groups = !kTail || *E.strict != 0 ? 0 : tail_groups_of(T, static_cast<int>(blockDim.x >> 5));
    const CtaView V{sh_ok, sh_held, sh_budget, sh_res_slot, sh_res_cnt, sh_res_base, sh_started, &sh_pool,
                    sh_warp_act, sh_warp_knd, &sh_share, &sh_tail, &sh_tail_groups, sh_act_count, sh_flags};
    for (int s = threadIdx.x; s < E.max_requests; s += blockDim.x) {
        sh_ok[s] = 0u;
        sh_held[s] = 0;
        sh_budget[s] = 0;
    }
    if (threadIdx.x == 0) {
        sh_pool = 0;
        sh_tail = 0;
        sh_done = 0;
        sh_tail_groups = tail_groups;
        // blocks per warp of this launch: the engine's full launch or a shorter one it chose
        const unsigned c = static_cast<unsigned>(*E.chunk_now);
        sh_chunk = c == 0u || c > E.chunk_blocks ? E.chunk_blocks : c;
        sh_share = sh_chunk - sh_chunk / kPoolDiv;
    }
    // this thread's lanes and this warp's kind, asked for before they are needed
    int lane_slot[T];
#pragma unroll
    for (int t = 0; t < T; ++t)
        lane_slot[t] = checked(E, t * nthreads + gtid < E.n_lanes, kChkLane) ? E.lanes.slot[t * nthreads + gtid] : -1;
    int kind = E.warp_kind[warp];
    unsigned cursor = E.warp_cursor[warp];
    if (threadIdx.x < kNumKinds) sh_act_count[threadIdx.x] = E.act_count[threadIdx.x];
    if (threadIdx.x < 2) sh_flags[threadIdx.x] = threadIdx.x == 0 ? *E.strict : *E.claim_warps;
    if (threadIdx.x < 32) {
        sh_res_slot[threadIdx.x] = -1;
        sh_res_cnt[threadIdx.x] = 0;
        sh_res_base[threadIdx.x] = 0ull;
        sh_started[threadIdx.x] = 0;
        sh_warp_act[threadIdx.x] = 0;
        sh_warp_knd[threadIdx.x] = 0;
    }
    __syncthreads();
    int listed = 0;
    for (int k = 0; k < kNumKinds; ++k) listed += sh_act_count[k];
    const auto listed_slot = [&](int i) {
        int k = 0;
        while (i >= sh_act_count[k]) i -= sh_act_count[k++];
        return E.act_list[k * E.max_requests + i];
    };
    {
        for (int i = threadIdx.x; i < listed; i += blockDim.x) {
            const int s = listed_slot(i);
            const SlotCtl &C = E.ctl[s];
            if (vload(C.state) != kSlotActive) continue;
            sh_ok[s] = (vload(C.head) < claim_end(E.slots[s].n_traj, E.slots[s].stop_block, C.claim_blocks) ? 1u : 0u) |
                       (vload(C.park_avail) > 0 ? 2u : 0u);
            // reservoir room: what the ring can still take beyond one entry per lane (the most
            // suspensions of this launch could add), shared equally by the CTAs
            const long long room = static_cast<long long>(E.slots[s].park_cap) - vload(C.park_used) -
                                   static_cast<long long>(E.n_lanes);
            sh_budget[s] = room > 0 ? static_cast<int>(room / gridDim.x) : 0;
        }
    }
    Lane L[T];
    int n_active = 0;
#pragma unroll
    for (int t = 0; t < T; ++t) {
        const unsigned i = t * nthreads + gtid;
        int s = lane_slot[t];
        if (s >= 0 && !checked(E, s < E.max_requests, kChkSlot)) s = -1;
        if (s >= 0 && vload(E.ctl[s].state) != kSlotActive) {   // request finished or cancelled
            atomicSub(&E.ctl[s].inflight, 1);
            s = -1;
        }
        if (s < 0) {
            set_idle(L[t]);
            continue;
        }
        load_lane(L[t], E, i, s);
        atomicAdd(&sh_held[s], 1);
        ++n_active;
    }
    __syncthreads();
    if (kind >= 0 && !checked(E, kind < kNumKinds, kChkKind)) kind = -1;
    if (!__any_sync(kFull, n_active > 0)) kind = -1;
    unsigned long long useful = 0;
    unsigned n_esc = 0, n_cens = 0;
    unsigned b = 0;
    if (kind >= 0) refill(L, E, V, kind, n_active, cursor, 0u);
    else kind = seek_work(L, E, V, n_active, cursor, 0u);
    // The CTA's pool holds the last 1/kPoolDiv of the launch's blocks of every warp that has work
    // now, so a CTA whose warps are partly idle (fewer trajectories than lanes) gives its busy
    // warps as many blocks as a full CTA does, and all CTAs end together.
    if (lane == 0 && kind >= 0) atomicAdd(&sh_pool, static_cast<int>(sh_chunk / kPoolDiv));
    {
        const unsigned m = __ballot_sync(kFull, n_active > 0);
        if (lane == 0) {
            sh_warp_act[threadIdx.x >> 5] = __popc(m);
            sh_warp_knd[threadIdx.x >> 5] = kind < 0 ? 0 : kind;
        }
    }
    // Dry from the start?  The queue heads as they are after this CTA's first claims.  One warp decides
    // for all, between two barriers: the counts it reads change as soon as a warp runs on.  Then they go
    // straight to the meeting.
    bool dry = false;
    {
        bool work = false;
        for (int i = threadIdx.x; i < listed; i += blockDim.x) {
            const int s = listed_slot(i);
            unsigned ok = vload(sh_ok[s]);
            if (T == 1 && (ok & 1u) &&
                vload(E.ctl[s].head) >= claim_end(E.slots[s].n_traj, E.slots[s].stop_block, E.ctl[s].claim_blocks))
                ok = atomicAnd(&sh_ok[s], ~1u) & ~1u;
            work |= (ok & 3u) != 0u;
        }
        work = __syncthreads_or(work) != 0;
        if (kTail && tail_groups > 0 && !work) {
            dry = __syncthreads_or(threadIdx.x < 32 && thinned_out(V)) != 0;
            if (dry && threadIdx.x == 0) sh_tail = 1;
        }
    }
    unsigned limit = 0;
    for (bool again = true; again;) {   // again: the warps have met and go on with fewer of them
        again = false;
        while (!dry && (b < limit || more(V, limit))) {
            if (kind < 0) {
                kind = seek_work(L, E, V, n_active, cursor, b);
                if (kind < 0) break;
                look_dry(L, E, V, kind);
            }
            switch (kind) {
#define FPT_KIND_CASE(M_, H_, R_)                                                              \
        case kind_of(M_, H_, R_):                                                                \
            b = run_blocks<M_, H_, R_, T>(L, E, V, b, n_active, cursor, useful, n_esc, n_cens, limit); \
            break;
            FPT_KIND_CASE(kUnder, kEuler, kConstBias)
            FPT_KIND_CASE(kOver, kEuler, kConstBias)
            FPT_KIND_CASE(kUnder, kHeun, kConstBias)
            FPT_KIND_CASE(kOver, kHeun, kConstBias)
            FPT_KIND_CASE(kUnder, kEuler, kRamp)
            FPT_KIND_CASE(kOver, kEuler, kRamp)
            FPT_KIND_CASE(kUnder, kHeun, kRamp)
            default:
                b = run_blocks<kOver, kHeun, kRamp, T>(L, E, V, b, n_active, cursor, useful, n_esc, n_cens, limit);
                break;
#undef FPT_KIND_CASE
            }
            if (kTail && !__all_sync(kFull, L[0].slot >= 0)) look_dry(L, E, V, kind);
            if (!__any_sync(kFull, n_active > 0)) kind = -1;
        }
        // Ids left in this warp's reservoir go back to their request as suspended trajectories that
        // have not started (state r0, v0, w0 at step 0: resuming one is starting it).  The CTA's
        // budget kept the ring's room for them.  Before the meeting: a warp that goes on from there
        // finds the claim flags cleared, so no reservoir is filled again, and tail_run ends the launch.
        {
            __syncwarp();
            const int wl = static_cast<int>(threadIdx.x >> 5);
            const int rs = sh_res_slot[wl], rc = sh_res_cnt[wl];
            if (rs >= 0 && rc > 0 && checked(E, rs < E.max_requests, kChkSlot)) {
                SlotCtl *C = E.ctl + rs;
                const SlotDev *S = E.slots + rs;
                for (int j = lane; j < rc; j += 32) {
                    const unsigned long long gid = S->traj_offset + sh_res_base[wl] + static_cast<unsigned long long>(j);
                    const int used = atomicAdd(&C->park_used, 1);
                    checked(E, used < static_cast<int>(S->park_cap), kChkPark);   // the budget's invariant
                    const unsigned pi = atomicAdd(&C->park_tail, 1u);
                    if (!checked(E, pi % S->park_cap < S->park_cap, kChkPark)) continue;
                    ParkEntry &P = S->park[pi % S->park_cap];
                    P.r = S->r0;
                    P.v = S->v0;
                    P.w = S->w0;
                    P.c_lo = P.c_hi = 0u;
                    P.gid_lo = static_cast<unsigned>(gid);
                    P.gid_hi = static_cast<unsigned>(gid >> 32);
                    P.pad = 0;
                }
            }
            __syncwarp();
            if (lane == 0) sh_res_cnt[wl] = 0;
        }
        if constexpr (kTail) {
            if (tail_groups > 0) {
                // the blocks left in this launch, after the furthest of the warps with trajectories
                if (lane == 0 && kind >= 0) atomicMax(&sh_done, static_cast<int>(b));
                __syncthreads();
                checked(E, !dry || sh_tail != 0, kChkDry);
                if (sh_tail != 0) {
                    const int groups = tail_pack(L, kind);
                    if (groups <= tail_groups) {
                        checked(E, vload(sh_res_cnt[threadIdx.x >> 5]) == 0, kChkReservoir);
                        if (lane == 0) E.warp_cursor[warp] = cursor;
                        add_counters(E, useful, n_esc, n_cens);
                        const unsigned done = static_cast<unsigned>(sh_done);
                        tail_run<-1>(E, sh_held, groups, sh_chunk > done ? sh_chunk - done : 0u);
                        return;
                    }
                    tail_spread(L, E, V, groups, kind, n_active);
                    dry = false;
                    again = true;
                }
            }
        }
    }
    // Preemption: a whole warp of this kind may be asked to vacate (so it can switch kind),
    // or single lanes of requests above their share to suspend.  Suspended state goes to the
    // request's ring; a push needs a free ring entry (park_used < park_cap).
    bool vacate = false;
    if (kind >= 0 && __any_sync(kFull, n_active > 0)) {
        int v = 0;
        if (lane == 0 && vload(E.vacate[kind]) > 0) v = atomicSub(&E.vacate[kind], 1) > 0 ? 1 : 0;
        vacate = __shfl_sync(kFull, v, 0) != 0;
    }
#pragma unroll
    for (int t = 0; t < T; ++t) {
        const int s = L[t].slot;
        if (s < 0) continue;
        bool park = vacate;
        if (!park && vload(E.preempt[s]) > 0) park = atomicSub(&E.preempt[s], 1) > 0;
        if (!park) continue;
        SlotCtl *C = E.ctl + s;
        const SlotDev *S = E.slots + s;
        if (atomicAdd(&C->park_used, 1) >= static_cast<int>(S->park_cap)) {
            atomicSub(&C->park_used, 1);
            continue;
        }
        const unsigned pi = atomicAdd(&C->park_tail, 1u);
        if (!checked(E, pi % S->park_cap < S->park_cap, kChkPark)) continue;
        ParkEntry &P = S->park[pi % S->park_cap];
        P.r = L[t].r;
        P.v = L[t].v;
        P.w = L[t].w;
        P.c_lo = L[t].c_lo;
        P.c_hi = L[t].c_hi;
        P.gid_lo = L[t].gid_lo;
        P.gid_hi = L[t].gid_hi;
        P.pad = 0;
        atomicSub(&C->inflight, 1);
        L[t].slot = -1;
        --n_active;
    }
    if (!__any_sync(kFull, n_active > 0)) kind = -1;
#pragma unroll
    for (int t = 0; t < T; ++t) store_lane(E, t * nthreads + gtid, L[t]);
    if (lane == 0) {
        E.warp_kind[warp] = kind;
        E.warp_cursor[warp] = cursor;
    }
    add_counters(E, useful, n_esc, n_cens);
}

__device__ __forceinline__ double u128_to_d(unsigned long long lo, unsigned long long hi) {
    return __dadd_rn(__dmul_rn(static_cast<double>(hi), 18446744073709551616.0),
                     static_cast<double>(lo));
}

// lo:hi (128 bits) += l0 + 2^32 l1 + 2^64 l2, exactly (l0, l1, l2 < 2^64).
__device__ __forceinline__ void add_limbs(unsigned long long &lo, unsigned long long &hi, unsigned long long l0,
                                          unsigned long long l1, unsigned long long l2) {
    const unsigned long long a = l1 << 32, ah = l1 >> 32;   // 2^32 l1 = ah:a
    lo += l0;
    hi += lo < l0 ? 1ull : 0ull;
    lo += a;
    hi += ah + (lo < a ? 1ull : 0ull) + l2;
}

// ---- one request without an engine ------------------------------------------------------------
// fpt_run_noalloc on the machinery above: each CTA is an engine of its own for a contiguous range of the ids, its slot,
// queue and accumulators in shared memory, so a call needs no scratch in device memory and shares
// nothing with other calls; it runs until its range is done and adds its exact sums and counts to
// the caller's.  Ranges of equal size differ in length by a few percent, less than the last
// trajectories take.  Against one event test per step, a full Philox per call and one queue for all
// CTAs (256 threads each): 200 003 trajectories of 19 000 steps 17-18 -> 6.0-6.2 ms.
template <int M, int H, int R>
__global__ void __launch_bounds__(kSoloThreads, 1) solo_kernel(const __grid_constant__ SoloArgs a) {
    const int warp = static_cast<int>(threadIdx.x >> 5), lane = threadIdx.x & 31;
    constexpr int kind = kind_of(M, H, R);
    __shared__ SlotDev slot;
    __shared__ SlotCtl ctl;
    __shared__ IdBlockAcc acc;
    __shared__ EngineDev E;
    __shared__ unsigned long long counters[kCntCount], res_base[32];
    __shared__ unsigned ok, share;
    __shared__ int held, budget, pool, tail, max_groups, flags[2], zeros[kNumKinds], counts[kNumKinds];
    __shared__ int res_slot[32], res_cnt[32], started[32], warp_act[32], warp_knd[32];
    unsigned *hist = reinterpret_cast<unsigned *>(tail_mem + tail_shared_bytes(kSoloThreads / 32));
    const CtaView V{&ok, &held, &budget, res_slot, res_cnt, res_base, started, &pool, warp_act, warp_knd, &share, &tail,
                    &max_groups, counts, flags};
    for (int b = threadIdx.x; b < a.nbins; b += blockDim.x) hist[b] = 0u;
    if (threadIdx.x < 32) {
        res_slot[threadIdx.x] = -1;
        res_cnt[threadIdx.x] = started[threadIdx.x] = warp_act[threadIdx.x] = 0;
        warp_knd[threadIdx.x] = kind;
        res_base[threadIdx.x] = 0ull;
    }
    if (threadIdx.x < kNumKinds) {
        zeros[threadIdx.x] = 0;
        counts[threadIdx.x] = threadIdx.x == kind ? 1 : 0;
    }
    if (threadIdx.x == 0) {
        const unsigned long long first = a.n * blockIdx.x / gridDim.x, end = a.n * (blockIdx.x + 1ull) / gridDim.x;
        slot = a.slot;
        slot.n_traj = end;
        slot.acc = &acc;
        slot.hist = a.nbins ? hist : nullptr;
        ctl = SlotCtl{};
        ctl.head = first;
        ctl.state = kSlotActive;
        acc = IdBlockAcc{};
        for (int i = 0; i < kCntCount; ++i) counters[i] = 0ull;
        E = EngineDev{};
        E.slots = &slot;
        E.ctl = &ctl;
        E.act_list = zeros;
        E.counters = counters;
        E.max_requests = 1;
        E.n_lanes = gridDim.x * blockDim.x;
        ok = first < end ? 1u : 0u;
        held = budget = pool = tail = 0;
        share = 0x80000000u;   // blocks before the warps meet in any case (they go on)
        const unsigned long long warps = (end - first + 31) / 32;
        max_groups = tail_groups_of(1, kSoloThreads / 32);
        flags[0] = 0;
        flags[1] = warps < kSoloThreads / 32 ? static_cast<int>(warps) : kSoloThreads / 32;
    }
    __syncthreads();
    Lane L[1];
    set_idle(L[0]);
    int n_active = 0;
    unsigned cursor = 0, n_esc = 0, n_cens = 0;
    unsigned long long useful = 0;
    refill(L, E, V, kind, n_active, cursor, 0u);
    {
        const unsigned m = __ballot_sync(kFull, n_active > 0);
        if (lane == 0) warp_act[warp] = __popc(m);
    }
    __syncthreads();
    if (warp == 0) {
        if (lane == 0 && ctl.head >= slot.n_traj) ok = 0u;
        __syncwarp();
        look_dry(L, E, V, kind);
    }
    for (;;) {
        unsigned b = 0, limit = 0;
        while (__any_sync(kFull, n_active > 0) && (b < limit || more(V, limit))) {
            b = run_blocks<M, H, R, 1>(L, E, V, b, n_active, cursor, useful, n_esc, n_cens, limit);
            if (!__all_sync(kFull, L[0].slot >= 0)) look_dry(L, E, V, kind);
        }
        __syncthreads();
        if (tail != 0) {
            const int groups = tail_pack(L, kind);
            if (groups <= *V.tail_groups) {
                tail_run<kind>(E, &held, groups, ~0ull);
                break;
            }
            int k = kind;
            tail_spread(L, E, V, groups, k, n_active);
            continue;
        }
        if (!__syncthreads_or(n_active > 0)) break;
    }
    __syncthreads();
    if (a.sums && threadIdx.x == 0) {
        unsigned long long s1lo = 0, s1hi = 0, s2lo = 0, s2hi = 0;
        add_limbs(s1lo, s1hi, acc.s1[0], acc.s1[1], 0ull);
        add_limbs(s2lo, s2hi, acc.s2[0], acc.s2[1], acc.s2[2]);
        unsigned long long *o = reinterpret_cast<unsigned long long *>(a.sums);
        atomicAdd(&o[0], static_cast<unsigned long long>(acc.done));
        if (acc.escaped) atomicAdd(&o[1], static_cast<unsigned long long>(acc.escaped));
        const unsigned long long p1 = atomicAdd(&o[2], s1lo);
        if (s1hi + (p1 + s1lo < p1 ? 1ull : 0ull)) atomicAdd(&o[3], s1hi + (p1 + s1lo < p1 ? 1ull : 0ull));
        const unsigned long long p2 = atomicAdd(&o[4], s2lo);
        if (s2hi + (p2 + s2lo < p2 ? 1ull : 0ull)) atomicAdd(&o[5], s2hi + (p2 + s2lo < p2 ? 1ull : 0ull));
        if (acc.under) atomicAdd(&o[6], static_cast<unsigned long long>(acc.under));
        if (acc.over) atomicAdd(&o[7], static_cast<unsigned long long>(acc.over));
    }
    for (int b = threadIdx.x; b < a.nbins; b += blockDim.x)
        if (hist[b]) atomicAdd(&a.hist[b], static_cast<unsigned long long>(hist[b]));
}

// A prefix's exact sums: trajectories, escapes, out-of-range counts, sums of k and k^2.
struct PrefixSums {
    unsigned long long done, esc, under, over, s1_lo, s1_hi, s2_lo, s2_hi;
    __device__ __forceinline__ void add(const PrefixSums &o) {
        done += o.done;
        esc += o.esc;
        under += o.under;
        over += o.over;
        s1_lo += o.s1_lo;
        s1_hi += o.s1_hi + (s1_lo < o.s1_lo ? 1ull : 0ull);
        s2_lo += o.s2_lo;
        s2_hi += o.s2_hi + (s2_lo < o.s2_lo ? 1ull : 0ull);
    }
    __device__ __forceinline__ PrefixSums from(int lane) const {
        PrefixSums r;
        r.done = __shfl_sync(kFull, done, lane);
        r.esc = __shfl_sync(kFull, esc, lane);
        r.under = __shfl_sync(kFull, under, lane);
        r.over = __shfl_sync(kFull, over, lane);
        r.s1_lo = __shfl_sync(kFull, s1_lo, lane);
        r.s1_hi = __shfl_sync(kFull, s1_hi, lane);
        r.s2_lo = __shfl_sync(kFull, s2_lo, lane);
        r.s2_hi = __shfl_sync(kFull, s2_hi, lane);
        return r;
    }
};

// The relative-standard-error rule on a prefix (IEEE double, each operation rounded): whether the
// standard error of the mean is at most stop_rse times the mean; `ids` gets the trajectories that
// the rule is expected to need at this prefix's spread.
__device__ __forceinline__ bool stop_rule(const SlotDev *S, const PrefixSums &P, double &ids) {
    ids = 0.0;
    if (P.esc < 2) return false;
    const double n = static_cast<double>(P.esc);
    const double s1 = u128_to_d(P.s1_lo, P.s1_hi);
    const double s2 = u128_to_d(P.s2_lo, P.s2_hi);
    const double mk = __ddiv_rn(s1, n);
    double vk = __ddiv_rn(__dsub_rn(s2, __dmul_rn(s1, mk)), __dsub_rn(n, 1.0));
    if (vk < 0.0) vk = 0.0;
    const double mx = S->output == FPT_OUT_TIME ? __dmul_rn(S->out_b, mk)
                                                : __dadd_rn(S->out_a, __dmul_rn(S->out_b, mk));
    const double se = __dmul_rn(fabs(S->out_b), __dsqrt_rn(__ddiv_rn(vk, n)));
    const double most = __dmul_rn(S->stop_rse, fabs(mx));
    const double over = se / most;
    ids = static_cast<double>(P.done) * over * over;
    return se <= most;
}

// After a launch, one warp per request: folds its completed id blocks, in id order and 32 at a time
// (each lane one block, sums to its block by a scan over the lanes, the stop rule on each prefix),
// into its running sums; it is finished at the first prefix that meets the rule, or when every
// block is complete.  Then the status of every slot in use and the counters go straight to the
// host's pinned memory, where two copies behind this kernel would each cost a step of the graph.
__global__ void engine_scan_kernel(EngineDev E, SlotCtl *h_ctl, unsigned long long *h_counters) {
    const int s = static_cast<int>((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (blockIdx.x == 0 && threadIdx.x < kCntCount) h_counters[threadIdx.x] = E.counters[threadIdx.x];
    if (s >= E.max_requests) return;
    SlotCtl *C = E.ctl + s;
    const int state = C->state;
    if (state == kSlotFree) return;
    if (state == kSlotActive) {
        const SlotDev *S = E.slots + s;
        const unsigned first = C->prefix;
        unsigned p = first;
        PrefixSums total{C->n_done, C->n_esc, C->under, C->over, C->s1_lo, C->s1_hi, C->s2_lo, C->s2_hi};
        bool finished = false;
        double need = 0.0;   // trajectories the stop rule is expected to take
        while (p < S->n_idblocks) {
            const unsigned ib = p + static_cast<unsigned>(lane);
            PrefixSums mine{};
            bool complete = false;
            if (ib < S->n_idblocks && ib >= p) {
                const unsigned long long left = S->n_traj - static_cast<unsigned long long>(ib) * S->stop_block;
                const unsigned need = left < S->stop_block ? static_cast<unsigned>(left) : S->stop_block;
                const IdBlockAcc &A = S->acc[ib];
                complete = A.done >= need;
                if (complete) {
                    mine.done = A.done;
                    mine.esc = A.escaped;
                    mine.under = A.under;
                    mine.over = A.over;
                    add_limbs(mine.s1_lo, mine.s1_hi, A.s1[0], A.s1[1], 0ull);
                    add_limbs(mine.s2_lo, mine.s2_hi, A.s2[0], A.s2[1], A.s2[2]);
                }
            }
            const unsigned gap = ~__ballot_sync(kFull, complete);
            const int run = gap ? __ffs(gap) - 1 : 32;   // complete blocks from p on
            if (run == 0) break;
            if (lane >= run) mine = PrefixSums{};
            if (lane == 0) mine.add(total);
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const PrefixSums o = mine.from((lane - off) & 31);
                if (lane >= off) mine.add(o);
            }
            double ids = 0.0;
            const bool stop = S->stop_rse > 0.0 && lane < run && stop_rule(S, mine, ids);
            const unsigned stops = __ballot_sync(kFull, stop);
            const int last = stops ? __ffs(stops) - 1 : run - 1;
            total = mine.from(last);
            need = __shfl_sync(kFull, ids, last);
            p += static_cast<unsigned>(last + 1);
            if (stops) {
                finished = true;
                break;
            }
            if (run < 32) break;
        }
        if (p >= S->n_idblocks) finished = true;
        if (lane == 0) {
            // entries suspended during the launch become available to the next launch's refills
            C->park_avail += static_cast<int>(C->park_tail - C->park_commit);
            C->park_commit = C->park_tail;
            C->n_done = total.done;
            C->n_esc = total.esc;
            C->under = total.under;
            C->over = total.over;
            C->s1_lo = total.s1_lo;
            C->s1_hi = total.s1_hi;
            C->s2_lo = total.s2_lo;
            C->s2_hi = total.s2_hi;
            C->prefix = p;
            if (finished) C->state = kSlotFinished;
            else if (C->claim_blocks != 0 && p > first) {
                const unsigned claim = claim_blocks_for(need, S->stop_block, p, E.sms);
                if (claim == 0 || claim > C->claim_blocks) C->claim_blocks = claim;
            }
        }
        __syncwarp();
    }
    static_assert(sizeof(SlotCtl) % 8 == 0, "copied as 8-byte words");
    const unsigned long long *src = reinterpret_cast<const unsigned long long *>(C);
    unsigned long long *dst = reinterpret_cast<unsigned long long *>(h_ctl + s);
    if (lane < static_cast<int>(sizeof(SlotCtl) / 8)) dst[lane] = src[lane];
}

}  // namespace

cudaError_t launch_engine_chunk(const EngineDev &E, int T, unsigned grid, unsigned block,
                                cudaStream_t s) {
    const size_t shared = tail_shared_bytes(static_cast<int>(block / 32));
    if (T != 1)
        engine_chunk_kernel<2, false><<<grid, block, 0, s>>>(E);
    else if (shared == 0)
        engine_chunk_kernel<1, false><<<grid, block, 0, s>>>(E);
    else
        engine_chunk_kernel<1, true><<<grid, block, shared, s>>>(E);
    return cudaGetLastError();
}

cudaError_t launch_solo(const Decoded &d, uint64_t seed, uint64_t traj_offset, uint64_t n, int64_t *steps,
                        fpt_sums *sums, unsigned long long *hist, cudaStream_t s) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    SoloArgs a{};
    slot_constants(d, seed, traj_offset, &a.slot);
    a.slot.n_traj = n;
    a.slot.stop_block = 0xFFFFFFFFu;
    a.slot.n_idblocks = 1;
    id_block_magic(a.slot.stop_block, a.slot.ib_magic, a.slot.ib_shift);
    a.slot.hist_per_block = 1;   // one row
    a.slot.hist_rows = 1;
    a.slot.per_traj = reinterpret_cast<long long *>(steps);
    a.slot.park_cap = 1;
    a.n = n;
    a.sums = sums;
    a.hist = hist;
    a.nbins = hist ? d.hist_bins : 0;
    void (*kernel)(SoloArgs) = nullptr;
    switch (d.kind) {
#define FPT_KIND_CASE(M_, H_, R_) \
    case kind_of(M_, H_, R_): kernel = solo_kernel<M_, H_, R_>; break;
    FPT_KIND_CASE(kUnder, kEuler, kConstBias)
    FPT_KIND_CASE(kOver, kEuler, kConstBias)
    FPT_KIND_CASE(kUnder, kHeun, kConstBias)
    FPT_KIND_CASE(kOver, kHeun, kConstBias)
    FPT_KIND_CASE(kUnder, kEuler, kRamp)
    FPT_KIND_CASE(kOver, kEuler, kRamp)
    FPT_KIND_CASE(kUnder, kHeun, kRamp)
#undef FPT_KIND_CASE
    default: kernel = solo_kernel<kOver, kHeun, kRamp>; break;
    }
    const size_t shared = tail_shared_bytes(kSoloThreads / 32) + static_cast<size_t>(a.nbins) * 4;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(tail_shared_bytes(kSoloThreads / 32) + kSoloMaxBins * 4));
    if (e != cudaSuccess) return e;
    const uint64_t warps = (n + 31) / 32;
    kernel<<<static_cast<unsigned>(warps < static_cast<uint64_t>(sms) ? warps : sms), kSoloThreads, shared, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_engine_scan(const EngineDev &E, SlotCtl *h_ctl, unsigned long long *h_counters, cudaStream_t s) {
    const unsigned block = 128;
    const unsigned grid = (static_cast<unsigned>(E.max_requests) * 32 + block - 1) / block;
    engine_scan_kernel<<<grid, block, 0, s>>>(E, h_ctl, h_counters);
    return cudaGetLastError();
}

cudaError_t engine_chunk_occupancy(int T, int block, int *blocks_per_sm) {
    const size_t shared = tail_shared_bytes(block / 32);
    if (T != 1) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, engine_chunk_kernel<2, false>, block, 0);
    if (shared == 0)
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, engine_chunk_kernel<1, false>, block, 0);
    // every engine asks before its first launch, so the kernel's shared-memory limit is set
    const cudaError_t e = cudaFuncSetAttribute(engine_chunk_kernel<1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               static_cast<int>(tail_shared_bytes(640 / 32)));
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, engine_chunk_kernel<1, true>, block, shared);
}

}  // namespace fpt
