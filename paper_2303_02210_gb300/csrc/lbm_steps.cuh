// Many steps in one launch: the TMA-staged update kernels (k_update_tma,
// k_update7_tma with FUSED) loop over time steps, and some of their CTAs run
// the planner between two updates (plan_step), in a cooperative launch.
//
// What bounds a step as two launches (the update, then k_plan) while the
// lattice is small: a fixed ~20 us of launches, ramps and the planner's latency
// (its instruction chain, fetched cold at every launch, and its grid barriers,
// an atomic, a poll and a reread each). Inside one launch the CTAs and their
// barriers stay set up, the planner's exchanges are single tagged words, and
// what does not depend on the update (the candidates' Philox blocks, the
// pending statistics) is done before it ends. Per step, two launches against
// one: 128 columns by 53 rows 20.5 -> 13.0 us, 1024 by 53 20.5 -> 15.7, 1501 by
// 53 in BF16 23.1 -> 17.6, 1024 by 490 26.1 -> 23.3, 2048 by 976 47.1 -> 43.5,
// D2Q7 4096 by 1003 66.2 -> 63.8 (which calls take it: fused_min_steps in
// lbm_api.cu). What is left at 128 columns: four hand-overs
// between CTAs of about 1 us each, the front's scan 0.9, the candidates'
// gathers 1.0, the divisions' atomics 1.6, the update itself 2.5.
//
// One step:
//   update    every CTA its tiles, as in the one-step launch; each CTA also
//             empties its share of the merge table and its division bucket,
//             which the selection below fills again;
//   up        every CTA counts itself in (release); the first G CTAs wait for
//             all of them (acquire);
//   plan_step those G CTAs observe the new state and select the divisions of
//             the next step;
//   done      they count themselves in; every CTA waits for them and goes on.
// Bulk tensor copies (the async proxy) read what other CTAs stored in either
// proxy, so each thread fences the proxies before `up` and the issuing thread
// again after `done`.
//
// The waits are bounded as elsewhere; one that runs out sets `st_quit`, which
// every waiting CTA sees: all leave, the last one puts the step count where
// the host expects it, and the status says LBM_STATUS_TIMEOUT.
#pragma once

#include "lbm_plan.cuh"

namespace lbm {

constexpr int kStepSleep = 100;    // ns between polls of the CTAs that wait for the planner
constexpr int kStepR = 8;          // candidates per thread in the first pass
constexpr int kStepWords = 4;      // mask words per warp up to which every planner CTA scans the whole front,
constexpr int kStepRough = 96;     // and rows of the front

__device__ __forceinline__ void fence_proxy_async_all() { asm volatile("fence.proxy.async;" ::: "memory"); }

__device__ __forceinline__ int ld_relaxed_s32(const int *p)
{
    int v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed_u64(unsigned long long *p, unsigned long long v)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void st_relaxed_v2(unsigned long long *p, unsigned long long a, unsigned long long b)
{
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}
__device__ __forceinline__ void ld_relaxed_v2(const unsigned long long *p, unsigned long long *a, unsigned long long *b)
{
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(*a), "=l"(*b) : "l"(p) : "memory");
}
__device__ __forceinline__ void red_relaxed_u64(unsigned long long *p, unsigned long long v)
{
    asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Gives up the launch: every CTA that waits sees it.
__device__ __forceinline__ void step_give_up(DevScalars *sc)
{
    atomicOr(&sc->status, ST_TIMEOUT);
    atomicExch(&sc->st_quit, 1);
}

// Polls until `done(value at p)`; false if the launch gave up. The caller
// fences (acquire) before it relies on what was written before the value.
// SLEEP: nanoseconds between polls.
template <int SLEEP, typename F>
__device__ __forceinline__ bool step_poll(const unsigned long long *p, DevScalars *sc, long long budget,
                                          unsigned long long *out, F done)
{
    unsigned long long v = ld_relaxed_u64(p);
    if (!done(v)) {
        const long long t0 = clock64();
        for (int n = 1;; ++n) {
            if (SLEEP > 0) __nanosleep(SLEEP);
            v = ld_relaxed_u64(p);
            if (done(v)) break;
            if ((n & 7) == 0) {
                if (ld_relaxed_s32(&sc->st_quit)) return false;
                if (clock64() - t0 > budget) {
                    step_give_up(sc);
                    return false;
                }
            }
        }
    }
    *out = v;
    return true;
}
template <int SLEEP>
__device__ __forceinline__ bool step_wait(const unsigned long long *ctr, unsigned long long target, DevScalars *sc,
                                          long long budget)
{
    unsigned long long v;
    const bool ok = step_poll<SLEEP>(ctr, sc, budget, &v, [&](unsigned long long c) { return c >= target; });
    __threadfence();
    return ok;
}

// What the planner keeps in shared memory (over a staged tile's room).
template <int NT>
struct StepScratch {
    static constexpr int WARPS = NT / 32;
    uint32_t key[NT * kStepR]; // first-pass candidates of this CTA: key,
    int lr[NT * kStepR];       // and rank among its accepted candidates (-1: rejected)
    unsigned short h[WARPS * kStepWords * 32]; // the front heights (when this CTA scans the whole front)
    long long cm[12], s2[WARPS], ll[WARPS], req;
    double carry, kcf, carry_in, ratio_in;
    unsigned long long kstop;
    int s1[WARPS], top[WARPS], low[WARPS], cnt[2][WARPS], bf[WARPS], tt[WARPS];
    int quit;
};

// Exchange of one value per planner CTA: each puts its words, tagged with the
// step (so that a stale word is told from a new one), into its own slot, and
// every CTA reads all slots (kXch words a CTA): 0-3 the front's sums and
// extrema, 4-5 the mass of the rows just frozen, 6-7 accepted candidates (two
// buffers: a CTA writes round r + 2 only after it has read every word of
// round r + 1, whose writers had read round r).

__device__ __forceinline__ unsigned long long xch_tag(uint32_t epoch, uint32_t v)
{
    return ((unsigned long long)epoch << 32) | v;
}
__device__ __forceinline__ bool xch_get(const SimDev &d, int blk, int word, uint32_t epoch, long long budget,
                                        uint32_t *v)
{
    unsigned long long r = 0;
    const bool ok = step_poll<0>(&d.xch[blk * kXch + word], d.sc, budget, &r,
                              [&](unsigned long long c) { return (uint32_t)(c >> 32) == epoch; });
    *v = (uint32_t)r;
    return ok;
}

// Two words at once (`word` even).
__device__ __forceinline__ bool xch_get2(const SimDev &d, int blk, int word, uint32_t epoch, long long budget,
                                         uint32_t *a, uint32_t *b)
{
    const unsigned long long *p = &d.xch[blk * kXch + word];
    unsigned long long u, v;
    ld_relaxed_v2(p, &u, &v);
    if ((uint32_t)(u >> 32) != epoch || (uint32_t)(v >> 32) != epoch) {
        if (!step_poll<0>(p, d.sc, budget, &u, [&](unsigned long long c) { return (uint32_t)(c >> 32) == epoch; }) ||
            !step_poll<0>(p + 1, d.sc, budget, &v, [&](unsigned long long c) { return (uint32_t)(c >> 32) == epoch; }))
            return false;
    }
    *a = (uint32_t)u;
    *b = (uint32_t)v;
    return true;
}

// Planner CTAs of a step (at most kStepMaxPlan), from the number of candidates
// that the selection before needed (an estimate): 16 candidates a CTA, up to
// 128 when there are many. A candidate gathers 9 (7) scattered populations and a
// division does three scattered atomics and stores, and an SM sends such
// requests at one per several clocks (72 candidates in one CTA: 4300 clocks), so
// few are spread thin; but every CTA reads every other's counts. A front of more
// than kStepWords words per warp is scanned by as many CTAs as it has words per
// warp, and their sums are exchanged; a narrower one by every planner CTA whole
// (no exchange), unless a warp has several words of it and it spans more than
// kStepRough rows, each 32 of which cost a round for each word (405 columns, 800
// rows: 48.3 us a step scanned whole, 33.4 exchanged, 44 as two launches; 200
// rows 23.8 and 21.8; 100 rows 17.6 whole).
template <int NT>
__device__ __forceinline__ int step_planners(const DevScalars *sc, int MW, int ctas, bool *whole)
{
    constexpr int WARPS = NT / 32;
    const long long kc = sc->plan_kc;
    *whole = MW <= WARPS * kStepWords && (MW <= WARPS || sc->H_top - sc->hmin <= kStepRough);
    const long long per = min(max(kc / 64, 16ll), 128ll);
    int G = (int)min((kc + per - 1) / per, (long long)kStepMaxPlan);
    if (!*whole) G = max(G, min((MW + WARPS - 1) / WARPS, kStepMaxPlan));
    return max(1, min(G, ctas));
}

// Warp sum of S2 < 2^40 per lane by two 32-bit reductions.
__device__ __forceinline__ long long step_sum_s2(long long v)
{
    const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)(v & 0xFFFFF));
    const unsigned hi = __reduce_add_sync(0xffffffffu, (unsigned)(v >> 20));
    return ((long long)hi << 20) + lo;
}

// The 32 x 32 bit transpose of a mask word's 32 rows (lane l holds row yb - l):
// lane c gets its column, bit l set iff row yb - l is occupied.
__device__ __forceinline__ unsigned step_transpose(unsigned col, int lane)
{
#pragma unroll
    for (int j = 16; j > 0; j >>= 1) {
        const unsigned keep = j == 16 ? 0x0000FFFFu
                            : j == 8  ? 0x00FF00FFu
                            : j == 4  ? 0x0F0F0F0Fu
                            : j == 2  ? 0x33333333u
                                      : 0x55555555u; // bits c with (c & j) == 0
        const unsigned other = __shfl_xor_sync(0xffffffffu, col, j);
        col = (lane & j) ? ((col & ~keep) | ((other & ~keep) >> j)) : ((col & keep) | ((other & keep) << j));
    }
    return col;
}

// Height of this lane's column of word m, from row yb down (the columns of
// `pending` have no occupied row above it).
__device__ __forceinline__ int step_height(const SimDev &d, int m, int yb, unsigned pending, int h, int lane)
{
    for (; yb >= 0 && pending; yb -= 32) {
        const int y = yb - lane;
        const unsigned col = step_transpose(y >= 0 ? d.mask[(long long)y * d.MW + m] : 0u, lane);
        if (((pending >> lane) & 1u) && col != 0u) h = yb - (__ffs(col) - 1) + 1;
        pending &= ~__ballot_sync(0xffffffffu, col != 0u);
    }
    return h;
}

// Exclusive rank of this thread's flag among the CTA's; *total gets their
// number. `buf` alternates between calls (one barrier a call).
template <int NT>
__device__ __forceinline__ int step_rank(bool a, int *total, int (*cnt)[NT / 32], int buf)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned b = __ballot_sync(0xffffffffu, a);
    if (lane == 0) cnt[buf][warp] = __popc(b);
    __syncthreads();
    int before = 0, all = 0;
#pragma unroll
    for (int i = 0; i < NT / 32; ++i) {
        const int c = cnt[buf][i];
        before += i < warp ? c : 0;
        all += c;
    }
    *total = all;
    return before + __popc(b & ((1u << lane) - 1u));
}

// The accepted-candidate counts of all planner CTAs: their sum and that of
// the CTAs before this one. False if the launch gave up.
template <int NT>
__device__ __forceinline__ bool step_counts(const SimDev &d, StepScratch<NT> &ps, int G, int blk, uint32_t epoch,
                                            int round, int mine, long long budget, long long *before,
                                            long long *total)
{
    constexpr int WARPS = NT / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (G == 1) {
        *before = 0;
        *total = mine;
        return true;
    }
    const int word = 6 + (round & 1);
    const uint32_t tag = (uint32_t)(round & 0xFFFF) << 16;
    // (the words say it all: nothing else is handed over here)
    if (tid == 0) st_relaxed_u64(&d.xch[blk * kXch + word], xch_tag(epoch, tag | (uint32_t)mine));
    int bf = 0, tt = 0;
    bool ok = true;
    for (int i = tid; i < G; i += NT) {
        unsigned long long r = 0;
        ok &= step_poll<0>(&d.xch[i * kXch + word], d.sc, budget, &r, [&](unsigned long long c) {
            return (uint32_t)(c >> 32) == epoch && ((uint32_t)c & 0xFFFF0000u) == tag;
        });
        const int c = (int)((uint32_t)r & 0xFFFFu);
        tt += c;
        bf += i < blk ? c : 0;
    }
    bf = __reduce_add_sync(0xffffffffu, bf);
    tt = __reduce_add_sync(0xffffffffu, tt);
    if (lane == 0) {
        ps.bf[warp] = bf;
        ps.tt[warp] = tt;
    }
    ok = __syncthreads_and(ok);
    bf = tt = 0;
#pragma unroll
    for (int i = 0; i < WARPS; ++i) {
        bf += ps.bf[i];
        tt += ps.tt[i];
    }
    __syncthreads(); // (ps.bf, ps.tt are written again next round)
    *before = bf;
    *total = tt;
    return ok;
}

// The planner between the update of step t and that of step t + 1 (the same
// arithmetic and draws as plan_body), by CTAs blk = 0 .. G - 1 of NT threads.
// False if the launch gave up.
template <typename S, typename LT, int NT>
__device__ __forceinline__ bool plan_step(const SimDev &d, StepScratch<NT> &ps, uint32_t t, int G, int blk, bool whole,
                                          long long budget, unsigned long long up, bool ok_in)
{
    using R = arith_t<S>;
    constexpr int WARPS = NT / 32;
    DevScalars *sc = d.sc;
    const uint32_t tn = t + 1u, epoch = t + 1u;
    const S *f = (const S *)d.f[tn & 1u];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool grow = d.growth_mode != GROW_NONE;

    // ---- before the other CTAs' updates are done: what they do not change.
    // The first pass draws about as many candidates as the selection before
    // needed (the selection does not depend on how many; more are drawn if
    // they fall short), so that its counters, and their Philox blocks, are
    // known now.
    const int C = (int)min((long long)NT * kStepR, max(1ll, (sc->plan_kc + G - 1) / G)); // candidates of this CTA
    const long long kc = (long long)G * C;                                               // and of the pass
    const int rounds = (C + NT - 1) / NT;
    const u32x4 r0 = grow ? philox4x32_10(u32x4{(uint32_t)(blk * C + tid), tn, STREAM_PROLIF, d.sim}, d.pk)
                          : u32x4{0u, 0u, 0u, 0u};
    const int y_r = sc->y_r, y_hi_old = sc->y_hi;
    // what block 0 commits about the step that ran
    if (blk == 0 && tid == 0) {
        ps.cm[0] = sc->pend_req;
        ps.cm[1] = sc->pend_acc;
        ps.cm[2] = sc->pend_nev;
        ps.cm[3] = sc->pend_cand;
        ps.cm[4] = sc->ns_total;
        ps.cm[5] = sc->div_total;
        ps.cm[6] = sc->starved_steps;
        ps.cm[7] = sc->node_updates;
        ps.cm[8] = sc->step;
        ps.cm[9] = sc->quiescent_fix;
        ps.cm[10] = sc->pend_starved;
        ps.cm[11] = __double_as_longlong(sc->pend_carry);
    }
    if (tid == 0) ps.kstop = 0ull;
    if (grow && tid == NT - 32) {
        ps.carry_in = sc->pend_carry;
        ps.ratio_in = sc->acc_ratio;
    }
    // ---- every CTA's update is done
    if (tid == 0) ok_in = ok_in && step_wait<0>(&sc->st_up, up, sc, budget);
    if (!__syncthreads_and(ok_in)) return false;
    const int maxmass = sc->maxmass_accum;
    const long long mass_acc = (long long)sc->mass_accum;

    // ---- A: front heights and their sums, from the window's top row down (it
    // is known without waiting for the mass's; the window's rows above the
    // mass are empty) unless the mass ends far below. The last warp first
    // works out n_s in FP64 (if no row is frozen now, almost always).
    const int per = (d.MW + WARPS - 1) / WARPS; // words per warp when each CTA scans the whole front
    int ytop = min(y_hi_old, d.H) - 1;
    auto row_word = [&](int m) -> unsigned {
        const int y = ytop - lane;
        return y >= 0 ? d.mask[(long long)y * d.MW + m] : 0u;
    };
    const int m0 = whole ? warp * per : blk * WARPS + warp; // this warp's first word
    unsigned w[kStepWords];                                   // (all loads in flight together)
    auto load_rows = [&]() {
        w[0] = m0 < d.MW ? row_word(m0) : 0u;
        if (whole && per > 1) {
#pragma unroll
            for (int j = 1; j < kStepWords; ++j) w[j] = j < per && m0 + j < d.MW ? row_word(m0 + j) : 0u;
        }
    };
    load_rows();
    if (grow && tid == NT - 32)
        plan_ns(d.growth_rate, d.rho_cell, mass_acc, ps.carry_in, ps.ratio_in, &ps.req, &ps.carry, &ps.kcf);
    const int yfar = min(max(maxmass, y_r - 1), d.H - 1);
    if (yfar < ytop - 16) { // uniform
        ytop = yfar;
        load_rows();
    }
    long long S2 = 0;
    int S1 = 0, top = 0, low = 0x7fffffff;
    // one word whose first 32 rows are in `col`, transposed
    auto take = [&](int m, unsigned col, bool store) {
        const int x = m * 32 + lane;
        int h = col != 0u ? ytop - (__ffs(col) - 1) + 1 : 0;
        const unsigned pending = __ballot_sync(0xffffffffu, x < d.W && col == 0u);
        if (pending) h = step_height(d, m, ytop - 32, pending, h, lane);
        if (x < d.W) {
            if (store) d.heights[x] = h;
            if (whole) ps.h[x] = (unsigned short)h;
            S1 += h;
            S2 += (long long)h * h;
            top = max(top, h);
            low = min(low, h);
        }
    };
    if (m0 < d.MW) take(m0, step_transpose(w[0], lane), !whole || blk == 0);
    if (whole && per > 1) {
        // (the transposes of the other words side by side: each is a chain of
        // shuffles)
#pragma unroll
        for (int j = 1; j < kStepWords; ++j) w[j] = step_transpose(w[j], lane);
#pragma unroll 1
        for (int j = 1; j < per; ++j) {
            const unsigned col = w[1];
#pragma unroll
            for (int i = 1; i + 1 < kStepWords; ++i) w[i] = w[i + 1];
            if (m0 + j < d.MW) take(m0 + j, col, blk == 0);
        }
    } else if (!whole) {
#pragma unroll 1
        for (int m = m0 + G * WARPS; m < d.MW; m += G * WARPS) take(m, step_transpose(row_word(m), lane), true);
    }
    S1 = __reduce_add_sync(0xffffffffu, S1);
    S2 = step_sum_s2(S2);
    top = __reduce_max_sync(0xffffffffu, top);
    low = __reduce_min_sync(0xffffffffu, low);
    if (lane == 0) {
        ps.s1[warp] = S1;
        ps.s2[warp] = S2;
        ps.top[warp] = top;
        ps.low[warp] = low;
    }
    __syncthreads();
    long long S1a = 0, S2a = 0;
    int topa = 0, lowa = 0x7fffffff;
#pragma unroll
    for (int i = 0; i < WARPS; ++i) {
        S1a += ps.s1[i];
        S2a += ps.s2[i];
        topa = max(topa, ps.top[i]);
        lowa = min(lowa, ps.low[i]);
    }
    const int Gs = whole ? 1 : min(G, (d.MW + WARPS - 1) / WARPS); // the CTAs whose sums are exchanged
    if (!whole && G > 1) {
        if (tid == 0 && blk < Gs) {
            unsigned long long *x = d.xch + blk * kXch;
            if (d.growth_mode == GROW_EDGE) __threadfence(); // the heights of all this CTA's threads come first
            st_relaxed_v2(x, xch_tag(epoch, (uint32_t)S1a), xch_tag(epoch, (uint32_t)S2a)); // (W h <= 2^30)
            st_relaxed_v2(x + 2, xch_tag(epoch, (uint32_t)(S2a >> 32) << 16 | (uint32_t)topa),
                          xch_tag(epoch, (uint32_t)lowa));
        }
        S1 = 0;
        S2 = 0;
        top = 0;
        low = 0x7fffffff;
        bool ok = true;
        for (int i = tid; i < Gs; i += NT) {
            uint32_t a, b, c, e;
            ok &= xch_get2(d, i, 0, epoch, budget, &a, &b);
            ok &= xch_get2(d, i, 2, epoch, budget, &c, &e);
            S1 += (int)a;
            S2 += (long long)(((unsigned long long)(c >> 16) << 32) | b);
            top = max(top, (int)(c & 0xFFFFu));
            low = min(low, (int)e);
        }
        if (d.growth_mode == GROW_EDGE) __threadfence();
        S1 = __reduce_add_sync(0xffffffffu, S1);
        S2 = warp_sum_ll(S2);
        top = __reduce_max_sync(0xffffffffu, top);
        low = __reduce_min_sync(0xffffffffu, low);
        __syncthreads(); // (the CTA's own partials have been read)
        if (lane == 0) {
            ps.s1[warp] = S1;
            ps.s2[warp] = S2;
            ps.top[warp] = top;
            ps.low[warp] = low;
        }
        if (!__syncthreads_and(ok)) return false;
        S1a = S2a = 0;
        topa = 0;
        lowa = 0x7fffffff;
#pragma unroll
        for (int i = 0; i < WARPS; ++i) {
            S1a += ps.s1[i];
            S2a += ps.s2[i];
            topa = max(topa, ps.top[i]);
            lowa = min(lowa, ps.low[i]);
        }
    }

    // ---- B: the rear wall, the active mass and the next plan (plan_body's
    // phase B)
    int nyr = y_r;
    if (d.wall_mode == 1 && !d.y_periodic) {
        const long long var = (long long)d.W * S2a - S1a * S1a;
        const float hf = (float)S1a / (float)d.W;
        const float wf = sqrtf((float)var) / (float)d.W;
        const float cf = hf - fmaxf((float)d.wall_min_gap, (float)d.wall_w_factor * wf);
        if (cf > (float)y_r + 0.9f) {
            const double hbar = (double)S1a / (double)d.W;
            const double wdt = sqrt((double)var) / (double)d.W;
            double gap = d.wall_min_gap;
            const double wg = d.wall_w_factor * wdt;
            if (wg > gap) gap = wg;
            double c = floor(hbar - gap);
            if (c > (double)(d.H - 1)) c = (double)(d.H - 1);
            const int cand = (int)c;
            if (cand > nyr) nyr = cand;
        }
    }
    long long frozen = 0;
    if (nyr > y_r) { // uniform across the planner CTAs
        const long long n = (long long)(nyr - y_r) * d.W;
        long long fm = 0;
        for (long long k = (long long)blk * NT + tid; k < n; k += (long long)G * NT) {
            const int y = y_r + (int)(k / d.W), x = (int)(k % d.W);
            const long long o = (long long)y * d.Wp + x;
            const Pop<S> pc(d);
            R r = pc.ld(f[o], 0);
#pragma unroll
            for (int i = 1; i < LT::Q; ++i) r = r + pc.ld(f[i * d.P + o], i);
            fm += fix24<R>(r);
        }
        auto block_sum = [&](long long v) {
            v = warp_sum_ll(v);
            if (lane == 0) ps.ll[warp] = v;
            __syncthreads();
            v = 0;
#pragma unroll
            for (int i = 0; i < WARPS; ++i) v += ps.ll[i];
            __syncthreads();
            return v;
        };
        frozen = block_sum(fm);
        if (G > 1) {
            if (tid == 0) {
                unsigned long long *x = d.xch + blk * kXch;
                st_relaxed_u64(x + 4, xch_tag(epoch, (uint32_t)frozen));
                st_relaxed_u64(x + 5, xch_tag(epoch, (uint32_t)((unsigned long long)frozen >> 32)));
            }
            long long a = 0;
            bool ok = true;
            for (int i = tid; i < G; i += NT) {
                uint32_t l, h;
                ok &= xch_get(d, i, 4, epoch, budget, &l);
                ok &= xch_get(d, i, 5, epoch, budget, &h);
                a += (long long)(((unsigned long long)h << 32) | l);
            }
            frozen = block_sum(a);
            if (!__syncthreads_and(ok)) return false;
        }
        if (grow && tid == 0)
            plan_ns(d.growth_rate, d.rho_cell, mass_acc - frozen, ps.carry_in, ps.ratio_in, &ps.req, &ps.carry,
                    &ps.kcf);
        __syncthreads();
    }
    const long long mass_fix = mass_acc - frozen;
    int yhi_next;
    if (d.y_periodic) {
        yhi_next = d.H;
    } else {
        yhi_next = maxmass + 2 < d.H ? maxmass + 2 : d.H;
        if (y_hi_old > yhi_next) yhi_next = y_hi_old;
    }
    long long ns_req = 0, ns = 0, kc_next = 0;
    int ylo = nyr, capacity = 0, nwin_zero = 0;
    unsigned long long nwin = 0ull;
    if (grow) {
        ns_req = ps.req;
        ns = ns_req;
        int yhi_c = topa;
        if (d.growth_mode == GROW_EDGE) {
            const int e = lowa - d.edge_depth;
            if (e > ylo) ylo = e;
        } else if (d.growth_mode == GROW_BAND) {
            if (nyr + d.band_rows < yhi_c) yhi_c = nyr + d.band_rows;
        }
        nwin = yhi_c > ylo ? (unsigned long long)(yhi_c - ylo) * (unsigned long long)d.W : 0ull;
        if (ns > d.ns_max || ns < 0 || mass_fix < 0) {
            capacity = 1;
            ns = 0;
        }
        nwin_zero = (ns > 0 && nwin == 0) ? 1 : 0;
        if (nwin == 0) ns = 0;
        kc_next = min((long long)ps.kcf, 64 * ns + 1024);
    }
    const size_t buf = (size_t)(tn & 1u) * (size_t)d.ns_max; // event list of step tn

    // ---- C/D: candidates in draw order, the first n_s accepted, merged (as
    // plan_body). Without divisions the counts are still exchanged when some
    // CTA has posted nothing so far (it has no word of the front): block 0 must
    // not commit while another CTA reads.
    long long acc = 0;
    auto accept = [&](const Candidate &c) -> bool {
        const R rs = rho_star<S, LT>(d, f, nyr, c.x, c.y);
        switch (d.growth_mode) {
        case GROW_BULK:
        case GROW_BAND: return rs >= rho_c_of<R>(d);
        case GROW_EDGE:
            return rs >= rho_c_of<R>(d) && ((whole ? (int)ps.h[c.x] : d.heights[c.x]) - c.y) <= d.edge_depth;
        case GROW_DENSITY: return (double)rs > d.rho_c && u01(c.u) < 1.0 - (double)rs / d.rho0; // Eq. 5
        default: return false;
        }
    };
    if (ns > 0 || G > Gs) { // uniform
        const long long cap = ns > 0 ? 64 * ns + 1024 : 0;
        int tot_b = 0;
#pragma unroll 1
        for (int i = 0; i < rounds; ++i) {
            const long long j = (long long)i * NT + tid;
            const long long k = (long long)blk * C + j;
            bool a = false;
            uint32_t key = 0u;
            if (j < C && k < cap && nwin > 0) {
                const Candidate c = i == 0 ? candidate_of<LT>(d, r0, ylo, nwin) : draw_candidate<LT>(d, k, tn, ylo, nwin);
                a = accept(c);
                key = pack_key(c.x, c.y, c.pair);
            }
            int t_i;
            const int pre = step_rank<NT>(a, &t_i, ps.cnt, i & 1);
            ps.key[j] = key;
            ps.lr[j] = a ? tot_b + pre : -1;
            tot_b += t_i;
        }
        long long before, total;
        if (!step_counts<NT>(d, ps, G, blk, epoch, 0, tot_b, budget, &before, &total)) return false;
#pragma unroll 1
        for (int i = 0; i < rounds; ++i) {
            const int j = i * NT + tid;
            const int lr = ps.lr[j];
            if (lr >= 0) {
                const long long rank = before + lr;
                if (rank == ns - 1) ps.kstop = (unsigned long long)((long long)blk * C + j + 1);
                if (rank < ns) plan_select<R, true, LT>(d, ps.key[j], (int)rank, buf, nyr);
            }
        }
        acc = total;
        long long base = kc;
        int round = 1;
        __syncthreads();
        while (acc < ns && base < cap) { // uniform
            const long long k0 = base + ((long long)blk * NT + tid) * kStepR;
            int mine = 0;
#pragma unroll 1
            for (int i = 0; i < kStepR; ++i) {
                const long long k = k0 + i;
                bool a = false;
                uint32_t key = 0u;
                if (k < cap) {
                    const Candidate c = draw_candidate<LT>(d, k, tn, ylo, nwin);
                    a = accept(c);
                    key = pack_key(c.x, c.y, c.pair);
                }
                ps.key[tid * kStepR + i] = key;
                ps.lr[tid * kStepR + i] = a ? mine : -1;
                mine += a ? 1 : 0;
            }
            // this thread's first rank in the CTA
            int incl = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += u;
            }
            if (lane == 31) ps.cnt[round & 1][warp] = incl;
            __syncthreads();
            int pr = incl - mine, tot_r = 0;
#pragma unroll
            for (int i = 0; i < WARPS; ++i) {
                const int c = ps.cnt[round & 1][i];
                pr += i < warp ? c : 0;
                tot_r += c;
            }
            long long bf, tt;
            if (!step_counts<NT>(d, ps, G, blk, epoch, round, tot_r, budget, &bf, &tt)) return false;
#pragma unroll 1
            for (int i = 0; i < kStepR; ++i) {
                const int lr = ps.lr[tid * kStepR + i];
                if (lr < 0) continue;
                const long long rank = acc + bf + pr + lr;
                if (rank == ns - 1) ps.kstop = (unsigned long long)(k0 + i + 1);
                if (rank < ns) plan_select<R, true, LT>(d, ps.key[tid * kStepR + i], (int)rank, buf, nyr);
            }
            acc += tt;
            base += (long long)G * NT * kStepR;
            ++round;
        }
        __syncthreads();
        if (tid == 0 && ps.kstop) {
            sc->pend_cand = (long long)ps.kstop;
            sc->acc_ratio = (double)((float)ps.kstop / (float)ns); // a work estimate only
        }
    }
    const int nsel = (int)(acc < ns ? acc : ns); // selected divisions (draw ranks)

    // ---- block 0: commit the step that ran, the observables, the new selection
    if (blk == 0 && tid == 0) {
        sc->ns_last = ps.cm[0];
        sc->ns_total = ps.cm[4] + ps.cm[0];
        sc->carry = __longlong_as_double(ps.cm[11]);
        sc->div_total = ps.cm[5] + ps.cm[1];
        sc->events_last = ps.cm[1];
        sc->n_events = (int)ps.cm[2];
        sc->cand_last = ps.cm[3];
        if (ps.cm[10]) {
            sc->starved_steps = ps.cm[6] + 1;
            atomicOr(&sc->status, ST_STARVED);
        }
        sc->node_updates = ps.cm[7] + (long long)d.W * (long long)(y_hi_old > y_r ? y_hi_old - y_r : 0);
        sc->step = ps.cm[8] + 1;
        sc->S1 = S1a;
        sc->S2 = S2a;
        sc->H_top = topa;
        sc->hmin = lowa;
        sc->mass_fix = mass_fix;
        sc->quiescent_fix = ps.cm[9] + frozen;
        sc->y_copy = y_r;
        sc->y_r = nyr;
        sc->y_hi = yhi_next;
        if (maxmass >= d.H - 1) atomicOr(&sc->status, ST_FRONT_AT_TOP);
        if (capacity) atomicOr(&sc->status, ST_CAPACITY);
        sc->mass_accum = 0ull;
        sc->maxmass_accum = -1;
        const long long cap = 64 * ns + 1024;
        const double carry_out = grow ? ps.carry : __longlong_as_double(ps.cm[11]);
        sc->pend_req = ns_req;
        sc->pend_carry = carry_out;
        sc->pend_acc = nsel;
        sc->pend_nev = nsel;
        sc->pend_starved = (nwin_zero || (ns > 0 && acc < ns)) ? 1 : 0;
        // (with n_s reached, the accepting CTA wrote pend_cand and acc_ratio)
        if (!(ns > 0 && acc >= ns)) sc->pend_cand = nwin_zero ? 0 : (ns > 0 ? cap : 0);
        sc->plan_req = ns_req;
        sc->plan_ns = ns;
        sc->plan_kc = kc_next;
        sc->plan_ylo = ylo;
        sc->plan_nwin = nwin;
        sc->plan_carry = carry_out;
        sc->rec_n = nsel;
    }
    return true;
}

// The end of a step in a fused update kernel: the CTA's stores and totals are
// out; planner CTAs select the next step's divisions; every CTA waits for
// them (not after the launch's last step). `planned`: planner CTAs of the
// launch's steps so far. False if the launch gave up.
template <typename S, typename LT, int NT>
__device__ __forceinline__ bool step_end(const SimDev &d, StepScratch<NT> &ps, uint32_t t, int it, bool last, int G,
                                         bool whole, long long budget, int extra, unsigned long long *planned,
                                         bool gave_up)
{
    DevScalars *sc = d.sc;
    fence_proxy_async_all(); // this thread's stores, before other CTAs' bulk copies
    bool ok = !__syncthreads_or(gave_up);
    if (threadIdx.x == 0) {
        if (!ok) step_give_up(sc);
        __threadfence();
        red_relaxed_u64(&sc->st_up, 1ull);
    }
    *planned += (unsigned long long)G;
    const int blk = (int)(gridDim.x - 1u - blockIdx.x); // (the last CTAs have a tile less to do)
    if (blk < G) {
        if (!plan_step<S, LT, NT>(d, ps, t, G, blk, whole, budget,
                                  (unsigned long long)gridDim.x * (unsigned)(it + 1) + (unsigned)extra, ok))
            return false;
        fence_proxy_async_smem(); // (the scratch lies where bulk copies will land)
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            red_relaxed_u64(&sc->st_done, 1ull);
        }
    }
    if (last) return ok;
    if (threadIdx.x == 0) {
        ok = ok && step_wait<kStepSleep>(&sc->st_done, *planned, sc, budget);
        fence_proxy_async_all();
    }
    return __syncthreads_and(ok);
}

// The last CTA out of a fused launch puts the counters back to zero, and after
// a launch that gave up the step count where the host expects it.
__device__ __forceinline__ void step_exit(DevScalars *sc, long long step_after)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&sc->st_exit, 1u) == gridDim.x - 1u) {
            sc->st_up = 0ull;
            sc->st_done = 0ull;
            sc->st_exit = 0u;
            if (sc->st_quit) {
                sc->st_quit = 0;
                sc->step = step_after;
            }
            __threadfence();
        }
    }
}

// Whether `ctas` CTAs of a fused kernel are resident at once. `per_sm`: the
// caller's record of what it was told before (a property of the device).
inline cudaError_t steps_fit(const void *kernel, int threads, size_t smem, int ctas, int (&per_sm)[64])
{
    int dev = 0, nsm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    int n = dev < 64 ? per_sm[dev] : 0;
    if (n == 0) {
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, threads, smem);
        if (e != cudaSuccess) return e;
        if (dev < 64) per_sm[dev] = n;
    }
    return (long long)n * nsm >= ctas ? cudaSuccess : cudaErrorCooperativeLaunchTooLarge;
}

} // namespace lbm
