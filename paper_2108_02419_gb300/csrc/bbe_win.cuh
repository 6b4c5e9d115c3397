// bbe_win.cuh -- the rollout kernel: the Section 3 dry-runs under Eq. 1, each rollout run to its
// first finisher (win counts) or, in place mode, to its K-th (place counts, ordered tallies and
// the finishing-order histogram).
//
// Layout.  A warp holds 32 V slots (V = 1..4 per lane; slot i = 32 v + lane, so the lanes of
// one register hold consecutive slots).  A race of n competitors takes floor(32 V / n)
// segments of n consecutive slots: slot s n + c holds competitor c for the whole work item, and
// each segment runs its own rollouts of the race.  A competitor never changes slot, so the four
// normals of its current Philox block live in registers, and so do its parameters (or, in the
// register-lean variant for three and four slots per lane, a shared-memory address of them).
//
// The nearest competitor strictly in front (i+).  Each step every slot publishes (d, previous
// step) in shared memory and reads the entry of its rank successor (rank order: ascending
// position, then index), whose address it keeps in a register.  In a segment where every
// successor is strictly in front, the successor is i+.  The same read detects an overtake or
// an equal position (successor not strictly in front); on that rare step the segment is
// re-ranked, and a slot whose successor stands level with it takes the first later rank strictly
// in front.
//
// The step loop goes by the four steps of a Philox block: a block draws one Philox4x32-10 output
// per slot (from words kept per rollout, StreamWords) and both of its Box-Muller pairs, then runs
// four steps whose normals are registers chosen at compile time.  Every rollout starts on a block boundary (a
// segment that finishes waits for the next one; the counter of step t is t >> 2 in any case).
// A finished segment takes the warp's next rollout index, so the segments of a work item stay busy until
// its rollouts run out.
//
// Who is advanced.  Only the competitors that can matter to the first finish, or the first K, are
// (bbe_contenders.cu); they take the slots, so a warp has room for more segments.  A work item is a
// ticket for some of a race's rollouts, and the warp takes as many as its segments can share.
//
// Finishing.  A rollout that ends waits for the block's end in any case, and what its slots do until
// then counts for nobody.  So the steps know nothing of the line: one vote a block finds the blocks
// with crossings (positions only grow), and the positions published in the block say which step each
// was.  The least key (step, within-step crossing time tau = (L - d) / S, slot) of a segment is the
// first finisher: the least tau and, on equal tau, the lowest competitor index.  Wins are tallied per
// competitor in shared memory and reach the global counts once per work item.  Place mode places a
// block's crossings in key order until the K-th place is filled.  The step limit is looked at in the
// same place, and a warp-uniform count-down rules it out until a block could reach it.  (With the
// finish found within its step, a vote a step and a copy of the step for blocks near the limit: 4096
// spread races of 20 52.0 instead of 50.0 ms, 10^4 uneven ones 80.3 instead of 78.4, 700 bunched of 13
// 15.5 instead of 14.7, places 19.5 instead of 18.3.)
//
// The arithmetic is the pinned binary32 round-to-nearest sequence of include/bbe.h (explicit
// intrinsics, file compiled with --fmad=false), so the counts are bit-identical to any
// implementation that follows it, whatever the layout.
#pragma once
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <type_traits>

#include "bbe_internal.h"
#include "bbe_rng.cuh"

namespace bbe {

namespace win {

constexpr unsigned kAll = 0xffffffffu;
constexpr unsigned long long kNoKey = ~0ull;
constexpr unsigned kRedo = 64;
constexpr int kPlaced = 128;           // place mode: a segment's K places are filled, at this step of the block
constexpr unsigned kNone = ~0u;       // win mode: a segment without a finish, ..
constexpr unsigned kCut = kNone - 1u;  // .. and one whose rollout has run its last step without one

template <int V, int MODE>
struct WinStage {
    static constexpr int NS = 32 * V;   // slots per warp
    // steps of a window, one Philox block: ends are looked for, and rollouts begun, between windows (two
    // blocks a window halve the ends to handle and waste as much: 31.7 instead of 32.2 ms for 4096 spread
    // races, 6.8 instead of 5.9 for the short rollouts of a bettor population)
    static constexpr int W = 4;
    static constexpr int ROW = NS + 2;  // entries per position row: slots, the sentinel, padding to 16 bytes
    float2 pos[W][ROW];                 // (d, previous step) per slot, one row per step of a window
    float4 pq[32];                      // per competitor: (mu, sigma, P, theta)
    float kr[32];                       // per competitor: kappa (2 rho - 1)
    unsigned pha[32];                   // per competitor: StreamWords::a, the same for all rollouts
    float d0[32], prev0[32];            // per competitor: start state of every rollout
    uint4 ph[NS];                       // per slot: the current rollout's Philox constants (StreamWords)
    unsigned segk[NS];                  // by segment base: its rollout
    // rollouts to run again with everybody: a warp takes no more new ones once kRedo are listed (16 or 256: the same
    // times, few rollouts are listed)
    static constexpr bool kContenders = MODE == 0 || V <= 2;
    unsigned redo[kContenders ? kRedo + NS : 1];
    unsigned n_redo, rest[2];           // how many; first and end of those not begun for their number
    int wins[MODE == 0 ? 32 : 1];       // wins per competitor in the current work item
    // by segment base; win mode: the window's least (step, slot) and, among several crossings in that
    // step, the least tau; place mode: the least crossing key not yet placed
    union {
        unsigned win[2][NS];
        unsigned long long place[NS];
    } key;
    // Rank order (ascending position, then slot).  A segment of n slots with first slot sb has the
    // entries of `order` from 1 + 2 sb on: its slots by rank and the sentinel behind them, so the entry
    // after a slot's own is its successor's (order[0] and flag[0] are nobody's); `at` is a slot's own
    // entry and `flag` marks the entries that swap with the next.
    uint8_t order[2 * NS + 4], flag[2 * NS + 4];
    uint8_t at[NS];
    uint8_t base[NS];                   // first slot of each slot's segment
    uint8_t rank0[32], byrank0[32];     // start rank of competitor c; competitor at start rank r
    uint8_t comp[32];                   // the race's index of competitor c (its stream and its count)
};

template <int DIST>
__device__ __forceinline__ void draw_block(const uint4 &q, uint32_t a, uint32_t blk, const uint32_t (&rkey)[20],
                                           float (&z)[4])
{
    const Words4 wd = philox4x32_10_from(StreamWords{a, q.x, q.y, q.z, q.w}, blk, rkey);
    if (DIST == BBE_DIST_NORMAL) {
        box_muller2(wd, z[0], z[1], z[2], z[3]);
    } else if (DIST == BBE_DIST_UNIFORM) {
        z[0] = uniform_z(wd.w0);
        z[1] = uniform_z(wd.w1);
        z[2] = uniform_z(wd.w2);
        z[3] = uniform_z(wd.w3);
    } else {
        z[0] = two_point_z(wd.w0);
        z[1] = two_point_z(wd.w1);
        z[2] = two_point_z(wd.w2);
        z[3] = two_point_z(wd.w3);
    }
}

// Registers per thread: 80 for two to four slots per lane (6 resident 4-warp blocks per SM); with 72 and
// 7 blocks it is the same (4096 races of 20 24.6 and 24.4 ms, places to the third of 512 12.6 and 12.5, full
// orders of 96 19.1 both).  One slot per lane: 64 for win counts, which spill nothing then (26 batches
// forced to that layout, 200 us or more each, 7 % faster at the mean than with 56; the smallest calls
// the same), 56 in place mode.  Three and four slots per lane read their parameters from shared memory.
template <int V, int MODE>
struct WinRegs {
    static constexpr int value = V == 1 ? (MODE == 0 ? 64 : 56) : 80;
};
// Parameters read from shared memory each step instead of held in registers.
template <int V>
struct WinLean {
    static constexpr bool value = V >= 3;
};

// MODE 0: win counts, each rollout run to its first finisher.  MODE 1: place counts (and the
// ordered tallies), each rollout run until K = min(l.places, n) competitors have crossed; the
// finished ones keep moving and blocking, a competitor has crossed exactly when its position is
// at least L (positions only grow), and the finishers of a step are placed in (tau, slot) order.
template <int DIST, int V, int LAW, int MODE>
__global__ void __maxnreg__((WinRegs<V, MODE>::value)) win_rollout_kernel(RolloutLaunch l)
{
    constexpr bool PS = WinLean<V>::value;
    using Stage = WinStage<V, MODE>;
    constexpr int NS = Stage::NS, W = Stage::W;
    constexpr int ROWB = Stage::ROW * int(sizeof(float2));
    constexpr int kSent = NS * int(sizeof(float2));  // byte offset of the sentinel (+inf: no one in front)
    extern __shared__ __align__(16) unsigned char win_smem[];
    Stage &st = reinterpret_cast<Stage *>(win_smem)[threadIdx.x >> 5];
    char *const posb = reinterpret_cast<char *>(&st.pos[0][0]);
    // place mode, per warp after all the stages: the finisher of each place (by segment base +
    // place), the places filled (by segment base), then the work item's [competitor][place] table
    uint8_t *pl_ord = nullptr, *pl_n = nullptr;
    int *pl_cnt = nullptr;
    if constexpr (MODE == 1) {
        pl_cnt = reinterpret_cast<int *>(win_smem + (blockDim.x >> 5) * sizeof(Stage)) +
                 (threadIdx.x >> 5) * (NS / 2 + l.place_cells);
        pl_ord = reinterpret_cast<uint8_t *>(pl_cnt + l.place_cells);
        pl_n = pl_ord + NS;
    }
    const DevBatch &b = l.b;
    const int lane = threadIdx.x & 31;
    if (lane == 0) {
        for (int j = 0; j < W; ++j) st.pos[j][NS] = make_float2(INFINITY, INFINITY);
    }
    for (;;) {
        int it = 0;
        if (lane == 0) it = atomicAdd(l.queue, 1);
        it = __shfl_sync(kAll, it, 0);
        if (it >= l.n_items) break;
        const WorkItem w = l.items[it];
        const int r = BBE_INDEX(w.race, b.n_races, l.status);
        const int off = b.race_off[r];
        const int n_race = BBE_INDEX(b.race_off[r + 1] - off - 1, 32, l.status) + 1;  // 1..32
        (void)BBE_INDEX(off + n_race - 1, b.n_total, l.status);
        const float L = b.L[r];
        const float invL = __fdiv_rn(1.0f, L);
        const float t0r = LAW == BBE_LAW_TIME ? b.t0[r] : 0.0f;     // time law: elapsed steps
        const float invTr = LAW == BBE_LAW_TIME ? b.invT[r] : 0.0f;  // time law: 1 / expected duration
        const uint32_t rid = b.race_ids ? uint32_t(b.race_ids[r]) : b.race_id0 + uint32_t(r);
        // a ticket: nothing to do once the race's rollouts have all been taken
        const int64_t Rr = b.R[r];
        if (l.next != nullptr) {
            int taken = 0;
            if (lane == 0) taken = *reinterpret_cast<volatile int *>(l.next + r);
            taken = __shfl_sync(kAll, taken, 0);
            if (int64_t(taken) * w.k_count >= Rr) continue;
        }
        unsigned k_begin = unsigned(w.k_begin), k_count = unsigned(w.k_count);
        const int K = MODE == 1 ? min(l.places, n_race) : 1;  // places run per rollout
        // First with the contenders alone; then, with everybody, the rollouts that ran past the horizon
        // that those were chosen for, and what was not begun for the number of those.
        enum { kFirst, kListed, kRest };
        for (int pass = kFirst;;) {
        __syncwarp();
        if (lane == 0) {
            st.n_redo = 0u;
            if (pass == kFirst) st.rest[0] = st.rest[1] = 0u;
        }
        // stage the race: lane j < n_race loads competitor j (coalesced)
        float my_d0 = INFINITY, my_mu = 1.0f, my_sg = 0.0f, my_P = 1.0f, my_th = 0.0f, my_kr = 0.0f, my_pv = 0.0f;
        if (lane < n_race) {
            const int ci = off + lane;
            my_mu = b.mu[ci];
            my_P = b.P[ci];
            my_sg = b.sigma[ci];
            my_th = b.theta[ci];
            my_d0 = b.d0[ci];
            my_kr = __fmul_rn(kKappa, __fsub_rn(__fmul_rn(2.0f, b.rho[ci]), 1.0f));
            my_pv = b.prev0 ? b.prev0[ci] : __fmul_rn(my_mu, my_P);
        }
        // the n competitors advanced, in the race's order: all of them, or the contenders
        unsigned keep = kAll >> (32 - n_race);
        int limit = l.max_steps;  // a rollout that reaches it ends undecided
        if constexpr (Stage::kContenders) {
            if (pass == kFirst && l.contenders != nullptr) {
                const Contenders who = l.contenders[r];
                if (who.keep != keep) BBE_SEEN(l, kSeenContenders, 1);
                keep = who.keep;
                limit = min(limit, who.horizon);
            }
        }
        const int n = __popc(keep);
        const int nseg = l.seg_cap > 0 ? min(NS / n, l.seg_cap) : NS / n;  // segments of this warp
        if (l.next != nullptr && pass == kFirst) {
            // as many rollouts as give every segment its share, in multiples of the ticket's
            const int mult = max(1, min(l.per_lane * nseg, l.most) / w.k_count);
            int first = 0;
            if (lane == 0) first = atomicAdd(l.next + r, mult);
            const int64_t k = int64_t(__shfl_sync(kAll, first, 0)) * w.k_count;
            if (k >= Rr) break;
            k_begin += unsigned(k);
            const int64_t share = int64_t(mult) * w.k_count;
            k_count = unsigned(share < Rr - k ? share : Rr - k);
        }
        const bool kept = (keep >> lane) & 1u;
        int rank = 0;  // by (d0, index)
        for (int i = 0; i < n_race; ++i) {
            const float di = __shfl_sync(kAll, my_d0, i);
            rank += ((keep >> i) & 1u) && (di < my_d0 || (di == my_d0 && i < lane)) ? 1 : 0;
        }
        __syncwarp();
        if (kept) {
            const int c = __popc(keep & ((1u << lane) - 1u));
            st.pq[c] = make_float4(my_mu, my_sg, my_P, my_th);
            st.kr[c] = my_kr;
            st.d0[c] = my_d0;
            st.prev0[c] = my_pv;
            st.comp[c] = uint8_t(lane);
            if constexpr (MODE == 0) st.wins[c] = 0;
            st.pha[c] = stream_words(0u, uint32_t(lane), rid, l.round_key).a;
            st.rank0[c] = uint8_t(rank);
            st.byrank0[BBE_INDEX(rank, 32, l.status)] = uint8_t(c);
        }
        for (int i = lane; i < NS; i += 32) {
            if constexpr (MODE == 1) {
                st.key.place[i] = kNoKey;
                pl_n[i] = 0;
            } else {
                st.key.win[0][i] = st.key.win[1][i] = kNone;
            }
            st.order[2 * i] = st.order[2 * i + 1] = uint8_t(NS);
            st.flag[2 * i] = st.flag[2 * i + 1] = 0;
        }
        if (lane < 4) {
            st.order[2 * NS + lane] = uint8_t(NS);
            st.flag[2 * NS + lane] = 0;
        }
        if constexpr (MODE == 1) {
            for (int i = lane; i < n * K; i += 32) pl_cnt[i] = 0;
        }
        __syncwarp();

        // unsigned: rollout indices stay below 2^31 + 2^7
        unsigned kend = k_begin + k_count;
        unsigned next_k = k_begin + unsigned(nseg);  // warp-uniform (as kend): the next segment that is free takes it

        // per slot: segment base, competitor parameters, state, front address, rollout, block
        int fo[V];
        unsigned blk[V], pha[V];
        float mu[V], sg[V], P[V], th[V], kr[V], d[V], pv[V];
        const float4 *pqa[V];  // register-lean variant: this slot's (mu, sigma, P, theta)
        const float *kra[V];   // register-lean variant: this slot's kappa (2 rho - 1)
        // a slot that runs no rollout has no position (NaN): it is never out of order, never over
        // the line, and stays so without a test in the step
        auto alive = [&](int v) { return d[v] == d[v]; };
        auto base = [&](int v) { return int(st.base[32 * v + lane]); };
        // slot's stream for rollout k (competitor c of the advanced ones)
        auto set_stream = [&](int slot, unsigned k, int c) {
            if (pass == kListed && k < kend) k = st.redo[BBE_INDEX(k, kRedo + NS, l.status)];
            const StreamWords q = stream_words(k, uint32_t(st.comp[c]), rid, l.round_key);
            st.ph[slot] = make_uint4(q.d, q.e, q.f, q.g);
        };
        const float kDead = __int_as_float(0x7fffffff);
        unsigned long long steps = 0;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const int slot = 32 * v + lane;
            const int seg = slot / n;
            const bool used = seg < nseg;
            const int sb = used ? seg * n : slot;
            const int c = used ? slot - seg * n : 0;
            const unsigned k = k_begin + unsigned(seg);
            const bool run = used && k < kend;
            if (slot == sb) st.segk[slot] = k;
            st.base[slot] = uint8_t(sb);
            const int rb = 1 + 2 * sb;
            st.at[slot] = uint8_t(rb);
            set_stream(slot, k, c);
            blk[v] = 0;
            if constexpr (PS) {
                pqa[v] = &st.pq[c];
                kra[v] = &st.kr[c];
            } else {
                pha[v] = st.pha[c];
                const float4 q = st.pq[c];
                mu[v] = q.x;
                sg[v] = q.y;
                P[v] = q.z;
                th[v] = q.w;
                kr[v] = st.kr[c];
            }
            d[v] = run ? st.d0[c] : kDead;
            pv[v] = st.prev0[c];
            const int r0 = st.rank0[c];
            fo[v] = (run && r0 + 1 < n) ? BBE_INDEX(sb + st.byrank0[r0 + 1], NS, l.status) * int(sizeof(float2)) : kSent;
            if (run) {
                st.order[BBE_INDEX(rb + r0, 2 * NS + 4, l.status)] = uint8_t(slot);
                st.at[slot] = uint8_t(rb + r0);
            }
        }
        __syncwarp();

        // A segment whose rank order broke in more than isolated pairs, or with equal positions: odd-even
        // transposition by (position, slot) from the order that there was, which a step leaves a few
        // swaps from sorted; then every slot takes its successor, or if that stands level with it the
        // first later rank strictly in front.  (A count of every slot's rank, over all of its segment, took
        // 727 instead of 346 us where chains of overtakes are the rule: 116 bunched races of 30 to the sixth
        // place, 170 rollouts each; 700 of 13 14.45 instead of 14.16 ms.)  pb is the step's row.
        // In a pass a slot whose turn it is not reads its successor's entry while the pair behind it may be
        // swapping: it finds one or the other, which only decides whether there is another pass, and there is
        // one wherever somebody swapped.  Entries that count are read in passes that write none of them.
        auto full_sort = [&](const char *pb, float (&fd)[V], float (&fp)[V]) {
            const float2 *row = reinterpret_cast<const float2 *>(pb);
            __syncwarp();
            for (int pass = 0; pass < 2 * 32 + 2; ++pass) {  // n passes sort any order of n
                int a[V];
#pragma unroll
                for (int v = 0; v < V; ++v) a[v] = st.at[32 * v + lane];
                __syncwarp();
                bool inv = false;
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    const int slot = 32 * v + lane;
                    const int s2 = st.order[BBE_INDEX(a[v] + 1, 2 * NS + 4, l.status)];
                    const float d2 = row[BBE_INDEX(s2, NS + 1, l.status)].x;
                    const bool swap = alive(v) && (d2 < d[v] || (d2 == d[v] && s2 < slot));
                    inv |= swap;
                    // the rank's parity: entries of a segment start behind an even number
                    if (swap && ((a[v] ^ pass) & 1)) {
                        st.order[a[v]] = uint8_t(s2);
                        st.order[a[v] + 1] = uint8_t(slot);
                        st.at[s2] = uint8_t(a[v]);
                        st.at[slot] = uint8_t(a[v] + 1);
                    }
                }
                const bool more = __any_sync(kAll, inv);
                __syncwarp();
                if (!more) break;
            }
#pragma unroll
            for (int v = 0; v < V; ++v) {
                if (!alive(v)) continue;
                float2 f;
                for (int a = int(st.at[32 * v + lane]) + 1, q = 0; q < n; ++a, ++q) {
                    const int o = st.order[BBE_INDEX(a, 2 * NS + 4, l.status)] * int(sizeof(float2));
                    if (q == 0) fo[v] = o;
                    f = *reinterpret_cast<const float2 *>(pb + o);
                    if (f.x > d[v]) break;  // the sentinel behind the last rank is
                }
                fd[v] = f.x;
                fp[v] = f.y;
            }
            __syncwarp();
        };

        // The common case first: isolated overtakes.  A slot whose successor is now strictly
        // behind it swaps entries with that successor, unless a neighbouring pair swaps too (a
        // chain); the slots whose successor that changed read it, and what is still out of order or
        // level goes to the full sort.
        auto repair = [&](const char *pb, float (&fd)[V], float (&fp)[V]) {
            int a[V];
            bool init[V];
#pragma unroll
            for (int v = 0; v < V; ++v) {
                init[v] = fd[v] < d[v];
                a[v] = st.at[32 * v + lane];
                if (init[v]) st.flag[a[v]] = 1;
            }
            __syncwarp();
            bool ok[V];
#pragma unroll
            for (int v = 0; v < V; ++v) ok[v] = init[v] && st.flag[a[v] - 1] == 0 && st.flag[a[v] + 1] == 0;
            __syncwarp();
#pragma unroll
            for (int v = 0; v < V; ++v) {
                if (!init[v]) continue;
                st.flag[a[v]] = 0;
                if (ok[v]) {
                    const int f = BBE_INDEX(fo[v] / int(sizeof(float2)), NS, l.status);
                    st.order[a[v]] = uint8_t(f);
                    st.order[a[v] + 1] = uint8_t(32 * v + lane);
                    st.at[f] = uint8_t(a[v]);
                    st.at[32 * v + lane] = uint8_t(a[v] + 1);
                }
            }
            __syncwarp();
            bool again = false;
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const int o = st.order[BBE_INDEX(int(st.at[32 * v + lane]) + 1, 2 * NS + 4, l.status)] * int(sizeof(float2));
                if (o != fo[v] && alive(v)) {
                    fo[v] = o;
                    const float2 f = *reinterpret_cast<const float2 *>(pb + o);
                    fd[v] = f.x;
                    fp[v] = f.y;
                }
                again |= fd[v] <= d[v];
            }
            if (__any_sync(kAll, again)) full_sort(pb, fd, fp);
        };

        // Steps of a window past a crossing, or past the step limit, change nothing that counts (the
        // rollout ends with the window in any case), so crossings are looked for once a window: positions
        // only grow, and the window's rows say which step it was.  The step in the window, for a slot that
        // has crossed in it, and its tau = (L - d) / S:
        auto crossing = [&](int v) {
            int J = 0;
#pragma unroll
            for (int j = 1; j < W; ++j) J += st.pos[j][32 * v + lane].x < L ? 1 : 0;
            return J;
        };
        auto crossing_tau = [&](int v, int J) {
            const int slot = 32 * v + lane;
            const float S = J + 1 < W ? st.pos[J + 1][slot].y : pv[v];
            return __float_as_uint(__fdiv_rn(__fsub_rn(L, st.pos[J][slot].x), S));
        };

        // Win mode, the end of a window with a crossing (or, chk, one in which a rollout may have run its
        // last step): the least (step, slot) of each segment.  Where several crossed in that step, the least
        // tau wins and, among equals, the least slot (tau >= 0, so its bits order like its value); alone,
        // a crossing needs no tau.
        auto win_end = [&](bool chk, bool (&pend)[V], bool (&again)[V]) {
            unsigned mine[V], kw[V];
#pragma unroll
            for (int v = 0; v < V; ++v) {
                mine[v] = kNone;
                if (d[v] >= L) {
                    const int J = crossing(v);
                    if (!chk || int(blk[v]) * 4 - W + J < limit) {
                        mine[v] = unsigned(J) << 8 | unsigned(32 * v + lane);
                        atomicMin(&st.key.win[0][base(v)], mine[v]);
                    }
                }
                if (chk && alive(v) && int(blk[v]) * 4 >= limit) atomicMin(&st.key.win[0][base(v)], kCut);
            }
            __syncwarp();
            bool tie = false;
#pragma unroll
            for (int v = 0; v < V; ++v) {
                kw[v] = alive(v) ? st.key.win[0][base(v)] : kNone;
                pend[v] = kw[v] != kNone;
                tie |= mine[v] > kw[v] && (mine[v] >> 8) == (kw[v] >> 8);
            }
            if (__any_sync(kAll, tie)) {
                unsigned tau[V];
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    tau[v] = kNone;
                    if (mine[v] != kNone && (mine[v] >> 8) == (kw[v] >> 8)) {
                        tau[v] = crossing_tau(v, int(mine[v] >> 8));
                        atomicMin(&st.key.win[1][base(v)], tau[v]);
                    }
                    if (pend[v] && kw[v] != kCut && 32 * v + lane == base(v)) st.key.win[0][base(v)] = kw[v] | 255u;
                }
                __syncwarp();
#pragma unroll
                for (int v = 0; v < V; ++v)
                    if (tau[v] != kNone && tau[v] == st.key.win[1][base(v)]) atomicMin(&st.key.win[0][base(v)], mine[v]);
                __syncwarp();
#pragma unroll
                for (int v = 0; v < V; ++v)
                    if (pend[v]) kw[v] = st.key.win[0][base(v)];
            }
            __syncwarp();
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const int slot = 32 * v + lane;
                if (!pend[v] || slot != base(v)) continue;
                if (kw[v] == kCut) {
                    if (limit >= l.max_steps) {
                        atomicOr(l.status, kStatusStepLimit);
                        steps += (unsigned long long)l.max_steps;
                    } else {
                        again[v] = true;
                    }
                } else {
                    atomicAdd(&st.wins[BBE_INDEX(int(kw[v] & 255u) - slot, 32, l.status)], 1);
                    steps += (unsigned long long)(blk[v] * 4u - unsigned(W - 1) + (kw[v] >> 8));
                }
                st.key.win[0][slot] = st.key.win[1][slot] = kNone;
            }
        };

        // Place mode, the same: the window's crossings of each segment take the next places one at a
        // time in key order (step, tau, slot), and a segment whose K-th place is filled ends its
        // rollout; one stopped at max_steps that did not end earlier counts for nobody.
        auto place_end = [&](bool chk, bool (&pend)[V], bool (&again)[V]) {
            unsigned long long fk[V];
            int sb[V];
            bool more = false;
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const int slot = 32 * v + lane;
                sb[v] = base(v);
                fk[v] = kNoKey;
                if (d[v] >= L && st.pos[0][slot].x < L) {
                    const int J = crossing(v);
                    if (!chk || int(blk[v]) * 4 - W + J < limit) {
                        fk[v] = (static_cast<unsigned long long>(J) << 40) |
                                (static_cast<unsigned long long>(crossing_tau(v, J)) << 8) | unsigned(slot);
                        more = true;
                    }
                }
            }
            // one crossing per segment per round; a segment has at most n of them
            for (int round = 0; round < NS && __any_sync(kAll, more); ++round) {
#pragma unroll
                for (int v = 0; v < V; ++v)
                    if (fk[v] != kNoKey) atomicMin(&st.key.place[sb[v]], fk[v]);
                __syncwarp();
                bool won[V];
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    won[v] = fk[v] != kNoKey && st.key.place[sb[v]] == fk[v];
                    if (won[v] && pl_n[sb[v]] < K) {
                        const int p = BBE_INDEX(int(pl_n[sb[v]]), K, l.status);
                        pl_ord[sb[v] + p] = uint8_t(32 * v + lane - sb[v]);
                        pl_n[sb[v]] = uint8_t(p + 1 < K ? p + 1 : kPlaced + int(fk[v] >> 40));
                    }
                }
                __syncwarp();
                more = false;
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    if (fk[v] != kNoKey) st.key.place[sb[v]] = kNoKey;
                    if (won[v]) fk[v] = kNoKey;
                    more |= fk[v] != kNoKey;
                }
                __syncwarp();
            }
#pragma unroll
            for (int v = 0; v < V; ++v) {
                if (!alive(v)) continue;
                const int slot = 32 * v + lane;
                const unsigned filled = pl_n[sb[v]];
                if (filled >= kPlaced) {
                    if (slot == sb[v]) steps += (unsigned long long)(blk[v] * 4u - unsigned(W - 1) + filled - kPlaced);
                    pend[v] = true;
                } else if (chk && int(blk[v]) * 4 >= limit) {
                    if (limit >= l.max_steps) {
                        if (slot == sb[v]) steps += (unsigned long long)l.max_steps;
                        atomicOr(l.status, kStatusStepLimit);
                    } else {
                        again[v] = slot == sb[v];
                    }
                    pend[v] = true;
                }
            }
        };

        // Place mode, at a block boundary: the segments that completed a rollout (K places filled;
        // a rollout cut off at max_steps fills fewer and counts for nobody) add one count per
        // place and, for the ordered tallies, their order: as one base-n number (the dense
        // tables, K <= 3) and as the order key, the mixed-radix number whose digit j (radix
        // n - j) is the place-j finisher's index among the competitors not yet placed.
        auto tally_completed = [&](const bool (&pend)[V]) {
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const int sb = base(v);
                if (!pend[v] || pl_n[sb] < kPlaced) continue;
                const int c = 32 * v + lane - sb;  // this slot's competitor
                if (c < K) atomicAdd(&pl_cnt[BBE_INDEX(pl_ord[sb + c] * K + c, n * K, l.status)], 1);
                if (c == 0 && (l.orders != nullptr || l.hist_keys != nullptr)) {
                    unsigned code = 0u, taken = 0u;
                    unsigned long long key = 0ull;
                    for (int j = 0; j < K; ++j) {
                        const int cj = st.comp[pl_ord[sb + j]];
                        code = code * unsigned(n_race) + unsigned(cj);
                        key = key * unsigned(n_race - j) + unsigned(__popc(((1u << cj) - 1u) & ~taken));
                        taken |= 1u << cj;
                    }
                    if (l.orders != nullptr) {
#if defined(BBE_CHECKED) && BBE_CHECKED
                        unsigned cells = 1u;  // n^K entries in the race's dense table
                        for (int j = 0; j < K; ++j) cells *= unsigned(n_race);
#endif
                        atomicAdd(&l.orders[l.order_off[r] + BBE_INDEX(code, cells, l.status)], 1);
                    }
                    if (l.hist_keys != nullptr) {
                        const int64_t h0 = l.hist_off[r];
                        hist_insert(l.hist_keys + h0, l.hist_counts + h0, l.hist_off[r + 1] - h0, key, l.status);
                    }
                }
            }
            __syncwarp();
        };

        // One step of every slot: step j0 + J of the window, with the normal z[v][J].
        int j0 = 0;
        auto step = [&](auto Jc, const float (&z)[V][4]) {
            constexpr int J = decltype(Jc)::value;
            const int BO = (j0 + J) * ROWB;
            // publish this step's (d, previous step) of every slot
#pragma unroll
            for (int v = 0; v < V; ++v)
                *reinterpret_cast<float2 *>(posb + BO + (32 * v + lane) * 8) = make_float2(d[v], pv[v]);
            __syncwarp();
            float fd[V], fp[V];
            bool bad = false;
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const float2 f = *reinterpret_cast<const float2 *>(posb + BO + BBE_INDEX(fo[v], kSent + 1, l.status));
                fd[v] = f.x;
                fp[v] = f.y;
                bad |= f.x <= d[v];
            }
            if (__any_sync(kAll, bad)) repair(posb + BO, fd, fp);
            // Eq. 1 (a successor at +inf is never within theta: the free branch)
#pragma unroll
            for (int v = 0; v < V; ++v) {
                float kv, thv, Pv, sgv, muv;
                if constexpr (PS) {
                    const float4 q = *pqa[v];
                    muv = q.x;
                    sgv = q.y;
                    Pv = q.z;
                    thv = q.w;
                    kv = *kra[v];
                } else {
                    muv = mu[v];
                    sgv = sg[v];
                    Pv = P[v];
                    thv = th[v];
                    kv = kr[v];
                }
                const float Rc = responsiveness<LAW>(kv, d[v], invL, t0r, int(blk[v]) * 4 + j0 + J, invTr);
                const bool blocked = !(__fsub_rn(fd[v], d[v]) > thv);
                float Sv = blocked ? __fmul_rn(Rc, fminf(pv[v], fp[v]))
                                   : __fmul_rn(__fmul_rn(Rc, Pv), __fmaf_rn(sgv, z[v][J], muv));
                Sv = fmaxf(Sv, kStepFloor);
                d[v] = __fadd_rn(d[v], Sv);
                pv[v] = Sv;
            }
        };

        // windows before one at whose end a rollout can have run `limit` steps: no slot is further into
        // its rollout than the windows the work item has run, so a warp-uniform count-down rules the
        // check out in all but the longest items
        unsigned left = unsigned(max(limit, 1) - 1) / unsigned(W);
        for (bool live = k_count > 0u; live;) {
            // a block's normals: one Philox4x32-10 output per slot, counter (k, t >> 2, c, race)
            float z[V][4];
            auto draw = [&]() {
#pragma unroll
                for (int v = 0; v < V; ++v)
                    draw_block<DIST>(st.ph[32 * v + lane], PS ? st.pha[kra[v] - st.kr] : pha[v], blk[v], l.round_key, z[v]);
            };
            if constexpr (MODE == 0) {
                // two copies of the step, run twice (the second time with the block's other two normals): with
                // four, the steps and their repairs overflow the instruction cache where overtakes are frequent
                // (700 bunched races of 13: 15.3 instead of 14.6 ms; spread races without overtakes lose 1 to 2 %)
#pragma unroll 1
                for (j0 = 0; j0 < W; j0 += 2) {
                    if (j0 == 0) {
                        draw();
                    } else {
#pragma unroll
                        for (int v = 0; v < V; ++v) {
                            z[v][0] = z[v][2];
                            z[v][1] = z[v][3];
                        }
                    }
                    step(std::integral_constant<int, 0>{}, z);
                    step(std::integral_constant<int, 1>{}, z);
                }
            } else {
                draw();
                step(std::integral_constant<int, 0>{}, z);
                step(std::integral_constant<int, 1>{}, z);
                step(std::integral_constant<int, 2>{}, z);
                step(std::integral_constant<int, 3>{}, z);
            }
            const bool chk = left == 0u;
            if (!chk) --left;
            bool event = false;
#pragma unroll
            for (int v = 0; v < V; ++v) {
                blk[v] += unsigned(W / 4);
                event |= d[v] >= L && (MODE == 0 || st.pos[0][32 * v + lane].x < L);
            }
            if (chk) {
#pragma unroll
                for (int v = 0; v < V; ++v) event |= alive(v) && int(blk[v]) * 4 >= limit;
            }
            if (!__any_sync(kAll, event)) continue;

            // rollouts have ended: the segments that ran them take the next ones
            bool pend[V], again[V];  // rollout ended; at a segment's base: it is to be run again with everybody
#pragma unroll
            for (int v = 0; v < V; ++v) pend[v] = again[v] = false;
            if constexpr (MODE == 0) {
                win_end(chk, pend, again);
            } else {
                place_end(chk, pend, again);
                __syncwarp();
                tally_completed(pend);
            }
            if (Stage::kContenders && chk && limit < l.max_steps) {
                unsigned n_redo = st.n_redo;
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    const unsigned m = __ballot_sync(kAll, again[v]);
                    if (again[v])
                        st.redo[BBE_INDEX(n_redo + unsigned(__popc(m & ((1u << lane) - 1u))), kRedo + NS, l.status)] =
                            st.segk[32 * v + lane];
                    n_redo += unsigned(__popc(m));
                }
                __syncwarp();
                if (lane == 0) st.n_redo = n_redo;
                if (n_redo >= kRedo && next_k < kend) {
                    if (lane == 0) {
                        st.rest[0] = next_k;
                        st.rest[1] = kend;
                    }
                    kend = next_k;
                }
            }
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const int slot = 32 * v + lane;
                const bool lead = pend[v] && slot == base(v);
                const unsigned m = __ballot_sync(kAll, lead);
                if (lead) {
                    st.segk[slot] = next_k + unsigned(__popc(m & ((1u << lane) - 1u)));
                    if constexpr (MODE == 1) pl_n[slot] = 0;
                }
                next_k += unsigned(__popc(m));
            }
            __syncwarp();
            live = false;
#pragma unroll
            for (int v = 0; v < V; ++v) {
                if (pend[v]) {
                    const int slot = 32 * v + lane, sb = base(v);
                    const unsigned knew = st.segk[sb];
                    d[v] = kDead;
                    fo[v] = kSent;
                    if (knew < kend) {
                        const int c = slot - sb;
                        set_stream(slot, knew, c);
                        blk[v] = 0;
                        d[v] = st.d0[c];
                        pv[v] = st.prev0[c];
                        const int r0 = st.rank0[c];
                        if (r0 + 1 < n) fo[v] = (sb + st.byrank0[r0 + 1]) * int(sizeof(float2));
                        const int a = 1 + 2 * sb + r0;
                        st.order[a] = uint8_t(slot);
                        st.at[slot] = uint8_t(a);
                    }
                }
                live |= alive(v);
            }
            live = __any_sync(kAll, live);
            __syncwarp();
        }

        // one global atomic per competitor with wins (per competitor and place in place mode), one
        // for the step total
        __syncwarp();
        if constexpr (MODE == 1) {
            for (int i = lane; i < n * K && l.counts != nullptr; i += 32) {
                const int cc = pl_cnt[i];
                if (cc != 0) atomicAdd(&l.counts[(off + st.comp[i / K]) * l.places + i % K], cc);
            }
        } else {
            if (lane < n && st.wins[lane] != 0) atomicAdd(&l.counts[off + st.comp[lane]], st.wins[lane]);
        }
        for (int o = 16; o > 0; o >>= 1) steps += __shfl_xor_sync(kAll, steps, o);
        if (lane == 0 && l.steps != nullptr) atomicAdd(l.steps + r, steps);
        __syncwarp();
        const unsigned listed = st.n_redo;
        if (listed > 0u) {
            BBE_SEEN(l, kSeenListed, listed);
            pass = kListed;
            k_begin = 0u;
            k_count = listed;
        } else {
            k_begin = st.rest[0];
            k_count = st.rest[1] - k_begin;
            if (pass == kRest || k_count == 0u) break;
            BBE_SEEN(l, kSeenRest, 1);
            pass = kRest;
        }
        }
    }
}

// Dynamic shared memory of a block: the warps' stages, then in place mode each warp's place
// lists (2 x 32 V bytes) and [competitor][place] table (place_cells ints).
template <int V, int MODE>
size_t win_stage_bytes(int block, int place_cells)
{
    const size_t warps = size_t(block / 32);
    return warps * sizeof(WinStage<V, MODE>) + (MODE == 1 ? warps * (16 * V + size_t(place_cells)) * sizeof(int) : 0);
}

// The largest place table a launch may ask for (32 competitors x 32 places).
constexpr int kMaxPlaceCells = 32 * 32;
static_assert(16 * (sizeof(WinStage<4, 1>) + 4 * (16 * 4 + kMaxPlaceCells)) <= 227 * 1024, "the largest block");

template <int V, int LAW, int MODE>
cudaError_t launch_win_vl(const RolloutLaunch &l, cudaStream_t stream)
{
    const size_t smem = win_stage_bytes<V, MODE>(l.block, l.place_cells);
    switch (l.b.dist) {
    case BBE_DIST_NORMAL: win_rollout_kernel<BBE_DIST_NORMAL, V, LAW, MODE><<<l.grid, l.block, smem, stream>>>(l); break;
    case BBE_DIST_UNIFORM: win_rollout_kernel<BBE_DIST_UNIFORM, V, LAW, MODE><<<l.grid, l.block, smem, stream>>>(l); break;
    default: win_rollout_kernel<BBE_DIST_TWO_POINT, V, LAW, MODE><<<l.grid, l.block, smem, stream>>>(l); break;
    }
    return cudaGetLastError();
}

// Blocks resident per SM.  Also lets the kernels take the dynamic shared memory of the largest
// block (16 warps may need more than the default 48 KB); every launch path asks this first.
template <int DIST, int V, int LAW, int MODE>
int win_resident_dvl(int block, int place_cells)
{
    const void *fn = reinterpret_cast<const void *>(win_rollout_kernel<DIST, V, LAW, MODE>);
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             int(win_stage_bytes<V, MODE>(512, MODE == 1 ? kMaxPlaceCells : 0))) != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    int nb = 0;
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, win_rollout_kernel<DIST, V, LAW, MODE>,
                                                                        block, win_stage_bytes<V, MODE>(block, place_cells));
    return e == cudaSuccess ? nb : 1;
}

// The launch and the residency query of the kernels of one responsiveness law and mode (each
// law's kernels are compiled in a translation unit of their own).
template <int LAW, int MODE>
cudaError_t launch_law(const RolloutLaunch &l, int slots_per_lane, cudaStream_t stream)
{
    switch (slots_per_lane) {
    case 4: return launch_win_vl<4, LAW, MODE>(l, stream);
    case 3: return launch_win_vl<3, LAW, MODE>(l, stream);
    case 2: return launch_win_vl<2, LAW, MODE>(l, stream);
    default: return launch_win_vl<1, LAW, MODE>(l, stream);
    }
}

template <int LAW, int MODE>
int resident_law(int dist, int slots_per_lane, int block, int place_cells)
{
    auto one = [&](auto Vc) {
        constexpr int V = decltype(Vc)::value;
        switch (dist) {
        case BBE_DIST_NORMAL: return win_resident_dvl<BBE_DIST_NORMAL, V, LAW, MODE>(block, place_cells);
        case BBE_DIST_UNIFORM: return win_resident_dvl<BBE_DIST_UNIFORM, V, LAW, MODE>(block, place_cells);
        default: return win_resident_dvl<BBE_DIST_TWO_POINT, V, LAW, MODE>(block, place_cells);
        }
    };
    switch (slots_per_lane) {
    case 4: return one(std::integral_constant<int, 4>{});
    case 3: return one(std::integral_constant<int, 3>{});
    case 2: return one(std::integral_constant<int, 2>{});
    default: return one(std::integral_constant<int, 1>{});
    }
}

cudaError_t launch_position_law(const RolloutLaunch &l, int slots_per_lane, cudaStream_t stream);
int resident_position_law(int dist, int slots_per_lane, int block);
cudaError_t launch_time_law(const RolloutLaunch &l, int slots_per_lane, cudaStream_t stream);
int resident_time_law(int dist, int slots_per_lane, int block);

}  // namespace win

}  // namespace bbe
