// Growing steps inside one launch: the pushed form of a Delta-growing step and the control loop of CLUSTER that runs
// steps and stages back to back, by the CTAs of one thread-block cluster (k_grow, large jobs of a batch) or by one CTA
// (the other jobs of a batch, served requests).
#pragma once

#include "cluster_dev.cuh"

namespace cld {

// a5, pushed form: the frontier's adjacency lists are one flattened range of E
// positions; each warp takes QC consecutive positions (4 groups of 32), finds
// the entries they span from the chunk table (cfirst, written by the frontier
// producers) and maps positions to entries with the start words.  A pushing
// entry (start-of-step key of its node) sends (d_u + w, c_u) to each
// neighbour: a key read (evict-last) filters candidates that cannot win, the
// rest lower the neighbour's key with a no-return atomic minimum.  A pulling
// entry (an unfrozen node that reads the candidates of its contracted
// neighbours, kPullTag | v) reduces its candidates over its lanes first, so
// it lowers its own key once per group segment.  No block barrier.
// RESIDENT: the kernel runs many steps (k_grow), so node state is read past L1, whose lines may be older than a
// stage's reset; a one-step launch reads through L1 (a stale line only lets an extra candidate through).  Its
// positions and ids come from lists that other CTAs wrote earlier in the same launch, so they are checked against the
// graph's sizes (n, nnz) before use; one outside them would set ctr->bad.
template <int WARPS>
struct PushSmem {
    unsigned long long skey[WARPS][QC + 2];
    uint32_t spre[WARPS][QC + 1];  // first positions of the entries after the chunk's first
    uint32_t sbase[WARPS][QC + 2];
    uint32_t sbuf[WARPS][PNB];
};

// A frontier that the warps hold in PushSmem instead of the lists: this warp's entries and their positions.
struct Held {
    uint32_t ne = 0, total = 0;
    bool on = false;
};

template <bool RESIDENT, int WARPS>
__device__ __forceinline__ void dev_push(const uint32_t* __restrict__ fbase, const unsigned long long* __restrict__ fkey,
                                         const uint32_t* __restrict__ fpre, const uint32_t* __restrict__ cfirst,
                                         uint32_t nf, uint32_t E, const uint2* __restrict__ adj,
                                         const uint32_t* __restrict__ center, const uint32_t* __restrict__ Dcum,
                                         unsigned long long* __restrict__ key, uint32_t delta,
                                         uint32_t* __restrict__ stamp, uint32_t stepid,
                                         uint32_t* __restrict__ next, Counters* ctr, PushSmem<WARPS>& smp, uint32_t br,
                                         uint32_t nb, uint32_t n = 0, uint32_t nnz = 0,
                                         const Held held = Held{}) {
    auto& spre = smp.spre;
    auto& sbase = smp.sbase;
    auto& skey = smp.skey;
    auto& sbuf = smp.sbuf;
    const uint32_t lane = lane_id(), warp = threadIdx.x >> 5;
    const uint64_t pol_stream = l2_evict_first_policy(), pol_keep = l2_evict_last_policy();
    const unsigned le_mask = 0xffffffffu >> (31u - lane);
    WarpNext wn{sbuf[warp], 0};
    unsigned long long newly = 0;
    bool bad = false;
    const uint32_t nq = (uint32_t)(((uint64_t)E + QC - 1) / QC);
    const uint32_t nwarps = nb * WARPS;
    const bool mine = RESIDENT && held.on;  // the warp's own entries, else chunks of the lists
    const uint32_t qend = mine ? (held.total + QC - 1) / QC : nq, qstep = mine ? 1u : nwarps;
    uint32_t B = 0;
    for (uint32_t q = mine ? 0u : br * WARPS + warp; q < qend; q += qstep) {
        const uint32_t p0 = q * QC, e1 = min(mine ? held.total : E, p0 + QC);
        uint32_t ne = held.ne;
        if (!mine) {
            // entry i0 holds p0; entries i0 + 1 .. il start inside (p0, p0 + QC] (at most QC of them)
            const uint32_t i0 = __ldcg(&cfirst[q]);
            const uint32_t il = q + 1 < nq ? __ldcg(&cfirst[q + 1]) : nf - 1;
            if (RESIDENT && (i0 > il || il >= nf)) {
                bad = true;
                continue;
            }
            ne = min(il - i0 + 1, (uint32_t)QC + 1);
            if (RESIDENT) __syncwarp();  // the previous chunk's entries have been read
            for (uint32_t j = lane; j < ne; j += 32) {
                if (j) spre[warp][j - 1] = __ldcg(&fpre[i0 + j]);
                sbase[warp][j] = __ldcg(&fbase[i0 + j]);
                skey[warp][j] = __ldcg(&fkey[i0 + j]);
            }
            __syncwarp();
            B = 0;
        }
        uint32_t word[4], own[4];
        {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                word[u] = group_starts(spre[warp] + B, ne - 1 - B, p0 + 32u * u, B, lane, le_mask, &own[u]);
                B += (uint32_t)__popc(word[u]);
            }
        }
        uint2 ed[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const uint32_t p = p0 + 32u * u + lane;
            bool in = p < e1;
            if (RESIDENT && in && (own[u] >= ne || sbase[warp][own[u]] + p >= nnz)) {
                bad = true;
                in = false;
            }
            ed[u] = in ? ld_stream_u2(adj + (sbase[warp][own[u]] + p), pol_stream) : make_uint2(0u, 0xFFFFFFFFu);
        }
        // RESIDENT: the groups' loads and exchanges are issued level by level for all four groups, since few warps
        // share the latency (one group after another, a push took 14,000 cycles, so 8,200)
        uint32_t pcu[4], pdu[4], tgt[4];
        unsigned long long cnk[4];
        if constexpr (RESIDENT) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                pcu[u] = kNone;
                pdu[u] = 0;
                if ((skey[warp][own[u]] & kPullTag) == kPullTag && ed[u].y <= delta) {
                    pcu[u] = __ldcg(&center[ed[u].x]);
                    if (Dcum) pdu[u] = __ldcg(&Dcum[ed[u].x]);
                }
            }
        }
        unsigned long long carry = kInfKey;  // pull entry still open at the previous group's end
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const unsigned long long ku = skey[warp][own[u]];
            const bool is_pull = (ku & kPullTag) == kPullTag;
            const bool live = p0 + 32u * u + lane < e1;
            unsigned long long nk = kInfKey;
            uint32_t target = 0;
            if (live && !is_pull) {
                const uint64_t cand = (ku >> 32) + ed[u].y;
                if (cand <= delta) {
                    target = ed[u].x;
                    nk = (cand << 32) | (ku & 0xFFFFFFFFull);
                }
            } else if (live && ed[u].y <= delta) {  // pull: candidate of a contracted neighbour
                uint32_t cu, du = 0;
                if constexpr (RESIDENT) {
                    cu = pcu[u];
                    du = pdu[u];
                } else {
                    cu = __ldg(&center[ed[u].x]);
                    if (cu != kNone && Dcum) du = __ldg(&Dcum[ed[u].x]);
                }
                const uint64_t cand = (uint64_t)du + ed[u].y;
                if (cu != kNone && cand <= delta) nk = (cand << 32) | cu;
            }
            // pulling entries: one candidate per segment (all lanes of an entry share its kind)
            if (__any_sync(0xffffffffu, is_pull)) {
                unsigned long long pv = is_pull ? nk : kInfKey;
                if (lane == 0 && !(word[u] & 1u)) pv = carry < pv ? carry : pv;
                pv = segment_min(pv, word[u], lane);
                const uint32_t last_head = word[u] ? 31u - (uint32_t)__clz(word[u]) : 0u;
                const bool cont = u < 3 && !(word[(u + 1) & 3] & 1u);
                carry = __shfl_sync(0xffffffffu, pv, last_head);
                const unsigned le = word[u] & le_mask;
                const uint32_t head = le ? 31u - (uint32_t)__clz(le) : 0u;
                if (is_pull) {
                    const bool flush = lane == head && !(cont && head == last_head);
                    nk = flush ? pv : kInfKey;
                    target = (uint32_t)ku;
                }
            } else {
                carry = kInfKey;
            }
            if constexpr (RESIDENT) {
                if (nk != kInfKey && target >= n) {
                    bad = true;
                    nk = kInfKey;
                }
                cnk[u] = nk;
                tgt[u] = target;
            } else {
                bool first = false;
                if (nk != kInfKey) {
                    // the target's key and stamp in one round trip, through L1 (a stale line only lets an
                    // extra candidate through: keys only fall within a launch, and the atomics decide); most
                    // candidates lose to the current key
                    const unsigned long long cur = ld_keep_u64(&key[target], pol_keep);
                    const uint32_t stp = ld_keep_u32(&stamp[target], pol_keep);
                    if (nk < cur) {
                        red_min_keep_u64(&key[target], nk, pol_keep);
                        if (stp != stepid) {  // hubs see many lowerings: only the first ones exchange
                            const uint32_t old = atomicExch(&stamp[target], stepid);
                            first = old != stepid;
                            newly += old == 0u ? 1 : 0;
                        }
                    }
                }
                wn.put(first, target, lane);
            }
        }
        if constexpr (RESIDENT) {
            unsigned long long cur[4];
            uint32_t stp[4], old[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const bool has = cnk[u] != kInfKey;
                cur[u] = has ? ld_cg_keep_u64(&key[tgt[u]], pol_keep) : 0ull;
                stp[u] = has ? ld_cg_keep_u32(&stamp[tgt[u]], pol_keep) : stepid;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                old[u] = stepid;
                if (cnk[u] < cur[u]) {
                    red_min_keep_u64(&key[tgt[u]], cnk[u], pol_keep);
                    if (stp[u] != stepid) old[u] = atomicExch(&stamp[tgt[u]], stepid);
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                newly += old[u] == 0u ? 1 : 0;
                wn.put(old[u] != stepid, tgt[u], lane);
            }
        }
        if (wn.cnt >= (uint32_t)PW) wn.flush(next, &ctr->nnext, lane);
    }
    if (wn.cnt) wn.flush(next, &ctr->nnext, lane);
    warp_add_u64(&ctr->newly_covered, newly);
    if (RESIDENT && __any_sync(0xffffffffu, bad) && lane == 0) atomicExch(&ctr->bad, 1u);
}

// ---------------------------------------------------------------- resident growth
// Small steps are latency: as separate launches a step is a push, a snapshot, a counter reset and a counter read
// that the host waits for, 37 us on a 1,001 x 1,001 mesh for frontiers of a few thousand entries.  k_grow runs them
// in one launch: one thread-block cluster (its CTAs are resident together, and its barrier orders their memory)
// takes growing steps back to back, every CTA deciding from the same counters, until a step is too large for it or
// the growth ends; on small graphs it runs whole stages (draw, listing, doubling, contraction) too.
// Bound by dependent L2 round trips.  With the next frontier in the warps' hands (hold_front) a step takes 15,500 cycles
// up to 3,000 entries, 19,000 at 24,000, 25,000 at 54,000, 35,000 at 99,000: the push (adjacency, keys and stamps,
// exchange, append) 7,000 to 21,000 of them, two cluster barriers 3,600, hold_front 2,600 to 7,000, the decision the
// rest.  (Through lists, that is chunk table, entries and two more appends, the steps of the 1,001^2 mesh took 3.09 ms
// in place of 2.23, those of the 64^2 mesh with its whole-node phases 400 us in place of 353.)  Clustering alone, host
// loop / resident: 64^2 mesh (44 steps) 1,636 / 502 us, 300^2 mesh (101) 3,073 / 1,043 us, 1,001^2 mesh (206) 7,492 /
// 4,059 us, road mesh 4,096^2 (134) 11,538 / 10,483 us.  Above 2^18 entries a step of the whole device (push and
// snapshot 13 to 40 us and 22 us between them) is the faster one; a whole-node pass over more than 2^17 nodes by 16
// SMs likewise.
constexpr int GT = 1024;                     // threads per CTA
constexpr int GCTAS = 16;                    // CTAs of the cluster
constexpr uint32_t kGrowEntries = 1u << 18;  // largest step: 16 passes of a warp's 128 positions over the cluster's warps
constexpr uint32_t kGrowNodes = 1u << 17;    // whole stages up to this many nodes: 8 rounds of a node per thread
constexpr uint32_t kGrowEpochs = 1u << 20;   // phases per launch of k_grow, after which the host launches it again

enum GrowPhase : uint32_t { kPhaseStage = 0, kPhaseStep = 1, kPhaseGrown = 2, kPhaseDone = 3, kPhaseFailed = 4 };

// The control state of CLUSTER between phases, kept by the host and by every CTA alike.
struct GrowState {
    uint64_t U;           // unfrozen nodes at the stage's start
    uint64_t covered;     // of them, nodes holding a key
    uint64_t frozen_deg;  // adjacency entries of frozen nodes
    uint64_t node_updates, edges_scanned, centers_drawn;
    uint64_t unfrozen;    // what the last draw saw
    uint32_t phase, stage, stepid, delta;
    uint32_t nf, E, cur;  // the frontier and which pair of buffers holds it
    uint32_t growth_steps;
    uint32_t steps, stages, doublings, guard_exits;
};

struct GrowArgs {
    const uint64_t* off;
    const uint2* adj;
    unsigned long long* key;
    unsigned long long* keyS;
    unsigned long long* fkey[2];
    uint32_t *center, *D, *R, *stamp, *next;
    uint32_t *fbase[2], *fpre[2], *cfirst[2];
    Counters* ring;       // three counter blocks, zeroed
    GrowState* out;
    const uint32_t* row;  // graphs that may be unconnected: the row of every entry, for the guard's edge scan
    double tau, L;
    uint64_t seed, nnz;
    uint32_t n, step_cap, max_entries, max_epochs;
    bool cumulative, pull_ok, stages, connected;
};

// what a CTA does next, decided by its thread 0
enum GrowWork : uint32_t { kWorkPush, kWorkDraw, kWorkList, kWorkGuard, kWorkFinal, kWorkLeave, kWorkSnap };

struct GrowSmem {
    PushSmem<GT / 32> push;
    unsigned long long scratch[33];
    GrowState g;
    uint64_t thr;  // draw threshold of the stage
    uint32_t work;
    uint32_t nn;       // changed nodes of the last push
    uint32_t light;    // the warps took them (hold_front) ...
    uint32_t held;     // ... and push them
    uint32_t no_hold;  // a warp's share was too much: lists until the launch ends
};

// The changed nodes become the next frontier in the warps' hands: each takes up to 128 of them, their end-of-step keys and
// its own prefix over their degrees into the arrays its next push reads, so a step goes without the lists (two appends
// and three dependent reads less).  Counted as dev_snapshot counts; a warp with more than kHeldMost positions (a hub)
// sets ctr->heavy, and the lists are written after all.
constexpr uint32_t kHeldMost = 4 * QC;
constexpr uint32_t kHeldNodes = QC;  // entries that the warp's arrays hold
template <int WARPS>
__device__ __forceinline__ Held hold_front(const uint32_t* __restrict__ next, uint32_t nn,
                                           const unsigned long long* __restrict__ key, const uint64_t* __restrict__ off,
                                           uint32_t delta, Counters* ctr, PushSmem<WARPS>& smp, uint32_t br, uint32_t nb,
                                           unsigned long long* __restrict__ keyS, uint32_t n) {
    const uint32_t lane = lane_id(), warp = threadIdx.x >> 5, nwarps = nb * WARPS;
    // fewer warps with more lanes for small steps; at most kHeldNodes a warp
    const uint32_t per = max((nn + nwarps - 1) / nwarps, 8u), base = (warp * nb + br) * per;
    constexpr int HU = kHeldNodes / 32;
    uint32_t v[HU], deg[HU], b0[HU];
    unsigned long long k[HU];
    __syncwarp();  // the last push's entries have been read
#pragma unroll
    for (int u = 0; u < HU; ++u) {
        const uint32_t x = u * 32 + lane;
        v[u] = x < per && base + x < nn ? __ldcg(&next[base + x]) : kNone;
    }
#pragma unroll
    for (int u = 0; u < HU; ++u) {
        deg[u] = b0[u] = 0;
        k[u] = kInfKey;
        if (v[u] < n) {
            k[u] = __ldcg(&key[v[u]]);
            const uint64_t o = off[v[u]];
            b0[u] = (uint32_t)o;
            deg[u] = (uint32_t)(off[v[u] + 1] - o);
        } else if (v[u] != kNone) {
            atomicExch(&ctr->bad, 1u);
        }
    }
    Held h;
    h.on = true;
#pragma unroll
    for (int u = 0; u < HU; ++u) {
        if (u > 0 && per <= u * 32u) break;
        if (keyS && v[u] < n) keyS[v[u]] = k[u];  // the next step's start-of-step key
        const bool take = (uint32_t)(k[u] >> 32) < delta && deg[u] > 0;
        const unsigned m = __ballot_sync(0xffffffffu, take);
        const uint32_t d = take ? deg[u] : 0u, incl = warp_incl_scan(d), pre = h.total + incl - d;
        if (take) {
            const uint32_t at = h.ne + (uint32_t)__popc(m & lanemask_lt());
            if (at) smp.spre[warp][at - 1] = pre;
            smp.sbase[warp][at] = b0[u] - pre;
            smp.skey[warp][at] = k[u];
        }
        h.ne += (uint32_t)__popc(m);
        h.total += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (lane == 0 && h.ne) {
        atomicAdd(&ctr->front, ((unsigned long long)h.ne << 32) | h.total);
        if (h.total > kHeldMost) atomicExch(&ctr->heavy, 1u);
    }
    __syncwarp();
    return h;
}

// barrier of a thread-block cluster: all its threads, and their memory in order
__device__ __forceinline__ void cluster_barrier() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
}
// Control decisions up to the next work (thread 0 of every CTA, from the same values).
__device__ __forceinline__ uint32_t grow_decide(const GrowArgs& a, GrowState& g, uint64_t* thr) {
    for (;;) {
        if (g.phase == kPhaseStep) {
            if (g.E > a.max_entries) return kWorkLeave;
            ++g.growth_steps;
            ++g.stepid;
            if (g.nf > 0) return kWorkPush;
            g.steps++;
            g.phase = kPhaseGrown;
        } else if (!a.stages) {
            return kWorkLeave;
        } else if (g.phase == kPhaseStage) {
            if (!stage_threshold(g.U, a.tau, a.L, thr)) {
                g.phase = kPhaseDone;
                return kWorkLeave;
            }
            if (g.stage > kMaxStages) {
                g.phase = kPhaseFailed;
                return kWorkLeave;
            }
            return kWorkDraw;
        } else if (g.phase == kPhaseGrown) {
            if (2 * g.covered >= g.U) return kWorkFinal;
            // (connected graph: some covered or frozen node touches an uncovered one iff any exists)
            if (g.delta < kDeltaMax && (g.covered > 0 || g.U < a.n)) {
                if (!a.connected) return kWorkGuard;
                g.delta = (g.delta > kDeltaMax / 2) ? kDeltaMax : 2 * g.delta;
                g.doublings++;
                return kWorkList;
            }
            g.guard_exits++;
            return kWorkFinal;
        } else {
            return kWorkLeave;
        }
    }
}

// What a finished work changes, from the epoch's counters; returns the next work.  `last`: the launch is to end here if
// the state can be resumed from, which it can before a decision (that counts a step or doubles Delta) but not between
// a draw, a doubling or a step and what they ask for next.
__device__ __forceinline__ uint32_t grow_apply(const GrowArgs& a, GrowSmem& sm, uint32_t work, const Counters* c,
                                               bool last) {
    GrowState& g = sm.g;
    sm.held = 0;  // (a held frontier is for the next work alone)
    if (work == kWorkPush) {
        // (all of the step's counters in one round trip)
        const uint32_t updated = __ldcg(&c->nnext), bad = __ldcg(&c->bad), heavy = __ldcg(&c->heavy);
        const unsigned long long front = __ldcg(&c->front), newly = __ldcg(&c->newly_covered);
        if (bad) {
            g.phase = kPhaseFailed;
            g.unfrozen = ~g.U;
            return kWorkLeave;
        }
        g.covered += newly;
        g.edges_scanned += g.E;
        g.nf = (uint32_t)(front >> 32);
        g.E = (uint32_t)front;
        g.cur ^= 1;
        g.steps++;
        g.node_updates += updated;
        if (!(updated != 0 && 2 * g.covered < g.U && (a.step_cap == 0 || g.growth_steps < a.step_cap))) {
            g.phase = kPhaseGrown;
        } else if (sm.light) {
            if (heavy) sm.no_hold = 1;
            sm.held = !sm.no_hold && g.E <= a.max_entries;
            if (!sm.held) return kWorkSnap;
        }
    } else if (work == kWorkSnap) {
        if (__ldcg(&c->front) != (((unsigned long long)g.nf << 32) | g.E)) {
            g.phase = kPhaseFailed;
            return kWorkLeave;
        }
    } else if (work == kWorkDraw) {
        g.covered = __ldcg(&c->selected);
        g.centers_drawn += g.covered;
        g.unfrozen = __ldcg(&c->unfrozen);
        if (g.unfrozen != g.U) {
            g.phase = kPhaseFailed;
            return kWorkLeave;
        }
        return kWorkList;
    } else if (work == kWorkList) {
        const unsigned long long front = __ldcg(&c->front);
        g.nf = (uint32_t)(front >> 32);
        g.E = (uint32_t)front;
        g.growth_steps = 0;
        g.phase = kPhaseStep;
    } else if (work == kWorkGuard) {
        if (!__ldcg(&c->growable)) {
            g.guard_exits++;
            return kWorkFinal;
        }
        g.delta = (g.delta > kDeltaMax / 2) ? kDeltaMax : 2 * g.delta;
        g.doublings++;
        return kWorkList;
    } else {
        if (__ldcg(&c->overflow)) {
            g.phase = kPhaseFailed;
            g.unfrozen = g.U = 0;
            return kWorkLeave;
        }
        g.U -= __ldcg(&c->frozen);
        g.frozen_deg += __ldcg(&c->frozen_deg);
        g.stages++;
        ++g.stage;
        g.phase = kPhaseStage;
    }
    return last ? (uint32_t)kWorkLeave : grow_decide(a, g, &sm.thr);
}

// The loop: works until one that this launch may not take (a step of more than max_entries entries, a whole-node phase
// when `stages` is off), the end, a failure, or the first state from max_epochs works on that a launch can start from;
// sm.g holds the control state before and after.  CTA br of nb that share the graph; `barrier` synchronises all their
// threads and orders their memory.  The state stays in shared memory and thread 0 decides (kept in every thread's
// registers it spilled the pushes' at 64 of them).
template <class Barrier>
__device__ __forceinline__ void grow_run(const GrowArgs& a, GrowSmem& sm, uint32_t br, uint32_t nb, Barrier barrier) {
    GrowState& g = sm.g;
    __syncthreads();  // the state is set
    if (threadIdx.x == 0) {
        sm.held = sm.no_hold = sm.light = 0;
        sm.work = grow_decide(a, g, &sm.thr);
    }
    __syncthreads();
    Held held;
    // Counter block of the current epoch (one work, up to its closing barrier).  An epoch clears the next one's block,
    // last read two epochs ago: every CTA has passed the barrier that closed the epoch in between.
    for (uint32_t epoch = 0; sm.work != kWorkLeave; ++epoch) {
        const uint32_t work = sm.work;
        Counters* ctr = a.ring + epoch % 3;
        if (work == kWorkPush) {
            const uint32_t c = g.cur, o = c ^ 1;
            dev_push<true>(a.fbase[c], a.fkey[c], a.fpre[c], a.cfirst[c], g.nf, g.E, a.adj, a.center,
                           a.cumulative ? a.D : nullptr, a.key, g.delta, a.stamp, g.stepid, a.next, ctr, sm.push, br, nb,
                           a.n, (uint32_t)a.nnz, held);
            barrier();
            const uint32_t nn = min(__ldcg(&ctr->nnext), a.n);
            // (a launch that ends leaves lists)
            const bool light = nn <= nb * (GT / 32) * kHeldNodes && !sm.no_hold && epoch + 1 < a.max_epochs;
            if (light)
                held = hold_front(a.next, nn, a.key, a.off, g.delta, ctr, sm.push, br, nb, a.keyS, a.n);
            else
                dev_snapshot(a.next, nn, a.key, a.off, g.delta, a.fbase[o], a.fkey[o], a.fpre[o], a.cfirst[o], ctr,
                             sm.scratch, br, nb, a.keyS, a.n);
            if (threadIdx.x == 0) {
                sm.nn = nn;
                sm.light = light;
            }
        } else if (work == kWorkSnap) {
            const uint32_t c = g.cur;
            dev_snapshot(a.next, sm.nn, a.key, a.off, g.delta, a.fbase[c], a.fkey[c], a.fpre[c], a.cfirst[c], ctr,
                         sm.scratch, br, nb, a.keyS, a.n);
        } else if (work == kWorkDraw) {
            dev_select(a.n, a.center, a.key, a.seed, g.stage, sm.thr, ctr, br, nb, a.keyS);
        } else if (work == kWorkList) {
            const bool pull = a.pull_ok && (a.nnz - g.frozen_deg) < g.frozen_deg;
            dev_rebuild(a.n, a.key, a.center, a.cumulative ? a.D : nullptr, a.off, g.delta, pull, a.fbase[g.cur],
                        a.fkey[g.cur], a.fpre[g.cur], a.cfirst[g.cur], ctr, sm.scratch, br, nb);
        } else if (work == kWorkGuard) {
            dev_growable(a.row, a.adj, a.nnz, a.key, ctr, br, nb);
        } else {
            dev_finalize_d(a.n, a.key, a.center, a.cumulative ? nullptr : a.R, a.D, ctr, br, nb);
            barrier();
            dev_finalize_freeze(a.n, a.key, a.center, a.R, a.D, a.off, ctr, br, nb, a.keyS, a.cumulative);
        }
        if (br == 0 && threadIdx.x < sizeof(Counters) / 8)
            reinterpret_cast<unsigned long long*>(a.ring + (epoch + 1) % 3)[threadIdx.x] = 0ull;
        barrier();
        if (threadIdx.x == 0) sm.work = grow_apply(a, sm, work, ctr, epoch + 1 >= a.max_epochs);
        __syncthreads();
        held.on = sm.held;
    }
}

// ---------------------------------------------------------------- launching a resident kernel
// Launch configuration of one cluster of `ctas` CTAs of GT threads.
inline void resident_config(cudaLaunchConfig_t* cfg, cudaLaunchAttribute* at, int ctas, size_t smem, cudaStream_t s) {
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = (unsigned)ctas;
    at->val.clusterDim.y = at->val.clusterDim.z = 1;
    cfg->gridDim = dim3((unsigned)ctas);
    cfg->blockDim = dim3(GT);
    cfg->dynamicSmemBytes = smem;
    cfg->stream = s;
    cfg->attrs = at;
    cfg->numAttrs = 1;
}
// CTAs of a resident kernel's cluster on the current device: 16 where such a cluster can be resident, else the portable
// 8, else 0 (not used).
template <class Kern>
int resident_cluster_size(Kern kern, size_t smem) {
    int size = 0;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) == cudaSuccess &&
        cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
        for (int c = GCTAS; c >= 8 && size == 0; c /= 2) {
            cudaLaunchConfig_t cfg{};
            cudaLaunchAttribute at{};
            resident_config(&cfg, &at, c, smem, nullptr);
            int m = 0;
            if (cudaOccupancyMaxActiveClusters(&m, kern, &cfg) == cudaSuccess && m > 0) size = c;
        }
    }
    cudaGetLastError();
    return size;
}

}  // namespace cld
