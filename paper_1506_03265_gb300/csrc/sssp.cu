// Delta-stepping SSSP (Meyer and Sanders, J. Algorithms 2003), the parallel
// SSSP the paper compares against (Sections 1 and 5): bucket i holds the
// nodes with tentative distance in [i Delta, (i+1) Delta).  The current
// bucket is settled by repeated rounds; the next non-empty bucket is then
// taken from the far pile.  Twice the source's eccentricity is the SSSP
// 2-approximation of the diameter.
//
// A round relaxes every edge of its nodes, light and heavy alike: with rows
// sorted by column a light round reads the heavy edges too, so settling the
// light ones first only adds a pass over the bucket's adjacency and its
// rounds (R-MAT 24 read 2.2G entries in 34 rounds that way).
//
// Dedup: a node enters a round's frontier at most once per round (round
// stamp) and the far pile once per bucket epoch (epoch stamp); stale far
// entries are dropped when the next bucket is taken.
//
// Work distribution: each round's node list becomes a frontier with the
// first position of every node's adjacency in one flattened range (one packed
// atomic per CTA hands out slots and positions) and a chunk table; each warp
// takes PW consecutive positions, so a hub's adjacency is spread over many
// warps instead of one (edge-balanced, as the growing step of CLUSTER).
//
// Small rounds run back to back in one launch by one thread-block cluster
// (k_ds_resident), as CLUSTER's growing steps do (grow.cuh): a round as
// separate launches costs 30 us however small it is, and a mesh takes a
// thousand.
#include <algorithm>
#include <atomic>

#include "grow.cuh"
#include "internal.cuh"
#include "prof.cuh"

namespace cld {

namespace {

// A count that either form of append can raise: 32-bit additions to `count`, or front_append_n's 64-bit ones, whose low
// words are 0 here.
struct DsCount {
    uint32_t zero;
    uint32_t count;
    __device__ unsigned long long* packed() { return reinterpret_cast<unsigned long long*>(this); }
};
// Far pile of one bucket epoch: two take turns (what a new bucket leaves is rewritten into the other).
struct __align__(8) DsPile {
    DsCount n;
    uint32_t min;  // smallest distance at which a node was put on it
    uint32_t pad;
};
// counters of one round or split
struct __align__(8) DsRound {
    unsigned long long front;  // listed frontier: (entries << 32) | adjacency positions
    DsCount next;              // nodes of the next round
    uint32_t bad;              // a list held an id out of range
    uint32_t pad;
};
struct DsCounters {
    DsRound r;  // reset before every round
    DsPile pile[2];
    uint32_t overflow;  // some candidate reached 2^32 - 1
    uint32_t pad;
};

// Most entries of a resident round's nodes.  The list's node count says little where degrees are skewed: 1,500 hubs of
// 53,000 entries made a list within its limit, and 16 SMs took 16.2 ms for what the whole device does in 4.9.  (2^18 to
// 2^21 measured alike; at 2^17 rounds of a ring lattice that the launch does faster leave it, 393 -> 678 ms.)
constexpr uint32_t kDsEntries = 1u << 19;

// The control state between rounds, kept by the host and by every CTA of k_ds_resident alike.
struct DsState {
    uint64_t hi;       // end of the current bucket
    uint64_t scanned;  // adjacency entries read
    uint32_t ncur;     // nodes of the next round, in list[cur]
    uint32_t cur;
    uint32_t pile;     // the far pile in use
    uint32_t nfar, min;  // its entries and smallest distance
    uint32_t round_id, epoch, rounds;
    uint32_t done, bad;
    uint32_t wide;     // the next round's nodes hold too many entries for the resident form
};

struct DsArgs {
    const uint64_t* off;
    const uint2* adj;
    uint32_t *dist, *rstamp, *fstamp;
    uint32_t *list[2], *far[2];
    uint32_t *fbase, *fdist, *fpre, *cfirst;
    DsCounters* ctr;        // host-driven rounds and the kept counters
    DsRound* ring;          // resident rounds: three blocks, zeroed
    DsState* out;
    uint64_t nnz;
    uint32_t n, delta;
    uint32_t max_list, max_far, max_epochs;  // resident rounds: largest list and pile, phases per launch
    uint32_t max_entries;                    // and the entries of a round's nodes
};

// A round's node list as a frontier: slot, first position and adjacency base of every node with entries, its distance
// when listed, and the chunk table.
__device__ __forceinline__ void ds_list(const DsArgs& a, const uint32_t* list, uint32_t nl, unsigned long long* front,
                                        unsigned long long* scratch, uint32_t br, uint32_t nb, uint32_t* bad) {
    const uint32_t per = nodes_per_thread(nl, nb);
    const uint64_t stride = (uint64_t)nb * blockDim.x * per;
    for (uint64_t base = (uint64_t)br * blockDim.x * per; base < nl; base += stride) {
        uint32_t v[NU], deg[NU], b0[NU], d[NU], slot[NU], pre[NU], kinds = 0;
#pragma unroll
        for (uint32_t u = 0; u < NU; ++u) {
            const uint64_t i = base + u * blockDim.x + threadIdx.x;
            v[u] = u < per && i < nl ? __ldcg(&list[i]) : kNone;
            if (u < per && i < nl && v[u] >= a.n) atomicExch(bad, 1u);
        }
#pragma unroll
        for (uint32_t u = 0; u < NU; ++u) {
            deg[u] = b0[u] = d[u] = 0;
            if (v[u] < a.n) {
                d[u] = __ldcg(&a.dist[v[u]]);
                const uint64_t o = a.off[v[u]];
                b0[u] = (uint32_t)o;
                deg[u] = (uint32_t)(a.off[v[u] + 1] - o);
            }
            kinds |= (deg[u] ? 1u : 0u) << u;
        }
        front_append_n<NU>(front, kinds, deg, slot, pre, scratch);
#pragma unroll
        for (uint32_t u = 0; u < NU; ++u) {
            if (!deg[u]) continue;
            a.fbase[slot[u]] = b0[u] - pre[u];
            a.fdist[slot[u]] = d[u];
            a.fpre[slot[u]] = pre[u];
            chunk_table_put(a.cfirst, slot[u], pre[u], deg[u]);
        }
    }
}

template <int WARPS>
struct DsPushSmem {
    uint32_t spre[WARPS][PW + 1];
    uint32_t sbase[WARPS][PW + 2];
    uint32_t sdist[WARPS][PW + 2];
    uint32_t snext[WARPS][PNB];
    uint32_t sfar[WARPS][PNB];
};

// One round over a listed frontier: each warp takes PW consecutive positions of the flattened adjacency; a candidate
// that undercuts the target's distance lowers it with an atomic minimum, and an improved target goes to the next round
// (below hi) or to the far pile, each deduplicated by its stamp.  RESIDENT: distances are read past L1 and positions
// and ids checked, as in dev_push.
template <bool RESIDENT, int WARPS>
__device__ __forceinline__ void ds_push(const DsArgs& a, uint32_t nf, uint32_t E, uint64_t hi, uint32_t round_id,
                                        uint32_t epoch, uint32_t* next, uint32_t* nnext, uint32_t* far, DsPile* pile,
                                        DsPushSmem<WARPS>& sm, uint32_t br, uint32_t nb, uint32_t* overflow,
                                        uint32_t* badp) {
    const uint32_t lane = lane_id(), warp = threadIdx.x >> 5;
    const uint64_t pol_stream = l2_evict_first_policy(), pol_keep = l2_evict_last_policy();
    const unsigned le_mask = 0xffffffffu >> (31u - lane);
    WarpNext wn{sm.snext[warp], 0}, wf{sm.sfar[warp], 0};
    bool ovf = false, bad = false;
    uint32_t fmin = kNone;
    const uint32_t nq = (uint32_t)(((uint64_t)E + PW - 1) / PW);
    const uint32_t nwarps = nb * WARPS;
    for (uint32_t q = br * WARPS + warp; q < nq; q += nwarps) {
        const uint32_t p0 = q * PW, e1 = min(E, p0 + PW);
        const uint32_t i0 = __ldcg(&a.cfirst[q]);
        const uint32_t il = q + 1 < nq ? __ldcg(&a.cfirst[q + 1]) : nf - 1;
        if (RESIDENT && (i0 > il || il >= nf)) {
            bad = true;
            continue;
        }
        const uint32_t ne = min(il - i0 + 1, (uint32_t)PW + 1);
        __syncwarp();  // the previous chunk's entries have been read
        for (uint32_t j = lane; j < ne; j += 32) {
            if (j) sm.spre[warp][j - 1] = __ldcg(&a.fpre[i0 + j]);
            sm.sbase[warp][j] = __ldcg(&a.fbase[i0 + j]);
            sm.sdist[warp][j] = __ldcg(&a.fdist[i0 + j]);
        }
        __syncwarp();
        uint32_t own[PWG];
        {
            uint32_t B = 0;
#pragma unroll
            for (int u = 0; u < PWG; ++u) {
                const uint32_t word =
                    group_starts(sm.spre[warp] + B, ne - 1 - B, p0 + 32u * u, B, lane, le_mask, &own[u]);
                B += (uint32_t)__popc(word);
            }
        }
        uint2 ed[PWG];
        uint32_t live = 0;
#pragma unroll
        for (int u = 0; u < PWG; ++u) {
            const uint32_t p = p0 + 32u * u + lane;
            bool in = p < e1;
            if (RESIDENT && in && (own[u] >= ne || sm.sbase[warp][own[u]] + p >= (uint32_t)a.nnz)) {
                bad = true;
                in = false;
            }
            live |= (in ? 1u : 0u) << u;
            ed[u] = in ? ld_stream_u2(a.adj + (sm.sbase[warp][own[u]] + p), pol_stream) : make_uint2(0u, 0u);
        }
        uint64_t nd[PWG];
        uint32_t cur[PWG];
#pragma unroll
        for (int u = 0; u < PWG; ++u) {
            nd[u] = (live >> u) & 1u ? (uint64_t)sm.sdist[warp][own[u]] + ed[u].y : ~0ull;
            cur[u] = 0;
            if ((live >> u) & 1u) {  // (a one-round launch filters through L1)
                if constexpr (RESIDENT) cur[u] = ld_cg_keep_u32(&a.dist[ed[u].x], pol_keep);
                else cur[u] = ld_keep_u32(&a.dist[ed[u].x], pol_keep);
            }
        }
        uint32_t old[PWG];
#pragma unroll
        for (int u = 0; u < PWG; ++u) {
            old[u] = 0;
            if (nd[u] >= 0xFFFFFFFFull) {
                ovf |= nd[u] != ~0ull;
                nd[u] = ~0ull;
            } else if (nd[u] < cur[u]) {
                old[u] = atomicMin(&a.dist[ed[u].x], (uint32_t)nd[u]);
            }
        }
        uint32_t st[PWG];
#pragma unroll
        for (int u = 0; u < PWG; ++u) {
            // an improved target: was it listed (next round or far pile) before?
            const bool better = nd[u] < old[u];
            const bool near = nd[u] < hi;
            st[u] = 0;
            if (better) st[u] = near ? atomicExch(&a.rstamp[ed[u].x], round_id) != round_id
                                     : atomicExch(&a.fstamp[ed[u].x], epoch) != epoch;
            if (better && !near) fmin = min(fmin, (uint32_t)nd[u]);
        }
#pragma unroll
        for (int u = 0; u < PWG; ++u) {
            wn.put(st[u] && nd[u] < hi, ed[u].x, lane);
            wf.put(st[u] && nd[u] >= hi, ed[u].x, lane);
        }
        if (wn.cnt >= (uint32_t)PW) wn.flush(next, nnext, lane);
        if (wf.cnt >= (uint32_t)PW) wf.flush(far, &pile->n.count, lane);
    }
    if (wn.cnt) wn.flush(next, nnext, lane);
    if (wf.cnt) wf.flush(far, &pile->n.count, lane);
    fmin = __reduce_min_sync(0xffffffffu, fmin);
    if (lane == 0 && fmin != kNone) atomicMin(&pile->min, fmin);
    if (__any_sync(0xffffffffu, ovf) && lane == 0) atomicExch(overflow, 1u);
    if (RESIDENT && __any_sync(0xffffffffu, bad) && lane == 0) atomicExch(badp, 1u);
}

// Split the far pile (nfar entries): those below hi become the next round's list, later ones move to the other pile
// (re-stamped); entries that were improved below lo meanwhile are dropped.  *taken and pile2->count are counters of
// front_append_n: the number of entries in their high words.
__device__ __forceinline__ void ds_split(const DsArgs& a, const uint32_t* far, uint32_t nfar, uint64_t lo, uint64_t hi,
                                         uint32_t epoch, uint32_t* next, unsigned long long* taken, uint32_t* far2,
                                         DsPile* pile2, unsigned long long* scratch, uint32_t br, uint32_t nb,
                                         uint32_t* bad) {
    unsigned long long* kept = pile2->n.packed();
    const uint32_t per = nodes_per_thread(nfar, nb);
    const uint64_t stride = (uint64_t)nb * blockDim.x * per;
    uint32_t kmin = kNone;
    for (uint64_t base = (uint64_t)br * blockDim.x * per; base < nfar; base += stride) {
        uint32_t v[NU], d[NU];
#pragma unroll
        for (uint32_t u = 0; u < NU; ++u) {
            const uint64_t i = base + u * blockDim.x + threadIdx.x;
            v[u] = u < per && i < nfar ? __ldcg(&far[i]) : kNone;
            if (u < per && i < nfar && v[u] >= a.n) atomicExch(bad, 1u);
        }
#pragma unroll
        for (uint32_t u = 0; u < NU; ++u) d[u] = v[u] < a.n ? __ldcg(&a.dist[v[u]]) : 0u;
        uint32_t takes = 0, keeps = 0, slot[NU], one[NU], pre[NU];
#pragma unroll
        for (uint32_t u = 0; u < NU; ++u) {
            one[u] = 0;
            if (v[u] >= a.n) continue;
            if ((uint64_t)d[u] >= hi) {
                keeps |= (atomicExch(&a.fstamp[v[u]], epoch) != epoch ? 1u : 0u) << u;
                kmin = min(kmin, d[u]);
            } else {
                takes |= ((uint64_t)d[u] >= lo ? 1u : 0u) << u;
            }
        }
        // one append per block and list (with one per warp the 6.5M entries of R-MAT 24's first split queued at the two
        // counters for 636 us; 68 us so)
        front_append_n<NU>(taken, takes, one, slot, pre, scratch);
#pragma unroll
        for (uint32_t u = 0; u < NU; ++u)
            if ((takes >> u) & 1u) next[slot[u]] = v[u];
        front_append_n<NU>(kept, keeps, one, slot, pre, scratch);
#pragma unroll
        for (uint32_t u = 0; u < NU; ++u)
            if ((keeps >> u) & 1u) far2[slot[u]] = v[u];
    }
    kmin = __reduce_min_sync(0xffffffffu, kmin);
    if (lane_id() == 0 && kmin != kNone) atomicMin(&pile2->min, kmin);
}

__global__ void __launch_bounds__(256) k_ds_list(const DsArgs a, uint32_t cur, uint32_t nl) {
    __shared__ unsigned long long scratch[33];
    ds_list(a, a.list[cur], nl, &a.ctr->r.front, scratch, blockIdx.x, gridDim.x, &a.ctr->r.bad);
}
__global__ void __launch_bounds__(PT, 6) k_ds_push(const DsArgs a, uint32_t cur, uint32_t pile, uint64_t hi,
                                                   uint32_t round_id, uint32_t epoch) {
    __shared__ DsPushSmem<PT / 32> sm;
    const unsigned long long fr = __ldcg(&a.ctr->r.front);
    ds_push<false>(a, (uint32_t)(fr >> 32), (uint32_t)fr, hi, round_id, epoch, a.list[cur ^ 1], &a.ctr->r.next.count,
                   a.far[pile], &a.ctr->pile[pile], sm, blockIdx.x, gridDim.x, &a.ctr->overflow, &a.ctr->r.bad);
}
__global__ void __launch_bounds__(256) k_ds_split(const DsArgs a, uint32_t cur, uint32_t pile, uint32_t nfar, uint64_t lo,
                                                  uint64_t hi, uint32_t epoch) {
    __shared__ unsigned long long scratch[33];
    if (blockIdx.x == 0 && threadIdx.x == 0) a.ctr->pile[pile] = DsPile{{0u, 0u}, kNone, 0u};  // (its values are known)
    ds_split(a, a.far[pile], nfar, lo, hi, epoch, a.list[cur], a.ctr->r.next.packed(), a.far[pile ^ 1],
             &a.ctr->pile[pile ^ 1], scratch, blockIdx.x, gridDim.x, &a.ctr->r.bad);
}

// What follows a finished round or split (host, or thread 0 of every CTA): false when the SSSP is done.
__host__ __device__ inline bool ds_next_bucket(DsState& g, uint32_t delta, uint64_t* lo) {
    if (g.nfar == 0) {
        g.done = 1;
        return false;
    }
    *lo = (uint64_t)g.min / delta * delta;
    if (*lo < g.hi) *lo = g.hi;  // (the pile's minimum may be a node that has moved below since)
    g.hi = (uint64_t)g.min / delta * delta + delta;
    if (g.hi <= *lo) g.hi = *lo + delta;
    ++g.epoch;
    return true;
}

struct DsSmem {
    DsPushSmem<GT / 32> push;
    unsigned long long scratch[33];
    DsState g;
    uint64_t lo;
    uint32_t work;
};
enum DsWork : uint32_t { kDsRound, kDsSplit, kDsLeave };

__device__ __forceinline__ uint32_t ds_decide(const DsArgs& a, DsState& g, uint64_t* lo) {
    if (g.ncur > 0) {
        if (g.ncur > a.max_list) return kDsLeave;
        ++g.round_id;
        return kDsRound;
    }
    if (g.nfar > a.max_far) return kDsLeave;
    return ds_next_bucket(g, a.delta, lo) ? kDsSplit : kDsLeave;
}

// Rounds and splits back to back by one thread-block cluster, until one that is too large for it (by its nodes, or by
// their entries once they are listed: `wide`, the host then runs that round), the phase limit, or the end.  The next work
// is decided at the head of an iteration, after the limit has been tested: a decision moves the state (a split's bucket),
// so one that no work followed would leave its bucket out of the next launch.
__global__ void __launch_bounds__(GT, 1) k_ds_resident(const DsArgs a, const DsState start) {
    extern __shared__ __align__(16) unsigned char ds_smem[];
    DsSmem& sm = *reinterpret_cast<DsSmem*>(ds_smem);
    DsState& g = sm.g;
    const uint32_t br = blockIdx.x, nb = gridDim.x;
    if (threadIdx.x == 0) g = start;
    // Counters of the epoch; an epoch clears the next one's, last read two epochs ago.
    for (uint32_t epoch = 0;; ++epoch) {
        if (threadIdx.x == 0) sm.work = epoch < a.max_epochs && !g.bad ? ds_decide(a, g, &sm.lo) : (uint32_t)kDsLeave;
        __syncthreads();
        if (sm.work == kDsLeave) break;
        DsRound* r = a.ring + epoch % 3;
        const uint32_t work = sm.work, p = g.pile;
        unsigned long long fr = 0;
        if (work == kDsRound) {
            ds_list(a, a.list[g.cur], g.ncur, &r->front, sm.scratch, br, nb, &r->bad);
            cluster_barrier();
            fr = __ldcg(&r->front);
            if ((uint32_t)fr > a.max_entries) {  // (the same at every CTA)
                if (threadIdx.x == 0) g.wide = 1;
                __syncthreads();
                break;
            }
            ds_push<true>(a, (uint32_t)(fr >> 32), (uint32_t)fr, g.hi, g.round_id, g.epoch, a.list[g.cur ^ 1],
                          &r->next.count, a.far[p], &a.ctr->pile[p], sm.push, br, nb, &a.ctr->overflow, &r->bad);
        } else {
            cluster_barrier();  // every CTA has read the old pile's counters
            if (br == 0 && threadIdx.x == 0) a.ctr->pile[p] = DsPile{{0u, 0u}, kNone, 0u};
            ds_split(a, a.far[p], g.nfar, sm.lo, g.hi, g.epoch, a.list[g.cur], r->next.packed(), a.far[p ^ 1],
                     &a.ctr->pile[p ^ 1], sm.scratch, br, nb, &r->bad);
        }
        if (br == 0 && threadIdx.x < sizeof(DsRound) / 8)
            reinterpret_cast<unsigned long long*>(a.ring + (epoch + 1) % 3)[threadIdx.x] = 0ull;
        cluster_barrier();
        if (threadIdx.x == 0) {
            if (work == kDsRound) {
                g.cur ^= 1;
                ++g.rounds;
                g.scanned += (uint32_t)fr;
            } else {
                g.pile ^= 1;
            }
            g.ncur = __ldcg(&r->next.count);
            g.bad = __ldcg(&r->bad);
            // (while a round follows, other CTAs may already be adding to the pile: its counters decide only when none
            // does, and then nobody writes them before the next barrier)
            g.nfar = __ldcg(&a.ctr->pile[g.pile].n.count);
            g.min = __ldcg(&a.ctr->pile[g.pile].min);
        }
    }
    if (br == 0 && threadIdx.x == 0) *a.out = g;
}

// some edge (u, v) of a reached node has dist[u] + w >= 2^32 - 1: a distance does not fit
__global__ void k_ds_overflow(const uint64_t* __restrict__ off, const uint2* __restrict__ adj, uint32_t n,
                              const uint32_t* __restrict__ dist, uint32_t* __restrict__ overflow) {
    const uint32_t warps = (gridDim.x * blockDim.x) >> 5;
    bool ovf = false;
    for (uint32_t v = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < n; v += warps) {
        const uint32_t d = dist[v];
        if (d == kNone) continue;
        for (uint64_t j = off[v] + lane_id(); j < off[v + 1]; j += 32) ovf |= (uint64_t)d + adj[j].y >= 0xFFFFFFFFull;
    }
    if (ovf) atomicExch(overflow, 2u);
}

__global__ void k_ds_init(uint32_t* __restrict__ dist, uint32_t* __restrict__ a, uint32_t* __restrict__ b, uint32_t n,
                          uint32_t source) {
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
        dist[v] = v == source ? 0u : 0xFFFFFFFFu;
        a[v] = 0;
        b[v] = 0;
    }
}

__global__ void k_ds_ecc(const uint32_t* __restrict__ dist, uint32_t n, uint32_t* __restrict__ out) {
    uint32_t m = 0;
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x)
        if (dist[v] != 0xFFFFFFFFu) m = max(m, dist[v]);
    m = block_reduce(m, [](uint32_t a, uint32_t b) { return a > b ? a : b; }, 0u);
    if (threadIdx.x == 0) atomicMax(out, m);
}

// CTAs of the resident form's cluster: 16, else 8, else 0 (not used); asked once per device, concurrent first calls
// store the same value
int ds_cluster_size(int dev) {
    static std::atomic<int> cached[64];  // 0 = not asked yet, else size + 1
    if (dev < 0 || dev >= 64) return 0;
    if (cached[dev].load() == 0) cached[dev].store(1 + resident_cluster_size(k_ds_resident, sizeof(DsSmem)));
    return cached[dev].load() - 1;
}

}  // namespace

cldiam_status sssp_delta(cldiam_graph* g, uint32_t source, uint32_t delta, uint32_t* dist_out, uint64_t* ecc,
                         uint64_t* rounds_out, uint64_t* scanned_out, uint32_t max_phases) {
    if (!g || !ecc) return fail(CLDIAM_ERR_INVALID_ARG, "NULL graph or ecc");
    if (source >= g->n) return fail(CLDIAM_ERR_INVALID_ARG, "source >= n");
    if (g->nnz >= 0xFFFFFFFFull) return fail(CLDIAM_ERR_UNSUPPORTED, "2^32 - 1 or more adjacency entries");
    const uint32_t n = g->n;
    const cudaStream_t s = g->stream;
    if (delta == 0) {
        uint32_t d0 = 1;
        CLD_TRY(cld::delta0(g, CLDIAM_DELTA0_AVG, 0, &d0));
        // Width of a bucket, in average weights.  Wide buckets have fewer rounds (10 to 30 us each), narrow ones read fewer
        // entries twice (8 ps each with the whole device).  Which counts, ms at 0.3 / 1 / 8 / 16:
        // - sparse graphs take rounds by the hundred: road mesh 3,000^2 21.0 / 11.8 / 6.7 / 6.4, 700^2 mesh 56.9 / 31.5 /
        //   17.2 / 15.6, a uniform graph of 12.6M entries 2.50 / 1.55 / 1.65 / 1.57;
        // - denser ones without hubs read everything six times and more at 8: uniform, 12.6M entries 1.20 / 1.08 / 1.52 /
        //   1.50, 100.7M 2.91 / 3.30 / 7.06 / 7.03; 160^3 grid of 26 neighbours 14.9 / 13.4 / 22.1 / 36.0;
        // - hubs bring every node within a few hops, at any width about the same reads, so the rounds decide: R-MAT of 1.8M
        //   entries 0.80 / 0.65 / 0.52 / 0.53, 7.6M 1.45 / 1.15 / 0.96 / 0.96, 31M 2.44 / 2.18 / 2.09 / 2.10, 128M 7.69 /
        //   7.52 / 7.77 / 7.75;
        // - above 2^27 entries the reads do: uniform, 201M 4.73 / 6.05 / 14.0 / 14.0; R-MAT, 259M 13.8 / 14.5 / 14.8 / 14.7,
        //   521M 10.1 / 14.8 / 14.1 / 14.1; 180^3 grid 18.8 / 16.8 / 30.1 / 51.3.
        // (Hub: eight times the average degree.  Uniform graphs of that degree end at four, R-MAT graphs start at ten.)
        double scale = (double)sssp_delta_scale_set(g->nnz);
        if (scale == 0.0) {
            const bool hub = (uint64_t)g->max_deg * n >= 8ull * g->nnz;
            scale = g->nnz < 8ull * n ? 16.0 : g->nnz >= (1ull << 27) ? 0.3 : hub && g->nnz < (1ull << 26) ? 8.0 : 1.0;
        }
        const double scaled = (double)d0 * scale;
        delta = (uint32_t)std::min(std::max(scaled, 1.0), 2147483648.0);
    }
    DBuf<uint32_t> dist, rstamp, fstamp, listA, listB, farA, farB, ecc_d, fbase, fdist, fpre, cfirst;
    DBuf<DsCounters> ctr;
    DBuf<DsRound> ring;
    DBuf<DsState> gdev;
    CLD_TRY(dist.alloc(n, s));
    CLD_TRY(rstamp.alloc(n, s));
    CLD_TRY(fstamp.alloc(n, s));
    CLD_TRY(listA.alloc(n, s));
    CLD_TRY(listB.alloc(n, s));
    CLD_TRY(farA.alloc(n, s));
    CLD_TRY(farB.alloc(n, s));
    CLD_TRY(ecc_d.alloc(1, s));
    CLD_TRY(ctr.alloc(1, s));
    CLD_TRY(fbase.alloc(n, s));
    CLD_TRY(fdist.alloc(n, s));
    CLD_TRY(fpre.alloc(n, s));
    CLD_TRY(cfirst.alloc(g->nnz / PW + 2, s));
    CLD_TRY(ring.alloc(3, s));
    CLD_TRY(gdev.alloc(1, s));
    DsCounters* hc = reinterpret_cast<DsCounters*>(static_cast<char*>(g->host.h) + 96);
    DsState* hg = reinterpret_cast<DsState*>(static_cast<char*>(g->host.h) + 176);
    uint32_t* he = reinterpret_cast<uint32_t*>(static_cast<char*>(g->host.h) + 240);
    static_assert(sizeof(DsCounters) <= 80 && sizeof(DsState) <= 64, "read-back blocks must fit the pinned area");
    DsArgs a{};
    a.off = g->off;
    a.adj = g->adj;
    a.dist = dist.get();
    a.rstamp = rstamp.get();
    a.fstamp = fstamp.get();
    a.list[0] = listA.get();
    a.list[1] = listB.get();
    a.far[0] = farA.get();
    a.far[1] = farB.get();
    a.fbase = fbase.get();
    a.fdist = fdist.get();
    a.fpre = fpre.get();
    a.cfirst = cfirst.get();
    a.ctr = ctr.get();
    a.ring = ring.get();
    a.out = gdev.get();
    a.nnz = g->nnz;
    a.n = n;
    a.delta = delta;
    // resident rounds: lists of about 2^18 adjacency entries, piles of 2^18 nodes (as CLUSTER's resident steps)
    a.max_list = (uint32_t)std::max<uint64_t>(1, (uint64_t)kGrowEntries / (g->nnz / n + 1));
    a.max_far = kGrowEntries;
    a.max_entries = kDsEntries;
    a.max_epochs = max_phases ? max_phases : kGrowEpochs;
    const unsigned gb = grid_for(n, 256);
    CLD_K(K_SSSP, s, k_ds_init<<<gb, 256, 0, s>>>(dist.get(), rstamp.get(), fstamp.get(), n, source));
    CLD_LAUNCH_CHECK();
    hc[0] = DsCounters{};
    hc->pile[0].min = hc->pile[1].min = kNone;
    CLD_CUDA(cudaMemcpyAsync(ctr.get(), hc, sizeof(DsCounters), cudaMemcpyHostToDevice, s));
    he[0] = source;
    CLD_CUDA(cudaMemcpyAsync(listA.get(), he, 4, cudaMemcpyHostToDevice, s));

    DsState st{};
    st.hi = delta;
    st.ncur = 1;
    st.min = kNone;
    st.epoch = 1;
    const auto bad_list = [] { return fail(CLDIAM_ERR_DIVERGED, "inconsistent list in a shortest-path round"); };
    const auto read = [&]() -> cldiam_status {
        CLD_CUDA(cudaMemcpyAsync(hc, ctr.get(), sizeof(DsCounters), cudaMemcpyDeviceToHost, s));
        CLD_CUDA(cudaStreamSynchronize(s));
        if (hc->r.bad) return bad_list();
        st.ncur = hc->r.next.count;
        st.nfar = hc->pile[st.pile].n.count;
        st.min = hc->pile[st.pile].min;
        return CLDIAM_OK;
    };
    static std::atomic<int> push_per_sm[64];  // concurrent first calls store the same value
    int dev = 0;
    CLD_CUDA(cudaGetDevice(&dev));
    const int di = (dev >= 0 && dev < 64) ? dev : 0;
    if (push_per_sm[di].load() == 0) {
        int b = 0;
        CLD_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_ds_push, PT, 0));
        push_per_sm[di] = std::max(1, b);
    }
    const unsigned push_grid = (unsigned)num_sms() * (unsigned)std::max(1, push_per_sm[di].load());
    const int ctas = serving_kernel_alive(dev) ? 0 : ds_cluster_size(dev);  // (beside a server the query would load the kernel and wait)
    while (!st.done && (st.ncur > 0 || st.nfar > 0)) {
        const bool small = st.ncur > 0 ? st.ncur <= a.max_list && !st.wide : st.nfar <= a.max_far;
        if (small && ctas && !serving_kernel_alive(dev)) {
            CLD_CUDA(cudaMemsetAsync(ring.get(), 0, 3 * sizeof(DsRound), s));
            cudaLaunchConfig_t cfg{};
            cudaLaunchAttribute at{};
            resident_config(&cfg, &at, ctas, sizeof(DsSmem), s);
            const uint64_t scanned0 = st.scanned;
            CLD_K(K_SSSP, s, CLD_CUDA(cudaLaunchKernelEx(&cfg, k_ds_resident, a, st)));
            CLD_CUDA(cudaMemcpyAsync(hg, gdev.get(), sizeof(DsState), cudaMemcpyDeviceToHost, s));
            CLD_TRY(read());
            st = *hg;
            if (st.bad) return bad_list();
            prof_add_bytes(K_SSSP, 18.0 * (double)(st.scanned - scanned0));
        } else if (st.ncur > 0) {
            ++st.round_id;
            CLD_CUDA(cudaMemsetAsync(ctr.get(), 0, sizeof(DsRound), s));
            CLD_K(K_SSSP, s, k_ds_list<<<grid_for(((size_t)st.ncur + NU - 1) / NU, 256), 256, 0, s>>>(a, st.cur, st.ncur));
            CLD_K(K_SSSP, s, k_ds_push<<<push_grid, PT, 0, s>>>(a, st.cur, st.pile, st.hi, st.round_id, st.epoch));
            CLD_LAUNCH_CHECK();
            CLD_TRY(read());
            st.cur ^= 1;
            st.wide = 0;
            ++st.rounds;
            st.scanned += (uint32_t)hc->r.front;
            // list: 16 B per node (+ its chunk-table share); relax: 8 B (col, w) + 4 B target distance per
            // position (+ 8 B per improved target: distance, stamp, list slot)
            prof_add_bytes(K_SSSP, 24.0 * (double)(uint32_t)(hc->r.front >> 32) + 12.0 * (double)(uint32_t)hc->r.front +
                                       8.0 * st.ncur);
        } else {
            uint64_t lo = 0;
            if (!ds_next_bucket(st, delta, &lo)) break;
            CLD_CUDA(cudaMemsetAsync(ctr.get(), 0, sizeof(DsRound), s));
            CLD_K(K_SSSP, s, k_ds_split<<<grid_for(((size_t)st.nfar + NU - 1) / NU, 256), 256, 0, s>>>(
                                 a, st.cur, st.pile, st.nfar, lo, st.hi, st.epoch));
            CLD_LAUNCH_CHECK();
            st.pile ^= 1;
            CLD_TRY(read());
        }
    }
    CLD_CUDA(cudaMemsetAsync(ecc_d.get(), 0, 4, s));
    CLD_K(K_SSSP, s, k_ds_ecc<<<gb, 256, 0, s>>>(dist.get(), n, ecc_d.get()));
    CLD_LAUNCH_CHECK();
    if (hc->overflow) {
        // a candidate did not fit: an error if one from a final distance does not (an unsettled one may be larger)
        CLD_K(K_SSSP, s, k_ds_overflow<<<gb, 256, 0, s>>>(g->off, g->adj, n, dist.get(), &ctr.get()->overflow));
        CLD_LAUNCH_CHECK();
        CLD_TRY(read());
        if (hc->overflow == 2u) return fail(CLDIAM_ERR_OVERFLOW, "a distance reached 2^32 - 1");
    }
    CLD_CUDA(cudaMemcpyAsync(he, ecc_d.get(), 4, cudaMemcpyDeviceToHost, s));
    if (dist_out) CLD_CUDA(cudaMemcpyAsync(dist_out, dist.get(), (size_t)n * 4, cudaMemcpyDefault, s));
    CLD_CUDA(cudaStreamSynchronize(s));
    *ecc = *he;
    if (rounds_out) *rounds_out = st.rounds;
    if (scanned_out) *scanned_out = st.scanned;
    return CLDIAM_OK;
}

cldiam_status load_sssp_kernels() {
    return load_kernels(k_ds_init, k_ds_list, k_ds_push, k_ds_split, k_ds_overflow, k_ds_ecc);
}

}  // namespace cld
