// Device bodies of the CLUSTER(tau) phases (Algorithm 1), shared by the
// one-graph path's grid kernels (rank br = blockIdx.x of nb CTAs) and the
// resident loop of grow.cuh (the CTAs of a thread-block cluster, or one CTA
// alone, run every body for their graph with a barrier between phases).
//
// Node state (Section 3) is one 64-bit word per node, key = d << 32 | c, so
// the paper's tie-break (smallest distance, then smallest center index) is
// the integer minimum and a Delta-growing step is an atomicMin per light
// edge.  Frozen nodes (clustered in an earlier stage; Procedure Contract)
// hold key 0, which no candidate can undercut, so the relaxation needs no
// frozen test; they are relaxers with the virtual key (0, c_u).
//
// In the cumulative contract mode (Dcum != nullptr) a frozen node relaxes
// with its own bound (D_u, c_u) instead, and only while D_u < Delta.
//
// Steps are synchronous: each frontier entry carries the key its node had
// at the start of the step, so in-place atomicMin gives exactly the
// start-of-step (Jacobi) semantics of the paper's "in parallel" step.  The
// next frontier is the set of nodes whose key decreased (deduplicated with a
// per-node step stamp); nodes whose key did not change would only repeat
// candidates that are already applied.  After a stage start or a Delta
// doubling every relaxer is listed again.
//
// A frontier entry is three parallel words: key (the start-of-step key of a
// pushing node, or kPullTag | v for a node that pulls), pre (its first
// position in the frontier's flattened adjacency) and base = off[v] - pre
// (mod 2^32), so that adjacency index = base + position.
//
// Mutable node state is read with L2 loads (__ldcg): inside one resident
// launch there is no kernel boundary to drop stale L1 lines between phases.
#pragma once

#include <cstddef>

#include "common.cuh"

namespace cld {

struct Counters {
    unsigned long long selected;       // centers drawn in this stage
    unsigned long long edges_scanned;  // adjacency entries read by relax
    unsigned long long frozen;         // nodes frozen by finalize
    unsigned long long frozen_deg;     // their degree sum
    // reset before every growing step (one contiguous block)
    unsigned long long newly_covered;  // nodes that got their first key this step
    unsigned long long front;          // next frontier: (entries << 32) | adjacency entries
    uint32_t nnext;                    // changed nodes this step
    uint32_t bad;                      // a list of the resident growth held an id out of range
    // others
    uint32_t growable;                 // some covered/frozen node touches an uncovered one
    uint32_t overflow;                 // a D_v reached 2^32 - 1
    unsigned long long unfrozen;       // unfrozen nodes the stage's draw saw (checks the tracked |U|)
    uint32_t heavy;                    // a warp that was to hold its part of the next frontier got too much of it
    uint32_t pad;
};
static_assert(offsetof(Counters, bad) + 4 - offsetof(Counters, newly_covered) == 24,
              "the per-step counters form one block");

constexpr int QC = 128;   // frontier positions per chunk-table slot (one warp chunk of the one-graph form)
// In shared memory a pull entry's key is kPullTag | v: a pushed key has
// d < Delta <= 2^31, so its high word is never all ones.
constexpr unsigned long long kPullTag = 0xFFFFFFFF00000000ull;

// Chunk table of a frontier: cfirst[c] = the entry whose adjacency range
// holds flattened position c * QC.  The producer of each entry writes the
// chunk starts that fall inside its range, so relax finds a chunk's entries
// with two loads instead of a search over the frontier.
__device__ __forceinline__ void chunk_table_put(uint32_t* __restrict__ cfirst, uint32_t slot, uint32_t pre,
                                                uint32_t deg) {
    const uint64_t end = (uint64_t)pre + deg;
    for (uint64_t c = ((uint64_t)pre + QC - 1) / QC; c * QC < end; ++c) cfirst[c] = slot;
}

// The same for the entries (`take`) of a whole warp, called by all its lanes: a lane writes a few slots itself, those of
// an entry with more are shared by the warp.  (By its own lane the 8,192 slots of a hub of 2^20 neighbours took 90 us of a
// resident step.)
__device__ __forceinline__ void chunk_table_put_warp(uint32_t* __restrict__ cfirst, bool take, uint32_t slot, uint32_t pre,
                                                     uint32_t deg) {
    constexpr uint32_t kOwn = 8 * QC;  // entries of at most this many positions are their lane's
    if (take && deg <= kOwn) chunk_table_put(cfirst, slot, pre, deg);
    for (unsigned m = __ballot_sync(0xffffffffu, take && deg > kOwn); m; m &= m - 1) {
        const int src = __ffs(m) - 1;
        const uint32_t s = __shfl_sync(0xffffffffu, slot, src);
        const uint64_t p = __shfl_sync(0xffffffffu, pre, src), end = p + __shfl_sync(0xffffffffu, deg, src);
        for (uint64_t c = (p + QC - 1) / QC + lane_id(); c * QC < end; c += 32) cfirst[c] = s;
    }
}

__device__ __forceinline__ void warp_add_u64(unsigned long long* p, unsigned long long v) {
    v = warp_sum(v);
    if (lane_id() == 0 && v) atomicAdd(p, v);
}

// Append to the frontier: one packed atomicAdd per CTA hands out both the
// entry slots (high word) and the entries' first positions in the flattened
// edge list (low word), so positions increase with slots and the frontier's
// degree prefix needs no separate scan.  All threads of the block must call
// it (it synchronises the block); `scratch` holds 33 words.
__device__ __forceinline__ void front_append(unsigned long long* ctr, bool pred, uint32_t deg, uint32_t& slot,
                                             uint32_t& pre, unsigned long long* scratch) {
    const unsigned mask = __ballot_sync(0xffffffffu, pred);
    const unsigned w = threadIdx.x >> 5, l = lane_id(), nw = blockDim.x >> 5;
    const uint32_t d = pred ? deg : 0u;
    const uint32_t incl = warp_incl_scan(d);
    if (l == 31) scratch[w] = ((unsigned long long)__popc(mask) << 32) | incl;
    __syncthreads();
    if (w == 0) {
        const unsigned long long v = l < nw ? scratch[l] : 0ull;
        const unsigned long long iv = warp_incl_scan(v);  // packed (count, entries): no carry, block sums < 2^32
        if (l < nw) scratch[l] = iv - v;
        if (l == 31) scratch[32] = iv ? atomicAdd(ctr, iv) : 0ull;
    }
    __syncthreads();
    const unsigned long long base = scratch[32] + scratch[w];
    slot = (uint32_t)(base >> 32) + (uint32_t)__popc(mask & lanemask_lt());
    pre = (uint32_t)base + (incl - d);
    __syncthreads();
}

// The same for NC candidate entries per thread (bit j of `kinds` set: entry j of deg[j] positions is taken), in the
// order entry 0 of every lane, entry 1 of every lane, ...: a warp's entries stay consecutive per j, so the writes of
// the frontier arrays are coalesced.
template <int NC>
__device__ __forceinline__ void front_append_n(unsigned long long* ctr, uint32_t kinds, const uint32_t (&deg)[NC],
                                               uint32_t (&slot)[NC], uint32_t (&pre)[NC], unsigned long long* scratch) {
    const unsigned w = threadIdx.x >> 5, l = lane_id(), nw = blockDim.x >> 5;
    uint32_t wc = 0, wd = 0;  // the warp's entries and positions so far
#pragma unroll
    for (int j = 0; j < NC; ++j) {
        const bool p = (kinds >> j) & 1u;
        const unsigned mask = __ballot_sync(0xffffffffu, p);
        const uint32_t d = p ? deg[j] : 0u;
        const uint32_t incl = warp_incl_scan(d);
        slot[j] = wc + (uint32_t)__popc(mask & lanemask_lt());
        pre[j] = wd + incl - d;
        wc += (uint32_t)__popc(mask);
        wd += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (l == 31) scratch[w] = ((unsigned long long)wc << 32) | wd;
    __syncthreads();
    if (w == 0) {
        const unsigned long long v = l < nw ? scratch[l] : 0ull;
        const unsigned long long iv = warp_incl_scan(v);
        if (l < nw) scratch[l] = iv - v;
        if (l == 31) scratch[32] = iv ? atomicAdd(ctr, iv) : 0ull;
    }
    __syncthreads();
    const unsigned long long at = scratch[32] + scratch[w];
#pragma unroll
    for (int j = 0; j < NC; ++j) {
        slot[j] += (uint32_t)(at >> 32);
        pre[j] += (uint32_t)at;
    }
    __syncthreads();
}

// ---------------------------------------------------------------- warp-chunk sweeps
// The one-graph kernels that sweep a flattened range of positions (a
// frontier's adjacency, or the whole CSR) give each warp PW consecutive
// positions (PWG groups of 32 lanes) and run without block barriers.
constexpr int PT = 256;          // threads per CTA of the warp-chunk kernels
constexpr int PW = 128;          // positions per warp chunk (== QC, the chunk-table granularity)
constexpr int PWG = PW / 32;     // groups of 32 positions per chunk
constexpr int PNB = 2 * PW + 8;  // per-warp buffer of changed nodes (flushed once >= PW)
static_assert(PW == QC, "one chunk-table slot per warp chunk");

// Row (or frontier entry) segments of a warp's 32-position group.  Entries
// start at strictly increasing positions and each holds at least one; B is
// the index of the entry that holds position g0 (the group's first), and
// starts[j] the first position of entry B + 1 + j for j < n_after.  Returns
// the group's start word (bit d = an entry starts at g0 + d); *own = the
// entry index of this lane's position.
__device__ __forceinline__ uint32_t group_starts(const uint32_t* starts, uint32_t n_after, uint32_t g0,
                                                 uint32_t B, uint32_t lane, unsigned le_mask, uint32_t* own) {
    const uint32_t d = (lane < n_after ? starts[lane] : 0xFFFFFFFFu) - g0;  // entries after B start after g0
    const uint32_t word = __reduce_or_sync(0xffffffffu, d < 32u ? 1u << d : 0u);
    *own = B + (uint32_t)__popc(word & le_mask);
    return word;
}

// Minimum of v over this lane's segment [head, tail] of a group (segments are
// runs of consecutive lanes bounded by the start word); valid at every lane,
// so the head lane holds the segment's minimum.
__device__ __forceinline__ unsigned long long segment_min(unsigned long long v, uint32_t word, uint32_t lane) {
    const unsigned above = lane == 31 ? 0u : word & (0xfffffffeu << lane);
    const uint32_t tail = above ? (uint32_t)__ffs(above) - 2u : 31u;
#pragma unroll
    for (uint32_t o = 1; o < 32; o <<= 1) {
        const unsigned long long t = __shfl_down_sync(0xffffffffu, v, o);
        if (lane + o <= tail) v = t < v ? t : v;
    }
    return v;
}

// Per-warp list of changed nodes, appended to the next list with one atomic per >= PW of them.
struct WarpNext {
    uint32_t* buf;
    uint32_t cnt;
    __device__ __forceinline__ void put(bool first, uint32_t r, uint32_t lane) {
        const unsigned m = __ballot_sync(0xffffffffu, first);
        if (first) buf[cnt + (uint32_t)__popc(m & lanemask_lt())] = r;
        cnt += (uint32_t)__popc(m);
    }
    __device__ __forceinline__ void flush(uint32_t* __restrict__ next, uint32_t* counter, uint32_t lane) {
        __syncwarp();
        uint32_t base = 0;
        if (lane == 0) base = atomicAdd(counter, cnt);
        base = __shfl_sync(0xffffffffu, base, 0);
        for (uint32_t j = lane; j < cnt; j += 32) next[base + j] = buf[j];
        cnt = 0;
        __syncwarp();
    }
};

// Passes over every node (or every changed node) give each thread NU of them a block apart and issue the loads of each
// level for all NU before the next level, one append per NU: with one node per thread and iteration the dependent
// loads and the append's barriers set the time (n = 16.8M: listing 136 -> 92 us, draw 33 -> 29, bounds of the
// contraction 41 -> 32; its freezing pass, 54 us, became slower, 67, and keeps one).
// Nodes that the threads hold one each stay one per thread, so that they spread over all of them.
constexpr uint32_t NU = 4;
__device__ __forceinline__ uint32_t nodes_per_thread(uint32_t n, uint32_t nb) {
    return (uint64_t)n > (uint64_t)nb * blockDim.x ? NU : 1u;
}

// a3: draw the new centers of this stage among unfrozen nodes, reset the others.
__device__ __forceinline__ void dev_select(uint32_t n, const uint32_t* __restrict__ center,
                                           unsigned long long* __restrict__ key, uint64_t seed, uint32_t stage,
                                           uint64_t thr, Counters* ctr, uint32_t br, uint32_t nb,
                                           unsigned long long* __restrict__ keyS = nullptr) {
    unsigned long long cnt = 0, unfrozen = 0;
    const uint32_t per = nodes_per_thread(n, nb);
    const uint64_t stride = (uint64_t)nb * blockDim.x * per;
    for (uint64_t base = (uint64_t)br * blockDim.x * per; base < n; base += stride) {
        uint32_t c[NU];
#pragma unroll
        for (uint32_t u = 0; u < NU; ++u) {
            const uint64_t v = base + u * blockDim.x + threadIdx.x;
            c[u] = u < per && v < n ? __ldcg(&center[v]) : 0u;
        }
#pragma unroll
        for (uint32_t u = 0; u < NU; ++u) {
            const uint32_t v = (uint32_t)base + u * blockDim.x + threadIdx.x;  // < n where c[u] is kNone
            if (c[u] != kNone) continue;
            const U4 r = philox4x32_10(seed, v, stage, 0u, 0u);
            const bool sel = (uint64_t)r.x < thr;
            key[v] = sel ? (unsigned long long)v : kInfKey;
            if (keyS) keyS[v] = sel ? (unsigned long long)v : kInfKey;
            cnt += sel ? 1 : 0;
            ++unfrozen;
        }
    }
    warp_add_u64(&ctr->selected, cnt);
    warp_add_u64(&ctr->unfrozen, unfrozen);
}

// a4: list every relaxer with its current key: unfrozen nodes with d < Delta
// push their key; the contracted clusters either push (0, c_u) from every
// frozen u, or (pull mode) every unfrozen node lists itself to pull
// (w, c_u) from its frozen neighbours -- the same candidates, read from the
// side with fewer adjacency entries.
__device__ __forceinline__ void dev_rebuild(uint32_t n, const unsigned long long* __restrict__ key,
                                            const uint32_t* __restrict__ center, const uint32_t* __restrict__ Dcum,
                                            const uint64_t* __restrict__ off, uint32_t delta, bool pull,
                                            uint32_t* __restrict__ fbase,
                                            unsigned long long* __restrict__ fkey, uint32_t* __restrict__ fpre,
                                            uint32_t* __restrict__ cfirst, Counters* ctr, unsigned long long* scratch,
                                            uint32_t br, uint32_t nb) {
    const uint32_t per = nodes_per_thread(n, nb);
    const uint64_t stride = (uint64_t)nb * blockDim.x * per;
    for (uint64_t base = (uint64_t)br * blockDim.x * per; base < n; base += stride) {
        uint32_t c[NU], b0[NU], deg[NU];
        unsigned long long k[NU];
#pragma unroll
        for (uint32_t u = 0; u < NU; ++u) {
            const uint64_t v = base + u * blockDim.x + threadIdx.x;
            c[u] = 0;
            k[u] = kInfKey;
            b0[u] = deg[u] = 0;
            if (u < per && v < n) {
                const uint64_t o = off[v];
                b0[u] = (uint32_t)o;
                deg[u] = (uint32_t)(off[v + 1] - o);
                c[u] = __ldcg(&center[v]);
            }
        }
#pragma unroll
        for (uint32_t u = 0; u < NU; ++u) {
            const uint64_t v = base + u * blockDim.x + threadIdx.x;
            if (c[u] == kNone) k[u] = __ldcg(&key[v]);
        }
        uint32_t pushes = 0, pulls = 0;
#pragma unroll
        for (uint32_t u = 0; u < NU; ++u) {
            const uint64_t v = base + u * blockDim.x + threadIdx.x;
            if (deg[u] == 0) continue;  // (also past the end)
            bool push;
            if (c[u] != kNone) {
                const uint32_t dd = Dcum ? __ldcg(&Dcum[v]) : 0u;  // (0, c_u), or (D_u, c_u) cumulative
                push = !pull && dd < delta;
                k[u] = ((unsigned long long)dd << 32) | c[u];
            } else {
                push = k[u] != kInfKey && (uint32_t)(k[u] >> 32) < delta;
                pulls |= (pull ? 1u : 0u) << u;
            }
            pushes |= (push ? 1u : 0u) << u;
        }
        for (int kind = 0; kind < (pull ? 2 : 1); ++kind) {
            const uint32_t kinds = kind ? pulls : pushes;
            uint32_t slot[NU], pre[NU];
            front_append_n<NU>(&ctr->front, kinds, deg, slot, pre, scratch);
#pragma unroll
            for (uint32_t u = 0; u < NU; ++u) {
                if (!((kinds >> u) & 1u)) continue;
                fbase[slot[u]] = b0[u] - pre[u];
                fkey[slot[u]] = kind ? kPullTag | (base + u * blockDim.x + threadIdx.x) : k[u];
                fpre[slot[u]] = pre[u];
                if (cfirst) chunk_table_put(cfirst, slot[u], pre[u], deg[u]);
            }
        }
    }
}

// the changed nodes become the next frontier, with their end-of-step keys
// (read after the step has finished, so they are the next step's
// start-of-step values); nodes that reached d = Delta do not relax.
__device__ __forceinline__ void dev_snapshot(const uint32_t* __restrict__ next, uint32_t nn,
                                             const unsigned long long* __restrict__ key,
                                             const uint64_t* __restrict__ off, uint32_t delta,
                                             uint32_t* __restrict__ fbase, unsigned long long* __restrict__ fkey,
                                             uint32_t* __restrict__ fpre, uint32_t* __restrict__ cfirst, Counters* ctr,
                                             unsigned long long* scratch, uint32_t br, uint32_t nb,
                                             unsigned long long* __restrict__ keyS = nullptr, uint32_t n = kNone) {
    for (uint32_t base = br * blockDim.x; base < nn; base += nb * blockDim.x) {
        const uint32_t i = base + threadIdx.x;
        bool take = false;
        uint32_t v = 0, deg = 0, b0 = 0;
        unsigned long long k = 0;
        if (i < nn) {
            v = __ldcg(&next[i]);
            if (v < n) {
                k = __ldcg(&key[v]);
                if (keyS) keyS[v] = k;  // the next step's start-of-step key
                const uint64_t o = off[v];
                b0 = (uint32_t)o;
                deg = (uint32_t)(off[v + 1] - o);
                take = (uint32_t)(k >> 32) < delta && deg > 0;
            } else {
                atomicExch(&ctr->bad, 1u);
            }
        }
        uint32_t slot = 0, pre = 0;
        front_append(&ctr->front, take, deg, slot, pre, scratch);
        if (take) {
            fbase[slot] = b0 - pre;
            fkey[slot] = k;
            fpre[slot] = pre;
        }
        chunk_table_put_warp(cfirst, take, slot, pre, deg);
    }
}

// guard of the doubling loop: does any covered or frozen node have an uncovered neighbour?
__device__ __forceinline__ void dev_growable(const uint32_t* __restrict__ row, const uint2* __restrict__ adj,
                                             uint64_t nnz, const unsigned long long* __restrict__ key, Counters* ctr,
                                             uint32_t br, uint32_t nb) {
    bool any = false;
    for (uint64_t i = (uint64_t)br * blockDim.x + threadIdx.x; i < nnz; i += (uint64_t)nb * blockDim.x) {
        if (__ldcg(&key[adj[i].x]) == kInfKey && __ldcg(&key[row[i]]) != kInfKey) any = true;
    }
    if (__any_sync(0xffffffffu, any) && lane_id() == 0) atomicExch(&ctr->growable, 1u);
}

// a7 (part 1): D_v = d_v + R[c_v] for the nodes covered in this stage (R as before the stage);
// D_v = d_v in the cumulative contract mode (R null), whose d_v already bounds dist_G(c_v, v).
__device__ __forceinline__ void dev_finalize_d(uint32_t n, const unsigned long long* __restrict__ key,
                                               const uint32_t* __restrict__ center, const uint32_t* __restrict__ R,
                                               uint32_t* __restrict__ D, Counters* ctr, uint32_t br, uint32_t nb) {
    const uint32_t per = nodes_per_thread(n, nb);
    const uint64_t stride = (uint64_t)nb * blockDim.x * per;
    for (uint64_t base = (uint64_t)br * blockDim.x * per; base < n; base += stride) {
        unsigned long long k[NU];
        uint32_t r[NU];
        bool take[NU];
#pragma unroll
        for (uint32_t u = 0; u < NU; ++u) {
            const uint64_t v = base + u * blockDim.x + threadIdx.x;
            take[u] = u < per && v < n && __ldcg(&center[v]) == kNone;
        }
#pragma unroll
        for (uint32_t u = 0; u < NU; ++u) k[u] = take[u] ? __ldcg(&key[base + u * blockDim.x + threadIdx.x]) : kInfKey;
#pragma unroll
        for (uint32_t u = 0; u < NU; ++u) {
            take[u] = take[u] && k[u] != kInfKey;
            r[u] = take[u] && R ? __ldcg(&R[(uint32_t)k[u]]) : 0u;  // cumulative mode: R null
        }
#pragma unroll
        for (uint32_t u = 0; u < NU; ++u) {
            if (!take[u]) continue;
            uint64_t dv = (k[u] >> 32) + (uint64_t)r[u];
            if (dv >= 0xFFFFFFFFull) {
                atomicExch(&ctr->overflow, 1u);
                dv = 0xFFFFFFFEull;
            }
            D[base + u * blockDim.x + threadIdx.x] = (uint32_t)dv;
        }
    }
}

// a7 (part 2): freeze them (key 0), record the center, grow R[c].
__device__ __forceinline__ void dev_finalize_freeze(uint32_t n, unsigned long long* __restrict__ key,
                                                    uint32_t* __restrict__ center, uint32_t* __restrict__ R,
                                                    const uint32_t* __restrict__ D, const uint64_t* __restrict__ off,
                                                    Counters* ctr, uint32_t br, uint32_t nb,
                                                    unsigned long long* __restrict__ keyS = nullptr,
                                                    bool cumulative = false) {
    unsigned long long cnt = 0, degs = 0;
    for (uint32_t base = br * blockDim.x; base < n; base += nb * blockDim.x) {
        const uint32_t v = base + threadIdx.x;
        bool take = false;
        uint32_t c = kNone, dv = 0;
        if (v < n && __ldcg(&center[v]) == kNone) {
            const unsigned long long k = __ldcg(&key[v]);
            if (k != kInfKey) {
                take = true;
                c = (uint32_t)k;
                dv = __ldcg(&D[v]);
                center[v] = c;
                key[v] = 0;
                // as a relaxer a contracted node holds (0, c_v), or (D_v, c_v) in the cumulative mode
                if (keyS) keyS[v] = ((cumulative ? (unsigned long long)dv : 0ull) << 32) | c;
                ++cnt;
                degs += off[v + 1] - off[v];
            }
        }
        // nodes of one cluster often share a warp: one atomicMax per distinct center
        const unsigned peers = __match_any_sync(0xffffffffu, take ? c : kNone);
        const uint32_t m = __reduce_max_sync(peers, dv);
        if (take && lane_id() == (unsigned)(__ffs(peers) - 1)) atomicMax(&R[c], m);
    }
    warp_add_u64(&ctr->frozen, cnt);
    warp_add_u64(&ctr->frozen_deg, degs);
}

// a8: leftover nodes become singleton clusters.
__device__ __forceinline__ void dev_singletons(uint32_t n, uint32_t* __restrict__ center, uint32_t* __restrict__ D,
                                               uint32_t br, uint32_t nb) {
    for (uint32_t v = br * blockDim.x + threadIdx.x; v < n; v += nb * blockDim.x)
        if (__ldcg(&center[v]) == kNone) {
            center[v] = v;
            D[v] = 0;
        }
}

// Stage control shared by both forms: the outer-loop test of Algorithm 1 and
// the center-draw threshold floor(p 2^32), p = gamma tau log2 n / |U|; log2 n
// comes from the host so both forms (and the oracle) use the same double.
__host__ __device__ inline bool stage_threshold(uint64_t U, double tau, double L, uint64_t* thr) {
    if (U == 0) return false;
    if ((double)U < 8.0 * tau * L) return false;
    const double p = kGamma * tau * L / (double)U;
    *thr = (p >= 1.0) ? 4294967296ull : (uint64_t)floor(p * 4294967296.0);
    return *thr != 0;
}

}  // namespace cld
