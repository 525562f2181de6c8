// CLUSTER2(G, tau) of Algorithm 2 (Section 4) on the GPU.
//
// Algorithm 2 contracts the clusters after every iteration and rescales an
// edge leaving a cluster to d_u + w - 2 R_CL (Contract2).  Rescaling by 2 R_CL
// per contraction is the same as giving every node a global offset instead:
// a center drawn in iteration i starts at g = (i - 1) 2 R_CL, a node reached
// from u over an edge of weight w gets g_u + w, and iteration i keeps exactly
// the nodes with g <= i 2 R_CL (distance <= 2 R_CL in the contracted graph
// G_i).  So the device keeps the original CSR and one offset per node: no
// edge list is rebuilt.  PartialGrowth2 runs growth to its fixed point
// (unique: the (distance, center id) minimum over the allowed paths), here by
// frontier rounds of relaxations, which reach the same fixed point as the
// paper's synchronous steps.  D_v = g_v - g_{c_v} is the length of the path
// the growth followed.
//
// A covered node's key is 0 during growth (below every candidate, whose high
// word is at least 1: a neighbour of an earlier iteration's node within
// g <= base was covered by then), so one gather of the key tells whether a
// neighbour is covered and filters candidates that cannot win.
#include <algorithm>
#include <atomic>
#include <cmath>

#include "cluster_dev.cuh"
#include "internal.cuh"
#include "prof.cuh"

namespace cld {

namespace {

constexpr uint32_t kC2Stream = 1;  // third Philox counter word of CLUSTER2's center draws

struct C2Counters {
    unsigned long long drawn;     // centers drawn
    unsigned long long updates;   // successful state decreases
    unsigned long long joined;    // nodes that joined a cluster by growth
    // reset before every round (one block)
    unsigned long long front;     // listed frontier: (entries << 32) | adjacency positions
    uint32_t nnext;               // nodes improved this round
    uint32_t pad0;
    // others
    uint32_t uncovered;           // nodes left without a center at the end
    uint32_t pad1;
};
static_assert(offsetof(C2Counters, pad0) + 4 - offsetof(C2Counters, front) == 16, "the per-round counters form one block");

// scan state of a node: never listed, listed with no uncovered neighbour over a usable edge (which stays true:
// coverage only grows), or listed with one
constexpr uint8_t kC2New = 0, kC2Done = 1, kC2Open = 2;

// iteration i: an uncovered v is drawn iff Philox(seed; (v, i, 1, 0)) word 0 < thr; it starts at g = base
__global__ void k_c2_select(uint32_t n, uint32_t* __restrict__ center, uint32_t* __restrict__ g,
                            unsigned long long* __restrict__ key, uint64_t seed, uint32_t it, uint64_t thr,
                            uint32_t base, C2Counters* ctr) {
    unsigned long long cnt = 0;
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
        if (center[v] != kNone) continue;
        const U4 r = philox4x32_10(seed, v, it, kC2Stream, 0u);
        if ((uint64_t)r.x < thr) {
            center[v] = v;
            g[v] = base;
            key[v] = 0;
            ++cnt;
        }
    }
    cnt = warp_sum(cnt);
    if (lane_id() == 0 && cnt) atomicAdd(&ctr->drawn, cnt);
}

// A round's frontier, with the first position of every node's adjacency in one flattened range and a chunk table
// (as a growing step of CLUSTER): the nodes of `list`, or (ALL: an iteration's first round) every covered node that
// may still have an uncovered neighbour.  An entry carries its node's value (g_u, c_u) at the start of the round:
// g_u when covered, else base + its current distance.  Every listed node counts as done until the push finds an
// uncovered neighbour.
template <bool ALL>
__global__ void __launch_bounds__(256) k_c2_list(const uint32_t* __restrict__ list, uint32_t nl,
                                                 const uint32_t* __restrict__ center, const uint32_t* __restrict__ g,
                                                 const unsigned long long* __restrict__ key, uint32_t base,
                                                 const uint64_t* __restrict__ off, uint8_t* __restrict__ state,
                                                 uint32_t* __restrict__ fnode, uint32_t* __restrict__ fbase,
                                                 unsigned long long* __restrict__ fval, uint32_t* __restrict__ fpre,
                                                 uint32_t* __restrict__ cfirst, C2Counters* ctr) {
    __shared__ unsigned long long scratch[33];
    for (uint32_t b = blockIdx.x * blockDim.x; b < nl; b += gridDim.x * blockDim.x) {
        const uint32_t i = b + threadIdx.x;
        bool take = false;
        uint32_t u = 0, deg = 0, b0 = 0;
        unsigned long long val = 0;
        if (i < nl) {
            u = ALL ? i : list[i];
            const uint32_t cc = center[u];
            if (!ALL || (cc != kNone && state[u] != kC2Done)) {
                if (cc != kNone) {
                    val = ((unsigned long long)g[u] << 32) | cc;
                } else {
                    const unsigned long long k = key[u];
                    val = ((unsigned long long)(base + (uint32_t)(k >> 32)) << 32) | (uint32_t)k;
                }
                const uint64_t o = off[u];
                b0 = (uint32_t)o;
                deg = (uint32_t)(off[u + 1] - o);
                take = deg > 0;
                state[u] = kC2Done;
            }
        }
        uint32_t slot = 0, pre = 0;
        front_append(&ctr->front, take, deg, slot, pre, scratch);
        if (take) {
            fnode[slot] = u;
            fbase[slot] = b0 - pre;
            fval[slot] = val;
            fpre[slot] = pre;
            chunk_table_put(cfirst, slot, pre, deg);
        }
    }
}

// One round over the listed frontier: each warp takes PW consecutive positions of the flattened adjacency, so a hub's
// entries spread over many warps (with a CTA per node above 256 entries, the hubs of R-MAT 20 took 231 us a round and
// the other nodes, a warp each, 95 us; together 86 us so).  Bound by the latency of the key gathers.  An uncovered neighbour (key not 0) over an edge of
// weight <= delta marks the entry's node open; the candidate (g_u + w - base, c_u) is kept when g_u + w <= base + delta
// and lowers the neighbour's key, and an improved node joins the next frontier once per round (stamp).
__global__ void __launch_bounds__(PT, 6) k_c2_push(const uint32_t* __restrict__ fnode, const uint32_t* __restrict__ fbase,
                                                   const unsigned long long* __restrict__ fval,
                                                   const uint32_t* __restrict__ fpre, const uint32_t* __restrict__ cfirst,
                                                   const uint2* __restrict__ adj, unsigned long long* __restrict__ key,
                                                   uint32_t base, uint32_t delta, uint32_t* __restrict__ stamp,
                                                   uint32_t round, uint32_t* __restrict__ next,
                                                   uint8_t* __restrict__ state, C2Counters* ctr) {
    __shared__ uint32_t spre[PT / 32][PW + 1];
    __shared__ uint32_t sbase[PT / 32][PW + 2];
    __shared__ uint32_t snode[PT / 32][PW + 2];
    __shared__ unsigned long long sval[PT / 32][PW + 2];
    __shared__ uint32_t sbuf[PT / 32][PNB];
    const uint32_t lane = lane_id(), warp = threadIdx.x >> 5;
    const uint64_t pol_stream = l2_evict_first_policy(), pol_keep = l2_evict_last_policy();
    const unsigned le_mask = 0xffffffffu >> (31u - lane);
    const unsigned long long fr = __ldcg(&ctr->front);
    const uint32_t nf = (uint32_t)(fr >> 32), E = (uint32_t)fr;
    const uint64_t limit = (uint64_t)base + delta;
    WarpNext wn{sbuf[warp], 0};
    unsigned long long upd = 0;
    const uint32_t nq = (uint32_t)(((uint64_t)E + PW - 1) / PW);
    const uint32_t nwarps = gridDim.x * (PT / 32);
    for (uint32_t q = blockIdx.x * (PT / 32) + warp; q < nq; q += nwarps) {
        const uint32_t p0 = q * PW, e1 = (uint32_t)min((uint64_t)E, (uint64_t)p0 + PW);
        const uint32_t i0 = __ldg(&cfirst[q]);
        const uint32_t il = q + 1 < nq ? __ldg(&cfirst[q + 1]) : nf - 1;
        const uint32_t ne = min(il - i0 + 1, (uint32_t)PW + 1);
        __syncwarp();  // the previous chunk's entries have been read
        for (uint32_t j = lane; j < ne; j += 32) {
            if (j) spre[warp][j - 1] = __ldg(&fpre[i0 + j]);
            sbase[warp][j] = __ldg(&fbase[i0 + j]);
            snode[warp][j] = __ldg(&fnode[i0 + j]);
            sval[warp][j] = __ldg(&fval[i0 + j]);
        }
        __syncwarp();
        uint32_t own[PWG], word[PWG];
        {
            uint32_t B = 0;
#pragma unroll
            for (int u = 0; u < PWG; ++u) {
                word[u] = group_starts(spre[warp] + B, ne - 1 - B, p0 + 32u * u, B, lane, le_mask, &own[u]);
                B += (uint32_t)__popc(word[u]);
            }
        }
        uint2 ed[PWG];
#pragma unroll
        for (int u = 0; u < PWG; ++u) {
            const uint32_t p = p0 + 32u * u + lane;
            ed[u] = p < e1 && p >= p0 ? ld_stream_u2(adj + (sbase[warp][own[u]] + p), pol_stream)
                                      : make_uint2(0u, 0xFFFFFFFFu);
        }
        unsigned long long cur[PWG];  // through L1: a stale line holds a larger key, or 0 as long as the node is covered
#pragma unroll
        for (int u = 0; u < PWG; ++u) {
            const uint32_t p = p0 + 32u * u + lane;
            cur[u] = p < e1 && p >= p0 && ed[u].y <= delta ? ld_keep_u64(&key[ed[u].x], pol_keep) : 0ull;
        }
#pragma unroll
        for (int u = 0; u < PWG; ++u) {
            const bool open = cur[u] != 0ull;
            const unsigned om = __ballot_sync(0xffffffffu, open);
            const unsigned le = word[u] & le_mask;
            const uint32_t head = le ? 31u - (uint32_t)__clz(le) : 0u;  // first lane of this lane's entry
            if (open && !(om & lanemask_lt() & (0xffffffffu << head))) state[snode[warp][own[u]]] = kC2Open;
            bool first = false;
            const unsigned long long val = sval[warp][own[u]];
            const uint64_t cg = (val >> 32) + ed[u].y;
            if (open && cg <= limit) {
                const unsigned long long ck = ((unsigned long long)(uint32_t)(cg - base) << 32) | (uint32_t)val;
                if (ck < cur[u] && ck < atomicMin(&key[ed[u].x], ck)) {
                    ++upd;
                    first = atomicExch(&stamp[ed[u].x], round) != round;
                }
            }
            wn.put(first, ed[u].x, lane);
        }
        if (wn.cnt >= (uint32_t)PW) wn.flush(next, &ctr->nnext, lane);
    }
    if (wn.cnt) wn.flush(next, &ctr->nnext, lane);
    warp_add_u64(&ctr->updates, upd);
}

// reached nodes join their clusters at g = base + distance; their keys become 0 (covered)
__global__ void k_c2_finalize(uint32_t n, uint32_t* __restrict__ center, uint32_t* __restrict__ g,
                              unsigned long long* __restrict__ key, uint32_t base, C2Counters* ctr) {
    unsigned long long cnt = 0;
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
        const unsigned long long k = key[v];
        if (k == kInfKey || k == 0ull) continue;
        center[v] = (uint32_t)k;
        g[v] = base + (uint32_t)(k >> 32);
        key[v] = 0;
        ++cnt;
    }
    cnt = warp_sum(cnt);
    if (lane_id() == 0 && cnt) atomicAdd(&ctr->joined, cnt);
}

// D_v = g_v - g_{c_v}; counts nodes left uncovered (none after the last iteration)
__global__ void k_c2_distances(uint32_t n, const uint32_t* __restrict__ center, const uint32_t* __restrict__ g,
                               uint32_t* __restrict__ D, C2Counters* ctr) {
    uint32_t bad = 0;
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
        const uint32_t c = center[v];
        if (c == kNone) {
            ++bad;
            D[v] = 0;
        } else {
            D[v] = g[v] - g[c];
        }
    }
    bad = warp_sum(bad);
    if (lane_id() == 0 && bad) atomicAdd(&ctr->uncovered, bad);
}

__global__ void k_c2_fill(uint32_t n, uint32_t* __restrict__ center, uint32_t* __restrict__ g,
                          unsigned long long* __restrict__ key, uint32_t* __restrict__ stamp,
                          uint8_t* __restrict__ state) {
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
        center[v] = kNone;
        g[v] = 0;
        key[v] = kInfKey;
        stamp[v] = 0;
        state[v] = kC2New;
    }
}

struct Owner {
    cldiam_clustering* c;
    explicit Owner(cldiam_clustering* x) : c(x) {}
    ~Owner() {
        if (c) free_clustering(c);
    }
};

}  // namespace

cldiam_status cluster2(cldiam_graph* g, double tau, uint64_t seed, const cldiam_opts* o, cldiam_clustering** out) {
    if (!g || !out) return fail(CLDIAM_ERR_INVALID_ARG, "NULL graph or out");
    *out = nullptr;
    // R_CL: the radius of CLUSTER(G, tau) under the same options
    cldiam_clustering* first = nullptr;
    CLD_TRY(cluster(g, tau, seed, o, &first));
    Owner own_first(first);
    const cudaStream_t s = g->stream;
    const uint32_t n = g->n;
    C2Counters* hc = static_cast<C2Counters*>(g->host.h);
    static_assert(sizeof(C2Counters) <= 128, "counter block must fit the pinned area");
    DBuf<C2Counters> ctr;
    CLD_TRY(ctr.alloc(1, s));
    uint32_t R = 0;
    {
        DBuf<uint32_t> rmax;
        CLD_TRY(rmax.alloc(1, s));
        CLD_TRY(reduce_max_u32(first->D, n, rmax.get(), s));
        CLD_CUDA(cudaMemcpyAsync(&hc->nnext, rmax.get(), 4, cudaMemcpyDeviceToHost, s));
        CLD_CUDA(cudaStreamSynchronize(s));
        R = hc->nnext;
    }
    uint32_t L = 1;
    while ((1ull << L) < (uint64_t)n) ++L;
    const uint64_t delta64 = 2ull * R;
    if (delta64 * L >= 0xFFFFFFFFull)
        return fail(CLDIAM_ERR_UNSUPPORTED, "CLUSTER2 offsets (log2 n x 2 R_CL) need more than 32 bits");
    const uint32_t delta = (uint32_t)delta64;

    Owner owner(new cldiam_clustering());
    cldiam_clustering* cl = owner.c;
    cl->g = g;
    cl->stream = g->stream;
    cl->max_fw_k = first->max_fw_k;
    cl->quotient_mode = first->quotient_mode;
    DBuf<uint32_t> center, D, cid, gv, stamp, frA, frB;
    DBuf<unsigned long long> key, fval;
    DBuf<uint8_t> state;
    DBuf<uint32_t> fnode, fbase, fpre, cfirst;
    CLD_TRY(state.alloc(n, s));
    CLD_TRY(fnode.alloc(n, s));
    CLD_TRY(fbase.alloc(n, s));
    CLD_TRY(fpre.alloc(n, s));
    CLD_TRY(fval.alloc(n, s));
    CLD_TRY(cfirst.alloc(g->nnz / PW + 2, s));  // a round lists a node at most once
    CLD_TRY(center.alloc(n, s));
    CLD_TRY(D.alloc(n, s));
    CLD_TRY(cid.alloc(n, s));
    CLD_TRY(gv.alloc(n, s));
    CLD_TRY(stamp.alloc(n, s));
    CLD_TRY(frA.alloc(n, s));
    CLD_TRY(frB.alloc(n, s));
    CLD_TRY(key.alloc(n, s));
    const unsigned gb = grid_for(n, 256);
    CLD_K(K_MISC, s, k_c2_fill<<<gb, 256, 0, s>>>(n, center.get(), gv.get(), key.get(), stamp.get(), state.get()));
    CLD_LAUNCH_CHECK();
    CLD_CUDA(cudaMemsetAsync(ctr.get(), 0, sizeof(C2Counters), s));
    auto read_counters = [&]() -> cldiam_status {
        CLD_CUDA(cudaMemcpyAsync(hc, ctr.get(), sizeof(C2Counters), cudaMemcpyDeviceToHost, s));
        CLD_CUDA(cudaStreamSynchronize(s));
        return CLDIAM_OK;
    };
    static std::atomic<int> push_per_sm[64];  // concurrent first calls store the same value
    int dev = 0;
    CLD_CUDA(cudaGetDevice(&dev));
    const int di = (dev >= 0 && dev < 64) ? dev : 0;
    if (push_per_sm[di].load() == 0) {
        int a = 0;
        CLD_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_c2_push, PT, 0));
        push_per_sm[di] = std::max(1, a);
    }
    const unsigned push_grid = (unsigned)num_sms() * (unsigned)push_per_sm[di].load();

    cldiam_result st{};
    uint32_t round = 0;
    uint64_t scanned = 0;
    const uint64_t max_rounds = (uint64_t)L * ((uint64_t)n + 2);  // each round settles some node for good
    for (uint32_t i = 1; i <= L; ++i) {
        const uint64_t thr = ((1ull << i) >= (uint64_t)n) ? (1ull << 32) : ((1ull << (32 + i)) / n);
        const uint32_t base = (uint32_t)((uint64_t)(i - 1) * delta);
        CLD_K(K_SELECT, s, k_c2_select<<<gb, 256, 0, s>>>(n, center.get(), gv.get(), key.get(), seed, i, thr, base,
                                                          ctr.get()));
        CLD_LAUNCH_CHECK();
        // PartialGrowth2: rounds until no state decreases
        uint32_t* fr = frA.get();
        uint32_t* fr2 = frB.get();
        uint32_t nf = 0;
        for (bool all = true; all || nf > 0; all = false) {
            CLD_CUDA(cudaMemsetAsync(&ctr.get()->front, 0, 16, s));  // front, nnext
            if (all)
                CLD_K(K_REBUILD, s, k_c2_list<true><<<gb, 256, 0, s>>>(nullptr, n, center.get(), gv.get(), key.get(), base,
                                                                       g->off, state.get(), fnode.get(), fbase.get(),
                                                                       fval.get(), fpre.get(), cfirst.get(), ctr.get()));
            else
                CLD_K(K_SNAPSHOT, s, k_c2_list<false><<<grid_for(nf, 256), 256, 0, s>>>(
                                         fr, nf, center.get(), gv.get(), key.get(), base, g->off, state.get(), fnode.get(),
                                         fbase.get(), fval.get(), fpre.get(), cfirst.get(), ctr.get()));
            CLD_K(K_RELAX, s, k_c2_push<<<push_grid, PT, 0, s>>>(fnode.get(), fbase.get(), fval.get(), fpre.get(),
                                                                 cfirst.get(), g->adj, key.get(), base, delta,
                                                                 stamp.get(), round + 1, fr2, state.get(), ctr.get()));
            CLD_LAUNCH_CHECK();
            CLD_TRY(read_counters());
            if (hc->front == 0) break;
            if (++round > max_rounds) return fail(CLDIAM_ERR_DIVERGED, "CLUSTER2 growth did not settle");
            scanned += (uint32_t)hc->front;
            nf = hc->nnext;
            std::swap(fr, fr2);
        }
        CLD_K(K_FINALIZE, s, k_c2_finalize<<<gb, 256, 0, s>>>(n, center.get(), gv.get(), key.get(), base, ctr.get()));
        CLD_LAUNCH_CHECK();
        // every node covered: the remaining iterations can neither draw nor grow anything
        CLD_TRY(read_counters());
        if (hc->drawn + hc->joined >= n) break;
    }
    CLD_K(K_FINALIZE, s, k_c2_distances<<<gb, 256, 0, s>>>(n, center.get(), gv.get(), D.get(), ctr.get()));
    CLD_LAUNCH_CHECK();
    CLD_TRY(read_counters());
    if (hc->uncovered) return fail(CLDIAM_ERR_DIVERGED, "CLUSTER2 left nodes uncovered");
    st.centers_drawn = hc->drawn;
    st.node_updates = hc->updates;
    st.edges_scanned = scanned;
    CLD_TRY(relabel_clusters(g, center.get(), cid.get(), &st.k));
    prof_flush();
    st.stages = L;
    st.steps = round;
    st.delta_end = delta;

    cl->center = center.detach();
    cl->D = D.detach();
    cl->cid = cid.detach();
    cl->k = st.k;
    cl->stats = st;
    *out = cl;
    owner.c = nullptr;
    return CLDIAM_OK;
}

cldiam_status load_cluster2_kernels() {
    return load_kernels(k_c2_fill, k_c2_select, k_c2_list<false>, k_c2_list<true>, k_c2_push, k_c2_finalize, k_c2_distances);
}

}  // namespace cld
