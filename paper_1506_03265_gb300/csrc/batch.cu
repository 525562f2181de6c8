// Many-graph form: graphs packed into one device CSR arena and processed by
// one persistent launch.  Each CTA (1024 threads, one per SM) takes whole
// graphs from a work queue (longest first) and runs CLUSTER(tau) (the growth
// loop of grow.cuh), the weighted quotient graph (Section 4) and the exact
// Phi(G_C) for it; large graphs are shared by a group of CTAs (a thread-block
// cluster) that run the same code, every phase split over them.  Results are
// identical to the one-graph-per-launch path: the same phase bodies run in
// the same order on the same data, and the stage control uses the same
// host-computed log2 n.
//
// The quotient is deduplicated in a dense k x k matrix (atomicMin per
// inter-cluster edge) instead of a sort; its row order equals the sorted
// quotient CSR of the other path.  Graphs whose quotient exceeds the dense
// capacity are finished with the one-graph path after the launch.
#include <algorithm>
#include <atomic>
#include <chrono>
#include <cmath>
#include <condition_variable>
#include <deque>
#include <mutex>
#include <numeric>
#include <thread>
#include <vector>

#include "bounds.cuh"
#include "grow.cuh"
#include "internal.cuh"
#include "prof.cuh"

namespace cld {

namespace {

// many-graph CTAs resident per SM.  One 1,024-thread CTA per SM: two 512-thread CTAs per SM (shared-memory
// carveout at its maximum, Floyd-Warshall cut-over 128) gave 16 % more aggregate work per second on the
// 2,000-graph mixture but 1.6x the time per large graph on one CTA, and its 111 R-MAT 16 graphs set the
// tail (17.4k against 25.4k graphs/s)
constexpr int kBatchCtasPerSm = 1;
constexpr int BT = GT;  // threads per CTA: those of the growth loop
constexpr int BW = BT / 32;
constexpr int kJobCtas = 8;  // CTAs that share a large job: the portable cluster size
constexpr uint32_t kDenseCap = 1024;  // largest quotient deduplicated in the dense matrix
constexpr uint64_t kSplitMinEntries = 1u << 16;  // graphs below this many entries always stay in the launch
// Time model of the many-graph split (GB300; unit = entry or node): a job on one CTA, on a group of kJobCtas CTAs, and
// on the one-graph path (launches and counter reads, then the whole device).  Graphs of fewer than 8 entries per node
// (meshes, roads) take many small steps, others few large ones.  Measured on one CTA: meshes 15 ns a unit from 10^5 to
// 10^6 units, R-MAT 4 to 5; on a group meshes of 4.6 / 6.2 / 10.7 x 10^5 units 2.4 / 3.0 / 3.6 ms, R-MAT 0.8 to 1.1 ns.
// A batch of 200 graphs (10^3 to 10^6 units): every job on one CTA 15.8 ms, with groups 5.9 ms.
inline double job_cta_s(double units, bool sparse) { return units * (sparse ? 15e-9 : 4.5e-9); }
inline double job_group_s(double units, bool sparse) {
    return sparse ? 1.6e-3 * std::min(1.0, units / 4e5) + units * 1.9e-9 : units * 1.0e-9;
}
inline double job_plain_s(double units, bool sparse) { return (sparse ? 3.0e-3 : 1.0e-3) + units * 0.1e-9; }
// quotients up to this size are closed by Floyd-Warshall in shared memory (the k x k matrix, next to the
// static shared memory, must fit kBatchCtasPerSm times per SM)
constexpr uint32_t kSmemFwK = kBatchCtasPerSm == 1 ? 200 : 128;
constexpr uint32_t kJobOk = 0, kJobNeedsPlain = 1, kJobOverflow = 2, kJobDiverged = 3, kJobTimeout = 4;

struct ArenaDesc {  // one graph of the arena (device copy)
    uint64_t off_base;  // into the arena's offset array (n + 1 entries, local values)
    uint64_t adj_base;  // into the arena's adjacency / row arrays
    uint64_t nnz;
    uint32_t n;
    uint32_t connected;
};

struct Job {
    double tau;
    double L;  // log2 n, computed on the host
    uint64_t seed;
    uint32_t graph;
    uint32_t delta0;
    uint32_t out;         // index in the caller's result array
    uint32_t step_cap;    // growing steps per PartialGrowth, 0 = no cap
    uint32_t cumulative;  // cumulative contract mode
    uint32_t fw_k;        // quotients up to this size (<= kSmemFwK) are closed by Floyd-Warshall in shared memory
    uint32_t pad;
};

// Results of a job's phases after CLUSTER, shared by its CTAs.
struct FinishCtl {
    unsigned long long entries;  // of the quotient
    unsigned long long wsum;     // sum over quotient nodes of their heaviest entry
    uint32_t wmax, rmax, best, nsrc, err, job;
    uint32_t part[kJobCtas];     // centers in each CTA's share of the nodes
};

struct Workspace {  // one slice per CTA, or per group of CTAs that share a job
    unsigned long long* key;
    unsigned long long* fkey[2];
    uint32_t* center;
    uint32_t* D;
    uint32_t* R;
    uint32_t* stamp;
    uint32_t* fbase[2];
    uint32_t* fpre[2];
    uint32_t* cfirst[2];
    uint32_t* next;
    uint32_t* M;      // dense quotient, kDenseCap^2
    uint32_t* qoff;   // quotient CSR extracted from M
    uint32_t* qcol;
    uint32_t* qw;
    Counters* ring;   // three counter blocks
    FinishCtl* fin;
};

struct JobOut {
    cldiam_result r;
    uint32_t status;
    uint32_t pad;
    uint64_t t_start, t_end;  // device global timer (ns) when the job started and ended
};


__device__ __forceinline__ uint32_t relax_min_u32(uint32_t c, uint32_t a, uint32_t b, bool& ovf) {
    const uint32_t s = a + b;
    const bool carry = s < a;
    const bool finite = (a != kNone) & (b != kNone);
    ovf |= finite & (carry | (s == kNone));
    return (carry | !finite) ? c : (s < c ? s : c);
}

// every thread gets op over the block's values; ident is op's identity (it fills the lanes past the
// block's warp count)
template <class T, class Op>
__device__ __forceinline__ T block_all_reduce(T v, Op op, T ident, T* red) {
    v = op(v, __shfl_xor_sync(0xffffffffu, v, 16));
    v = op(v, __shfl_xor_sync(0xffffffffu, v, 8));
    v = op(v, __shfl_xor_sync(0xffffffffu, v, 4));
    v = op(v, __shfl_xor_sync(0xffffffffu, v, 2));
    v = op(v, __shfl_xor_sync(0xffffffffu, v, 1));
    const unsigned w = threadIdx.x >> 5, l = lane_id(), nw = blockDim.x >> 5;
    if (l == 0) red[w] = v;
    __syncthreads();
    if (w == 0) {
        T x = l < nw ? red[l] : ident;
        x = op(x, __shfl_xor_sync(0xffffffffu, x, 16));
        x = op(x, __shfl_xor_sync(0xffffffffu, x, 8));
        x = op(x, __shfl_xor_sync(0xffffffffu, x, 4));
        x = op(x, __shfl_xor_sync(0xffffffffu, x, 2));
        x = op(x, __shfl_xor_sync(0xffffffffu, x, 1));
        if (l == 0) red[32] = x;
    }
    __syncthreads();
    const T r = red[32];
    __syncthreads();
    return r;
}

struct BatchSmem {  // (a CTA's copies of what every thread would otherwise hold in registers)
    GrowArgs args;
    GrowState grown;  // CLUSTER's control state at its end
    Workspace ws;
    Job job;
    uint32_t red32[33];
    uint32_t woff[33];
    uint32_t word;
};

constexpr uint32_t kFinishU = 4;  // nodes, rows' columns or entries per thread whose loads are issued together

// Centers among nodes [lo, hi) (4,096 per iteration, 128 consecutive ones per warp): returns their number; with `rank`
// also rank[c] = first + the number of smaller centers of the range.
__device__ uint32_t block_centers(uint32_t lo, uint32_t hi, const uint32_t* center, uint32_t* rank, uint32_t first,
                                  BatchSmem& sm) {
    const unsigned w = threadIdx.x >> 5, l = lane_id();
    uint32_t running = 0;
    for (uint64_t base = lo; base < hi; base += BT * kFinishU) {
        unsigned bal[kFinishU];
        uint32_t mine = 0;
        const uint64_t v0 = base + w * (32 * kFinishU) + l;
        uint32_t c[kFinishU];
#pragma unroll
        for (uint32_t u = 0; u < kFinishU; ++u) c[u] = v0 + 32 * u < hi ? __ldcg(&center[v0 + 32 * u]) : kNone;
#pragma unroll
        for (uint32_t u = 0; u < kFinishU; ++u) {
            bal[u] = __ballot_sync(0xffffffffu, c[u] != kNone && c[u] == (uint32_t)v0 + 32 * u);
            mine += (uint32_t)__popc(bal[u]);
        }
        if (l == 0) sm.woff[w] = mine;
        __syncthreads();
        if (w == 0) {
            const uint32_t x = l < BW ? sm.woff[l] : 0u;
            const uint32_t incl = warp_incl_scan(x);
            sm.woff[l] = incl - x;
            if (l == 31) sm.woff[32] = incl;
        }
        __syncthreads();
        if (rank) {
            uint32_t at = first + running + sm.woff[w];
#pragma unroll
            for (uint32_t u = 0; u < kFinishU; ++u) {
                if ((bal[u] >> l) & 1u) rank[v0 + 32 * u] = at + (uint32_t)__popc(bal[u] & lanemask_lt());
                at += (uint32_t)__popc(bal[u]);
            }
        }
        running += sm.woff[32];
        __syncthreads();
    }
    return running;
}

// Floyd-Warshall of the k x k matrix M in shared memory (k <= kSmemFwK); row p and column p are fixed during iteration p
__device__ uint32_t block_floyd_warshall(uint32_t k, const uint32_t* M, uint32_t* dyn, bool& ovf) {
    const unsigned w = threadIdx.x >> 5, l = lane_id();
    for (uint32_t i = threadIdx.x; i < k * k; i += BT) dyn[i] = __ldcg(&M[i]);
    __syncthreads();
    for (uint32_t p = 0; p < k; ++p) {
        for (uint32_t i = w; i < k; i += BW) {
            const uint32_t a = dyn[i * k + p];
            for (uint32_t j = l; j < k; j += 32) dyn[i * k + j] = relax_min_u32(dyn[i * k + j], a, dyn[p * k + j], ovf);
        }
        __syncthreads();
    }
    uint32_t best = 0;
    for (uint32_t i = threadIdx.x; i < k * k; i += BT)
        if (dyn[i] != kNone && dyn[i] > best) best = dyn[i];
    return best;
}

// Every source of the quotient CSR by one CTA, with overflow checks (quotients whose path sums might reach 2^32 - 1):
// worklist multi-source Bellman-Ford, 8 sources at a time: dist[v][s] and one word of change bits per node (two rounds)
// in shared memory; a changed node pushes to its neighbours
__device__ uint32_t block_all_sources(uint32_t k, const Workspace& ws, uint32_t* dyn, bool& ovf) {
    const unsigned w = threadIdx.x >> 5, l = lane_id();
    constexpr uint32_t S = 8;
    uint32_t best = 0;
    uint32_t* dist = dyn;  // k x S
    uint32_t* chg0 = dyn + (size_t)k * S;
    uint32_t* chg1 = chg0 + k;
    for (uint32_t s0 = 0; s0 < k; s0 += S) {
        for (uint32_t i = threadIdx.x; i < k * S; i += BT) dist[i] = (s0 + i % S == i / S) ? 0u : kNone;
        for (uint32_t v = threadIdx.x; v < k; v += BT) {
            chg0[v] = (v >= s0 && v < s0 + S) ? 1u << (v - s0) : 0u;
            chg1[v] = 0;
        }
        __syncthreads();
        for (uint32_t round = 0;; ++round) {
            uint32_t* cur = (round & 1) ? chg1 : chg0;
            uint32_t* nxt = (round & 1) ? chg0 : chg1;
            for (uint32_t v = w; v < k; v += BW) {
                const uint32_t bits = cur[v];
                if (!bits) continue;
                const uint32_t beg = __ldcg(&ws.qoff[v]), end = __ldcg(&ws.qoff[v + 1]);
                for (uint32_t j = beg + l; j < end; j += 32) {
                    const uint32_t u = __ldcg(&ws.qcol[j]), wj = __ldcg(&ws.qw[j]);
                    for (uint32_t b = bits; b; b &= b - 1) {
                        const uint32_t si = (uint32_t)__ffs(b) - 1;
                        const uint32_t dv = dist[v * S + si];
                        if (dv == kNone) continue;
                        const uint64_t nd = (uint64_t)dv + wj;
                        if (nd >= kNone) {
                            ovf = true;
                            continue;
                        }
                        uint32_t* du = &dist[u * S + si];
                        if ((uint32_t)nd < *du && (uint32_t)nd < atomicMin(du, (uint32_t)nd))
                            atomicOr(&nxt[u], 1u << si);
                    }
                }
            }
            __syncthreads();
            bool any = false;
            for (uint32_t v = threadIdx.x; v < k; v += BT) {
                cur[v] = 0;
                any |= nxt[v] != 0;
            }
            if (!__syncthreads_or(any)) break;
            if (round > k * S + 64) {  // distances only decrease: far above any real count, reported
                ovf = true;
                break;
            }
        }
        for (uint32_t i = threadIdx.x; i < k * S; i += BT)
            if (s0 + i % S < k && dist[i] != kNone && dist[i] > best) best = dist[i];
        __syncthreads();
    }
    return best;
}

// The quotient CSR as the SSSPs of one CTA read it: staged in shared memory when it fits beside them.
struct QuotientView {
    const uint32_t* off;   // [k + 1], shared
    const uint16_t* scol;  // shared, or null
    const uint32_t* sw;
    const uint32_t* gcol;
    const uint32_t* gw;
};

// Exact SSSP from `source` by one warp, in its own memory: dist[k], one bit per node to be relaxed again and the list of
// a round's nodes.  A round lists the nodes of the set bits and clears them, then a lane relaxes one node's entries and
// gives improved nodes their bit back; the last round sets none.  (A lane per node of a 32-node word, without the list,
// left most lanes idle: 90 of 480 nodes are improved in a round of a mesh's quotient.)  No path sum can reach 2^32 - 1.
// Returns the largest distance at every lane; *err when the rounds exceed their limit.
__device__ __forceinline__ uint32_t warp_sssp(uint32_t k, const QuotientView& q, uint32_t source, uint32_t* dist,
                                              uint32_t* bits, uint16_t* list, uint32_t* err) {
    const uint32_t l = lane_id(), words = (k + 31) / 32;
    for (uint32_t v = l; v < k; v += 32) dist[v] = v == source ? 0u : kNone;
    for (uint32_t i = l; i < words; i += 32) bits[i] = i == source / 32 ? 1u << (source % 32) : 0u;
    __syncwarp();
    for (uint32_t round = 0;; ++round) {
        uint32_t m = 0;  // listed nodes; words <= 32: one word per lane
        {
            const uint32_t b = l < words ? bits[l] : 0u;
            const uint32_t c = (uint32_t)__popc(b), incl = warp_incl_scan(c);
            m = __shfl_sync(0xffffffffu, incl, 31);
            if (m == 0) break;
            uint32_t at = incl - c;
            for (uint32_t x = b; x; x &= x - 1) list[at++] = (uint16_t)(32 * l + (uint32_t)__ffs(x) - 1);
            if (l < words) bits[l] = 0;
        }
        __syncwarp();
        if (round > 4 * k + 64) {  // far above any real count: a guard, reported as an error
            if (l == 0) atomicExch(err, 1u);
            break;
        }
        for (uint32_t g = l; g < m; g += 32) {
            const uint32_t v = list[g], d = *(volatile uint32_t*)&dist[v];
            for (uint32_t j = q.off[v]; j < q.off[v + 1]; ++j) {
                const uint32_t u = q.scol ? q.scol[j] : __ldcg(&q.gcol[j]);
                const uint32_t nd = d + (q.scol ? q.sw[j] : __ldcg(&q.gw[j]));
                if (nd < *(volatile uint32_t*)&dist[u] && nd < atomicMin(&dist[u], nd))
                    atomicOr(&bits[u / 32], 1u << (u % 32));
            }
        }
        __syncwarp();
    }
    uint32_t ecc = 0;
    for (uint32_t v = l; v < k; v += 32) ecc = dist[v] != kNone ? max(ecc, dist[v]) : ecc;
    return __reduce_max_sync(0xffffffffu, ecc);
}
static_assert(kDenseCap <= 1024, "one word of a round's bits per lane");

constexpr size_t kBatchDyn = 208 * 1024;  // dynamic shared memory of a CTA
static_assert(kBatchDyn >= sizeof(GrowSmem) && kBatchDyn >= (size_t)kSmemFwK * kSmemFwK * 4 &&
                  kBatchDyn >= (size_t)kDenseCap * (8 * 4 + 8),
              "the growth loop, the shared Floyd-Warshall matrix and the all-source SSSP share the dynamic memory");

// Exact diameter of a symmetric quotient whose path sums cannot reach 2^32 - 1, by eccentricity bounds (bounds.cuh): a
// warp per source, the warps of all CTAs of the job at once.  ub, lb and src are global scratch, ub and lb preset.
template <class Barrier>
__device__ void group_bound_diameter(uint32_t k, uint32_t entries, const Workspace& ws, uint32_t* ub, uint32_t* lb,
                                     uint32_t* src, uint32_t* soff, BatchSmem& sm, uint32_t br, uint32_t nb,
                                     Barrier barrier) {
    // shared memory behind the offsets: the CSR if it leaves room for 16 warps, then dist, bits and list per warp
    const uint32_t words = (k + 31) / 32, per = k + words + (k + 1) / 2;  // words of one warp's SSSP
    uint32_t* mem = soff + k + 1;
    const size_t room = kBatchDyn / 4 - (k + 1);
    const size_t csr = entries + (entries + 1) / 2;
    QuotientView q{soff, nullptr, nullptr, ws.qcol, ws.qw};
    size_t left = room;
    if (csr + 16 * (size_t)per <= room) {
        uint32_t* sw = mem;
        uint16_t* scol = reinterpret_cast<uint16_t*>(mem + entries);
        for (uint32_t j = threadIdx.x; j < entries; j += BT) {
            sw[j] = __ldcg(&ws.qw[j]);
            scol[j] = (uint16_t)__ldcg(&ws.qcol[j]);
        }
        q.scol = scol;
        q.sw = sw;
        mem += csr;
        left -= csr;
    }
    const uint32_t warps = (uint32_t)min((size_t)BW, left / per);  // sources at once in this CTA
    const uint32_t w = threadIdx.x >> 5, l = lane_id();
    __syncthreads();
    uint32_t ns = min(k, warps * nb);
    for (bool first = true; ns > 0; first = false) {
        const uint32_t i = br * warps + w;
        if (w < warps && i < ns) {
            uint32_t* dist = mem + (size_t)w * per;
            const uint32_t source = first ? (uint32_t)((uint64_t)i * k / ns) : __ldcg(&src[i]);
            const uint32_t ecc = warp_sssp(k, q, source, dist, dist + k,
                                           reinterpret_cast<uint16_t*>(dist + k + words), &ws.fin->err);
            if (l == 0) atomicMax(&ws.fin->best, ecc);
            for (uint32_t v = l; v < k; v += 32) {
                const uint32_t d = dist[v];
                if (d == kNone) continue;
                atomicMin(&ub[v], (uint32_t)min((uint64_t)d + ecc, (uint64_t)(kNone - 1)));
                atomicMax(&lb[v], max(d, ecc - d));
            }
        }
        barrier();
        if (ns == k) break;  // every node was a source
        if (br == 0) {
            // (the SSSPs' memory is free between batches)
            uint32_t* sub = mem;
            uint32_t* slb = mem + k;
            for (uint32_t v = threadIdx.x; v < k; v += BT) {
                sub[v] = __ldcg(&ub[v]);
                slb[v] = __ldcg(&lb[v]);
            }
            __syncthreads();
            const uint32_t n = bound_select(k, warps * nb, __ldcg(&ws.fin->best), sub, slb, src, sm.word);
            if (threadIdx.x == 0) ws.fin->nsrc = __ldcg(&ws.fin->err) ? 0u : n;
        }
        barrier();
        ns = __ldcg(&ws.fin->nsrc);
    }
}

// The end of a job: singletons, relabel, the dense quotient and Phi(G_C); CTA 0 stores the result, with the counters of
// sm.grown.  Every phase is split over the job's CTAs (br of nb), a barrier between phases.
template <class Barrier>
__device__ void finish_job(const Job& job, const ArenaDesc& d, const uint64_t* __restrict__ off,
                           const uint2* __restrict__ adj, const uint32_t* __restrict__ row, const Workspace& ws,
                           BatchSmem& sm, uint32_t* dyn, JobOut* out, uint32_t status, uint32_t br, uint32_t nb,
                           Barrier barrier) {
    const unsigned tid = threadIdx.x, w = tid >> 5, l = lane_id();
    const uint32_t n = d.n, gt = br * BT + tid, gw = br * BW + w;  // thread and warp among the job's
    const uint32_t nt = nb * BT, nw = nb * BW;
    FinishCtl* fin = ws.fin;
    uint2* cd = reinterpret_cast<uint2*>(ws.fkey[0]);  // (cluster id, D) of every node
    const auto pack = [](uint2 x) { return (unsigned long long)x.y << 32 | x.x; };
    uint32_t k = 0, qe = 0;
    if (status == kJobOk) {
        dev_singletons(n, ws.center, ws.D, br, nb);
        barrier();
        // cluster id = rank of the center among the centers: counts of the CTAs' shares, then ranks
        const uint32_t share = (uint32_t)(((uint64_t)n + (uint64_t)nb * 4096 - 1) / ((uint64_t)nb * 4096) * 4096);
        const uint32_t lo = min(n, br * share), hi = (uint32_t)min((uint64_t)n, (uint64_t)lo + share);
        uint32_t first = 0;
        if (nb > 1) {
            const uint32_t c = block_centers(lo, hi, ws.center, nullptr, 0, sm);
            if (tid == 0) fin->part[br] = c;
            barrier();
            for (uint32_t i = 0; i < nb; ++i) {
                const uint32_t x = __ldcg(&fin->part[i]);
                first += i < br ? x : 0u;
                k += x;
            }
        }
        const uint32_t mine = block_centers(lo, hi, ws.center, ws.stamp, first, sm);  // stamp reused as rank
        if (nb == 1) k = mine;
        barrier();
        uint32_t* ub = ws.R;
        uint32_t* lb = ws.next;
        uint32_t rmax = 0;
        for (uint64_t base = gt; base < n; base += (uint64_t)nt * kFinishU) {
            uint32_t c[kFinishU], dd[kFinishU];
#pragma unroll
            for (uint32_t u = 0; u < kFinishU; ++u) {
                const uint64_t v = base + (uint64_t)u * nt;
                c[u] = v < n ? __ldcg(&ws.center[v]) : 0u;
                dd[u] = v < n ? __ldcg(&ws.D[v]) : 0u;
            }
#pragma unroll
            for (uint32_t u = 0; u < kFinishU; ++u) c[u] = __ldcg(&ws.stamp[c[u]]);
#pragma unroll
            for (uint32_t u = 0; u < kFinishU; ++u) {
                const uint64_t v = base + (uint64_t)u * nt;
                if (v < n) cd[v] = make_uint2(c[u], dd[u]);
                rmax = max(rmax, dd[u]);
            }
        }
        rmax = __reduce_max_sync(0xffffffffu, rmax);
        if (l == 0 && rmax) atomicMax(&fin->rmax, rmax);
        if (k > kDenseCap) {
            status = kJobNeedsPlain;
        } else {
            // weighted quotient graph, deduplicated densely: each undirected edge once, into both of its entries
            uint32_t* M = ws.M;
            for (uint32_t a = gw; a < k; a += nw)
                for (uint32_t b = l; b < k; b += 32) M[a * k + b] = a == b ? 0u : kNone;
            for (uint32_t v = gt; v < k; v += nt) {
                ub[v] = kNone;
                lb[v] = 0;
            }
            barrier();
            bool ovf = false;
            for (uint64_t base = gt; base < d.nnz; base += (uint64_t)nt * kFinishU) {
                uint32_t r[kFinishU];
                uint2 e[kFinishU];
#pragma unroll
                for (uint32_t u = 0; u < kFinishU; ++u) {
                    const uint64_t i = base + (uint64_t)u * nt;
                    r[u] = i < d.nnz ? row[i] : 0u;
                    e[u] = i < d.nnz ? adj[i] : make_uint2(0u, 0u);
                }
                unsigned long long pu[kFinishU], pv[kFinishU];
#pragma unroll
                for (uint32_t u = 0; u < kFinishU; ++u) {
                    const bool take = r[u] < e[u].x;
                    pu[u] = take ? pack(__ldcg(&cd[r[u]])) : 0ull;
                    pv[u] = take ? pack(__ldcg(&cd[e[u].x])) : 0ull;
                }
                uint32_t at[kFinishU], cur[kFinishU], s32[kFinishU];
#pragma unroll
                for (uint32_t u = 0; u < kFinishU; ++u) {
                    const uint32_t a = (uint32_t)pu[u], b = (uint32_t)pv[u];
                    uint64_t sw = (pu[u] >> 32) + e[u].y + (pv[u] >> 32);
                    const bool take = r[u] < e[u].x && a != b;
                    if (take && sw >= 0xFFFFFFFFull) {
                        ovf = true;
                        sw = 0xFFFFFFFEull;
                    }
                    s32[u] = (uint32_t)sw;
                    at[u] = a * k + b;
                    cur[u] = take ? __ldcg(&M[at[u]]) : 0u;
                }
#pragma unroll
                for (uint32_t u = 0; u < kFinishU; ++u)
                    if (s32[u] < cur[u]) {
                        atomicMin(&M[at[u]], s32[u]);
                        atomicMin(&M[(uint32_t)pv[u] * k + (uint32_t)pu[u]], s32[u]);
                    }
            }
            if (__any_sync(0xffffffffu, ovf) && l == 0) atomicExch(&fin->err, 2u);
            barrier();
            // entries per row, and the guard of the bounds: sum over rows of the heaviest entry
            unsigned long long entries = 0, wsum = 0;
            uint32_t wmax = 0;
            for (uint32_t a = gw; a < k; a += nw) {
                uint32_t c = 0, m = 0;
                for (uint32_t b0 = 0; b0 < k; b0 += 32 * kFinishU) {
                    uint32_t x[kFinishU];
#pragma unroll
                    for (uint32_t u = 0; u < kFinishU; ++u) {
                        const uint32_t b = b0 + 32 * u + l;
                        x[u] = b < k && b != a ? __ldcg(&M[a * k + b]) : kNone;
                    }
#pragma unroll
                    for (uint32_t u = 0; u < kFinishU; ++u) {
                        c += x[u] != kNone ? 1u : 0u;
                        m = x[u] != kNone ? max(m, x[u]) : m;
                    }
                }
                c = __reduce_add_sync(0xffffffffu, c);
                m = __reduce_max_sync(0xffffffffu, m);
                if (l == 0) ws.qoff[a] = c;
                entries += c;
                wsum += m;
                wmax = max(wmax, m);
            }
            if (l == 0 && entries) {
                atomicAdd(&fin->entries, entries);
                atomicAdd(&fin->wsum, wsum);
                atomicMax(&fin->wmax, wmax);
            }
            barrier();
            qe = (uint32_t)__ldcg(&fin->entries);
            bool ovf2 = false;
            // No path sum of an SSSP can reach 2^32 - 1 when the sum of the rows' heaviest entries and one more entry do
            // not; Floyd-Warshall also adds two paths.  Up to fw_k nodes it takes dense quotients, and those whose two
            // paths might overflow, so that OVERFLOW is reported as it always was (sparse ones are faster by bounds).
            const unsigned long long longest = __ldcg(&fin->wsum), heaviest = __ldcg(&fin->wmax);
            const bool dense = (uint64_t)qe * 8 >= (uint64_t)k * k || 2 * longest + heaviest >= 0xFFFFFFFFull;
            if (k > 1 && k <= min(job.fw_k, kSmemFwK) && dense) {
                if (br == 0) {
                    const uint32_t best = block_floyd_warshall(k, M, dyn, ovf2);
                    const uint32_t m = __reduce_max_sync(0xffffffffu, best);
                    if (l == 0) atomicMax(&fin->best, m);
                }
            } else if (k > 1) {
                // quotient CSR from M: row starts by a block scan of the counts (k <= 1,024), in every CTA; a warp per
                // row, ballot compaction keeps the columns sorted
                uint32_t* soff = dyn;
                const uint32_t c = tid < k ? __ldcg(&ws.qoff[tid]) : 0u;
                const uint32_t incl = warp_incl_scan(c);
                if (l == 31) sm.woff[w] = incl;
                __syncthreads();
                uint32_t before = 0;
                for (uint32_t i = 0; i < w; ++i) before += sm.woff[i];
                if (tid < k) soff[tid] = before + incl - c;
                if (tid == 0) soff[k] = qe;
                __syncthreads();
                for (uint32_t a = gw; a < k; a += nw) {
                    uint32_t pos = soff[a];
                    for (uint32_t b0 = 0; b0 < k; b0 += 32 * kFinishU) {
                        uint32_t x[kFinishU];
#pragma unroll
                        for (uint32_t u = 0; u < kFinishU; ++u) {
                            const uint32_t b = b0 + 32 * u + l;
                            x[u] = b < k && b != a ? __ldcg(&M[a * k + b]) : kNone;
                        }
#pragma unroll
                        for (uint32_t u = 0; u < kFinishU; ++u) {
                            const unsigned bal = __ballot_sync(0xffffffffu, x[u] != kNone);
                            if (x[u] != kNone) {
                                const uint32_t p = pos + (uint32_t)__popc(bal & lanemask_lt());
                                ws.qcol[p] = b0 + 32 * u + l;
                                ws.qw[p] = x[u];
                            }
                            pos += (uint32_t)__popc(bal);
                        }
                    }
                }
                barrier();
                if (longest + heaviest < 0xFFFFFFFFull) {
                    group_bound_diameter(k, qe, ws, ub, lb, ws.fbase[0], soff, sm, br, nb, barrier);
                } else if (br == 0) {
                    for (uint32_t i = tid; i <= k; i += BT) ws.qoff[i] = soff[i];
                    __syncthreads();
                    const uint32_t best = block_all_sources(k, ws, dyn, ovf2);
                    const uint32_t m = __reduce_max_sync(0xffffffffu, best);
                    if (l == 0) atomicMax(&fin->best, m);
                }
            }
            if (__any_sync(0xffffffffu, ovf2) && l == 0) atomicExch(&fin->err, 2u);
            barrier();
            if (const uint32_t err = __ldcg(&fin->err)) status = err == 1u ? kJobDiverged : kJobOverflow;
        }
    }
    if (br == 0 && tid == 0) {
        const GrowState& g = sm.grown;
        cldiam_result res;
        memset(&res, 0, sizeof res);
        res.stages = g.stages;
        res.steps = g.steps;
        res.doublings = g.doublings;
        res.delta_end = g.delta;
        res.guard_exits = g.guard_exits;
        res.node_updates = g.node_updates;
        res.edges_scanned = g.edges_scanned;
        res.centers_drawn = g.centers_drawn;
        res.k = k;
        res.quotient_edges = qe;
        res.radius = __ldcg(&fin->rmax);
        res.phi_gc = __ldcg(&fin->best);
        res.phi_approx = res.phi_gc + 2ull * res.radius;
        out->r = res;
        out->status = status;
    }
}

// One job: CLUSTER + quotient + Phi(G_C) of one arena graph by CTA br of nb; CTA 0 stores the result.
template <class Barrier>
__device__ void run_job(const Job& job, const ArenaDesc& d, const uint64_t* __restrict__ arena_off,
                        const uint2* __restrict__ arena_adj, const uint32_t* __restrict__ arena_row,
                        const Workspace& ws, BatchSmem& sm, uint32_t* dyn, JobOut* out, uint32_t br, uint32_t nb,
                        Barrier barrier) {
    const unsigned tid = threadIdx.x;
    const uint32_t n = d.n;
    const uint64_t* off = arena_off + d.off_base;
    const uint2* adj = arena_adj + d.adj_base;
    const uint32_t* row = arena_row + d.adj_base;
    for (uint32_t v = br * BT + tid; v < n; v += nb * BT) {
        ws.center[v] = kNone;
        ws.D[v] = 0;
        ws.R[v] = 0;
        ws.stamp[v] = 0;
        ws.key[v] = kInfKey;
    }
    if (br == 0 && tid == 0) {
        memset(ws.ring, 0, 3 * sizeof(Counters));
        FinishCtl* fin = ws.fin;
        fin->entries = fin->wsum = 0;
        fin->wmax = fin->rmax = fin->best = fin->nsrc = fin->err = 0;
    }
    if (tid == 0) {
        GrowArgs& a = sm.args;
        a.off = off;
        a.adj = adj;
        a.key = ws.key;
        a.keyS = nullptr;
        for (int i = 0; i < 2; ++i) {
            a.fkey[i] = ws.fkey[i];
            a.fbase[i] = ws.fbase[i];
            a.fpre[i] = ws.fpre[i];
            a.cfirst[i] = ws.cfirst[i];
        }
        a.center = ws.center;
        a.D = ws.D;
        a.R = ws.R;
        a.stamp = ws.stamp;
        a.next = ws.next;
        a.ring = ws.ring;
        a.out = nullptr;
        a.row = row;
        a.tau = job.tau;
        a.L = job.L;
        a.seed = job.seed;
        a.nnz = d.nnz;
        a.n = n;
        a.step_cap = job.step_cap;
        a.max_entries = a.max_epochs = 0xFFFFFFFFu;
        a.cumulative = job.cumulative != 0;
        a.pull_ok = d.nnz < 0x80000000ull;
        a.stages = true;
        a.connected = d.connected != 0;
    }
    GrowSmem& gsm = *reinterpret_cast<GrowSmem*>(dyn);
    GrowState& g = gsm.g;
    if (tid == 0) {
        memset(&g, 0, sizeof g);
        g.U = n;
        g.phase = kPhaseStage;
        g.stage = 1;
        g.delta = job.delta0;
    }
    barrier();
    grow_run(sm.args, gsm, br, nb, barrier);
    uint32_t status = kJobOk;
    if (g.phase != kPhaseDone)
        status = g.stage > kMaxStages || g.unfrozen != g.U ? kJobDiverged : kJobOverflow;
    if (tid == 0) sm.grown = g;
    __syncthreads();  // the state has been read: the end of the job uses its shared memory
    finish_job(job, d, off, adj, row, ws, sm, dyn, out, status, br, nb, barrier);
}

// The jobs of a queue (largest first), one after another, by one CTA each (GROUP: by a thread-block cluster each).
template <bool GROUP>
__global__ void __launch_bounds__(BT, kBatchCtasPerSm)
    k_batch(const ArenaDesc* __restrict__ descs, const Job* __restrict__ jobs, uint32_t count,
            const uint64_t* __restrict__ arena_off, const uint2* __restrict__ arena_adj,
            const uint32_t* __restrict__ arena_row, Workspace* __restrict__ wss, uint32_t* __restrict__ queue,
            JobOut* __restrict__ outs) {
    extern __shared__ __align__(16) uint32_t dyn[];
    __shared__ BatchSmem sm;
    uint32_t br = 0, nb = 1;
    if constexpr (GROUP) {
        asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(br));
        asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(nb));
    }
    const auto barrier = [] {
        if constexpr (GROUP) cluster_barrier();
        else __syncthreads();
    };
    if (threadIdx.x == 0) sm.ws = wss[blockIdx.x / nb];
    __syncthreads();
    for (;;) {
        uint32_t j;
        if constexpr (GROUP) {
            if (br == 0 && threadIdx.x == 0) sm.ws.fin->job = atomicAdd(queue, 1u);
            barrier();
            j = __ldcg(&sm.ws.fin->job);
        } else {
            if (threadIdx.x == 0) sm.word = atomicAdd(queue, 1u);
            __syncthreads();
            j = sm.word;
            __syncthreads();
        }
        if (j >= count) break;
        if (threadIdx.x == 0) sm.job = jobs[j];
        __syncthreads();
        const uint64_t t0 = global_ns();
        run_job(sm.job, descs[sm.job.graph], arena_off, arena_adj, arena_row, sm.ws, sm, dyn, &outs[sm.job.out], br, nb,
                barrier);
        barrier();  // (every CTA is done with the job and its workspace)
        if (br == 0 && threadIdx.x == 0) {
            outs[sm.job.out].t_start = t0;
            outs[sm.job.out].t_end = global_ns();
        }
    }
}

// ---------------------------------------------------------------------------- serving
// Host-mapped control block of the serving kernel.
struct ServeCtl {
    uint32_t tail;   // requests published by the host (store-release)
    uint32_t stop;   // host asks the CTAs to leave
    uint32_t idle;   // a CTA left after the idle limit with no request
    uint32_t pad;
};

__device__ __forceinline__ uint32_t ld_acquire_sys(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.acquire.sys.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release_sys(uint32_t* p, uint32_t v) {
    asm volatile("st.release.sys.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Continuous batching: every CTA takes the next published request as soon as
// it finishes its previous one, so requests that arrive while others run join
// immediately.  Waiting for work is bounded by idle_cycles; the host
// relaunches the kernel when a request arrives after the CTAs left.
__global__ void __launch_bounds__(BT, kBatchCtasPerSm)
    k_serve(const ArenaDesc* __restrict__ descs, const uint64_t* __restrict__ arena_off,
            const uint2* __restrict__ arena_adj, const uint32_t* __restrict__ arena_row,
            Workspace* __restrict__ wss, const Job* ring, ServeCtl* ctl, uint32_t* head, JobOut* outs,
            uint32_t* done, long long idle_cycles) {
    extern __shared__ __align__(16) uint32_t dyn[];
    __shared__ BatchSmem sm;
    if (threadIdx.x == 0) sm.ws = wss[blockIdx.x];
    for (;;) {
        if (threadIdx.x == 0) {
            uint32_t claimed = kNone;
            const long long t0 = clock64();
            for (;;) {
                const uint32_t t = ld_acquire_sys(&ctl->tail);
                const uint32_t h = atomicAdd(head, 0u);
                if (h < t) {
                    if (atomicCAS(head, h, h + 1) == h) {
                        claimed = h;
                        break;
                    }
                    continue;
                }
                if (ld_acquire_sys(&ctl->stop)) break;
                if (clock64() - t0 > idle_cycles) {
                    atomicExch(&ctl->idle, 1u);
                    break;
                }
                __nanosleep(2000);
            }
            sm.word = claimed;
            if (claimed != kNone) {
                const volatile Job* vj = ring + claimed;
                sm.job.tau = vj->tau;
                sm.job.L = vj->L;
                sm.job.seed = vj->seed;
                sm.job.graph = vj->graph;
                sm.job.delta0 = vj->delta0;
                sm.job.out = vj->out;
                sm.job.step_cap = vj->step_cap;
                sm.job.cumulative = vj->cumulative;
                sm.job.fw_k = vj->fw_k;
            }
        }
        __syncthreads();
        const uint32_t slot = sm.word;
        if (slot == kNone) break;
        __syncthreads();
        run_job(sm.job, descs[sm.job.graph], arena_off, arena_adj, arena_row, sm.ws, sm, dyn, &outs[sm.job.out], 0u, 1u,
                [] { __syncthreads(); });
        if (threadIdx.x == 0) {
            __threadfence_system();
            st_release_sys(&done[sm.job.out], 1u);
        }
        __syncthreads();
    }
}

}  // namespace

}  // namespace cld

// ---------------------------------------------------------------------------- arena
struct cldiam_arena {
    int device = 0;
    cudaStream_t stream = nullptr;
    uint64_t budget = 0;
    std::vector<cld::ArenaDesc> graphs;
    std::vector<uint64_t> wsum_upper;
    std::vector<uint32_t> wmin, max_deg;
    uint64_t* off = nullptr;
    uint2* adj = nullptr;
    uint32_t* row = nullptr;
    uint64_t off_cap = 0, adj_cap = 0, off_used = 0, adj_used = 0;
    void* ws = nullptr;  // cached per-CTA workspaces
    size_t ws_bytes = 0;
    void* gws = nullptr;  // cached workspaces of the groups that share large jobs
    size_t gws_bytes = 0;
    cudaStream_t aux = nullptr;  // the one-CTA jobs run here beside the groups' on `stream`
    std::vector<double> last_start, last_end;  // per-job device times of the last batch (seconds)
};

namespace cld {

// the workspaces are a cache for the next batch: given back where their bytes stand in the way of a budget
static void release_workspaces(cldiam_arena* a) {
    dfree(a->ws, a->stream);
    dfree(a->gws, a->stream);
    a->ws = a->gws = nullptr;
    a->ws_bytes = a->gws_bytes = 0;
}

static uint64_t arena_bytes(const cldiam_arena* a) { return a->off_cap * 8 + a->adj_cap * 12 + a->ws_bytes + a->gws_bytes; }

// grow a device array to hold `need` elements (doubling), keeping the first `used`
template <class T>
static cldiam_status grow(T** p, uint64_t* cap, uint64_t used, uint64_t need, cudaStream_t s) {
    if (need <= *cap) return CLDIAM_OK;
    uint64_t nc = std::max<uint64_t>(need, *cap * 2 + 1024);
    T* q = nullptr;
    CLD_TRY(dmalloc(reinterpret_cast<void**>(&q), nc * sizeof(T), s));
    if (used) CLD_CUDA(cudaMemcpyAsync(q, *p, used * sizeof(T), cudaMemcpyDeviceToDevice, s));
    dfree(*p, s);
    *p = q;
    *cap = nc;
    return CLDIAM_OK;
}

cldiam_status arena_create(uint64_t budget, cudaStream_t s, cldiam_arena** out) {
    if (!out) return fail(CLDIAM_ERR_INVALID_ARG, "NULL out");
    cldiam_arena* a = new cldiam_arena();
    cudaGetDevice(&a->device);
    a->stream = s;
    a->budget = budget;
    *out = a;
    return CLDIAM_OK;
}

void arena_free(cldiam_arena* a) {
    if (!a) return;
    dfree(a->off, a->stream);
    dfree(a->adj, a->stream);
    dfree(a->row, a->stream);
    release_workspaces(a);
    cudaStreamSynchronize(a->stream);
    if (a->aux) cudaStreamDestroy(a->aux);
    delete a;
}

cldiam_status arena_add(cldiam_arena* a, const uint32_t* src, const uint32_t* dst, const uint32_t* w, uint64_t m,
                        uint32_t n, uint32_t flags, uint32_t* id) {
    if (!a || !id) return fail(CLDIAM_ERR_INVALID_ARG, "NULL arena or id");
    cldiam_graph* g = nullptr;
    CLD_TRY(build_csr(src, dst, w, m, n, flags, a->stream, &g));
    struct Free {
        cldiam_graph* g;
        ~Free() { free_graph(g); }
    } fg{g};
    const uint64_t need_off = a->off_used + g->n + 1, need_adj = a->adj_used + g->nnz;
    const uint64_t extra = (need_off > a->off_cap ? (need_off - a->off_cap) * 8 : 0) +
                           (need_adj > a->adj_cap ? (need_adj - a->adj_cap) * 12 : 0);
    if (a->budget && arena_bytes(a) + extra > a->budget) release_workspaces(a);
    if (a->budget && arena_bytes(a) + extra > a->budget)
        return fail(CLDIAM_ERR_OOM, "graph does not fit the arena's device memory budget");
    CLD_TRY(grow(&a->off, &a->off_cap, a->off_used, need_off, a->stream));
    {
        uint64_t cap = a->adj_cap;
        CLD_TRY(grow(&a->adj, &cap, a->adj_used, need_adj, a->stream));
        uint64_t cap2 = a->adj_cap;
        CLD_TRY(grow(&a->row, &cap2, a->adj_used, need_adj, a->stream));
        a->adj_cap = std::max(cap, cap2);
    }
    CLD_CUDA(cudaMemcpyAsync(a->off + a->off_used, g->off, (g->n + 1) * 8, cudaMemcpyDeviceToDevice, a->stream));
    if (g->nnz) {
        CLD_CUDA(cudaMemcpyAsync(a->adj + a->adj_used, g->adj, g->nnz * 8, cudaMemcpyDeviceToDevice, a->stream));
        if (g->row) {
            CLD_CUDA(cudaMemcpyAsync(a->row + a->adj_used, g->row, g->nnz * 4, cudaMemcpyDeviceToDevice, a->stream));
        } else {
            CLD_TRY(fill_rows(g->off, g->n, a->row + a->adj_used, a->stream));
        }
    }
    ArenaDesc dsc{};
    dsc.off_base = a->off_used;
    dsc.adj_base = a->adj_used;
    dsc.nnz = g->nnz;
    dsc.n = g->n;
    dsc.connected = g->connected ? 1u : 0u;
    a->graphs.push_back(dsc);
    a->wsum_upper.push_back(g->wsum_upper);
    a->wmin.push_back(g->wmin);
    a->max_deg.push_back(g->max_deg);
    a->off_used = need_off;
    a->adj_used = need_adj;
    *id = (uint32_t)(a->graphs.size() - 1);
    CLD_CUDA(cudaStreamSynchronize(a->stream));
    return CLDIAM_OK;
}

// a non-owning graph handle over one arena graph (for the one-graph path)
static void arena_view(const cldiam_arena* a, uint32_t id, cldiam_graph* g) {
    const ArenaDesc& d = a->graphs[id];
    g->device = a->device;
    g->stream = a->stream;
    g->n = d.n;
    g->nnz = d.nnz;
    g->off = a->off + d.off_base;
    g->adj = a->adj + d.adj_base;
    g->row = a->row + d.adj_base;
    g->orig = nullptr;
    g->wsum_upper = a->wsum_upper[id];
    g->wmin = a->wmin[id];
    g->max_deg = a->max_deg[id];
    g->connected = d.connected != 0;
    g->borrowed = true;
}

cldiam_status arena_graph(cldiam_arena* a, uint32_t id, cldiam_graph** out) {
    if (!a || !out || id >= a->graphs.size()) return fail(CLDIAM_ERR_INVALID_ARG, "bad arena or graph id");
    cldiam_graph* g = new cldiam_graph();
    arena_view(a, id, g);
    CLD_TRY(g->host.alloc(256));
    *out = g;
    return CLDIAM_OK;
}

uint32_t arena_count(const cldiam_arena* a) { return (uint32_t)a->graphs.size(); }
cudaStream_t arena_stream(const cldiam_arena* a) { return a->stream; }
cldiam_status arena_job_times(const cldiam_arena* a, uint32_t count, double* start_s, double* end_s) {
    if (!a || (count && (!start_s || !end_s))) return fail(CLDIAM_ERR_INVALID_ARG, "NULL argument");
    if (count > a->last_start.size()) return fail(CLDIAM_ERR_INVALID_ARG, "count exceeds the last batch");
    for (uint32_t i = 0; i < count; ++i) {
        start_s[i] = a->last_start[i];
        end_s[i] = a->last_end[i];
    }
    return CLDIAM_OK;
}
uint64_t arena_entries(const cldiam_arena* a, const uint32_t* ids, uint32_t count) {
    uint64_t e = 0;
    for (uint32_t i = 0; i < count; ++i)
        if (ids[i] < a->graphs.size()) e += a->graphs[ids[i]].nnz;
    return e;
}
uint64_t arena_device_bytes(const cldiam_arena* a) { return arena_bytes(a); }

// Workspaces for graphs of up to nmax nodes and zmax entries, one per CTA (or group of CTAs), carved from one (cached)
// device buffer.
static cldiam_status make_workspaces(uint32_t nmax, uint64_t zmax, int ctas, cudaStream_t s, void** buf,
                                     size_t* buf_bytes, std::vector<Workspace>* out) {
    auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
    const size_t n8 = al((size_t)nmax * 8), n4 = al((size_t)nmax * 4), f8 = al((size_t)nmax * 16),
                 f4 = al((size_t)nmax * 8), mm = al((size_t)kDenseCap * kDenseCap * 4),
                 cf = al((size_t)(2 * zmax / QC + 2) * 4),  // a frontier has at most 2 x nnz entries (push + pull)
                 qo = al(((size_t)kDenseCap + 1) * 4), ctrb = al(3 * sizeof(Counters)), finb = al(sizeof(FinishCtl));
    const size_t slice = n8 + 2 * f8 + 5 * n4 + 4 * f4 + 2 * cf + mm + qo + 2 * mm + ctrb + finb;
    const size_t need = slice * ctas;
    if (need > *buf_bytes) {
        dfree(*buf, s);
        *buf = nullptr;
        *buf_bytes = 0;
        CLD_TRY(dmalloc(buf, need, s));
        *buf_bytes = need;
    }
    out->assign(ctas, Workspace{});
    for (int b = 0; b < ctas; ++b) {
        char* p = static_cast<char*>(*buf) + (size_t)b * slice;
        Workspace& w = (*out)[b];
        w.key = reinterpret_cast<unsigned long long*>(p); p += n8;
        w.fkey[0] = reinterpret_cast<unsigned long long*>(p); p += f8;
        w.fkey[1] = reinterpret_cast<unsigned long long*>(p); p += f8;
        w.center = reinterpret_cast<uint32_t*>(p); p += n4;
        w.D = reinterpret_cast<uint32_t*>(p); p += n4;
        w.R = reinterpret_cast<uint32_t*>(p); p += n4;
        w.stamp = reinterpret_cast<uint32_t*>(p); p += n4;
        w.next = reinterpret_cast<uint32_t*>(p); p += n4;
        w.fbase[0] = reinterpret_cast<uint32_t*>(p); p += f4;
        w.fbase[1] = reinterpret_cast<uint32_t*>(p); p += f4;
        w.fpre[0] = reinterpret_cast<uint32_t*>(p); p += f4;
        w.fpre[1] = reinterpret_cast<uint32_t*>(p); p += f4;
        w.cfirst[0] = reinterpret_cast<uint32_t*>(p); p += cf;
        w.cfirst[1] = reinterpret_cast<uint32_t*>(p); p += cf;
        w.M = reinterpret_cast<uint32_t*>(p); p += mm;
        w.qoff = reinterpret_cast<uint32_t*>(p); p += qo;
        w.qcol = reinterpret_cast<uint32_t*>(p); p += mm;
        w.qw = reinterpret_cast<uint32_t*>(p); p += mm;
        w.ring = reinterpret_cast<Counters*>(p); p += ctrb;
        w.fin = reinterpret_cast<FinishCtl*>(p);
    }
    return CLDIAM_OK;
}

struct CudaEvent {
    cudaEvent_t e = nullptr;
    cldiam_status create() {
        CLD_CUDA(cudaEventCreate(&e));
        return CLDIAM_OK;
    }
    ~CudaEvent() {
        if (e) cudaEventDestroy(e);
    }
};

static size_t batch_dyn_smem() { return kBatchDyn; }

template <class Kern>
static cldiam_status set_dyn_smem(Kern k, std::atomic<bool>* done_flags) {
    int dev = 0;
    CLD_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64 || !done_flags[dev]) {
        CLD_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)batch_dyn_smem()));
        if (kBatchCtasPerSm > 1)  // room for several CTAs' shared memory on one SM
            CLD_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout,
                                          (int)cudaSharedmemCarveoutMaxShared));
        if (dev >= 0 && dev < 64) done_flags[dev] = true;
    }
    return CLDIAM_OK;
}

// CTAs of a persistent many-graph kernel resident on one SM: kBatchCtasPerSm when they fit, else what does
template <class Kern>
static cldiam_status resident_per_sm(Kern k, std::atomic<bool>* done_flags, int* out) {
    CLD_TRY(set_dyn_smem(k, done_flags));
    int nb = 0;
    CLD_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, BT, batch_dyn_smem()));
    *out = std::max(1, std::min(nb, kBatchCtasPerSm));
    return CLDIAM_OK;
}

// launch configuration of `groups` job groups, one CTA per SM each of kJobCtas in a thread-block cluster
static void job_group_config(cudaLaunchConfig_t* cfg, cudaLaunchAttribute* at, int groups) {
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = kJobCtas;
    at->val.clusterDim.y = at->val.clusterDim.z = 1;
    cfg->gridDim = dim3((unsigned)groups * kJobCtas);
    cfg->blockDim = dim3(BT);
    cfg->dynamicSmemBytes = batch_dyn_smem();
    cfg->attrs = at;
    cfg->numAttrs = 1;
}
// job groups that this device holds at once (0: none); asked once per device, concurrent first calls store the same
static cldiam_status max_job_groups(int dev, int* out) {
    static std::atomic<int> cached[64];  // 0 = not asked yet, else number + 1
    *out = 0;
    if (dev < 0 || dev >= 64) return CLDIAM_OK;
    if (cached[dev].load() == 0) {
        CLD_CUDA(cudaFuncSetAttribute(k_batch<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)batch_dyn_smem()));
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute at{};
        job_group_config(&cfg, &at, 1);
        int m = 0;
        if (cudaOccupancyMaxActiveClusters(&m, k_batch<true>, &cfg) != cudaSuccess) {
            cudaGetLastError();
            m = 0;
        }
        cached[dev].store(m + 1);
    }
    *out = cached[dev].load() - 1;
    return CLDIAM_OK;
}

cldiam_status batch_run(cldiam_arena* a, const uint32_t* ids, const double* tau, const uint64_t* seed, uint32_t count,
                        const cldiam_opts* o, cldiam_result* out, cldiam_status* status) {
    if (!a || (count && (!ids || !tau || !seed || !out))) return fail(CLDIAM_ERR_INVALID_ARG, "NULL argument");
    if (count == 0) return CLDIAM_OK;
    cldiam_opts opts{};
    if (o) opts = *o;
    if (opts.contract_mode != CLDIAM_CONTRACT_RESET && opts.contract_mode != CLDIAM_CONTRACT_CUMULATIVE)
        return fail(CLDIAM_ERR_INVALID_ARG, "unknown contract_mode");
    if (opts.reserved[0] || opts.reserved[1]) return fail(CLDIAM_ERR_INVALID_ARG, "reserved options must be 0");
    const cudaStream_t s = a->stream;
    const uint32_t fw_k = tuning_for_batch(arena_entries(a, ids, count)).batch_fw_k;
    std::vector<Job> jobs(count);
    for (uint32_t i = 0; i < count; ++i) {
        if (ids[i] >= a->graphs.size()) return fail(CLDIAM_ERR_INVALID_ARG, "graph id out of range");
        if (!(tau[i] > 0.0) || !std::isfinite(tau[i])) return fail(CLDIAM_ERR_INVALID_ARG, "tau must be positive");
        cldiam_graph view;
        arena_view(a, ids[i], &view);
        uint32_t d0 = 0;
        CLD_TRY(delta0(&view, opts.delta0_mode, opts.delta0, &d0));
        jobs[i].tau = tau[i];
        jobs[i].L = std::log2((double)view.n);
        jobs[i].seed = seed[i];
        jobs[i].graph = ids[i];
        jobs[i].delta0 = d0;
        jobs[i].out = i;
        jobs[i].step_cap = opts.step_cap;
        jobs[i].cumulative = opts.contract_mode == CLDIAM_CONTRACT_CUMULATIVE ? 1u : 0u;
        jobs[i].fw_k = fw_k;
    }
    // longest jobs first: the work queue then balances the tail
    const auto units = [&](const Job& j) { return (double)(a->graphs[j.graph].nnz + a->graphs[j.graph].n); };
    const auto sparse = [&](const Job& j) { return a->graphs[j.graph].nnz < 8ull * a->graphs[j.graph].n; };
    std::stable_sort(jobs.begin(), jobs.end(), [&](const Job& x, const Job& y) {
        return job_cta_s(units(x), sparse(x)) > job_cta_s(units(y), sparse(y));
    });
    static std::atomic<bool> attr[64];
    int cps = 1;
    CLD_TRY(resident_per_sm(k_batch<false>, attr, &cps));
    const int nsm = num_sms() * cps;  // CTAs of the launch
    // The launch ends with its largest graph on one CTA, or with the even split of all work over the CTAs, whichever is
    // later.  So the largest graphs may run elsewhere (batch_split = 2; 1 keeps every graph on one CTA): on groups of
    // kJobCtas CTAs beside the others, or, larger still, first on the one-graph path, each with the whole device at a
    // fixed cost per graph.  Both are prefixes of the jobs, chosen to minimise the estimated end.  Work = adjacency
    // entries + nodes.
    const uint32_t split = tuning_for_batch(arena_entries(a, ids, count)).batch_split;
    int dev = 0;
    CLD_CUDA(cudaGetDevice(&dev));
    int max_groups = 0;
    if (split == 2 && !serving_kernel_alive(dev)) CLD_TRY(max_job_groups(dev, &max_groups));
    std::vector<double> one(count + 1, 0.0), grp(count + 1, 0.0);          // seconds of job j on one CTA, on a group
    std::vector<double> one_from(count + 1, 0.0), grp_from(count + 1, 0.0);  // their sums over jobs[j ..)
    for (uint32_t j = count; j-- > 0;) {
        one[j] = job_cta_s(units(jobs[j]), sparse(jobs[j]));
        grp[j] = job_group_s(units(jobs[j]), sparse(jobs[j]));
        one_from[j] = one_from[j + 1] + one[j];
        grp_from[j] = grp_from[j + 1] + grp[j];
    }
    uint32_t nbig = 0, ngrp = 0;  // jobs[0 .. nbig): one-graph path; jobs[nbig .. nbig + ngrp): groups
    if (split == 2) {
        const auto big = [&](uint32_t j) { return a->graphs[jobs[j].graph].nnz >= kSplitMinEntries; };
        // end of the launch when jobs[k .. k + g) run on groups and jobs[k + g ..) on one CTA each
        const auto launch_s = [&](uint32_t k, uint32_t g) {
            const double group_s = grp_from[k] - grp_from[k + g];
            const double even = (group_s * kJobCtas + one_from[k + g]) / nsm;
            const double groups = g ? std::max(grp[k], group_s / max_groups) : 0.0;
            return std::max(std::max(even, groups), one[k + g]);
        };
        double plain_s = 0.0, best = -1.0;
        for (uint32_t k = 0; k <= count; ++k) {
            if (k > 0) plain_s += job_plain_s(units(jobs[k - 1]), sparse(jobs[k - 1]));
            if (best >= 0.0 && plain_s >= best) break;
            for (uint32_t g = 0; k + g <= count; ++g) {
                if (g > 0 && (max_groups == 0 || !big(k + g - 1))) break;
                const double t = plain_s + launch_s(k, g);
                if (best < 0.0 || t < best) {
                    best = t;
                    nbig = k;
                    ngrp = g;
                }
            }
            if (k < count && !big(k)) break;
        }
    }
    a->last_start.assign(count, 0.0);
    a->last_end.assign(count, 0.0);
    std::vector<JobOut> ho(count);
    for (auto& h : ho) h.status = kJobOk;
    double big_s = 0.0;  // device time of the one-graph runs, the offset of the launch's job times
    std::vector<cldiam_status> big_st(count, CLDIAM_OK);
    if (nbig > 0) {
        CudaEvent e0, e1;
        CLD_TRY(e0.create());
        CLD_TRY(e1.create());
        for (uint32_t j = 0; j < nbig; ++j) {
            const uint32_t i = jobs[j].out;
            cldiam_graph view;
            arena_view(a, ids[i], &view);
            CLD_TRY(view.host.alloc(256));
            CLD_CUDA(cudaEventRecord(e0.e, s));
            cldiam_clustering* c = nullptr;
            cldiam_quotient* q = nullptr;
            cldiam_status st = cluster(&view, tau[i], seed[i], &opts, &c);
            if (st == CLDIAM_OK) st = quotient(c, &q);
            if (st == CLDIAM_OK) st = cldiam_estimate(q, &ho[i].r);
            free_quotient(q);
            free_clustering(c);
            CLD_CUDA(cudaEventRecord(e1.e, s));
            CLD_CUDA(cudaEventSynchronize(e1.e));
            float ms = 0.f;
            CLD_CUDA(cudaEventElapsedTime(&ms, e0.e, e1.e));
            a->last_start[i] = big_s;
            big_s += ms * 1e-3;
            a->last_end[i] = big_s;
            big_st[i] = st;
        }
    }
    const uint32_t nrest = count - nbig;
    if (nrest > 0) {
        const auto workspaces = [&](uint32_t j0, uint32_t j1, int slices, void** buf, size_t* bytes,
                                    std::vector<Workspace>* out) {
            uint32_t nmax = 1;
            uint64_t zmax = 0;
            for (uint32_t j = j0; j < j1; ++j) {
                nmax = std::max(nmax, a->graphs[jobs[j].graph].n);
                zmax = std::max(zmax, a->graphs[jobs[j].graph].nnz);
            }
            return make_workspaces(nmax, zmax, slices, s, buf, bytes, out);
        };
        std::vector<Workspace> wsh, gwsh;
        const int groups = std::min<int>((int)ngrp, max_groups);
        if (ngrp > 0 && workspaces(nbig, nbig + ngrp, groups, &a->gws, &a->gws_bytes, &gwsh) != CLDIAM_OK)
            ngrp = 0;  // no memory for the groups' workspaces: every job on one CTA
        const uint32_t nones = nrest - ngrp;  // jobs on one CTA each
        const uint32_t one_ctas = std::min<uint32_t>(nsm, nones);
        if (nones > 0) CLD_TRY(workspaces(nbig + ngrp, count, (int)one_ctas, &a->ws, &a->ws_bytes, &wsh));
        if (ngrp > 0) wsh.insert(wsh.end(), gwsh.begin(), gwsh.end());
        DBuf<ArenaDesc> ddesc;
        DBuf<Job> djobs;
        DBuf<Workspace> dws;
        DBuf<uint32_t> queue;
        DBuf<JobOut> douts;
        CLD_TRY(ddesc.alloc(a->graphs.size(), s));
        CLD_TRY(djobs.alloc(nrest, s));
        CLD_TRY(dws.alloc(wsh.size(), s));
        CLD_TRY(queue.alloc(2, s));
        CLD_TRY(douts.alloc(count, s));
        CLD_CUDA(cudaMemcpyAsync(ddesc.get(), a->graphs.data(), a->graphs.size() * sizeof(ArenaDesc),
                                 cudaMemcpyHostToDevice, s));
        CLD_CUDA(cudaMemcpyAsync(djobs.get(), jobs.data() + nbig, nrest * sizeof(Job), cudaMemcpyHostToDevice, s));
        CLD_CUDA(cudaMemcpyAsync(dws.get(), wsh.data(), wsh.size() * sizeof(Workspace), cudaMemcpyHostToDevice, s));
        CLD_CUDA(cudaMemsetAsync(queue.get(), 0, 8, s));
        const size_t dyn = batch_dyn_smem();
        cudaStream_t ones = s;
        CudaEvent fork, join;
        if (ngrp > 0) {
            // the groups first, on s; the one-CTA jobs beside them on the arena's second stream, on the SMs left and
            // those that the groups leave.  Everything they use was allocated and filled on s before the fork, and s
            // waits for them before anything is read or released.
            if (nones > 0 && !a->aux) CLD_CUDA(cudaStreamCreateWithFlags(&a->aux, cudaStreamNonBlocking));
            if (nones > 0) {
                ones = a->aux;
                CLD_TRY(fork.create());
                CLD_TRY(join.create());
                CLD_CUDA(cudaEventRecord(fork.e, s));
                CLD_CUDA(cudaStreamWaitEvent(ones, fork.e, 0));
            }
            cudaLaunchConfig_t cfg{};
            cudaLaunchAttribute at{};
            job_group_config(&cfg, &at, groups);
            cfg.stream = s;
            const uint64_t* off = a->off;
            const uint2* adj = a->adj;
            const uint32_t* row = a->row;
            CLD_K(K_MISC, s, CLD_CUDA(cudaLaunchKernelEx(&cfg, k_batch<true>, (const ArenaDesc*)ddesc.get(),
                                                         (const Job*)djobs.get(), ngrp, off, adj, row,
                                                         dws.get() + one_ctas, queue.get() + 1, douts.get())));
        }
        if (nones > 0) {
            CLD_K(K_MISC, ones, k_batch<false><<<one_ctas, BT, dyn, ones>>>(
                                    ddesc.get(), djobs.get() + ngrp, nones, a->off, a->adj, a->row, dws.get(), queue.get(),
                                    douts.get()));
            CLD_LAUNCH_CHECK();
            if (ones != s) {
                CLD_CUDA(cudaEventRecord(join.e, ones));
                CLD_CUDA(cudaStreamWaitEvent(s, join.e, 0));
            }
        }
        std::vector<JobOut> hl(count);
        CLD_CUDA(cudaMemcpyAsync(hl.data(), douts.get(), count * sizeof(JobOut), cudaMemcpyDeviceToHost, s));
        CLD_CUDA(cudaStreamSynchronize(s));
        // per-job device times of the launch, relative to its first job's start, after the one-graph runs
        uint64_t t0 = ~0ull;
        for (uint32_t j = nbig; j < count; ++j) t0 = std::min(t0, hl[jobs[j].out].t_start);
        for (uint32_t j = nbig; j < count; ++j) {
            const uint32_t i = jobs[j].out;
            ho[i] = hl[i];
            a->last_start[i] = big_s + (double)(hl[i].t_start - t0) * 1e-9;
            a->last_end[i] = big_s + (double)(hl[i].t_end - t0) * 1e-9;
        }
    }
    cldiam_status first_err = CLDIAM_OK;
    for (uint32_t i = 0; i < count; ++i) {
        cldiam_status st = big_st[i];
        if (ho[i].status == kJobNeedsPlain) {
            // quotient larger than the dense capacity: finish this graph with the one-graph path
            cldiam_graph view;
            arena_view(a, ids[i], &view);
            CLD_TRY(view.host.alloc(256));
            cldiam_clustering* c = nullptr;
            cldiam_quotient* q = nullptr;
            st = cluster(&view, tau[i], seed[i], &opts, &c);
            if (st == CLDIAM_OK) st = quotient(c, &q);
            if (st == CLDIAM_OK) st = cldiam_estimate(q, &ho[i].r);
            free_quotient(q);
            free_clustering(c);
        } else if (ho[i].status == kJobOverflow) {
            st = CLDIAM_ERR_OVERFLOW;
        } else if (ho[i].status == kJobDiverged) {
            st = CLDIAM_ERR_DIVERGED;
        } else if (ho[i].status != kJobOk) {
            st = CLDIAM_ERR_TIMEOUT;
        }
        out[i] = ho[i].r;
        if (status) status[i] = st;
        if (st != CLDIAM_OK && first_err == CLDIAM_OK) first_err = st;
    }
    if (first_err != CLDIAM_OK) return fail(first_err, "one or more graphs of the batch failed (see status[])");
    return CLDIAM_OK;
}

// ---------------------------------------------------------------------------- server
namespace {
inline void host_store_release(uint32_t* p, uint32_t v) { __atomic_store_n(p, v, __ATOMIC_RELEASE); }
inline uint32_t host_load_acquire(const uint32_t* p) { return __atomic_load_n(p, __ATOMIC_ACQUIRE); }
}  // namespace

}  // namespace cld

struct cldiam_server {
    cldiam_arena* arena = nullptr;
    int device = 0;
    cudaStream_t kstream = nullptr, bstream = nullptr;
    uint32_t ctas = 0, cap = 0, big_nodes = 0;
    uint64_t budget = 0;
    long long idle_cycles = 0;
    // host-mapped (pinned) memory, shared with the serving kernel
    cld::ServeCtl* ctl = nullptr;
    cld::Job* ring = nullptr;
    cld::JobOut* outs = nullptr;
    uint32_t* done = nullptr;
    // device memory
    uint32_t* head = nullptr;
    cld::Workspace* wss = nullptr;
    cld::ArenaDesc* descs = nullptr;
    void* ws = nullptr;
    size_t ws_bytes = 0;
    // host state
    std::mutex mu;
    uint32_t next_ticket = 0, next_ring = 0;
    bool kernel_live = false;
    std::vector<uint32_t> big_graph;
    std::vector<double> big_tau;
    std::vector<uint64_t> big_seed;
    std::thread big;
    std::mutex bmu;
    std::condition_variable bcv;
    std::deque<uint32_t> bq;
    bool bstop = false;
    cld::Pinned bhost;  // counter block of the big lane's one-graph runs
    bool counted = false;  // counted among the device's live servers
};

namespace cld {

static std::atomic<bool> g_serve_attr[64];

static cldiam_status server_launch(cldiam_server* sv) {
    CLD_TRY(set_dyn_smem(k_serve, g_serve_attr));
    sv->ctl->idle = 0;
    CLD_K(K_MISC, sv->kstream,
          k_serve<<<sv->ctas, BT, batch_dyn_smem(), sv->kstream>>>(sv->descs, sv->arena->off, sv->arena->adj,
                                                                   sv->arena->row, sv->wss, sv->ring, sv->ctl,
                                                                   sv->head, sv->outs, sv->done, sv->idle_cycles));
    CLD_LAUNCH_CHECK();
    sv->kernel_live = true;
    return CLDIAM_OK;
}

// relaunch the serving kernel if its CTAs left after the idle limit (caller holds sv->mu)
static cldiam_status server_ensure_live(cldiam_server* sv) {
    if (sv->kernel_live) {
        cudaError_t q = cudaStreamQuery(sv->kstream);
        if (q == cudaErrorNotReady) return CLDIAM_OK;
        if (q != cudaSuccess) return cuda_fail(q, "serving kernel", __FILE__, __LINE__);
        sv->kernel_live = false;
    }
    return server_launch(sv);
}

static void big_lane(cldiam_server* sv) {
    cudaSetDevice(sv->device);
    for (;;) {
        uint32_t t;
        {
            std::unique_lock<std::mutex> lk(sv->bmu);
            sv->bcv.wait(lk, [&] { return sv->bstop || !sv->bq.empty(); });
            if (sv->bq.empty()) return;
            t = sv->bq.front();
            sv->bq.pop_front();
        }
        cldiam_graph view;
        arena_view(sv->arena, sv->big_graph[t], &view);
        view.stream = sv->bstream;
        view.host.h = sv->bhost.h;  // borrowed pinned block; released with the server
        cldiam_result r{};
        cldiam_status st = CLDIAM_OK;
        // admission by device memory: the one-graph path needs ~100 B per node plus ~40 B per entry
        const uint64_t need = (uint64_t)view.n * 100 + view.nnz * 40;
        if (sv->budget && arena_bytes(sv->arena) + sv->ws_bytes + need > sv->budget) {
            st = fail(CLDIAM_ERR_OOM, "request does not fit the server's device memory budget");
        } else {
            cldiam_clustering* c = nullptr;
            cldiam_quotient* q = nullptr;
            cldiam_opts o{};
            st = cluster(&view, sv->big_tau[t], sv->big_seed[t], &o, &c);
            if (st == CLDIAM_OK) st = quotient(c, &q);
            if (st == CLDIAM_OK) st = cldiam_estimate(q, &r);
            free_quotient(q);
            free_clustering(c);
        }
        view.host.h = nullptr;
        sv->outs[t].r = r;
        sv->outs[t].status = st == CLDIAM_OK ? kJobOk
                             : st == CLDIAM_ERR_OVERFLOW ? kJobOverflow
                             : st == CLDIAM_ERR_DIVERGED ? kJobDiverged : kJobTimeout;
        host_store_release(&sv->done[t], 1u);
    }
}

cldiam_status server_free(cldiam_server* sv);

// Servers alive on each device: a server's persistent kernel holds its SMs until it has been idle for long, and the
// few SMs it leaves need not include a cluster's worth in one GPC, so thread-block clusters are not launched beside it.
// A server counts until it is freed, also while its kernel is gone: the next request launches it again, possibly before
// a cluster that was launched in between is running, which would then wait for the whole idle limit.
static std::atomic<int> g_live_servers[64];
bool serving_kernel_alive(int dev) { return dev < 0 || dev >= 64 || g_live_servers[dev].load() > 0; }

cldiam_status server_create(cldiam_arena* a, const cldiam_server_opts* o, cldiam_server** out) {
    if (!a || !out) return fail(CLDIAM_ERR_INVALID_ARG, "NULL arena or out");
    *out = nullptr;
    cldiam_server_opts opts{};
    if (o) opts = *o;
    cldiam_server* sv = new cldiam_server();
    sv->arena = a;
    CLD_CUDA(cudaGetDevice(&sv->device));
    const int nsm = num_sms();
    int cps = 1;
    if (cldiam_status st = resident_per_sm(k_serve, g_serve_attr, &cps); st != CLDIAM_OK) {
        delete sv;
        return st;
    }
    sv->ctas = opts.ctas ? std::min<uint32_t>(opts.ctas, (uint32_t)(nsm * cps)) : (uint32_t)(std::max(1, nsm - 24) * cps);
    sv->cap = opts.capacity ? opts.capacity : (1u << 20);
    sv->big_nodes = opts.big_nodes ? opts.big_nodes : (1u << 19);
    sv->budget = opts.hbm_budget_bytes;
    int khz = 0;
    cudaDeviceGetAttribute(&khz, cudaDevAttrClockRate, sv->device);
    const double idle_s = opts.idle_seconds > 0 ? opts.idle_seconds : 10.0;
    sv->idle_cycles = (long long)(idle_s * (khz > 0 ? khz : 2000000) * 1e3);
    auto cleanup = [&](cldiam_status st) {
        server_free(sv);
        return st;
    };
    if (cudaStreamCreateWithFlags(&sv->kstream, cudaStreamNonBlocking) != cudaSuccess ||
        cudaStreamCreateWithFlags(&sv->bstream, cudaStreamNonBlocking) != cudaSuccess)
        return cleanup(fail(CLDIAM_ERR_CUDA, "stream creation failed"));
    void* p = nullptr;
    const size_t host_bytes = sizeof(ServeCtl) + (size_t)sv->cap * (sizeof(Job) + sizeof(JobOut) + sizeof(uint32_t));
    if (cudaHostAlloc(&p, host_bytes, cudaHostAllocMapped) != cudaSuccess) {
        cudaGetLastError();
        return cleanup(fail(CLDIAM_ERR_OOM, "pinned host memory for the request ring"));
    }
    memset(p, 0, host_bytes);
    char* c = static_cast<char*>(p);
    sv->ctl = reinterpret_cast<ServeCtl*>(c); c += sizeof(ServeCtl);
    sv->ring = reinterpret_cast<Job*>(c); c += (size_t)sv->cap * sizeof(Job);
    sv->outs = reinterpret_cast<JobOut*>(c); c += (size_t)sv->cap * sizeof(JobOut);
    sv->done = reinterpret_cast<uint32_t*>(c);
    cldiam_status st = sv->bhost.alloc(256);
    if (st != CLDIAM_OK) return cleanup(st);
    // device state: descriptors, head counter, workspaces for the graphs the kernel serves
    uint32_t nmax = 1;
    uint64_t zmax = 0;
    for (const ArenaDesc& d : a->graphs)
        if (d.n <= sv->big_nodes) {
            nmax = std::max(nmax, d.n);
            zmax = std::max(zmax, d.nnz);
        }
    std::vector<Workspace> wsh;
    if ((st = make_workspaces(nmax, zmax, (int)sv->ctas, sv->kstream, &sv->ws, &sv->ws_bytes, &wsh)) != CLDIAM_OK)
        return cleanup(st);
    if (sv->budget) release_workspaces(a);
    if (sv->budget && arena_bytes(a) + sv->ws_bytes > sv->budget)
        return cleanup(fail(CLDIAM_ERR_OOM, "arena plus serving workspace exceed the budget"));
    if ((st = dmalloc((void**)&sv->head, 4, sv->kstream)) != CLDIAM_OK ||
        (st = dmalloc((void**)&sv->wss, wsh.size() * sizeof(Workspace), sv->kstream)) != CLDIAM_OK ||
        (st = dmalloc((void**)&sv->descs, std::max<size_t>(1, a->graphs.size()) * sizeof(ArenaDesc), sv->kstream)) !=
            CLDIAM_OK)
        return cleanup(st);
    cudaMemsetAsync(sv->head, 0, 4, sv->kstream);
    cudaMemcpyAsync(sv->wss, wsh.data(), wsh.size() * sizeof(Workspace), cudaMemcpyHostToDevice, sv->kstream);
    if (!a->graphs.empty())
        cudaMemcpyAsync(sv->descs, a->graphs.data(), a->graphs.size() * sizeof(ArenaDesc), cudaMemcpyHostToDevice,
                        sv->kstream);
    if (cudaStreamSynchronize(sv->kstream) != cudaSuccess) return cleanup(fail(CLDIAM_ERR_CUDA, "server set-up"));
    sv->big_graph.resize(sv->cap);
    sv->big_tau.resize(sv->cap);
    sv->big_seed.resize(sv->cap);
    for (auto load : {load_prims_kernels, load_csr_kernels, load_cluster_kernels, load_cluster2_kernels,
                      load_quotient_kernels, load_apsp_kernels, load_sssp_kernels, load_api_kernels})
        if ((st = load()) != CLDIAM_OK) return cleanup(st);
    if ((st = load_kernels(k_batch<false>)) != CLDIAM_OK) return cleanup(st);
    {
        std::lock_guard<std::mutex> lk(sv->mu);
        if (sv->device >= 0 && sv->device < 64) {
            g_live_servers[sv->device].fetch_add(1);
            sv->counted = true;
        }
        if ((st = server_launch(sv)) != CLDIAM_OK) return cleanup(st);
    }
    sv->big = std::thread(big_lane, sv);
    *out = sv;
    return CLDIAM_OK;
}

cldiam_status server_submit(cldiam_server* sv, uint32_t graph_id, double tau, uint64_t seed, uint64_t* ticket) {
    if (!sv || !ticket) return fail(CLDIAM_ERR_INVALID_ARG, "NULL server or ticket");
    if (graph_id >= sv->arena->graphs.size()) return fail(CLDIAM_ERR_INVALID_ARG, "graph id out of range");
    if (!(tau > 0.0) || !std::isfinite(tau)) return fail(CLDIAM_ERR_INVALID_ARG, "tau must be positive");
    cldiam_graph view;
    arena_view(sv->arena, graph_id, &view);
    uint32_t d0 = 0;
    CLD_TRY(delta0(&view, CLDIAM_DELTA0_AVG, 0, &d0));
    std::lock_guard<std::mutex> lk(sv->mu);
    if (sv->next_ticket >= sv->cap) return fail(CLDIAM_ERR_BUSY, "server request capacity exhausted");
    const uint32_t t = sv->next_ticket++;
    if (view.n > sv->big_nodes) {
        // large graph: the one-graph path on the big-lane stream, using the SMs the kernel leaves free
        sv->big_graph[t] = graph_id;
        sv->big_tau[t] = tau;
        sv->big_seed[t] = seed;
        {
            std::lock_guard<std::mutex> bl(sv->bmu);
            sv->bq.push_back(t);
        }
        sv->bcv.notify_one();
    } else {
        Job j{};
        j.tau = tau;
        j.L = std::log2((double)view.n);
        j.seed = seed;
        j.graph = graph_id;
        j.delta0 = d0;
        j.out = t;
        j.fw_k = tuning_for_batch(sv->arena->adj_used).batch_fw_k;
        sv->ring[sv->next_ring] = j;
        host_store_release(&sv->ctl->tail, ++sv->next_ring);  // publish after the entry is written
        CLD_TRY(server_ensure_live(sv));
    }
    *ticket = t;
    return CLDIAM_OK;
}

cldiam_status server_poll(cldiam_server* sv, uint64_t ticket, cldiam_result* out) {
    if (!sv || !out) return fail(CLDIAM_ERR_INVALID_ARG, "NULL server or out");
    if (ticket >= sv->next_ticket) return fail(CLDIAM_ERR_INVALID_ARG, "unknown ticket");
    if (!host_load_acquire(&sv->done[ticket])) {
        std::lock_guard<std::mutex> lk(sv->mu);
        CLD_TRY(server_ensure_live(sv));
        return CLDIAM_ERR_BUSY;
    }
    *out = sv->outs[ticket].r;
    switch (sv->outs[ticket].status) {
        case kJobOk: return CLDIAM_OK;
        case kJobOverflow: return fail(CLDIAM_ERR_OVERFLOW, "distance overflow");
        case kJobDiverged: return fail(CLDIAM_ERR_DIVERGED, "stage limit exceeded");
        case kJobNeedsPlain: return fail(CLDIAM_ERR_UNSUPPORTED, "quotient above the serving kernel's capacity");
        default: return fail(CLDIAM_ERR_TIMEOUT, "request failed");
    }
}

cldiam_status server_free(cldiam_server* sv) {
    if (!sv) return CLDIAM_OK;
    if (sv->ctl) host_store_release(&sv->ctl->stop, 1u);
    if (sv->big.joinable()) {
        {
            std::lock_guard<std::mutex> bl(sv->bmu);
            sv->bstop = true;
        }
        sv->bcv.notify_all();
        sv->big.join();
    }
    if (sv->kstream) cudaStreamSynchronize(sv->kstream);
    if (sv->bstream) cudaStreamSynchronize(sv->bstream);
    if (sv->counted) g_live_servers[sv->device].fetch_sub(1);
    dfree(sv->head, sv->kstream);
    dfree(sv->wss, sv->kstream);
    dfree(sv->descs, sv->kstream);
    dfree(sv->ws, sv->kstream);
    if (sv->kstream) cudaStreamSynchronize(sv->kstream);
    if (sv->ctl) cudaFreeHost(sv->ctl);
    if (sv->kstream) cudaStreamDestroy(sv->kstream);
    if (sv->bstream) cudaStreamDestroy(sv->bstream);
    delete sv;
    return CLDIAM_OK;
}

// Replay an arrival trace: request i is submitted at arrival[i] seconds after the start and its
// latency is completion minus arrival.  plain != 0 serves the same trace one request at a time
// in arrival order on the one-graph path instead (the one-query-per-call baseline).
cldiam_status server_replay(cldiam_server* sv, const uint32_t* ids, const double* tau, const uint64_t* seed,
                            const double* arrival, uint32_t count, int plain, cldiam_result* out, double* latency,
                            double* elapsed) {
    using clk = std::chrono::steady_clock;
    if (!sv || (count && (!ids || !tau || !seed || !arrival || !out || !latency)))
        return fail(CLDIAM_ERR_INVALID_ARG, "NULL argument");
    const auto t0 = clk::now();
    auto since = [&](clk::time_point t) { return std::chrono::duration<double>(t - t0).count(); };
    auto wait_until = [&](double at) {
        for (;;) {
            const double now = since(clk::now());
            if (now >= at) return;
            if (at - now > 200e-6) std::this_thread::sleep_for(std::chrono::microseconds(50));
        }
    };
    cldiam_status first = CLDIAM_OK;
    if (plain) {
        cldiam_graph view;
        for (uint32_t i = 0; i < count; ++i) {
            wait_until(arrival[i]);
            arena_view(sv->arena, ids[i], &view);
            view.stream = sv->bstream;
            view.host.h = sv->bhost.h;
            cldiam_clustering* c = nullptr;
            cldiam_quotient* q = nullptr;
            cldiam_opts o{};
            cldiam_status st = cluster(&view, tau[i], seed[i], &o, &c);
            if (st == CLDIAM_OK) st = quotient(c, &q);
            if (st == CLDIAM_OK) st = cldiam_estimate(q, &out[i]);
            free_quotient(q);
            free_clustering(c);
            view.host.h = nullptr;
            latency[i] = since(clk::now()) - arrival[i];
            if (st != CLDIAM_OK && first == CLDIAM_OK) first = st;
        }
    } else {
        std::vector<uint64_t> tickets(count, ~0ull);
        std::atomic<uint32_t> submitted{0};
        cldiam_status sub_err = CLDIAM_OK;
        std::thread submitter([&] {
            cudaSetDevice(sv->device);
            for (uint32_t i = 0; i < count; ++i) {
                wait_until(arrival[i]);
                uint64_t t = 0;
                cldiam_status st = server_submit(sv, ids[i], tau[i], seed[i], &t);
                if (st != CLDIAM_OK) {
                    sub_err = st;
                    break;
                }
                tickets[i] = t;
                submitted.store(i + 1, std::memory_order_release);
            }
        });
        std::vector<uint32_t> pending;
        uint32_t seen = 0, finished = 0;
        while (finished < count) {
            const uint32_t s = submitted.load(std::memory_order_acquire);
            while (seen < s) pending.push_back(seen++);
            if (sub_err != CLDIAM_OK && pending.empty()) break;
            size_t keep = 0;
            for (uint32_t i : pending) {
                if (host_load_acquire(&sv->done[tickets[i]])) {
                    latency[i] = since(clk::now()) - arrival[i];
                    cldiam_status st = server_poll(sv, tickets[i], &out[i]);
                    if (st != CLDIAM_OK && first == CLDIAM_OK) first = st;
                    ++finished;
                } else {
                    pending[keep++] = i;
                }
            }
            const bool progressed = keep < pending.size();
            pending.resize(keep);
            static thread_local auto last_check = clk::now();
            if (!pending.empty() && !progressed && clk::now() - last_check > std::chrono::milliseconds(1)) {
                last_check = clk::now();
                std::lock_guard<std::mutex> lk(sv->mu);
                CLD_TRY(server_ensure_live(sv));
            }
        }
        submitter.join();
        if (sub_err != CLDIAM_OK) return sub_err;
    }
    if (elapsed) *elapsed = since(clk::now());
    if (first != CLDIAM_OK) return first;
    return CLDIAM_OK;
}

}  // namespace cld
