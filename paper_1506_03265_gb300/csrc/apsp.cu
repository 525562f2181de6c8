// Phi(G_C) (Section 4): the largest finite shortest-path distance of the
// quotient graph, by exact blocked Floyd-Warshall over the dense k x k
// distance matrix in (min, +) arithmetic on the integer ALUs (min-plus is not
// a tensor-core contraction).
//
// Blocked FW with 64 x 64 tiles (Venkataraman, Sahni, Mukhopadhyaya): for
// each pivot tile r, (1) close the diagonal tile, (2) update the tiles of
// row r and column r through it, (3) update every other tile from its row-r
// and column-r tiles.  Two arithmetic forms share the kernels: the checked
// form keeps uint32 entries with 0xFFFFFFFF = no path, and a sum of two
// finite entries that reaches 2^32 - 1 raises the overflow flag instead of
// wrapping; the fast form uses 0x7FFFFFFF = no path, so a sum never wraps and
// one fused add-min per relaxation suffices (a path that would reach
// 0x7FFFFFFF stays "no path").  The fast form runs first; its result is
// exact when every pair ends up connected, otherwise the checked form
// recomputes the matrix.
#include <algorithm>
#include <atomic>
#include <mutex>

#include "bounds.cuh"
#include "cluster_dev.cuh"
#include "internal.cuh"
#include "prof.cuh"

namespace cld {

namespace {

constexpr uint32_t INF = 0xFFFFFFFFu;
constexpr uint32_t INFF = 0x7FFFFFFFu;  // "no path" of the fast form

__device__ __forceinline__ uint32_t relax_min(uint32_t c, uint32_t a, uint32_t b, bool& ovf) {
    uint32_t s = a + b;
    bool carry = s < a;
    bool finite = (a != INF) & (b != INF);
    ovf |= finite & (carry | (s == INF));
    return (carry | !finite) ? c : (s < c ? s : c);
}

// one relaxation c = min(c, a + b) in the form's arithmetic
template <bool FAST>
__device__ __forceinline__ uint32_t fw_relax(uint32_t c, uint32_t a, uint32_t b, bool& ovf) {
    if constexpr (FAST) return __viaddmin_u32(a, b, c);
    else return relax_min(c, a, b, ovf);
}

__global__ void k_fw_init(uint32_t* __restrict__ M, uint32_t kp, uint32_t k, uint32_t none) {
    size_t total = (size_t)kp * kp;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        uint32_t r = (uint32_t)(i / kp), c = (uint32_t)(i % kp);
        M[i] = (r == c) ? 0u : none;
    }
}

// caller-supplied CSR: offsets must start at 0, never decrease, end at nnz; columns < k
__global__ void k_fw_validate(const uint64_t* __restrict__ off, const uint32_t* __restrict__ col, uint32_t k,
                              uint64_t nnz, uint32_t* __restrict__ bad) {
    bool b = false;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i <= (uint64_t)k + nnz;
         i += (uint64_t)gridDim.x * blockDim.x) {
        if (i <= k) {
            uint64_t o = off[i];
            if (o > nnz || (i == 0 && o != 0) || (i == k && o != nnz) || (i > 0 && off[i - 1] > o)) b = true;
        } else if (col[i - k - 1] >= k) {
            b = true;
        }
    }
    if (b) atomicExch(bad, 1u);
}

// edge weights into the matrix; a weight of 0x7FFFFFFF or more sets *wide (the fast form cannot hold it)
__global__ void k_fw_scatter(const uint64_t* __restrict__ off, const uint32_t* __restrict__ col,
                             const uint32_t* __restrict__ w, uint32_t k, uint32_t kp, uint32_t* __restrict__ M,
                             uint32_t* __restrict__ wide) {
    bool wd = false;
    for (uint32_t a = blockIdx.x; a < k; a += gridDim.x)
        for (uint64_t j = off[a] + threadIdx.x; j < off[a + 1]; j += blockDim.x) {
            uint32_t b = col[j];
            wd |= w[j] >= INFF;
            if (b != a) atomicMin(&M[(size_t)a * kp + b], w[j]);
        }
    if (wd && wide) atomicExch(wide, 1u);
}

// Tiles are T x T = 64 x 64; 256 threads hold a tile as 4 x 4 registers each (rows 4*ty.., cols 4*tx..).
constexpr int FT = 64;
constexpr int FQ = 4;       // 4 x 4 entries per thread
constexpr int FTH = 256;    // 16 x 16 threads
constexpr int FS = 32;      // columns (row tiles) or rows (column tiles) of a phase 2 strip
constexpr int FA = FT + 4;  // padded row of a transposed tile, 16-byte aligned

__device__ __forceinline__ void fw_load4x4(uint32_t (&c)[FQ][FQ], const uint32_t* M, uint32_t kp, size_t y, size_t x) {
#pragma unroll
    for (int i = 0; i < FQ; ++i) {
        const uint4 v = *reinterpret_cast<const uint4*>(&M[(y + i) * kp + x]);
        c[i][0] = v.x; c[i][1] = v.y; c[i][2] = v.z; c[i][3] = v.w;
    }
}
__device__ __forceinline__ void fw_store4x4(const uint32_t (&c)[FQ][FQ], uint32_t* M, uint32_t kp, size_t y, size_t x) {
#pragma unroll
    for (int i = 0; i < FQ; ++i)
        *reinterpret_cast<uint4*>(&M[(y + i) * kp + x]) = make_uint4(c[i][0], c[i][1], c[i][2], c[i][3]);
}
template <bool FAST>
__device__ __forceinline__ void fw_relax4x4(uint32_t (&c)[FQ][FQ], const uint4 av, const uint4 bv, bool& ovf) {
    const uint32_t a[FQ] = {av.x, av.y, av.z, av.w};
    const uint32_t b[FQ] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
    for (int i = 0; i < FQ; ++i)
#pragma unroll
        for (int j = 0; j < FQ; ++j) c[i][j] = fw_relax<FAST>(c[i][j], a[i], b[j], ovf);
}

// Phase 1: closes the pivot tile held in registers.  Iteration p needs row p and column p, which it cannot change
// itself (D[p][p] = 0): their owners publish them in one of two shared buffers, one barrier per p.  A serial chain
// of 64 barriers on one CTA; with the tile in shared memory (16 read-modify-writes per thread and p) it took 40 us,
// from registers 7 us.
struct FwLine {
    __align__(16) uint32_t row[2][FT], col[2][FT];
};
template <bool FAST>
__device__ __forceinline__ void fw_close(uint32_t (&c)[FQ][FQ], FwLine& s, int ty, int tx, bool& ovf) {
    for (int p4 = 0; p4 < FT / FQ; ++p4) {
#pragma unroll
        for (int j = 0; j < FQ; ++j) {
            const int b = j & 1;
            if (ty == p4) *reinterpret_cast<uint4*>(&s.row[b][tx * FQ]) = make_uint4(c[j][0], c[j][1], c[j][2], c[j][3]);
            if (tx == p4) *reinterpret_cast<uint4*>(&s.col[b][ty * FQ]) = make_uint4(c[0][j], c[1][j], c[2][j], c[3][j]);
            __syncthreads();
            fw_relax4x4<FAST>(c, *reinterpret_cast<const uint4*>(&s.col[b][ty * FQ]),
                              *reinterpret_cast<const uint4*>(&s.row[b][tx * FQ]), ovf);
        }
    }
}

template <bool FAST>
__global__ void __launch_bounds__(FTH) k_fw_phase1(uint32_t* __restrict__ M, uint32_t kp, uint32_t r,
                                                   uint32_t* __restrict__ ovf_flag) {
    __shared__ FwLine line;
    const int ty = threadIdx.x / 16, tx = threadIdx.x % 16;
    const size_t y = (size_t)r * FT + ty * FQ, x = (size_t)r * FT + tx * FQ;
    uint32_t c[FQ][FQ];
    fw_load4x4(c, M, kp, y, x);
    bool ovf = false;
    fw_close<FAST>(c, line, ty, tx, ovf);
    fw_store4x4(c, M, kp, y, x);
    if (!FAST && ovf) atomicExch(ovf_flag, 1u);
}

// Phase 2, tiles in pivot row r (blockIdx.y == 0) and pivot column r (blockIdx.y == 1).
// Fast form: the pivot tile is closed, so one min-plus product with the tile as it was gives the same values as 64
// dependent iterations (any path through the pivot nodes is one closed hop and one old entry), without a barrier
// per p.  A tile is cut into two strips of 32, one CTA of 128 threads each, since 2 (nt - 1) tiles alone leave half
// of the SMs idle: 47 us as dependent iterations, 5.2 us so (nt = 32).
__global__ void __launch_bounds__(FTH / 2) k_fw_phase2_fast(uint32_t* __restrict__ M, uint32_t kp, uint32_t r) {
    __shared__ __align__(16) uint32_t At[FT][FA];  // left operand, transposed (row strip: the whole pivot tile)
    __shared__ __align__(16) uint32_t B[FT][FT];
    const bool is_row = blockIdx.y == 0;
    uint32_t o = blockIdx.x >> 1;
    const uint32_t strip = blockIdx.x & 1;
    if (o >= r) ++o;
    // output block: 64 rows x 32 columns of a row tile, or 32 rows x 64 columns of a column tile
    const size_t y0 = (size_t)(is_row ? r : o) * FT + (is_row ? 0 : strip * FS);
    const size_t x0 = (size_t)(is_row ? o : r) * FT + (is_row ? strip * FS : 0);
    const int h = is_row ? FT : FS, w = is_row ? FS : FT;
    for (int i = threadIdx.x; i < h * FT; i += FTH / 2) At[i % FT][i / FT] = M[(y0 + i / FT) * kp + (size_t)r * FT + i % FT];
    for (int i = threadIdx.x; i < FT * w; i += FTH / 2) B[i / w][i % w] = M[((size_t)r * FT + i / w) * kp + x0 + i % w];
    const int tx = threadIdx.x % (w / FQ), ty = threadIdx.x / (w / FQ);
    uint32_t c[FQ][FQ];
    fw_load4x4(c, M, kp, y0 + ty * FQ, x0 + tx * FQ);
    __syncthreads();
    bool ovf = false;
#pragma unroll 8
    for (int p = 0; p < FT; ++p)
        fw_relax4x4<true>(c, *reinterpret_cast<const uint4*>(&At[p][ty * FQ]),
                          *reinterpret_cast<const uint4*>(&B[p][tx * FQ]), ovf);
    fw_store4x4(c, M, kp, y0 + ty * FQ, x0 + tx * FQ);
}

// Checked form: dependent iterations (a product with the old tile would look at larger candidate sums and report
// OVERFLOW on inputs that these accept), the tile in registers, row or column p published as in phase 1.
__global__ void __launch_bounds__(FTH) k_fw_phase2_checked(uint32_t* __restrict__ M, uint32_t kp, uint32_t r,
                                                           uint32_t* __restrict__ ovf_flag) {
    __shared__ __align__(16) uint32_t piv[FT][FA];  // row tiles: the pivot tile transposed; column tiles: as it is
    __shared__ __align__(16) uint32_t line[2][FT];
    const int ty = threadIdx.x / 16, tx = threadIdx.x % 16;
    const bool is_row = blockIdx.y == 0;
    uint32_t o = blockIdx.x;
    if (o >= r) ++o;
    const size_t y = (size_t)(is_row ? r : o) * FT + ty * FQ, x = (size_t)(is_row ? o : r) * FT + tx * FQ;
    for (int i = threadIdx.x; i < FT * FT; i += FTH) {
        const uint32_t v = M[((size_t)r * FT + i / FT) * kp + (size_t)r * FT + i % FT];
        if (is_row) piv[i % FT][i / FT] = v;
        else piv[i / FT][i % FT] = v;
    }
    uint32_t c[FQ][FQ];
    fw_load4x4(c, M, kp, y, x);
    bool ovf = false;
    for (int p4 = 0; p4 < FT / FQ; ++p4) {
#pragma unroll
        for (int j = 0; j < FQ; ++j) {
            const int b = j & 1, p = p4 * FQ + j;
            if (is_row && ty == p4)
                *reinterpret_cast<uint4*>(&line[b][tx * FQ]) = make_uint4(c[j][0], c[j][1], c[j][2], c[j][3]);
            if (!is_row && tx == p4)
                *reinterpret_cast<uint4*>(&line[b][ty * FQ]) = make_uint4(c[0][j], c[1][j], c[2][j], c[3][j]);
            __syncthreads();
            const uint32_t* a = is_row ? piv[p] : line[b];
            const uint32_t* bb = is_row ? line[b] : piv[p];
            fw_relax4x4<false>(c, *reinterpret_cast<const uint4*>(a + ty * FQ),
                               *reinterpret_cast<const uint4*>(bb + tx * FQ), ovf);
        }
    }
    fw_store4x4(c, M, kp, y, x);
    if (ovf) atomicExch(ovf_flag, 1u);
}

// Phase 3: every other tile from its pivot-column and pivot-row tiles; no barrier inside the p loop.  The
// pivot-column tile is held transposed, so a thread reads its 4 rows of column p as one vector.  Bound by the
// integer add-min rate.  The first CTA takes the next pivot tile and closes it when it is done (phase 1 of the next
// round), hidden behind the other tiles instead of a launch of its own.
template <bool FAST>
__global__ void __launch_bounds__(FTH) k_fw_phase3(uint32_t* __restrict__ M, uint32_t kp, uint32_t r,
                                                   uint32_t* __restrict__ ovf_flag) {
    __shared__ __align__(16) uint32_t At[FT][FA];
    __shared__ __align__(16) uint32_t B[FT][FT];
    __shared__ FwLine line;
    const int ty = threadIdx.x / 16, tx = threadIdx.x % 16;
    uint32_t ti = blockIdx.y, tj = blockIdx.x;
    // (in the grid's numbering, which leaves the pivot out, the next pivot is number r: swap it with number 0)
    const bool has_next = r < gridDim.x;
    const bool next = has_next && ti == 0 && tj == 0;
    if (next) ti = tj = r;
    else if (has_next && ti == r && tj == r) ti = tj = 0;
    if (ti >= r) ++ti;
    if (tj >= r) ++tj;
    for (int i = threadIdx.x; i < FT * FT; i += FTH) {
        int y = i / FT, x = i % FT;
        At[x][y] = M[((size_t)ti * FT + y) * kp + (size_t)r * FT + x];
        B[y][x] = M[((size_t)r * FT + y) * kp + (size_t)tj * FT + x];
    }
    uint32_t c[FQ][FQ];
    const size_t y0 = (size_t)ti * FT + ty * FQ, x0 = (size_t)tj * FT + tx * FQ;
    fw_load4x4(c, M, kp, y0, x0);
    __syncthreads();
    bool ovf = false;
#pragma unroll 8
    for (int p = 0; p < FT; ++p)
        fw_relax4x4<FAST>(c, *reinterpret_cast<const uint4*>(&At[p][ty * FQ]),
                          *reinterpret_cast<const uint4*>(&B[p][tx * FQ]), ovf);
    if (next) fw_close<FAST>(c, line, ty, tx, ovf);
    fw_store4x4(c, M, kp, y0, x0);
    if (!FAST && ovf) atomicExch(ovf_flag, 1u);
}

// all rounds of blocked Floyd-Warshall on the padded matrix of nt x nt tiles
template <bool FAST>
cldiam_status fw_rounds(uint32_t* M, uint32_t kp, uint32_t nt, uint32_t* ovf, cudaStream_t s) {
    CLD_K(K_FW, s, k_fw_phase1<FAST><<<1, FTH, 0, s>>>(M, kp, 0, ovf));
    for (uint32_t r = 0; r < nt && nt > 1; ++r) {
        if constexpr (FAST) CLD_K(K_FW, s, k_fw_phase2_fast<<<dim3(2 * (nt - 1), 2), FTH / 2, 0, s>>>(M, kp, r));
        else CLD_K(K_FW, s, k_fw_phase2_checked<<<dim3(nt - 1, 2), FTH, 0, s>>>(M, kp, r, ovf));
        CLD_K(K_FW, s, k_fw_phase3<FAST><<<dim3(nt - 1, nt - 1), FTH, 0, s>>>(M, kp, r, ovf));
    }
    CLD_LAUNCH_CHECK();
    return CLDIAM_OK;
}

// largest entry below `none` among the k x k real entries; *missing = 1 if some entry is `none`
__global__ void k_fw_max_finite(const uint32_t* __restrict__ M, uint32_t kp, uint32_t k, uint32_t none,
                                uint32_t* __restrict__ out, uint32_t* __restrict__ missing) {
    uint32_t m = 0;
    bool miss = false;
    size_t total = (size_t)k * kp;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        uint32_t c = (uint32_t)(i % kp);
        uint32_t v = M[i];
        if (c < k && v != none && v > m) m = v;
        miss |= c < k && v == none;
    }
    if (missing && __any_sync(0xffffffffu, miss) && lane_id() == 0) atomicExch(missing, 1u);
    m = block_reduce(m, [](uint32_t a, uint32_t b) { return a > b ? a : b; }, 0u);
    if (threadIdx.x == 0) atomicMax(out, m);
}

// Batched exact SSSP on the quotient CSR (multi-source Bellman-Ford): a CTA
// owns S consecutive sources and keeps dist[v][s] for all k nodes in shared
// memory; in each round one warp per node v pulls min(dist[u][s] + w(u,v))
// over its neighbours u for all S sources at once (lane = (neighbour slot,
// source)), and only v's warp writes row v.  Rounds repeat until no distance
// changes.  Exact, so the eccentricities and their maximum equal
// Floyd-Warshall's, with about rounds x entries x k work instead of k^3,
// which wins on sparse quotients.
template <int S, bool kCsrInSmem>
__global__ void __launch_bounds__(1024) k_apsp_msbf(const uint64_t* __restrict__ goff, const uint32_t* __restrict__ gcol,
                                                    const uint32_t* __restrict__ gw, uint32_t k, uint32_t nnz,
                                                    uint32_t* __restrict__ out_max, uint32_t* __restrict__ ovf_flag) {
    extern __shared__ __align__(16) uint32_t sm[];
    uint32_t* dist = sm;  // k x S
    // when it fits, the quotient CSR itself is staged in shared memory too (32-bit offsets)
    uint32_t* soff = sm + (size_t)k * S;
    uint32_t* scol = soff + (k + 1);
    uint32_t* sw = scol + nnz;
    // "some distance changed" flag of round r lives in slot r % 3: it is written during round r and
    // read after its closing barrier, and slot (r + 1) % 3 is cleared during round r, when no thread
    // can still be reading it (round r - 2) or writing it yet (round r + 1)
    __shared__ uint32_t s_changed[3];
    const uint32_t s0 = blockIdx.x * S;
    const uint32_t warp = threadIdx.x >> 5, lane = lane_id(), nwarps = blockDim.x >> 5;
    const uint32_t my_s = lane % S, slot = lane / S;
    constexpr uint32_t kSlots = 32 / S;
    for (uint32_t i = threadIdx.x; i < k * S; i += blockDim.x) {
        const uint32_t v = i / S, s = i % S;
        dist[i] = (s0 + s == v) ? 0u : INF;
    }
    if (kCsrInSmem) {
        for (uint32_t i = threadIdx.x; i <= k; i += blockDim.x) soff[i] = (uint32_t)goff[i];
        for (uint32_t i = threadIdx.x; i < nnz; i += blockDim.x) {
            scol[i] = gcol[i];
            sw[i] = gw[i];
        }
    }
    bool ovf = false;
    if (threadIdx.x == 0) s_changed[0] = s_changed[1] = s_changed[2] = 0;
    __syncthreads();
    for (uint32_t round = 0; round < k; ++round) {
        const uint32_t slot_r = round % 3;
        if (threadIdx.x == 0) s_changed[(round + 1) % 3] = 0;
        bool changed = false;
        for (uint32_t v = warp; v < k; v += nwarps) {
            const uint32_t beg = kCsrInSmem ? soff[v] : (uint32_t)goff[v];
            const uint32_t end = kCsrInSmem ? soff[v + 1] : (uint32_t)goff[v + 1];
            uint32_t best = INF;
            for (uint32_t j = beg + slot; j < end; j += kSlots) {
                const uint32_t u = kCsrInSmem ? scol[j] : gcol[j];
                const uint32_t wj = kCsrInSmem ? sw[j] : gw[j];
                const uint32_t du = dist[u * S + my_s];
                if (du != INF) {
                    const uint64_t nd = (uint64_t)du + wj;
                    if (nd >= INF) ovf = true;
                    else best = min(best, (uint32_t)nd);
                }
            }
#pragma unroll
            for (uint32_t o = S; o < 32; o <<= 1) best = min(best, __shfl_xor_sync(0xffffffffu, best, o));
            if (lane < S && best < dist[v * S + lane]) {
                dist[v * S + lane] = best;
                changed = true;
            }
        }
        if (__any_sync(0xffffffffu, changed) && lane == 0) s_changed[slot_r] = 1;
        __syncthreads();
        if (!s_changed[slot_r]) break;
    }
    uint32_t best = 0;
    for (uint32_t i = threadIdx.x; i < k * S; i += blockDim.x)
        if (s0 + i % S < k && dist[i] != INF && dist[i] > best) best = dist[i];
    best = block_reduce(best, [](uint32_t a, uint32_t b) { return a > b ? a : b; }, 0u);
    if (threadIdx.x == 0) atomicMax(out_max, best);
    if (__any_sync(0xffffffffu, ovf) && lane == 0) atomicExch(ovf_flag, 1u);
}

template <int S>
cldiam_status launch_msbf(uint32_t k, const uint64_t* off, const uint32_t* col, const uint32_t* w, uint64_t nnz,
                          cudaStream_t s, uint32_t* out_max, uint32_t* ovf) {
    constexpr int kMax = 220 * 1024;
    static std::atomic<bool> attr[64];  // first call per device sets the attribute (idempotent)
    int dev = 0;
    CLD_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64 || !attr[dev]) {
        CLD_CUDA(cudaFuncSetAttribute(k_apsp_msbf<S, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMax));
        CLD_CUDA(cudaFuncSetAttribute(k_apsp_msbf<S, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMax));
        if (dev >= 0 && dev < 64) attr[dev] = true;
    }
    const size_t dist_bytes = (size_t)k * S * 4;
    const size_t csr_bytes = ((size_t)k + 1 + 2 * nnz) * 4;
    const unsigned grid = (k + S - 1) / S;
    if (dist_bytes + csr_bytes <= (size_t)kMax) {
        CLD_K(K_FW, s, k_apsp_msbf<S, true><<<grid, 1024, dist_bytes + csr_bytes, s>>>(off, col, w, k, (uint32_t)nnz,
                                                                                     out_max, ovf));
    } else {
        CLD_K(K_FW, s, k_apsp_msbf<S, false><<<grid, 1024, dist_bytes, s>>>(off, col, w, k, (uint32_t)nnz, out_max, ovf));
    }
    CLD_LAUNCH_CHECK();
    return CLDIAM_OK;
}

// Batched exact SSSP on the quotient with a worklist (multi-source Bellman-Ford
// that only pushes from changed nodes): a CTA owns S consecutive sources and
// keeps dist[v][s] for all k nodes in shared memory, plus one word of change
// bits per node (bit s: dist[v][s] decreased).  In each round one warp per
// node v with change bits pushes dist[v][s] + w(v, u) to every neighbour u
// (lanes = neighbours) with a shared-memory atomicMin for each changed
// source s, and marks u for the next round when that lowers dist[u][s].
// Distances only ever decrease and stay lengths of real paths, so when no
// node is marked they are exact; the work is the number of distance
// decreases times the degree, instead of rounds x entries, which wins on
// quotients with many rounds (high hop diameter).
template <int S, bool kCsrInSmem>
__global__ void __launch_bounds__(1024) k_apsp_wl(const uint64_t* __restrict__ goff, const uint32_t* __restrict__ gcol,
                                                  const uint32_t* __restrict__ gw, uint32_t k, uint32_t nnz,
                                                  uint32_t* __restrict__ out_max, uint32_t* __restrict__ ovf_flag,
                                                  uint32_t* __restrict__ err) {
    extern __shared__ __align__(16) uint32_t sm[];
    uint32_t* dist = sm;                   // k x S
    uint32_t* chg0 = sm + (size_t)k * S;   // change bits, two rounds
    uint32_t* chg1 = chg0 + k;
    uint32_t* soff = chg1 + k;
    uint32_t* scol = soff + (k + 1);
    uint32_t* sw = scol + nnz;
    const uint32_t s0 = blockIdx.x * S;
    const uint32_t warp = threadIdx.x >> 5, lane = lane_id(), nwarps = blockDim.x >> 5;
    for (uint32_t i = threadIdx.x; i < k * S; i += blockDim.x) {
        const uint32_t v = i / S, s = i % S;
        dist[i] = (s0 + s == v) ? 0u : INF;
    }
    for (uint32_t v = threadIdx.x; v < k; v += blockDim.x) {
        chg0[v] = (v >= s0 && v < s0 + S) ? 1u << (v - s0) : 0u;
        chg1[v] = 0;
    }
    if (kCsrInSmem) {
        for (uint32_t i = threadIdx.x; i <= k; i += blockDim.x) soff[i] = (uint32_t)goff[i];
        for (uint32_t i = threadIdx.x; i < nnz; i += blockDim.x) {
            scol[i] = gcol[i];
            sw[i] = gw[i];
        }
    }
    bool ovf = false;
    __syncthreads();
    const uint32_t max_rounds = 4 * k + 64;  // far above any real count: a guard, reported as an error
    uint32_t round = 0;
    for (;; ++round) {
        uint32_t* cur = (round & 1) ? chg1 : chg0;
        uint32_t* nxt = (round & 1) ? chg0 : chg1;
        for (uint32_t v = warp; v < k; v += nwarps) {
            const uint32_t bits = cur[v];
            if (!bits) continue;
            const uint32_t beg = kCsrInSmem ? soff[v] : (uint32_t)goff[v];
            const uint32_t end = kCsrInSmem ? soff[v + 1] : (uint32_t)goff[v + 1];
            for (uint32_t j = beg + lane; j < end; j += 32) {
                const uint32_t u = kCsrInSmem ? scol[j] : gcol[j];
                const uint32_t wj = kCsrInSmem ? sw[j] : gw[j];
                for (uint32_t b = bits; b; b &= b - 1) {
                    const uint32_t sidx = (uint32_t)__ffs(b) - 1;
                    const uint32_t dv = dist[v * S + sidx];
                    if (dv == INF) continue;
                    const uint64_t nd = (uint64_t)dv + wj;
                    if (nd >= INF) {
                        ovf = true;
                        continue;
                    }
                    uint32_t* du = &dist[u * S + sidx];
                    if ((uint32_t)nd < *du && (uint32_t)nd < atomicMin(du, (uint32_t)nd))
                        atomicOr(&nxt[u], 1u << sidx);
                }
            }
        }
        __syncthreads();
        bool any = false;
        for (uint32_t v = threadIdx.x; v < k; v += blockDim.x) {
            cur[v] = 0;
            any |= nxt[v] != 0;
        }
        if (!__syncthreads_or(any)) break;
        if (round >= max_rounds) {
            if (threadIdx.x == 0) atomicExch(err, 1u);
            break;
        }
    }
    uint32_t best = 0;
    for (uint32_t i = threadIdx.x; i < k * S; i += blockDim.x)
        if (s0 + i % S < k && dist[i] != INF && dist[i] > best) best = dist[i];
    best = block_reduce(best, [](uint32_t a, uint32_t b) { return a > b ? a : b; }, 0u);
    if (threadIdx.x == 0) atomicMax(out_max, best);
    if (__any_sync(0xffffffffu, ovf) && lane == 0) atomicExch(ovf_flag, 1u);
}

template <int S>
cldiam_status launch_wl(uint32_t k, const uint64_t* off, const uint32_t* col, const uint32_t* w, uint64_t nnz,
                        cudaStream_t s, uint32_t* out_max, uint32_t* ovf, uint32_t* err) {
    constexpr int kMax = 220 * 1024;
    static std::atomic<bool> attr[64];  // first call per device sets the attribute (idempotent)
    int dev = 0;
    CLD_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64 || !attr[dev]) {
        CLD_CUDA(cudaFuncSetAttribute(k_apsp_wl<S, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMax));
        CLD_CUDA(cudaFuncSetAttribute(k_apsp_wl<S, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMax));
        if (dev >= 0 && dev < 64) attr[dev] = true;
    }
    const size_t dist_bytes = (size_t)k * S * 4 + (size_t)k * 8;
    const size_t csr_bytes = ((size_t)k + 1 + 2 * nnz) * 4;
    const unsigned grid = (k + S - 1) / S;
    if (dist_bytes + csr_bytes <= (size_t)kMax) {
        CLD_K(K_FW, s, k_apsp_wl<S, true><<<grid, 1024, dist_bytes + csr_bytes, s>>>(off, col, w, k, (uint32_t)nnz,
                                                                                   out_max, ovf, err));
    } else {
        CLD_K(K_FW, s, k_apsp_wl<S, false><<<grid, 1024, dist_bytes, s>>>(off, col, w, k, (uint32_t)nnz, out_max, ovf,
                                                                          err));
    }
    CLD_LAUNCH_CHECK();
    return CLDIAM_OK;
}

// ---------------------------------------------------------------- diameter of a symmetric quotient by bounds
// The largest distance needs the eccentricity of few nodes (bounds.cuh).  Batches of sources run until no node is left:
// first an even sample of the ids, then the nodes of the largest upper and of the smallest lower bounds.  Two or three
// batches are enough on meshes, road meshes and R-MAT graphs alike, whatever k is.
// One CTA per source, so that a round costs little: the nodes improved in the last round are a list in shared memory,
// their adjacency is one flattened range (a block scan of the degrees), and each warp takes 128 positions of it; an SSSP
// on a road mesh's quotient (k = 4,082, 98,000 entries) is 12 to 20 rounds and 140,000 positions, bound by the issue
// and latency of the position lookups and shared atomics.  Every source by the worklist above / bounds: road mesh
// 4,096^2 2,702 / 1,082 us, R-MAT 24 (k = 4,023) 2,617 / 390 us, R-MAT 22 (k = 1,897) 354 / 107 us, 1,001^2 mesh
// (k = 840) 269 / 168 us.
struct BoundCtl {
    unsigned long long wsum;  // sum over nodes of their heaviest entry
    uint32_t wmax;
    uint32_t wide;            // a path might reach 2^32 - 1: nothing is pruned, the caller takes every source
    uint32_t nsrc;            // sources of the next batch
    uint32_t best;            // largest eccentricity so far
    uint32_t err;             // an SSSP exceeded its round limit
    uint32_t pad;
};
constexpr uint32_t kBoundFirst = 152, kBoundNext = 304;  // sources of the first and of later batches

// heaviest entry of every row, and the first sources
__global__ void __launch_bounds__(256) k_bound_prep(const uint64_t* __restrict__ off, const uint32_t* __restrict__ w,
                                                    uint32_t k, uint32_t nsrc, uint32_t* __restrict__ ub,
                                                    uint32_t* __restrict__ lb, uint32_t* __restrict__ src,
                                                    BoundCtl* ctl) {
    const uint32_t warps = (gridDim.x * blockDim.x) >> 5, lane = lane_id();
    unsigned long long sum = 0;
    uint32_t mx = 0;
    for (uint32_t v = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < k; v += warps) {
        uint32_t m = 0;
        for (uint64_t j = off[v] + lane; j < off[v + 1]; j += 32) m = max(m, w[j]);
        m = __reduce_max_sync(0xffffffffu, m);
        sum += m;
        mx = max(mx, m);
        if (lane == 0) {
            ub[v] = INF;
            lb[v] = 0;
            if (v < nsrc) src[v] = (uint32_t)((uint64_t)v * k / nsrc);
        }
    }
    if (lane == 0) {
        atomicAdd(&ctl->wsum, sum);
        atomicMax(&ctl->wmax, mx);
        if (blockIdx.x == 0 && threadIdx.x == 0) ctl->nsrc = nsrc;
    }
}

template <int T>
struct BoundSmem {  // one tile of a round's list
    uint32_t pre[T + 1];  // first positions of the nodes after the tile's first
    uint32_t base[T];
    uint32_t dist[T];
    uint32_t wsum[T / 32];
    uint32_t total, count[2];
};

// Largest distance from src[blockIdx.x], and the bounds it gives every node (ub only falls, lb only rises).
template <int T>
__global__ void __launch_bounds__(T) k_bound_sssp(const uint64_t* __restrict__ off, const uint32_t* __restrict__ col,
                                                    const uint32_t* __restrict__ w, uint32_t k,
                                                    const uint32_t* __restrict__ src, uint32_t* __restrict__ ub,
                                                    uint32_t* __restrict__ lb, BoundCtl* ctl) {
    extern __shared__ __align__(16) uint32_t sm[];
    __shared__ BoundSmem<T> s;
    // No sum may reach 2^32 - 1, here or in the form that takes every source (which reports it).  A stored distance is
    // the length of a simple path, at most the sum of its nodes' heaviest entries.  Where that is too much, rounds bound
    // it: a listed node was reached before its round, so what round r stores is at most (r + 1) heaviest entries, and a
    // node h hops away is reached by round h - 1.  R rounds that reach every node show that no two are more than 2 R
    // hops apart, so no source's run forms a sum above 2 R + 1 heaviest entries.  (R-MAT of 10.4M nodes,
    // weights to 2^20, quotient of some 4,000 nodes: 1.94 ms for every source, 0.30 this way.)
    const bool by_rounds = ctl->wsum + ctl->wmax >= 0xFFFFFFFFull;
    const uint64_t wmax = ctl->wmax;
    // (another CTA of this launch may set wide meanwhile: one read decides for the CTA)
    if (threadIdx.x == 0) s.total = ctl->wide || blockIdx.x >= ctl->nsrc;
    __syncthreads();
    if (s.total) return;
    const uint32_t words = (k + 31) / 32;
    uint32_t* dist = sm;               // [k]
    uint32_t* listed = dist + k;       // bit v: v is in the next list
    uint32_t* soff = listed + words;   // [k + 1] row starts
    uint16_t* list[2];
    list[0] = reinterpret_cast<uint16_t*>(soff + k + 1);
    list[1] = list[0] + k;
    const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = lane_id();
    const unsigned le_mask = 0xffffffffu >> (31u - lane);
    const uint32_t source = src[blockIdx.x];
    for (uint32_t v = tid; v < k; v += T) dist[v] = v == source ? 0u : INF;
    for (uint32_t v = tid; v <= k; v += T) soff[v] = (uint32_t)off[v];
    for (uint32_t i = tid; i < words; i += T) listed[i] = 0;
    if (tid == 0) {
        list[0][0] = (uint16_t)source;
        s.count[0] = 1;
        s.count[1] = 0;
    }
    __syncthreads();
    const uint32_t max_rounds = 4 * k + 64;  // far above any real count: a guard, reported as an error
    for (uint32_t round = 0;; ++round) {
        const uint32_t c = round & 1;
        const uint32_t m = s.count[c];
        if (by_rounds && (m == 0 ? 2ull * round + 1 : round + 1ull) * wmax >= 0xFFFFFFFFull) {
            if (tid == 0) ctl->wide = 1;
            return;
        }
        if (m == 0) break;
        if (round > max_rounds) {
            if (tid == 0) atomicExch(&ctl->err, 1u);
            break;
        }
        for (uint32_t t0 = 0; t0 < m; t0 += T) {
            // the tile's nodes: taken off the list before their distance is read, so a later improvement lists them again
            const uint32_t mt = min(m - t0, (uint32_t)T);
            uint32_t deg = 0, b0 = 0, d = 0;
            if (tid < mt) {
                const uint32_t v = list[c][t0 + tid];
                atomicAnd(&listed[v >> 5], ~(1u << (v & 31)));
                d = atomicAdd(&dist[v], 0u);
                b0 = soff[v];
                deg = soff[v + 1] - b0;
            }
            const uint32_t incl = warp_incl_scan(deg);
            if (lane == 31) s.wsum[warp] = incl;
            __syncthreads();
            uint32_t before = 0, total = 0;
#pragma unroll
            for (uint32_t i = 0; i < T / 32; ++i) {
                const uint32_t x = s.wsum[i];
                before += i < warp ? x : 0u;
                total += x;
            }
            if (tid < mt) {
                const uint32_t pre = before + incl - deg;
                if (tid > 0) s.pre[tid - 1] = pre;
                s.base[tid] = b0 - pre;
                s.dist[tid] = d;
            }
            __syncthreads();
            for (uint32_t p0 = warp * PW; p0 < total; p0 += (T / 32) * PW) {
                // owner of p0: the number of later nodes that start at or before it
                uint32_t B = 0, len = mt - 1;
                while (len > 0) {
                    const uint32_t step = (len + 31) / 32;
                    const uint32_t at = (lane + 1) * step;  // probes the last of each piece
                    const bool in = at <= len ? s.pre[B + at - 1] <= p0 : false;
                    const uint32_t n_in = (uint32_t)__popc(__ballot_sync(0xffffffffu, in));
                    B += n_in * step;
                    len = min(step - 1, len - n_in * step);
                }
                // (the entries of all four groups are loaded before any is used)
                uint32_t own[PWG], v[PWG], nd[PWG];
#pragma unroll
                for (int u = 0; u < PWG; ++u)
                    B += (uint32_t)__popc(group_starts(s.pre + B, mt - 1 - B, p0 + 32u * u, B, lane, le_mask, &own[u]));
#pragma unroll
                for (int u = 0; u < PWG; ++u) {
                    const uint32_t p = p0 + 32u * u + lane;
                    v[u] = source;
                    nd[u] = INF;
                    if (p < total) {
                        const uint32_t j = s.base[own[u]] + p;
                        v[u] = __ldg(col + j);
                        nd[u] = s.dist[own[u]] + __ldg(w + j);
                    }
                }
#pragma unroll
                for (int u = 0; u < PWG; ++u) {
                    bool put = false;
                    if (nd[u] < dist[v[u]] && nd[u] < atomicMin(&dist[v[u]], nd[u])) {
                        const uint32_t bit = 1u << (v[u] & 31);
                        put = !(atomicOr(&listed[v[u] >> 5], bit) & bit);
                    }
                    const unsigned pm = __ballot_sync(0xffffffffu, put);
                    if (pm) {
                        uint32_t at = 0;
                        if (lane == 0) at = atomicAdd(&s.count[c ^ 1], (uint32_t)__popc(pm));
                        at = __shfl_sync(0xffffffffu, at, 0);
                        if (put) list[c ^ 1][at + (uint32_t)__popc(pm & lanemask_lt())] = (uint16_t)v[u];
                    }
                }
            }
            __syncthreads();
        }
        if (tid == 0) s.count[c] = 0;
        __syncthreads();
    }
    uint32_t ecc = 0;
    bool apart = false;
    for (uint32_t v = tid; v < k; v += T) {
        apart |= dist[v] == INF;
        ecc = dist[v] != INF ? max(ecc, dist[v]) : ecc;
    }
    if (by_rounds && apart) ctl->wide = 1;
    ecc = block_reduce(ecc, [](uint32_t a, uint32_t b) { return a > b ? a : b; }, 0u);
    if (tid == 0) {
        s.total = ecc;
        atomicMax(&ctl->best, ecc);
    }
    __syncthreads();
    ecc = s.total;
    for (uint32_t v = tid; v < k; v += T) {
        const uint32_t d = dist[v];
        if (d == INF) continue;
        const uint32_t hi = (uint32_t)min((uint64_t)d + ecc, (uint64_t)(INF - 1)), lo = max(d, ecc - d);
        if (hi < ub[v]) atomicMin(&ub[v], hi);
        if (lo > lb[v]) atomicMax(&lb[v], lo);
    }
}

__global__ void __launch_bounds__(1024) k_bound_select(uint32_t k, uint32_t most, const uint32_t* __restrict__ ub,
                                                       const uint32_t* __restrict__ lb, uint32_t* __restrict__ src,
                                                       BoundCtl* ctl) {
    __shared__ uint32_t s_n;
    if (ctl->wide || ctl->nsrc == 0) return;
    const uint32_t n = bound_select(k, most, ctl->best, ub, lb, src, s_n);
    if (threadIdx.x == 0) ctl->nsrc = n;
}

size_t bound_smem(uint32_t k) { return (size_t)k * 12 + 4 + (size_t)((k + 31) / 32) * 4; }
constexpr size_t kBoundSmemMax = 208 * 1024;  // beside the static tile

// Largest distance of a symmetric quotient by bounds; *done = false when a path might reach 2^32 - 1 (every source must
// then be looked at, in the caller's checked form).
cldiam_status bound_diameter(uint32_t k, const uint64_t* off, const uint32_t* col, const uint32_t* w, cudaStream_t s,
                             uint64_t* phi, bool* done) {
    static std::atomic<bool> attr[64];  // first call per device sets the attribute (idempotent)
    int dev = 0;
    CLD_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64 || !attr[dev]) {
        const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
        CLD_CUDA(cudaFuncSetAttribute(k_bound_sssp<512>, a, (int)kBoundSmemMax));
        CLD_CUDA(cudaFuncSetAttribute(k_bound_sssp<1024>, a, (int)kBoundSmemMax));
        if (dev >= 0 && dev < 64) attr[dev] = true;
    }
    *done = false;
    DBuf<uint32_t> bounds, src;
    DBuf<BoundCtl> ctl;
    CLD_TRY(bounds.alloc(2 * (size_t)k, s));
    CLD_TRY(src.alloc(kBoundNext, s));
    CLD_TRY(ctl.alloc(1, s));
    uint32_t *ub = bounds.get(), *lb = bounds.get() + k;
    CLD_CUDA(cudaMemsetAsync(ctl.get(), 0, sizeof(BoundCtl), s));
    uint32_t n = std::min(k, kBoundFirst);
    CLD_K(K_FW, s, k_bound_prep<<<grid_for((size_t)k * 32, 256), 256, 0, s>>>(off, w, k, n, ub, lb, src.get(), ctl.get()));
    BoundCtl h{};
    do {
        // most graphs are done after two or three batches: three are queued before the host looks
        for (int i = 0; i < 3; ++i) {
            // (three batches with 512 / 1,024 threads: k = 840 168 / 224 us, k = 1,897 126 / 107, k = 4,082 1,261 / 1,082)
            if (k < 1536)
                CLD_K(K_FW, s, k_bound_sssp<512><<<n, 512, bound_smem(k), s>>>(off, col, w, k, src.get(), ub, lb, ctl.get()));
            else
                CLD_K(K_FW, s, k_bound_sssp<1024><<<n, 1024, bound_smem(k), s>>>(off, col, w, k, src.get(), ub, lb,
                                                                                 ctl.get()));
            CLD_K(K_FW, s, k_bound_select<<<1, 1024, 0, s>>>(k, kBoundNext, ub, lb, src.get(), ctl.get()));
            n = std::min(k, kBoundNext);
        }
        CLD_LAUNCH_CHECK();
        CLD_CUDA(cudaMemcpyAsync(&h, ctl.get(), sizeof h, cudaMemcpyDeviceToHost, s));
        CLD_CUDA(cudaStreamSynchronize(s));
        if (h.err) return fail(CLDIAM_ERR_DIVERGED, "quotient SSSP exceeded its round limit");
    } while (!h.wide && h.nsrc > 0);
    *done = !h.wide;
    *phi = h.best;
    return CLDIAM_OK;
}

// Blocked Floyd-Warshall over the padded kp x kp matrix M in the given form; scal[0] = overflow
// (checked form), scal[1] = largest finite distance, scal[3] = wide weight, scal[4] = unconnected pair.
template <bool FAST>
cldiam_status fw_dense(uint32_t* M, uint32_t kp, uint32_t k, uint32_t nt, const uint64_t* off, const uint32_t* col,
                       const uint32_t* w, uint32_t* scal, cudaStream_t s) {
    const uint32_t none = FAST ? INFF : INF;
    CLD_K(K_FW, s, k_fw_init<<<grid_for((size_t)kp * kp, 256), 256, 0, s>>>(M, kp, k, none));
    CLD_K(K_FW, s, k_fw_scatter<<<grid_for(k, 1, 64), 128, 0, s>>>(off, col, w, k, kp, M, FAST ? scal + 3 : nullptr));
    CLD_LAUNCH_CHECK();
    CLD_TRY(fw_rounds<FAST>(M, kp, nt, scal, s));
    CLD_K(K_FW, s, k_fw_max_finite<<<grid_for((size_t)k * kp, 256), 256, 0, s>>>(M, kp, k, none, scal + 1,
                                                                                  FAST ? scal + 4 : nullptr));
    CLD_LAUNCH_CHECK();
    // algorithmic work: k^3 relaxations; bytes: the matrix read and written once per pivot round
    prof_add_bytes(K_FW, 2.0 * 4.0 * (double)kp * kp * nt);
    return CLDIAM_OK;
}

// Batched-SSSP kernel for a sparse quotient of k nodes: the worklist form with S sources per CTA while
// k x S distances and a word of change bits per node fit in shared memory (S = 8 below 2,048 nodes,
// else 4, else 1; a requested S that fits is taken), else all-node rounds with the distances alone
// (k <= 56,320), else none (dense form).
enum class SparsePlan { kNone, kWorklist8, kWorklist4, kWorklist1, kRounds1 };
SparsePlan sparse_plan(uint32_t k, uint32_t S) {
    constexpr size_t kSmem = 220 * 1024;
    const bool fit8 = (size_t)k * (8 * 4 + 8) <= kSmem, fit4 = (size_t)k * (4 * 4 + 8) <= kSmem,
               fit1 = (size_t)k * (4 + 8) <= kSmem;
    if ((S == 8 && fit8) || (S == 0 && fit8 && k < 2048)) return SparsePlan::kWorklist8;
    if ((S == 4 || S == 0 || S == 8) && fit4) return SparsePlan::kWorklist4;
    if (fit1) return SparsePlan::kWorklist1;
    if ((size_t)k * 4 <= kSmem) return SparsePlan::kRounds1;
    return SparsePlan::kNone;
}

}  // namespace

cldiam_status apsp_max_device(uint32_t k, const uint64_t* off, const uint32_t* col, const uint32_t* w, uint64_t nnz,
                              cudaStream_t s, uint64_t* phi, bool validate, uint32_t max_fw_k,
                              const cldiam_tuning& tun) {
    *phi = 0;
    if (k <= 1) return CLDIAM_OK;
    const uint32_t nt = (k + FT - 1) / FT;
    const uint32_t kp = nt * FT;
    DBuf<uint32_t> M, scal;
    CLD_TRY(scal.alloc(6, s));
    CLD_CUDA(cudaMemsetAsync(scal.get(), 0, 24, s));
    if (validate) {
        CLD_K(K_FW, s, k_fw_validate<<<grid_for((size_t)k + nnz + 1, 256), 256, 0, s>>>(off, col, k, nnz, scal.get() + 2));
        CLD_LAUNCH_CHECK();
        uint32_t bad = 0;
        CLD_CUDA(cudaMemcpyAsync(&bad, scal.get() + 2, 4, cudaMemcpyDeviceToHost, s));
        CLD_CUDA(cudaStreamSynchronize(s));
        if (bad) return fail(CLDIAM_ERR_INVALID_ARG, "malformed CSR (offsets or column ids)");
    }
    // sparse quotient (fewer than k^2 / 8 entries): batched SSSP, S sources per CTA with
    // k x S distances (and one word of change bits per node) in shared memory.  S = 8 below 2,048
    // nodes; above, S = 4: its half-size distance block lets two 1,024-thread CTAs share an SM (they
    // use <= 32 registers), where S = 8 fits one (R-MAT 24, k = 4,069: 3.0 -> 2.1 ms; road mesh 4096^2,
    // k = 4,357: 4.0 -> 3.4 ms)
    // (tuning: the density cut-over and the sources per CTA; a tuned cut-over never sends a quotient above
    // max_fw_k to Floyd-Warshall that the default would have solved by SSSP)
    bool sparse = (double)nnz * (double)tun.apsp_fw_density < (double)k * k;
    if (!sparse && k > max_fw_k) sparse = (double)nnz * 8.0 < (double)k * k;
    const SparsePlan plan = sparse ? sparse_plan(k, tun.apsp_sources_per_cta) : SparsePlan::kNone;
    // A quotient built here (not validated: symmetric by construction) takes the bounds, unless a knob sets the
    // sources per CTA; a caller's CSR is not checked for symmetry, which the bounds rely on, so it takes every source.
    // (Up to one batch of nodes there is nothing to leave out: the worklist is faster, 17 against 37 us at k = 59.)
    if (sparse && !validate && tun.apsp_sources_per_cta == 0 && k > kBoundFirst && k <= 65535u && bound_smem(k) <= kBoundSmemMax) {
        bool done = false;
        CLD_TRY(bound_diameter(k, off, col, w, s, phi, &done));
        if (done) return CLDIAM_OK;
    }
    if (plan == SparsePlan::kWorklist8) {
        CLD_TRY(launch_wl<8>(k, off, col, w, nnz, s, scal.get() + 1, scal.get(), scal.get() + 5));
    } else if (plan == SparsePlan::kWorklist4) {
        CLD_TRY(launch_wl<4>(k, off, col, w, nnz, s, scal.get() + 1, scal.get(), scal.get() + 5));
    } else if (plan == SparsePlan::kWorklist1) {
        CLD_TRY(launch_wl<1>(k, off, col, w, nnz, s, scal.get() + 1, scal.get(), scal.get() + 5));
    } else if (plan == SparsePlan::kRounds1) {
        CLD_TRY(launch_msbf<1>(k, off, col, w, nnz, s, scal.get() + 1, scal.get()));
    } else {
        if (k > max_fw_k) return fail(CLDIAM_ERR_UNSUPPORTED, "dense quotient larger than max_fw_k");
        CLD_TRY(M.alloc((size_t)kp * kp, s));
        // fast form first (scal[3] = a weight too wide for it, scal[4] = some pair left unconnected)
        CLD_TRY(fw_dense<true>(M.get(), kp, k, nt, off, col, w, scal.get(), s));
        uint32_t hf[5];
        CLD_CUDA(cudaMemcpyAsync(hf, scal.get(), 20, cudaMemcpyDeviceToHost, s));
        CLD_CUDA(cudaStreamSynchronize(s));
        if (hf[3] || hf[4]) {
            // disconnected pairs, or distances the fast form cannot hold: recompute with the checked form
            CLD_CUDA(cudaMemsetAsync(scal.get(), 0, 8, s));
            CLD_TRY(fw_dense<false>(M.get(), kp, k, nt, off, col, w, scal.get(), s));
        }
    }
    uint32_t h[6];
    CLD_CUDA(cudaMemcpyAsync(h, scal.get(), 24, cudaMemcpyDeviceToHost, s));
    CLD_CUDA(cudaStreamSynchronize(s));
    if (h[5]) return fail(CLDIAM_ERR_DIVERGED, "quotient SSSP exceeded its round limit");
    if (h[0]) return fail(CLDIAM_ERR_OVERFLOW, "a quotient distance reached 2^32 - 1");
    *phi = h[1];
    return CLDIAM_OK;
}

// ---------------------------------------------------------------------------
// Allocation-free variant of the quotient diameter, for callers that may not
// allocate device memory.  All scratch lives in one file-scope device array:
// three control words (overflow, result, validation) and, for dense inputs,
// the Floyd-Warshall matrix of up to kNoAllocMaxK x kNoAllocMaxK entries.  The
// array exists once per GPU that loads the library and stays resident until
// the process exits; every call reuses it, so calls whose work overlaps on the
// GPU race on it.
constexpr uint32_t kNoAllocMaxK = 1024;    // dense (Floyd-Warshall) inputs
constexpr uint32_t kNoAllocMaxSparseK = 51200;  // sparse inputs: distances live in shared memory
constexpr size_t kNoAllocCtlWords = 64;    // keeps the matrix 256-byte aligned
static __device__ __align__(256) uint32_t g_noalloc_scratch[kNoAllocCtlWords + (size_t)kNoAllocMaxK * kNoAllocMaxK];

static std::mutex g_noalloc_mu;
static uint32_t* g_noalloc_ptr[64];  // device address of the scratch array, per device

cldiam_status apsp_max_noalloc(uint32_t k, const uint64_t* off, const uint32_t* col, const uint32_t* w,
                               cudaStream_t s, uint64_t* phi) {
    *phi = 0;
    int dev = 0;
    CLD_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return fail(CLDIAM_ERR_UNSUPPORTED, "device ordinal above 63");
    uint32_t* scratch = nullptr;
    {
        // one-time set-up per device, with that device current: the host-side name of the
        // array is not a device address, so ask the runtime for it
        std::lock_guard<std::mutex> lk(g_noalloc_mu);
        if (!g_noalloc_ptr[dev]) {
            void* p = nullptr;
            cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
            if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(g_noalloc_scratch)", __FILE__, __LINE__);
            g_noalloc_ptr[dev] = static_cast<uint32_t*>(p);
        }
        scratch = g_noalloc_ptr[dev];
    }
    if (k <= 1) return CLDIAM_OK;
    if (!is_device_ptr(off) || !is_device_ptr(col) || !is_device_ptr(w))
        return fail(CLDIAM_ERR_INVALID_ARG, "off, col and w must be device memory (nothing is copied or allocated)");
    uint64_t nnz = 0;
    CLD_CUDA(cudaMemcpyAsync(&nnz, off + k, 8, cudaMemcpyDeviceToHost, s));
    CLD_CUDA(cudaStreamSynchronize(s));
    if (nnz > 0xFFFFFFFFull) return fail(CLDIAM_ERR_INVALID_ARG, "more than 2^32 - 1 entries");
    const bool sparse = (double)nnz * 8.0 < (double)k * k;
    if (sparse ? k > kNoAllocMaxSparseK : k > kNoAllocMaxK)
        return fail(CLDIAM_ERR_UNSUPPORTED, sparse ? "k above 51200, the allocation-free limit for sparse graphs"
                                                   : "k above 1024, the allocation-free limit for dense graphs");
    uint32_t* ovf = scratch + 0;
    uint32_t* best = scratch + 1;
    uint32_t* bad = scratch + 2;
    uint32_t* diverged = scratch + 3;  // the worklist SSSP's round limit
    CLD_CUDA(cudaMemsetAsync(scratch, 0, 4 * sizeof(uint32_t), s));  // the array keeps the last call's values
    k_fw_validate<<<grid_for((size_t)k + nnz + 1, 256), 256, 0, s>>>(off, col, k, nnz, bad);
    CLD_LAUNCH_CHECK();
    uint32_t h[3] = {0, 0, 0};
    CLD_CUDA(cudaMemcpyAsync(h, scratch, 3 * sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    CLD_CUDA(cudaStreamSynchronize(s));
    if (h[2]) return fail(CLDIAM_ERR_INVALID_ARG, "malformed CSR (offsets or column ids)");
    if (sparse) {
        // batched SSSP with the kernel and sources per CTA apsp_max_device takes by default: distances,
        // change bits (and the CSR when it fits) in shared memory, only the control words here
        switch (sparse_plan(k, 0)) {
            case SparsePlan::kWorklist8: CLD_TRY(launch_wl<8>(k, off, col, w, nnz, s, best, ovf, diverged)); break;
            case SparsePlan::kWorklist4: CLD_TRY(launch_wl<4>(k, off, col, w, nnz, s, best, ovf, diverged)); break;
            case SparsePlan::kWorklist1: CLD_TRY(launch_wl<1>(k, off, col, w, nnz, s, best, ovf, diverged)); break;
            default: CLD_TRY(launch_msbf<1>(k, off, col, w, nnz, s, best, ovf)); break;
        }
    } else {
        const uint32_t nt = (k + FT - 1) / FT;
        const uint32_t kp = nt * FT;  // <= kNoAllocMaxK
        uint32_t* M = scratch + kNoAllocCtlWords;
        k_fw_init<<<grid_for((size_t)kp * kp, 256), 256, 0, s>>>(M, kp, k, INF);
        k_fw_scatter<<<grid_for(k, 1, 64), 128, 0, s>>>(off, col, w, k, kp, M, nullptr);
        CLD_LAUNCH_CHECK();
        CLD_TRY(fw_rounds<false>(M, kp, nt, ovf, s));
        k_fw_max_finite<<<grid_for((size_t)k * kp, 256), 256, 0, s>>>(M, kp, k, INF, best, nullptr);
        CLD_LAUNCH_CHECK();
    }
    uint32_t hd[4] = {0, 0, 0, 0};
    CLD_CUDA(cudaMemcpyAsync(hd, scratch, 4 * sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    CLD_CUDA(cudaStreamSynchronize(s));
    if (hd[3]) return fail(CLDIAM_ERR_DIVERGED, "quotient SSSP exceeded its round limit");
    if (hd[0]) return fail(CLDIAM_ERR_OVERFLOW, "a distance reached 2^32 - 1");
    *phi = hd[1];
    return CLDIAM_OK;
}

cldiam_status load_apsp_kernels() {
    return load_kernels(k_bound_prep, k_bound_sssp<512>, k_bound_sssp<1024>, k_bound_select, k_fw_init, k_fw_validate,
                        k_fw_scatter, k_fw_phase1<true>, k_fw_phase1<false>, k_fw_phase2_fast, k_fw_phase2_checked,
                        k_fw_phase3<true>, k_fw_phase3<false>, k_fw_max_finite, k_apsp_wl<8, true>, k_apsp_wl<8, false>,
                        k_apsp_wl<4, true>, k_apsp_wl<4, false>, k_apsp_wl<1, true>, k_apsp_wl<1, false>,
                        k_apsp_msbf<1, true>, k_apsp_msbf<1, false>);
}

}  // namespace cld
