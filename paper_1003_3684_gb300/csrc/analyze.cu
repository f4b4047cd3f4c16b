// Graph-property checks on generated graphs (Sec. 4 examines the degree
// distribution and path lengths of the generated graphs): vertex degrees,
// their histogram, and breadth-first search distances from a source.
//
// Every result is exact integer work. Degrees and histogram counts are sums
// (atomic order does not change them); BFS distances are unique even though
// the order in which a level's vertices are found depends on the schedule.
#include <cstddef>
#include <cstring>

#include "../../include/pgen.h"
#include "pg_internal.h"
#include "pg_trace.h"

namespace pgen {
namespace {

constexpr uint32_t kBfsWarps = 8;          // warps per CTA of the BFS level kernel
constexpr uint32_t kHistSmem = 8192;   // histograms up to this many buckets count in smem

// A generated list often names one source on several edges in a row, so a
// warp counts equal neighbouring sources first and the first lane of each run
// adds the run's length. Bound by the L2's atomics while the counters (C) stay
// in it, by DRAM sectors read and written back for one count when they don't;
// the sources of a grouped list alone by reading it, which takes two groups of
// edges in flight per warp (2^24 vertices, m = 5: 0.264 -> 0.231 ms; without runs
// 0.248). Six CTAs per SM: with eight, lists of uniform ids lose 3 % by the second
// group.
constexpr int kDegreePlaces = 6;
template <typename Id, typename C>
__global__ void __launch_bounds__(256) degree_kernel(const Id* __restrict__ e, uint64_t M,
                                                     uint64_t N, int which, C* __restrict__ deg)
{
    constexpr int kU = 2;   // groups of 32 edges in flight per warp
    const uint32_t lane = threadIdx.x & 31;
    for (uint64_t i0 = kU * ((uint64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u)); i0 < M;
         i0 += (uint64_t)kU * gridDim.x * blockDim.x) {
        Id s[kU], d[kU];
#pragma unroll
        for (int t = 0; t < kU; ++t) {
            const uint64_t i = i0 + 32 * t + lane;
            s[t] = i < M ? e[2 * i] : 0;
            d[t] = i < M ? e[2 * i + 1] : 0;
        }
#pragma unroll
        for (int t = 0; t < kU; ++t) {
            const bool in = i0 + 32 * t + lane < M;
            if (which != PG_DEG_IN) {
                const Id before = __shfl_up_sync(0xFFFFFFFFu, s[t], 1);
                const uint32_t live = __ballot_sync(0xFFFFFFFFu, in);
                const uint32_t first = __ballot_sync(0xFFFFFFFFu, in && (lane == 0 || before != s[t]));
                if (((first >> lane) & 1u) && s[t] < N) {
                    // up to the next run's first lane, or the last live one
                    const uint32_t above = lane == 31 ? 0u : first >> (lane + 1);
                    const uint32_t len = above ? (uint32_t)__ffs(above) : __popc(live >> lane);
                    atomicAdd(&deg[s[t]], (C)len);
                }
            }
            if (which != PG_DEG_OUT && in && d[t] < N) atomicAdd(&deg[d[t]], (C)1);
        }
    }
}

// Counts of many vertices are taken in 32 bits, in the upper half of the
// result's own memory, so that they fit the L2 (2^24 vertices: 67 MB instead of
// 134), and widened in place: deg[i] covers the counts 2i - N and 2i - N + 1,
// neither above i. So the lower half of what is left can be widened at once,
// its results lie below every count; and a CTA that has read all counts left
// can write them.
constexpr uint64_t kNarrowVertices = 13u << 20;
constexpr uint32_t kWidenLast = 8192;   // results of the last CTA
__global__ void __launch_bounds__(256) widen_kernel(uint64_t* deg, uint64_t N, uint64_t begin,
                                                    uint64_t end)
{
    const uint32_t* cnt = reinterpret_cast<const uint32_t*>(deg) + N;
    const uint64_t i = begin + (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < end) deg[i] = cnt[i];
}
__global__ void __launch_bounds__(1024) widen_last_kernel(uint64_t* deg, uint64_t N, uint64_t begin)
{
    const uint32_t* cnt = reinterpret_cast<const uint32_t*>(deg) + N;
    uint32_t c[kWidenLast / 1024];
#pragma unroll
    for (uint32_t t = 0; t < kWidenLast / 1024; ++t) {
        const uint64_t i = begin + t * 1024 + threadIdx.x;
        c[t] = i < N ? cnt[i] : 0;
    }
    __syncthreads();
#pragma unroll
    for (uint32_t t = 0; t < kWidenLast / 1024; ++t) {
        const uint64_t i = begin + t * 1024 + threadIdx.x;
        if (i < N) deg[i] = c[t];
    }
}

// hist[d] = #{v : deg[v] = d} for d <= max_deg, hist[max_deg + 1] = the rest.
__global__ void __launch_bounds__(256) histogram_kernel(const uint64_t* __restrict__ deg, uint64_t N,
                                                        uint32_t max_deg,
                                                        unsigned long long* __restrict__ hist)
{
    __shared__ uint32_t h[kHistSmem];
    const uint32_t nb = max_deg + 2;
    const bool in_smem = nb <= kHistSmem;
    if (in_smem) {
        for (uint32_t t = threadIdx.x; t < nb; t += blockDim.x) h[t] = 0;
        __syncthreads();
    }
    constexpr int kU = 4;   // degrees in flight per thread
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t v0 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; v0 < N; v0 += kU * stride) {
        uint64_t d[kU];
#pragma unroll
        for (int t = 0; t < kU; ++t) d[t] = v0 + t * stride < N ? deg[v0 + t * stride] : 0;
#pragma unroll
        for (int t = 0; t < kU; ++t) {
            if (v0 + t * stride >= N) break;
            const uint32_t b = d[t] <= max_deg ? (uint32_t)d[t] : max_deg + 1;
            if (in_smem) atomicAdd(&h[b], 1u);
            else atomicAdd(&hist[b], 1ull);
        }
    }
    if (in_smem) {
        __syncthreads();
        for (uint32_t t = threadIdx.x; t < nb; t += blockDim.x)
            if (h[t]) atomicAdd(&hist[t], (unsigned long long)h[t]);
    }
}

// Adjacency entries are read once per search: streaming loads, so that they
// do not push the visited bitmap out of L2.
__device__ __forceinline__ uint64_t load_streaming(const uint32_t* p) { return __ldcs(p); }
__device__ __forceinline__ uint64_t load_streaming(const uint64_t* p)
{
    return __ldcs(reinterpret_cast<const unsigned long long*>(p));
}

// Claims for one step of 32 adjacency entries: lane l holds neighbour u when
// `have`. A neighbour whose bit in the visited bitmap (N bits, small enough
// to stay in L2) is clear is claimed by an atomic OR of that bit; the claimer
// writes its distance. Claimed vertices collect in the warp's buffer (64
// slots, fewer than 32 held between steps) and leave for the next frontier
// 32 at a time, so the frontier's counter takes one atomic per 32 claims (the
// frontier's order is not part of the result).
struct BfsQueue {
    uint32_t* buf;       // this warp's 64 shared-memory slots
    uint32_t held;       // warp-uniform, < 32 between steps
    uint32_t* next;
    uint32_t* nsize;
    uint32_t* dist;
    uint32_t* vis;
    uint32_t level;
    uint64_t N;

    __device__ __forceinline__ void step(bool have, uint32_t u, uint32_t lane, uint32_t lt)
    {
        bool claim = false;
        if (have) {
            const uint32_t bit = 1u << (u & 31);
            // a stale cached word only costs an atomic that finds the bit set
            if ((vis[u >> 5] & bit) == 0) claim = (atomicOr(&vis[u >> 5], bit) & bit) == 0;
        }
        if (claim) dist[u] = level + 1;
        push(claim, u, lane, lt);
    }

    // appends u (where `take`) to the next frontier
    __device__ __forceinline__ void push(bool take, uint32_t u, uint32_t lane, uint32_t lt)
    {
        const uint32_t m = __ballot_sync(0xFFFFFFFFu, take);
        if (take) buf[held + __popc(m & lt)] = u;
        held += __popc(m);
        if (held >= 32) {
            __syncwarp();
            uint32_t at = 0;
            if (lane == 0) at = atomicAdd(nsize, 32u);
            at = __shfl_sync(0xFFFFFFFFu, at, 0);
            if (PG_CHECK(at + lane, N)) next[at + lane] = buf[lane];
            const uint32_t rest = held - 32;
            const uint32_t x = lane < rest ? buf[32 + lane] : 0;
            __syncwarp();
            if (lane < rest) buf[lane] = x;
            __syncwarp();
            held = rest;
        }
    }

    __device__ __forceinline__ void flush(uint32_t lane)
    {
        __syncwarp();
        if (held) {
            uint32_t at = 0;
            if (lane == 0) at = atomicAdd(nsize, held);
            at = __shfl_sync(0xFFFFFFFFu, at, 0);
            if (lane < held && PG_CHECK(at + lane, N)) next[at + lane] = buf[lane];
        }
    }
};

// Slices, and frontier vertices per warp, are short while the frontier is: a
// level is a chain of dependent loads per step of a warp, and few vertices
// must not become many steps of few warps. (2^24 vertices: levels of 7, 96 and
// 3630 frontier vertices took 14, 76 and 96 us with 32 vertices per warp and
// slices of 512 entries.)
constexpr uint32_t kWideFrontier = 1u << 15;
__device__ __forceinline__ uint32_t slice_of(uint32_t fsize)
{
    return fsize < kWideFrontier ? 64u : 512u;
}
// Rows of this many entries or more are cut into slices spread over all warps:
// few in a wide level, whose warps have work enough, and where a list of rows
// that are one slice each costs a search per row (2^22 vertices with 64 neighbours on
// average, a level of all: 4.1 -> 1.7 ms; two-phase graphs, whose narrow levels
// hold the hubs, lose 2 to 4 % by 128 everywhere).
__device__ __forceinline__ uint32_t long_row(uint32_t fsize)
{
    return fsize < (1u << 17) ? 64u : 128u;
}

// What the levels count: the next frontier's vertices, and long rows << 32 |
// their slices. Every warp reads both at a level's end, in one request, as
// thousands of them queue at one place of the L2 (2^20 vertices: 8 us of a
// search's 0.2 ms when bottom-up levels read them one by one).
struct __align__(16) BfsCounts {
    unsigned long long longs;
    uint32_t size, pad;
    __device__ __forceinline__ BfsCounts now() const
    {
        const uint4 x = __ldcg(reinterpret_cast<const uint4*>(this));
        return BfsCounts{(unsigned long long)x.y << 32 | x.x, x.z, 0};
    }
};

// Counters of a search, in its workspace. The counts have a slot per level mod
// 4: a slot is cleared a level before its use, three levels after its last
// reader passed a barrier.
struct BfsState {
    BfsCounts counts[4];
    unsigned long long scanned;
    uint32_t arrived, error;       // grid barrier: arrivals so far, a wait that gave up
    uint32_t level, fsize, cur, pad;
    unsigned long long visited;
};
static_assert(sizeof(BfsState) <= 256, "the counters' region of the workspace");

// One step of two adjacency entries per lane, both loads in flight.
template <typename F>
__device__ __forceinline__ void bfs_claim_two(BfsQueue& Q, uint64_t N, uint32_t lane, uint32_t lt,
                                              F&& entry)
{
    uint64_t u[2];
    bool have[2];
#pragma unroll
    for (int t = 0; t < 2; ++t) have[t] = entry(t, u[t]) && u[t] < N;
#pragma unroll
    for (int t = 0; t < 2; ++t) Q.step(have[t], (uint32_t)u[t], lane, lt);
}

// A top-down level's short rows. Each warp takes `chunk` (1 to 32) frontier
// vertices at a time and walks their rows as one concatenated range, 64
// adjacency entries per step: a lane finds the vertex owning an entry by a
// binary search over the rows' starts (a warp scan of their degrees, kept in
// shared memory), so short rows (most rows of a power-law graph) do not leave
// lanes idle. A long row is appended to the long-row list instead: one 64-bit
// atomic on long_ctr adds 1 to the row count (high word) and its slice count
// to the slice total (low word), so the slice bases of the list ascend with
// its index.
template <typename Id>
__device__ __forceinline__ void bfs_short_rows(const uint64_t* __restrict__ row_ptr,
                                               const Id* __restrict__ col,
                                               const uint32_t* frontier, uint32_t fsize,
                                               uint32_t ctas, BfsQueue& Q, uint64_t* st, uint64_t* rw,
                                               unsigned long long* long_ctr, uint32_t* long_v,
                                               uint32_t* long_base)
{
    const uint64_t N = Q.N;
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t lt = (1u << lane) - 1u;
    const uint64_t warps = (uint64_t)ctas * kBfsWarps;
    const uint64_t warp = (uint64_t)blockIdx.x * kBfsWarps + (threadIdx.x >> 5);
    const uint32_t slice = slice_of(fsize);
    uint64_t chunk = (fsize + warps - 1) / warps;
    if (chunk > 32) chunk = 32;
    for (uint64_t c = warp * chunk; c < fsize; c += warps * chunk) {
        uint64_t a = 0, d = 0;
        if (lane < chunk && c + lane < fsize) {
            const uint32_t v = __ldcg(frontier + c + lane);
            if (PG_CHECK(v, N)) {
                a = row_ptr[v];
                d = row_ptr[v + 1] - a;
                if (d >= long_row(fsize)) {
                    const uint64_t ns = (d + slice - 1) / slice;
                    const unsigned long long old = atomicAdd(long_ctr, (1ull << 32) | ns);
                    const uint32_t r = (uint32_t)(old >> 32);
                    if (PG_CHECK(r, N)) {
                        long_v[r] = v;
                        long_base[r] = (uint32_t)old;
                    }
                    d = 0;
                }
            }
        }
        // inclusive scan of the short rows' lengths over the warp
        uint64_t incl = d;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint64_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= (uint32_t)o) incl += y;
        }
        const uint64_t total = __shfl_sync(0xFFFFFFFFu, incl, 31);
        st[lane] = incl - d;
        rw[lane] = a;
        __syncwarp();
        for (uint64_t base = 0; base < total; base += 64)
            bfs_claim_two(Q, N, lane, lt, [&](int t, uint64_t& u) {
                const uint64_t k = base + 32 * t + lane;
                if (k >= total) return false;
                // the last row whose start is at or below k owns entry k (an
                // empty row starts where the next one does)
                uint32_t o = 0;
#pragma unroll
                for (uint32_t step = 16; step > 0; step >>= 1)
                    if (st[o + step] <= k) o += step;
                u = load_streaming(col + rw[o] + (k - st[o]));
                return true;
            });
        __syncwarp();   // the next chunk rewrites the row tables
    }
}

// Slice t of a level's long rows: the `slice` entries from (t - long_base[r]) *
// slice on of row r without its first `skip` ones, r the last row whose base is
// at or below t. A warp finds r by a 32-way search (each round the lanes test
// 32 evenly spaced bases and a ballot keeps the interval below the first base
// above t). The list's first search rounds are the same for all warps and are
// served by the L1 (read past it, a graph of 2^20 vertices and 16 edges each: 0.46
// -> 0.48 ms per search).
struct BfsSlice {
    uint32_t v;
    uint64_t e0, e1;
};
__device__ __forceinline__ BfsSlice bfs_slice(const uint64_t* __restrict__ row_ptr, uint64_t N,
                                              uint32_t t, uint32_t rows, uint32_t skip,
                                              uint32_t slice, const uint32_t* long_v,
                                              const uint32_t* long_base)
{
    const uint32_t lane = threadIdx.x & 31;
    uint32_t lo = 0, n = rows;   // r lies in [lo, lo + n); long_base[lo] <= t
    while (n > 1) {
        const uint32_t step = (n + 31) / 32;
        const uint32_t off = lane * step;
        const bool le = off < n && PG_CHECK(lo + off, rows) && long_base[lo + off] <= t;
        const uint32_t m = __ballot_sync(0xFFFFFFFFu, le);   // lane 0 always set
        const uint32_t k = 31 - __clz(m);
        lo += k * step;
        n = (n - k * step < step) ? n - k * step : step;
    }
    BfsSlice s{0, 0, 0};
    if (PG_CHECK(lo, rows)) {
        s.v = long_v[lo];
        if (PG_CHECK(s.v, N)) {
            const uint64_t a = row_ptr[s.v] + skip, end = row_ptr[s.v + 1];
            s.e0 = a + (uint64_t)(t - long_base[lo]) * slice;
            s.e1 = (s.e0 + slice < end) ? s.e0 + slice : end;
            if (s.e0 > s.e1) s.e0 = s.e1;
        }
    }
    return s;
}

// A top-down level's long rows. Warps take slices t = warp, warp + warps, ...
template <typename Id>
__device__ __forceinline__ void bfs_long_rows(const uint64_t* __restrict__ row_ptr,
                                              const Id* __restrict__ col, uint32_t ctas,
                                              BfsQueue& Q, unsigned long long ctr, uint32_t slice,
                                              const uint32_t* long_v, const uint32_t* long_base)
{
    const uint64_t N = Q.N;
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t lt = (1u << lane) - 1u;
    const uint32_t rows = (uint32_t)(ctr >> 32), slices = (uint32_t)ctr;
    const uint32_t warps = ctas * kBfsWarps;
    for (uint32_t t = blockIdx.x * kBfsWarps + (threadIdx.x >> 5); t < slices; t += warps) {
        const BfsSlice s = bfs_slice(row_ptr, N, t, rows, 0, slice, long_v, long_base);
        for (uint64_t e = s.e0; e < s.e1; e += 64)
            bfs_claim_two(Q, N, lane, lt, [&](int k, uint64_t& u) {
                if (e + 32 * k + lane >= s.e1) return false;
                u = load_streaming(col + e + 32 * k + lane);
                return true;
            });
    }
}

// Top-down levels from the state's on, in one cooperative launch with a
// grid barrier between levels instead of a launch and a host round trip (a
// level of a small frontier is a few microseconds of latency): until the
// frontier is empty, or until bottom-up would be chosen on an undirected
// graph (never for the first level). Leaves where it stopped in the state. The
// first `few` CTAs do it all unless the rows have `dense` entries on average.
template <typename Id>
__global__ void __launch_bounds__(kBfsWarps * 32, 8) bfs_top_down_kernel(
    const uint64_t* __restrict__ row_ptr, const Id* __restrict__ col, uint32_t* f0, uint32_t* f1,
    uint32_t undirected, uint32_t* dist, uint32_t* vis, uint64_t N, uint32_t* long_v,
    uint32_t* long_base, BfsState* state, uint32_t few, uint32_t dense, BarrierLimits barrier)
{
    const uint32_t ctas = few < gridDim.x && row_ptr[N] < dense * N ? few : gridDim.x;
    if (blockIdx.x >= ctas) return;
    __shared__ uint32_t wbuf[kBfsWarps][64];
    __shared__ uint64_t wstart[kBfsWarps][32];   // the rows' starts in the concatenation
    __shared__ uint64_t wrow[kBfsWarps][32];     // and in col
    const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t epoch = 0, cur = state->cur, fsize = state->fsize, level = state->level;
    uint64_t visited = state->visited;
    for (bool first = true; fsize > 0; first = false) {
        if (visited >= N) {   // nothing left to find: the last level is empty
            fsize = 0;
            ++level;
            break;
        }
        if (!first && undirected && (uint64_t)fsize * 30 > N - visited) break;
        uint32_t* frontier = cur ? f1 : f0;
        uint32_t* next = cur ? f0 : f1;
        const uint32_t slot = level & 3, after = (level + 1) & 3;
        if (blockIdx.x == 0 && threadIdx.x == 0) state->counts[after] = BfsCounts{0, 0, 0};
        BfsCounts* counts = &state->counts[slot];
        BfsQueue Q{wbuf[wid], 0, next, &counts->size, dist, vis, level, N};
        bfs_short_rows(row_ptr, col, frontier, fsize, ctas, Q, wstart[wid], wrow[wid],
                       &counts->longs, long_v, long_base);
        Q.flush(lane);
        if (!grid_barrier(&state->arrived, &state->error, barrier, epoch, ctas)) return;
        BfsCounts c = counts->now();
        if (c.longs) {   // the same in every CTA
            Q.held = 0;
            bfs_long_rows(row_ptr, col, ctas, Q, c.longs, slice_of(fsize), long_v, long_base);
            Q.flush(lane);
            if (!grid_barrier(&state->arrived, &state->error, barrier, epoch, ctas)) return;
            c = counts->now();
        }
        fsize = c.size;
        visited += fsize;
        cur ^= 1;
        ++level;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        state->level = level;
        state->fsize = fsize;
        state->cur = cur;
        state->visited = visited;
    }
}

// The frontier of `level` as a bitmap, from the distances.
__device__ __forceinline__ void bfs_bitmap(const uint32_t* dist, uint32_t level, uint64_t N,
                                           uint32_t* bits)
{
    constexpr int kU = 8;   // words in flight per warp
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x >> 5);
    for (uint64_t b = (((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * (32 * kU); b < N;
         b += warps * (32 * kU)) {
        uint32_t d[kU], mine = 0;
#pragma unroll
        for (int t = 0; t < kU; ++t) {
            const uint64_t v = b + 32 * t + lane;
            d[t] = v < N ? dist[v] : 0xFFFFFFFFu;
        }
#pragma unroll
        for (int t = 0; t < kU; ++t) {
            const uint32_t m = __ballot_sync(0xFFFFFFFFu, d[t] == level);
            if (lane == (uint32_t)t) mine = m;
        }
        if (lane < kU && b + 32 * lane < N) bits[(b >> 5) + lane] = mine;
    }
}

// The vertices of a bitmap as a list (in any order), *count of them.
__device__ __forceinline__ void bfs_list(const uint32_t* bits, uint64_t N, uint32_t* list,
                                         uint32_t* count)
{
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t words = (N + 31) / 32, stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t w0 = (uint64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); w0 < words;
         w0 += stride) {
        const uint64_t w = w0 + lane;
        uint32_t m = w < words ? bits[w] : 0u;
        uint32_t incl = __popc(m);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= (uint32_t)o) incl += y;
        }
        uint32_t at = 0;
        if (lane == 31 && incl) at = atomicAdd(count, incl);
        at = __shfl_sync(0xFFFFFFFFu, at, 31) + incl - __popc(m);
        for (; m; m &= m - 1, ++at)
            if (PG_CHECK(at, N)) list[at] = (uint32_t)(w * 32 + __ffs(m) - 1);
    }
}

// One level bottom-up (Beamer, Asanovic and Patterson, "Direction-
// Optimizing Breadth-First Search", SC'12), for a symmetric CSR: every vertex
// not yet visited looks through its row for a neighbour in the frontier and,
// at the first one, takes distance level + 1. The frontier is a bitmap (2 MB
// for 2^24 vertices, in L2, where the distances, 64 MB, miss: the widest level
// of 2^24 vertices took 0.64-0.87 ms with those, 0.33-0.56 now, bound by the
// L2's sectors). A warp owns the 32 vertices of a word: one visited word and
// one word of the next frontier's bitmap, written with plain stores, as no
// other warp writes them during the level. It looks at eight words at once, so
// that late levels, whose words are full, cost no wait per word; the words are
// a grid stride apart, since neighbouring ids share hubs (eight neighbouring
// words: 0.95 ms). A lane reads at most kWalk entries; most rows are shorter or
// have their neighbour among those. The others go to a list, as long rows do
// top-down, and are read in slices by all warps: a hub of another component, of
// 2^22 entries, held its level up for 0.48 s, and larger ones would have let the
// barrier's wait give up.
constexpr uint32_t kWalk = 256, kWalkSlice = 2048;
template <typename Id>
__device__ __forceinline__ void bfs_bottom_up_level(
    const uint64_t* __restrict__ row_ptr, const Id* __restrict__ col, const uint32_t* front,
    uint32_t* next, BfsCounts* counts, uint32_t* dist, uint32_t* vis, uint32_t level, uint64_t N,
    uint32_t* long_v, uint32_t* long_base)
{
    constexpr uint32_t kWords = 8;
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t words = (N + 31) / 32;
    const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x >> 5);
    uint32_t found_all = 0;
    for (uint64_t w0 = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w0 < words;
         w0 += warps * kWords) {
        // lane t < kWords keeps word w0 + t * warps (neighbouring vertices, hubs
        // among them, go to different warps); past the last vertex every bit
        // is set
        const uint64_t my_w = w0 + lane * warps;
        const bool has = lane < kWords && my_w < words;
        uint32_t mine = 0xFFFFFFFFu, out = 0;
        if (has) {
            mine = vis[my_w];
            const uint64_t left = N - my_w * 32;
            if (left < 32) mine |= ~0u << left;
        }
        uint32_t todo = __ballot_sync(0xFFFFFFFFu, mine != 0xFFFFFFFFu);
        for (; todo; todo &= todo - 1) {
            const uint32_t t = __ffs(todo) - 1;
            const uint32_t word = __shfl_sync(0xFFFFFFFFu, mine, t);
            const uint64_t v = (w0 + t * warps) * 32 + lane;
            bool found = false;
            if (((word >> lane) & 1u) == 0) {
                const Id* at = col + row_ptr[v];
                const uint64_t len = row_ptr[v + 1] - row_ptr[v];
                const bool more = len > kWalk;
                for (uint32_t left = more ? kWalk : (uint32_t)len; left > 0; --left, ++at) {
                    const uint64_t u = __ldg(at);
                    if (u < N && ((front[u >> 5] >> (u & 31)) & 1u)) {
                        found = true;
                        break;
                    }
                }
                if (!found && more) {
                    const uint64_t rest = row_ptr[v + 1] - row_ptr[v] - kWalk;
                    const uint64_t ns = (rest + kWalkSlice - 1) / kWalkSlice;
                    const unsigned long long old = atomicAdd(&counts->longs, (1ull << 32) | ns);
                    const uint32_t r = (uint32_t)(old >> 32);
                    if (PG_CHECK(r, N)) {
                        long_v[r] = (uint32_t)v;
                        long_base[r] = (uint32_t)old;
                    }
                }
            }
            const uint32_t m = __ballot_sync(0xFFFFFFFFu, found);
            if (found) dist[v] = level + 1;
            if (lane == t) out = m;
            found_all += __popc(m);
        }
        if (has) {
            next[my_w] = out;
            if (out) vis[my_w] = mine | out;
        }
    }
    if (lane == 0 && found_all) atomicAdd(&counts->size, found_all);
}

// The rest of the listed rows, a slice per warp at a time. The first neighbour
// found in the frontier claims the vertex; slices of a claimed one are left out.
template <typename Id>
__device__ __forceinline__ void bfs_bottom_up_long(
    const uint64_t* __restrict__ row_ptr, const Id* __restrict__ col, const uint32_t* front,
    uint32_t* next, BfsCounts* counts, uint32_t* dist, uint32_t* vis, uint32_t level, uint64_t N,
    unsigned long long ctr, const uint32_t* long_v, const uint32_t* long_base)
{
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t rows = (uint32_t)(ctr >> 32), slices = (uint32_t)ctr;
    const uint32_t warps = gridDim.x * kBfsWarps;
    for (uint32_t t = blockIdx.x * kBfsWarps + (threadIdx.x >> 5); t < slices; t += warps) {
        const BfsSlice s = bfs_slice(row_ptr, N, t, rows, kWalk, kWalkSlice, long_v, long_base);
        const uint32_t word = s.v >> 5, bit = 1u << (s.v & 31);
        // one lane's view, as another warp may claim it meanwhile
        if (__shfl_sync(0xFFFFFFFFu, lane == 0 ? __ldcg(vis + word) : 0u, 0) & bit) continue;
        for (uint64_t e = s.e0; e < s.e1; e += 64) {
            bool hit = false;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const uint64_t at = e + 32 * k + lane;
                const uint64_t u = at < s.e1 ? (uint64_t)load_streaming(col + at) : N;
                hit |= u < N && ((front[u >> 5] >> (u & 31)) & 1u);
            }
            if (!__any_sync(0xFFFFFFFFu, hit)) continue;
            if (lane == 0 && (atomicOr(&vis[word], bit) & bit) == 0) {
                atomicOr(&next[word], bit);
                dist[s.v] = level + 1;
                atomicAdd(&counts->size, 1u);
            }
            break;
        }
    }
}

// Bottom-up levels from the state's on, as the top-down kernel runs its: from
// the frontier's bitmap until the frontier is empty, or until it is under 1/24
// of all vertices; then its vertices go back to a list.
template <typename Id>
__global__ void __launch_bounds__(kBfsWarps * 32, 8) bfs_bottom_up_kernel(
    const uint64_t* __restrict__ row_ptr, const Id* __restrict__ col, uint32_t* front, uint32_t* next,
    uint32_t* list, uint32_t* long_base, uint32_t* dist, uint32_t* vis, uint64_t N, BfsState* state,
    BarrierLimits barrier)
{
    uint32_t epoch = 0, fsize = state->fsize, level = state->level;
    uint64_t visited = state->visited;
    if (fsize == 0) return;   // the search is over
    bfs_bitmap(dist, level, N, front);
    if (!grid_barrier(&state->arrived, &state->error, barrier, epoch)) return;
    do {
        BfsCounts* counts = &state->counts[level & 3];
        if (blockIdx.x == 0 && threadIdx.x == 0) state->counts[(level + 1) & 3] = BfsCounts{0, 0, 0};
        bfs_bottom_up_level(row_ptr, col, front, next, counts, dist, vis, level, N, list, long_base);
        if (!grid_barrier(&state->arrived, &state->error, barrier, epoch)) return;
        BfsCounts c = counts->now();
        if (c.longs) {   // the same in every CTA
            bfs_bottom_up_long(row_ptr, col, front, next, counts, dist, vis, level, N, c.longs, list,
                               long_base);
            if (!grid_barrier(&state->arrived, &state->error, barrier, epoch)) return;
            c = counts->now();
        }
        fsize = c.size;
        visited += fsize;
        ++level;
        uint32_t* f = front;
        front = next;
        next = f;
        if (fsize > 0 && visited >= N) {   // the last level finds nothing
            fsize = 0;
            ++level;
        }
    } while (fsize > 0 && (uint64_t)fsize * 24 >= N);
    if (fsize > 0) bfs_list(front, N, list, &state->counts[level & 3].size);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        state->level = level;
        state->fsize = fsize;
        state->cur = 0;
        state->visited = visited;
    }
}

// scanned = the sum of the reached vertices' row lengths (what a top-down
// search reads, whichever direction each level ran), once the search is over.
__global__ void __launch_bounds__(256) bfs_reach_kernel(const uint64_t* __restrict__ row_ptr,
                                                        const uint32_t* __restrict__ dist,
                                                        uint64_t N, BfsState* __restrict__ state)
{
    if (state->fsize > 0) return;
    unsigned long long* scanned = &state->scanned;
    constexpr int kU = 4;   // vertices in flight per thread
    unsigned long long sum = 0;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t v0 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; v0 < N; v0 += kU * stride) {
        uint64_t a[kU], b[kU];
        uint32_t d[kU];
#pragma unroll
        for (int t = 0; t < kU; ++t) {
            const uint64_t v = v0 + t * stride < N ? v0 + t * stride : N - 1;
            d[t] = v0 + t * stride < N ? dist[v] : 0xFFFFFFFFu;
            a[t] = row_ptr[v];
            b[t] = row_ptr[v + 1];
        }
#pragma unroll
        for (int t = 0; t < kU; ++t)
            if (d[t] != 0xFFFFFFFFu) sum += b[t] - a[t];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_down_sync(0xFFFFFFFFu, sum, o);
    if ((threadIdx.x & 31) == 0 && sum) atomicAdd(scanned, sum);
}

__global__ void bfs_seed_kernel(uint32_t* dist, uint32_t* vis, uint32_t* frontier, BfsState* state,
                                uint32_t source)
{
    dist[source] = 0;
    vis[source >> 5] = 1u << (source & 31);
    frontier[0] = source;
    state->fsize = 1;   // of zeroed counters
    state->visited = 1;
}

bool aligned(const void* p, size_t a) { return ((uintptr_t)p & (a - 1)) == 0; }

int grid_cap(uint64_t items)
{
    const uint64_t full = (uint64_t)device_sm_count() * 8;
    const uint64_t need = (items + 255) / 256;
    return (int)(need < 1 ? 1 : (need < full ? need : full));
}

// Every CTA of a cooperative launch resident, and no more of them than the
// graph can use. The counters and the barrier start at zero.
template <typename F>
cudaError_t launch_levels(F* kernel, uint64_t N, uint32_t per_cta, int most, void** args,
                          BfsState* state, cudaStream_t s)
{
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kBfsWarps * 32, 0);
    if (e != cudaSuccess) return e;
    if (per_sm > most) per_sm = most;
    const uint64_t full = (uint64_t)device_sm_count() * (per_sm > 0 ? per_sm : 1);
    const uint64_t want = (N + per_cta - 1) / per_cta;
    const unsigned grid = (unsigned)(want < full ? want : full);
    // scanned, error and where the search stands are kept
    e = cudaMemsetAsync(state, 0, offsetof(BfsState, scanned), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(&state->arrived, 0, 4, s);
    if (e != cudaSuccess) return e;
    e = cudaLaunchCooperativeKernel((const void*)kernel, dim3(grid), dim3(kBfsWarps * 32), args, 0, s);
    note_launch();
    return e;
}

// The buffers of a search; bottom-up levels keep their bitmaps in the place of
// the long-row list of top-down ones.
struct BfsBuffers {
    uint32_t *fr[2], *dist, *vis, *long_v, *long_base;
    BfsState* state;
};

template <typename Id>
cudaError_t launch_top_down(const uint64_t* row_ptr, const Id* col, BfsBuffers W, uint32_t undirected,
                            uint64_t N, cudaStream_t s)
{
    // CTAs per SM: few where levels are short, as a barrier of 608 costs less than
    // one of 1216 (2^20 vertices 0.350 -> 0.237 ms per search), more where wide levels
    // run top-down, and all that fit where those read many entries per vertex
    // (Kronecker graphs of 16 edges per vertex, four / six / eight per SM, ms: 2^20
    // vertices 0.46 / 0.42 / 0.44, 2^22 1.30 / 1.10 / 1.02, 2^23 - / 1.82 / 1.66;
    // uniform ones of 2: 2^24 - / 2.38 / 2.51, 2^25 - / 4.69 / 4.88). Undirected
    // searches leave the wide levels to the other kernel, most of them (2^23 vertices,
    // four / six: Kronecker 0.82 / 0.74, two-phase 0.52 / 0.56).
    const bool large = N > (5u << 20);
    const int most = undirected ? (large ? 6 : 4) : N <= (5u << 18) ? 4 : large ? 8 : 6;
    uint32_t few = (uint32_t)device_sm_count() * (undirected ? 4 : 6), dense = undirected ? 24 : 8;
    BarrierLimits barrier = barrier_limits();
    void* args[] = {&row_ptr,  &col,         &W.fr[0], &W.fr[1], &undirected, &W.dist, &W.vis, &N,
                    &W.long_v, &W.long_base, &W.state, &few,     &dense,      &barrier};
    return launch_levels(bfs_top_down_kernel<Id>, N, 64, most, args, W.state, s);
}

template <typename Id>
cudaError_t launch_bottom_up(const uint64_t* row_ptr, const Id* col, BfsBuffers W, uint64_t N,
                             cudaStream_t s)
{
    TraceScope trace("bfs_bottom_up", s);
    BarrierLimits barrier = barrier_limits();
    // the frontier lists are free meanwhile: they take the level's long rows
    void* args[] = {&row_ptr, &col,    &W.long_v, &W.long_base, &W.fr[0], &W.fr[1],
                    &W.dist,  &W.vis,  &N,        &W.state,     &barrier};
    // six CTAs per SM up to five million vertices (2^20: 0.219 -> 0.191 ms per
    // search, 2^21 0.252 -> 0.234, 2^22 0.365 -> 0.357), where a barrier and the
    // slowest CTA weigh more than the loads in flight; eight above (2^23: 0.551
    // against 0.567)
    return launch_levels(bfs_bottom_up_kernel<Id>, N, 256, N <= (5u << 20) ? 6 : 8, args, W.state, s);
}

// The search from the seeded state on. A round is a run of top-down levels, on
// an undirected graph a run of bottom-up ones, and the count of what was
// scanned, which each find from the state what is left to do, and one read of
// the state by the host; most searches take one round (a read per run and per
// bottom-up level before; 2^24 vertices, undirected, per search: 0.933 -> 0.900 ms,
// 160,000: 0.195 -> 0.142, 8000: 0.161 -> 0.099).
// Direction of a level (Beamer et al.'s rule with vertex counts standing in for
// edge counts): bottom-up once the frontier is more than 1/30 of the vertices
// not yet visited, top-down again once it is under 1/24 of all.
template <typename Id>
pg_status search(const uint64_t* row_ptr, const Id* col, const BfsBuffers& W, uint32_t undirected,
                 uint64_t N, BfsState& h, cudaStream_t s)
{
    TraceScope trace("bfs", s);
    bool bottom_up = undirected && 30 > N - 1;
    do {
        if (!bottom_up && launch_top_down(row_ptr, col, W, undirected, N, s) != cudaSuccess)
            return PG_ECUDA;
        if (undirected && launch_bottom_up(row_ptr, col, W, N, s) != cudaSuccess) return PG_ECUDA;
        bottom_up = false;
        { bfs_reach_kernel<<<grid_cap(N), 256, 0, s>>>(row_ptr, W.dist, N, W.state); note_launch(); }
        if (cudaMemcpyAsync(&h, W.state, sizeof(h), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess)
            return PG_ECUDA;
        if (h.error) return PG_ETIMEOUT;
    } while (h.fsize > 0);
    return PG_OK;
}

}  // namespace

PG_CHECK_UNIT(analyze)

}  // namespace pgen

using namespace pgen;

extern "C" {

pg_status pg_degrees(const void* d_edges, uint64_t n_edges, uint64_t n_vertices, pg_idwidth w,
                     int which, uint64_t* d_deg, void* stream)
{
    if (w != PG_ID32 && w != PG_ID64) return PG_EINVAL;
    if (which != PG_DEG_OUT && which != PG_DEG_IN && which != PG_DEG_TOTAL) return PG_EINVAL;
    if (n_vertices > 0 && !d_deg) return PG_EINVAL;
    if (n_edges > 0 && !d_edges) return PG_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    // 32-bit counts where no count can reach 2^32 and 64-bit ones would nearly
    // fill the L2 (a list by two-phase attachment, of Kronecker and of uniform
    // cells: 15 million vertices 0.74 -> 0.62, 3.05 -> 2.60 and 3.29 -> 1.34 ms, 2^24
    // vertices 0.88 -> 0.70, 3.82 -> 3.71 and 4.28 -> 1.52; 11 million 0.47 -> 0.48, 2.17
    // -> 2.05 and 1.48 -> 1.00; fewer lose). One end alone gains less, and the sources
    // of a grouped list lose. Few edges don't pay for the widening: half an edge
    // per vertex gains on 2^24 vertices (uniform and grouped: 0.31 -> 0.20 and 0.22
    // -> 0.17 ms) but not in a grouped list on 2^28 (6.73 -> 6.83), and 1000 edges
    // on 2^24 took 0.114 ms instead of 0.035.
    const bool narrow = n_vertices >= kNarrowVertices && which == PG_DEG_TOTAL &&
                        n_edges >= n_vertices - n_vertices / 4 && n_edges < (1ull << 31);
    uint32_t* cnt = reinterpret_cast<uint32_t*>(d_deg) + n_vertices;
    if (n_vertices > 0 && (narrow ? cudaMemsetAsync(cnt, 0, n_vertices * 4, s)
                                  : cudaMemsetAsync(d_deg, 0, n_vertices * 8, s)) != cudaSuccess)
        return PG_ECUDA;
    if (n_edges == 0) return PG_OK;
    TraceScope trace("degrees", s);
    const int full = device_sm_count() * kDegreePlaces, need = grid_cap(n_edges);
    const int grid = need < full ? need : full;
    auto count = [&](auto id, auto* deg) {
        using Id = decltype(id);
        { degree_kernel<Id><<<grid, 256, 0, s>>>((const Id*)d_edges, n_edges, n_vertices, which, deg); note_launch(); }
    };
    auto count_in = [&](auto* deg) {
        if (w == PG_ID64) count(uint64_t{}, deg);
        else count(uint32_t{}, deg);
    };
    if (narrow) count_in(cnt);
    else count_in((unsigned long long*)d_deg);
    if (narrow) {
        uint64_t begin = 0;
        while (n_vertices - begin > kWidenLast) {
            const uint64_t end = begin + (n_vertices - begin) / 2;
            { widen_kernel<<<(unsigned)((end - begin + 255) / 256), 256, 0, s>>>(d_deg, n_vertices, begin, end); note_launch(); }
            begin = end;
        }
        { widen_last_kernel<<<1, 1024, 0, s>>>(d_deg, n_vertices, begin); note_launch(); }
    }
    return cudaGetLastError() == cudaSuccess ? PG_OK : PG_ECUDA;
}

pg_status pg_degree_histogram(const uint64_t* d_deg, uint64_t n_vertices, uint32_t max_degree,
                              uint64_t* d_hist, void* stream)
{
    if (!d_hist || (n_vertices > 0 && !d_deg) || max_degree > 0xFFFFFFF0u) return PG_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    if (cudaMemsetAsync(d_hist, 0, ((size_t)max_degree + 2) * 8, s) != cudaSuccess) return PG_ECUDA;
    if (n_vertices == 0) return PG_OK;
    TraceScope trace("degree_histogram", s);
    { histogram_kernel<<<grid_cap(n_vertices), 256, 0, s>>>(d_deg, n_vertices, max_degree,
                                                         (unsigned long long*)d_hist); note_launch(); }
    return cudaGetLastError() == cudaSuccess ? PG_OK : PG_ECUDA;
}

size_t pg_bfs_workspace_size(uint64_t n_vertices)
{
    // two frontiers of n_vertices uint32, the counters, the visited bitmap,
    // and the long-row list (a vertex and a slice base per row)
    return 4 * (((size_t)n_vertices * 4 + 255) & ~(size_t)255) + 256 +
           ((((size_t)n_vertices + 31) / 32 * 4 + 255) & ~(size_t)255);
}

pg_status pg_bfs(const uint64_t* d_row_ptr, const void* d_col, uint64_t n_vertices, pg_idwidth w,
                 uint64_t source, uint32_t flags, uint32_t* d_dist, void* d_ws, size_t ws_bytes,
                 uint32_t* levels_out, uint64_t* scanned_out, void* stream)
{
    if (w != PG_ID32 && w != PG_ID64) return PG_EINVAL;
    if (flags & ~(uint32_t)PG_BFS_UNDIRECTED) return PG_EINVAL;
    if (n_vertices == 0 || n_vertices >= 0xFFFFFFFFull || source >= n_vertices) return PG_EINVAL;
    if (!d_row_ptr || !d_col || !d_dist || !d_ws || !aligned(d_ws, 256)) return PG_EINVAL;
    if (ws_bytes < pg_bfs_workspace_size(n_vertices)) return PG_ENOMEM;
    cudaStream_t s = (cudaStream_t)stream;
    const size_t fbytes = ((size_t)n_vertices * 4 + 255) & ~(size_t)255;
    unsigned char* ws = (unsigned char*)d_ws;
    uint32_t* fr[2] = {(uint32_t*)ws, (uint32_t*)(ws + fbytes)};
    BfsState* state = (BfsState*)(ws + 2 * fbytes);
    uint32_t* vis = (uint32_t*)(ws + 2 * fbytes + 256);
    const size_t vbytes = ((size_t)n_vertices + 31) / 32 * 4;
    unsigned char* lists = ws + 2 * fbytes + 256 + ((vbytes + 255) & ~(size_t)255);
    // the long-row list of top-down levels; bottom-up ones keep the frontier's
    // and the next frontier's bitmaps there
    uint32_t* long_v = (uint32_t*)lists;
    uint32_t* long_base = (uint32_t*)(lists + fbytes);
    if (cudaMemsetAsync(d_dist, 0xFF, n_vertices * 4, s) != cudaSuccess) return PG_ECUDA;
    if (cudaMemsetAsync(ws + 2 * fbytes, 0, 256, s) != cudaSuccess) return PG_ECUDA;
    if (cudaMemsetAsync(vis, 0, vbytes, s) != cudaSuccess) return PG_ECUDA;
    { bfs_seed_kernel<<<1, 1, 0, s>>>(d_dist, vis, fr[0], state, (uint32_t)source); note_launch(); }
    const uint32_t undirected = (flags & PG_BFS_UNDIRECTED) ? 1 : 0;
    const BfsBuffers W{{fr[0], fr[1]}, d_dist, vis, long_v, long_base, state};
    BfsState h;
    const pg_status st =
        w == PG_ID64 ? search(d_row_ptr, (const uint64_t*)d_col, W, undirected, n_vertices, h, s)
                     : search(d_row_ptr, (const uint32_t*)d_col, W, undirected, n_vertices, h, s);
    if (st != PG_OK) return st;
    if (levels_out) *levels_out = h.level;
    if (scanned_out) *scanned_out = h.scanned;
    return PG_OK;
}

}  // extern "C"
