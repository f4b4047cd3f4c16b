// CSR assembly of a generated edge list.
//
// Rows hold their destinations in ascending order (duplicates kept), so the
// result is unique for a given multiset of edges.
//
// Grouped lists (non-decreasing src, as gen_pba and serial BA write them,
// rows of at most kGroupedMaxRow edges): csr_grouped finds the list grouped as
// it goes, places each destination at its rank within its own row and marks
// each row's end in row_ptr.
//
// Any other list: least-significant-digit radix sort of the (src, dst) keys,
// from the low bits of dst to the high bits of src, up to 8 bits per pass (9 for short lists):
//   radix_hist     one read of the list counts the digits of every pass
//                  (the totals do not depend on the order a pass leaves);
//   radix_dstart   per pass, where each digit's run starts in the output;
//   radix_scatter  per pass: stable rank of each element within its tile
//                  among equal digits (shared-memory peer words + per-warp
//                  counters + cross-warp scan), a reorder in shared memory, the tile's
//                  start in each digit's run by decoupled look-back over the
//                  earlier tiles' published counts, and coalesced writes.
// A short list does the three in one launch, radix_sort.
// Ranks come from counts in entry order, never from atomics racing for a
// slot, so the result does not depend on the schedule, and a power-law row
// (a hub with 10^5 edges) costs no more than any other key. The last pass
// writes the destinations to col itself and raises row_ptr[src + 1] at the
// last pair of each source in each tile. Both paths then take a parallel
// prefix maximum over row_ptr, which fills the rows without edges. The sort
// kernels read the flag that csr_grouped sets and return at once when the
// grouped path applied, so no host round trip decides the path.
//
// Ids at or above n_vertices are never used as an index, so a bad list cannot
// make a kernel write out of bounds, and such a source ends no row.
#include <atomic>
#include <cstring>
#include <type_traits>

#include "pg_internal.h"
#include "pg_trace.h"

namespace pgen {
namespace {

constexpr int kSortWarps = 16;
constexpr int kFly = 2;   // items a warp ranks at a time
// which items of a thread find their peers by ballots: three of eight
__host__ __device__ constexpr bool by_ballot(int r) { return 0x92 >> (r & 7) & 1; }
constexpr int kSortThreads = kSortWarps * 32;
constexpr uint32_t kScanTile = 4096;
constexpr uint32_t kGroupedMaxRow = 32;
constexpr uint32_t kHistCopies = 8;   // copies of each digit counter, half as many in the short-list kernel

template <typename Id>
struct PairOf;
template <>
struct PairOf<uint32_t> {
    using T = uint2;
};
template <>
struct PairOf<uint64_t> {
    using T = ulonglong2;
};

// What the sort moves (K): pairs of 32-bit ids wherever the ids fit, also of a
// list with 64-bit ids, else pairs of 64-bit ids. A pass is bound by the
// shared-memory pipe and moves half the bytes in the narrow form: the CSR of
// 2 * 10^7 pairs of 64-bit ids, k = 21, went from 1.243 to 0.921 ms. (One
// 64-bit key (src << nd) | dst per pair instead: 1.001 ms, and 0.662 instead
// of 0.586 ms for the passes of k = 20, whose digits then take 64-bit shifts.)
// The first pass reads the call's list itself, reversed pairs of a symmetrised
// list included.
//
// The digit of a pass: field 0 = dst and field 1 = src take `mask` bits at
// `shift` of that id; field 2 is a digit of the key (src << nd) | dst that
// starts in dst (shift < nd) and ends in src.
struct Digit {
    int field, shift, nd;
    uint32_t mask;
};
template <typename K>
__device__ __forceinline__ uint32_t digit_of(const K& e, const Digit& g)
{
    if (g.field == 2)
        return (uint32_t)(((uint64_t)e.y >> g.shift) | ((uint64_t)e.x << (g.nd - g.shift))) & g.mask;
    return (uint32_t)((g.field ? e.x : e.y) >> g.shift) & g.mask;
}

// The list of a call: its pairs, each twice when sym (the second time
// reversed), in the width the sort moves. Where that is the narrower one, an id
// it cannot hold becomes ~0, which is no vertex of such a call: its low word
// may name one. A source like that takes its destination along, so that the
// pair goes behind every row. Such ids are rare, so the readers take low words
// and collect the high ones in `far`, and read again what that shows to be
// wide (simple CSR of 2 * 10^7 pairs of 64-bit ids: 1.63 ms, with a test and a
// choice per id 1.65).
template <typename K, typename P>
struct PairList {
    const P* p;
    uint32_t sym;   // 0 or 1
    // from an even position on
    __device__ __forceinline__ PairList operator+(uint64_t i) const
    {
        return PairList{p + (i >> sym), sym};
    }
    template <typename I>
    __device__ __forceinline__ K operator[](I i) const { return again(i); }
    template <typename I>
    __device__ __forceinline__ K read(I i, uint32_t& far) const
    {
        const P e = p[i >> sym];
        const bool back = (uint32_t)i & sym;
        K k;
        k.x = (decltype(k.x))(back ? e.y : e.x);
        k.y = (decltype(k.y))(back ? e.x : e.y);
        if constexpr (sizeof(K) < sizeof(P)) far |= (uint32_t)(e.x >> 32) | (uint32_t)(e.y >> 32);
        return k;
    }
    template <typename I>
    __device__ __forceinline__ K again(I i) const
    {
        uint32_t wide = 0;
        K k = read(i, wide);
        if constexpr (sizeof(K) < sizeof(P)) {
            const P e = p[i >> sym];
            const bool back = (uint32_t)i & sym;
            if ((back ? e.y : e.x) >> 32) k.x = k.y = ~0u;
            if ((back ? e.x : e.y) >> 32) k.y = ~0u;
        }
        return k;
    }
};
template <typename K, typename I>
__device__ __forceinline__ K read_pair(const K* list, I i, uint32_t&) { return list[i]; }
template <typename K, typename P, typename I>
__device__ __forceinline__ K read_pair(const PairList<K, P>& list, I i, uint32_t& far)
{
    return list.read(i, far);
}
template <typename K, typename I>
__device__ __forceinline__ K read_again(const K* list, I i) { return list[i]; }
template <typename K, typename P, typename I>
__device__ __forceinline__ K read_again(const PairList<K, P>& list, I i) { return list.again(i); }

// A sort tile and the widest digit. Long lists: 16 pairs of 32-bit ids (8 of
// 64-bit) per thread and digits of at most 8 bits. Short lists, up to
// kShortList pairs, are fewer tiles than the GPU has places, so a pass takes a
// tile's latency: tiles of half the size, and digits of 9 bits for fewer
// passes (100,003 pairs, k = 13: 0.088 -> 0.071 ms, 2^19 pairs: 0.114 -> 0.108, both
// with a launch per pass; 2^20 pairs lose, 0.120 -> 0.135).
template <typename K, bool kShort>
struct SortShape {
    static constexpr int items = (sizeof(K) == 8 ? 16 : 8) / (kShort ? 2 : 1);
    static constexpr uint32_t tile = kSortThreads * items;
    static constexpr uint32_t buckets = kShort ? 512 : 256;
};
constexpr uint32_t kMaxBuckets = 512, kLongBuckets = 256;
constexpr uint64_t kShortList = 3u << 18;
constexpr uint32_t kShortPasses = 8;   // 64 key bits in digits of 9

// The digits of every LSD pass, from the host: pass k sorts by `bits[k]`
// bits of the destination (field 0) or source (field 1) at `shift[k]`, or
// (field 2) by the bits [shift[k], shift[k] + bits[k]) of the key
// (src << nd) | dst, which straddle the two ids.
constexpr int kMaxPasses = 16;   // 64-bit ids: 128 key bits in digits of 8
struct PassList {
    uint32_t n;
    uint32_t buckets;   // of the widest digit: stride of the passes' tables
    int nd;             // bits of the dst field
    int field[kMaxPasses], shift[kMaxPasses], bits[kMaxPasses];
    __host__ __device__ Digit digit(uint32_t k) const
    {
        return Digit{field[k], shift[k], nd, (1u << bits[k]) - 1};
    }
};
// Digit totals of every pass in one read of the list: tot[k][d] += number of
// pairs whose pass-k digit is d. Each CTA counts into shared memory
// (n passes x pl.buckets counters, kCopies copies of each) and adds its
// counts once. Bound by the shared-memory atomics, one per pair and pass (2^30
// pairs, 7 passes: 3.7 ms, of which reading the list takes 1.3).
template <typename K, uint32_t kCopies, typename In>
__device__ __forceinline__ void count_digits(const In in, uint64_t M, const PassList& pl,
                                             unsigned long long* tot)
{
    extern __shared__ __align__(16) unsigned char smem[];
    uint32_t* h = reinterpret_cast<uint32_t*>(smem);
    // the copies of a counter are interleaved, lane l adding to copy l mod
    // kCopies: lanes whose digits agree (the skewed digits of a power-law
    // graph) mostly hit different words
    const uint32_t cells = pl.n * pl.buckets;
    for (uint32_t t = threadIdx.x; t < cells * kCopies; t += blockDim.x) h[t] = 0;
    __syncthreads();
    const uint32_t copy = threadIdx.x & (kCopies - 1);
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    constexpr int kU = 4;
    for (uint64_t i0 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i0 < M; i0 += kU * stride) {
        K e[kU];
        uint32_t far = 0;
#pragma unroll
        for (int u = 0; u < kU; ++u)
            if (i0 + u * stride < M) e[u] = read_pair(in, i0 + u * stride, far);
        if (far)
#pragma unroll
            for (int u = 0; u < kU; ++u)
                if (i0 + u * stride < M) e[u] = read_again(in, i0 + u * stride);
        // pass by pass, so that each pass's digit rule is read once for the
        // kU elements
#pragma unroll 2
        for (uint32_t k = 0; k < pl.n; ++k) {
            const Digit dg = pl.digit(k);
            uint32_t* hk = h + (k * pl.buckets) * kCopies + copy;
#pragma unroll
            for (int u = 0; u < kU; ++u)
                if (i0 + u * stride < M) atomicAdd(&hk[digit_of(e[u], dg) * kCopies], 1u);
        }
    }
    __syncthreads();
    for (uint32_t t = threadIdx.x; t < cells; t += blockDim.x) {
        uint32_t c = 0;
        for (uint32_t r = 0; r < kCopies; ++r) c += h[t * kCopies + r];
        if (c) atomicAdd(&tot[t], (unsigned long long)c);
    }
}

// Tile status words, one per (tile, digit): bits 63..59 the pass (1 + its
// index, so the words of an earlier pass read as not ready), bits 58..57 the
// kind, a pair count below. kAgg: the tile's own count of the digit; kInc: the
// count of the digit in this tile and every earlier one. The array is zeroed
// once per call.
constexpr int kPassShift = 59;
constexpr unsigned long long kAgg = 1ull << 57, kInc = 2ull << 57;
constexpr unsigned long long kCountMask = (1ull << 57) - 1;
static_assert(kMaxPasses < 32, "the pass tag fits bits 63..59");
constexpr uint32_t kSpinLimit = 1u << 18;   // polls of one status word
constexpr int kLookWindow = 4;              // earlier tiles read per round trip

// Test hook (host-set, off by default): a shorter poll limit, and one tile
// per pass that never publishes its counts, so that the tiles after it give
// up waiting and set the error word. The values are passed to each launch.
struct CsrWaitHook {
    uint32_t spin_limit, withhold;
};
std::atomic<uint32_t> g_hook_spin{kSpinLimit};
std::atomic<uint32_t> g_hook_withhold{0xFFFFFFFFu};
CsrWaitHook csr_wait_hook() { return CsrWaitHook{g_hook_spin.load(), g_hook_withhold.load()}; }
// The same for the barriers of cooperative launches: one CTA never arrives.
std::atomic<uint32_t> g_barrier_polls{kBarrierPolls};
std::atomic<uint32_t> g_barrier_withhold{0xFFFFFFFFu};

// Exclusive scan of the CTA's values, and their sum.
__device__ __forceinline__ uint64_t block_exclusive_scan(uint64_t v, uint64_t* s_warp,
                                                         uint64_t& total)
{
    const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t nw = blockDim.x >> 5;
    uint64_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= (uint32_t)o) x += y;
    }
    if (lane == 31) s_warp[wid] = x;
    __syncthreads();
    if (wid == 0) {
        uint64_t w = lane < nw ? s_warp[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint64_t y = __shfl_up_sync(0xFFFFFFFFu, w, o);
            if (lane >= (uint32_t)o) w += y;
        }
        if (lane < nw) s_warp[lane] = w;   // inclusive warp totals
    }
    __syncthreads();
    total = s_warp[nw - 1];
    const uint64_t before = wid ? s_warp[wid - 1] : 0;
    __syncthreads();
    return before + x - v;
}

// What a sort works on. The words are the workspace's, in order: a ticket per
// pass, the wait error, the passes in which a wait gave up (a bit each), and
// the grid barrier's two.
constexpr int kWordErr = kMaxPasses, kWordFailed = kWordErr + 1, kWordBarrier = kWordFailed + 1;
template <typename K, typename P, typename Id>
struct SortJob {
    PairList<K, P> first;
    const K* plain;   // the list where it is what the passes move already, else null
    K* buf[2];
    uint64_t M, N, n_status16, n_rows;
    unsigned long long *status, *tot;
    uint32_t* words;
    const uint32_t* sort_needed;   // null: always
    Id* col;                       // null: the last pass writes pairs, too
    uint64_t* row_ptr;
    CsrWaitHook hook;
    BarrierLimits barrier;
    PassList pl;
};

// One LSD pass over a tile: load once, rank stably (per warp by match, then
// across warps), reorder the tile by digit in shared memory, and write each
// digit's run to its place in the output with consecutive threads on
// consecutive elements. Where a tile's run of digit d starts is dstart[d]
// (from the pass's digit totals) plus the count of d in earlier tiles, found
// by decoupled look-back over the status words. A long list's CTA takes its
// tile index from a ticket, so every earlier tile belongs to a CTA already
// running or done; a short list's CTAs take theirs by block index and are all
// resident, in one cooperative launch. A CTA publishes its own counts before it
// waits on anything, and it sums earlier tiles' counts, kLookWindow at a time,
// until it meets an inclusive one (windows of 3, 6 and 8: 2 to 4 % slower at k
// = 20). The look-back runs after the reorder, when the tile's pairs no longer
// occupy registers.
//
// Bound by the shared-memory pipe: 28 wavefronts per 32 pairs and 8 more for
// global memory, 71 % of its rate, the vector ALU 53 %. So three of eight
// items find their peers on the ALU (none: 10 %, a quarter: 3 %, half: 2 to
// 5 % slower, all: 26 %), two items are in flight, a CTA loops over tiles with
// as few barriers as it can, and the reorder takes one table lookup per pair.
// k = 20 (2^24 pairs, 5 passes) 0.645 -> 0.500 ms, k = 26 (2^30 pairs, 7 passes)
// 44.3 -> 36.6, 0.48 of the HBM rate. Every poll loop is bounded: after spin_limit polls of
// one word (kSpinLimit unless a test hook shortened it) it sets *err and
// goes on with the partial sum, which can only be too small, so every write
// stays inside the output.
template <typename K, typename In, typename Id, bool kShort, typename D>
__device__ __forceinline__ void scatter_pass(
    const In in, K* __restrict__ out, Id* __restrict__ col_out, uint64_t* __restrict__ row_ptr,
    const uint64_t M, const uint64_t N, const Digit dg, const uint32_t pass,
    const D* __restrict__ dstart, unsigned long long* __restrict__ status,
    uint32_t* __restrict__ words, const uint32_t spin_limit, const uint32_t withhold)
{
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int kItems = SortShape<K, kShort>::items;
    constexpr uint32_t kTile = SortShape<K, kShort>::tile;
    constexpr uint32_t kBuckets = SortShape<K, kShort>::buckets;
    constexpr int kBits = kBuckets == 512 ? 9 : 8;
    uint16_t (*wcnt)[kBuckets] = reinterpret_cast<uint16_t (*)[kBuckets]>(smem);
    uint64_t* tbase = reinterpret_cast<uint64_t*>(smem + kSortWarps * kBuckets * 2);
    uint32_t* loff = reinterpret_cast<uint32_t*>(tbase + kBuckets);
    K* buf = reinterpret_cast<K*>(loff + kBuckets);                                  // tile
    __shared__ uint32_t s_part[kSortWarps + 1];
    __shared__ uint32_t s_tile;
    const uint32_t nb = dg.mask + 1;
    const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t wbase = wid * (32 * kItems);
    K e[kItems];
    auto zero_counters = [&] {   // the warp's own
        for (uint32_t t = lane; t < kBuckets / 8; t += 32)
            reinterpret_cast<uint4*>(wcnt[wid])[t] = make_uint4(0u, 0u, 0u, 0u);
    };
    if (!kShort && threadIdx.x == 0) s_tile = atomicAdd(words + pass, 1u);
    zero_counters();
    __syncthreads();
    // (a short list's CTAs are all resident and need no ticket)
    uint32_t tile = kShort ? blockIdx.x : s_tile;
    while ((uint64_t)tile * kTile < M) {   // uniform
        const uint32_t n = (uint32_t)(M - (uint64_t)tile * kTile < kTile ? M - (uint64_t)tile * kTile
                                                                        : kTile);
        const auto tile_in = in + (uint64_t)tile * kTile;
        uint32_t far = 0;
#pragma unroll
        for (int r = 0; r < kItems; ++r) {
            const uint32_t t = wbase + r * 32 + lane;
            if (t < n) e[r] = read_pair(tile_in, t, far);
        }
        if (far)
#pragma unroll
            for (int r = 0; r < kItems; ++r) {
                const uint32_t t = wbase + r * 32 + lane;
                if (t < n) e[r] = read_again(tile_in, t);
            }
        // ranks within the warp (< 32 * kItems <= 512), two per register; the
        // digits are recomputed from e[] where needed, so no array holds them
        uint32_t rk[kItems / 2];
        const uint32_t lt = (1u << lane) - 1u;
        // kFly items of every lane at a time, in lane order within an item. The
        // lanes holding equal digits of an item find each other either by a ballot
        // per digit bit, or through a word per digit (each ORs in its lane bit,
        // then all read the word back and clear it; every item in flight has its
        // own table of kBuckets words per warp, in the reorder buffer, unused until
        // the ranks are done). Then, item by item, the lanes read the warp's
        // counter of their digit, and the last lane of each group adds the group's
        // size. A warp's shared-memory operations execute in order, so the accesses
        // of the items in flight need no wait between them.
        uint32_t* pmask = reinterpret_cast<uint32_t*>(buf) + wid * (kFly * kBuckets);
        for (uint32_t t = lane; t < kFly * kBuckets / 4; t += 32)
            reinterpret_cast<uint4*>(pmask)[t] = make_uint4(0u, 0u, 0u, 0u);
        __syncwarp();
        uint16_t* wc = wcnt[wid];
#pragma unroll
        for (int r0 = 0; r0 < kItems; r0 += kFly) {
            uint32_t d[kFly], peers[kFly];
            bool valid[kFly];
#pragma unroll
            for (int u = 0; u < kFly; ++u) {
                valid[u] = wbase + (r0 + u) * 32 + lane < n;
                d[u] = digit_of(e[r0 + u], dg);
                if (!by_ballot(r0 + u) && valid[u]) atomicOr(&pmask[u * kBuckets + d[u]], 1u << lane);
            }
            __syncwarp();
#pragma unroll
            for (int u = 0; u < kFly; ++u) {
                if (by_ballot(r0 + u)) {
                    peers[u] = __ballot_sync(0xFFFFFFFFu, valid[u]);
#pragma unroll
                    for (int b = 0; b < kBits; ++b) {
                        if (b >= 7 && !(dg.mask >> b)) break;
                        const bool one = d[u] & (1u << b);
                        const uint32_t same = __ballot_sync(0xFFFFFFFFu, one);
                        peers[u] &= one ? same : ~same;
                    }
                } else if (valid[u])
                    peers[u] = pmask[u * kBuckets + d[u]];
            }
            __syncwarp();
#pragma unroll
            for (int u = 0; u < kFly; ++u) {
                const int r = r0 + u;
                uint32_t rank = 0;
                if (valid[u]) {
                    if (!by_ballot(r)) pmask[u * kBuckets + d[u]] = 0;
                    rank = wc[d[u]] + __popc(peers[u] & lt);
                }
                __syncwarp();
                if (valid[u] && peers[u] >> lane == 1) wc[d[u]] = (uint16_t)(rank + 1);
                __syncwarp();
                if (r & 1) rk[r >> 1] |= rank << 16;
                else rk[r >> 1] = rank;
            }
        }
        __syncthreads();
        // per digit (one thread each): the tile total, published at once so that
        // later tiles can sum it; where the digit's run starts in the sorted tile
        // (loff), and where each warp's part of the run does (in wcnt)
        const unsigned long long tag = (unsigned long long)(pass + 1) << kPassShift;
        volatile unsigned long long* st = status + (uint64_t)tile * nb;
        {
            const uint32_t d = threadIdx.x;
            uint32_t acc = 0;
            if (d < nb) {
#pragma unroll
                for (int w = 0; w < kSortWarps; ++w) acc += wcnt[w][d];
                if (tile != withhold) st[d] = tag | (tile == 0 ? kInc : kAgg) | acc;
            }
            uint32_t x = acc;   // inclusive over the warp's digits
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
                if (lane >= (uint32_t)o) x += y;
            }
            if (lane == 31) s_part[wid] = x;
            __syncthreads();
            const uint32_t before = __reduce_add_sync(0xFFFFFFFFu, lane < wid ? s_part[lane] : 0u);
            if (d < nb) {
                uint32_t at = before + x - acc;
                loff[d] = at;
#pragma unroll
                for (int w = 0; w < kSortWarps; ++w) {
                    const uint32_t c = wcnt[w][d];
                    wcnt[w][d] = (uint16_t)at;   // below the tile's size
                    at += c;
                }
            }
        }
        __syncthreads();
        // reorder the tile by digit in shared memory
#pragma unroll
        for (int r = 0; r < kItems; ++r) {
            const uint32_t t = wbase + r * 32 + lane;
            if (t < n) {
                const uint32_t d = digit_of(e[r], dg);
                const uint32_t rank = (rk[r >> 1] >> ((r & 1) * 16)) & 0xFFFFu;
                const uint32_t at = wcnt[wid][d] + rank;
                if (PG_CHECK(at, n)) buf[at] = e[r];
            }
        }
        __syncwarp();
        zero_counters();   // for the next tile
        // look back through up to kLookWindow earlier tiles per round trip
        for (uint32_t d = threadIdx.x; d < nb; d += blockDim.x) {
            unsigned long long excl = 0;
            if (tile > 0) {
                uint32_t next = tile - 1;   // nearest tile not yet summed (tile 0 is inclusive)
                uint32_t polls = 0;
                bool found = false;
                while (!found) {
                    unsigned long long w[kLookWindow];
#pragma unroll
                    for (int u = 0; u < kLookWindow; ++u)
                        w[u] = (next >= (uint32_t)u)
                                   ? *((volatile const unsigned long long*)status +
                                       (uint64_t)(next - u) * nb + d)
                                   : 0ull;
                    // counts add up in the low bits; the tags above them are
                    // masked off at the end
                    uint32_t used = 0;
                    bool go = true;
#pragma unroll
                    for (int u = 0; u < kLookWindow; ++u) {
                        const uint32_t kind = (uint32_t)(w[u] >> 57) - 4 * (pass + 1);
                        go = go && kind - 1u < 2u;   // kAgg or kInc of this pass
                        if (go) {
                            excl += w[u];
                            ++used;
                        }
                        found |= go && kind == 2;
                        go = go && kind == 1;
                    }
                    if (found) break;
                    next -= used;
                    if (!go) {
                        if (++polls > spin_limit) {
                            atomicOr(words + kWordErr, 1u);
                            atomicOr(words + kWordFailed, 1u << pass);
                            break;
                        }
                        __nanosleep(32);
                    } else {
                        polls = 0;
                    }
                }
                excl &= kCountMask;
                const uint32_t cnt_d = (d + 1 < nb ? loff[d + 1] : n) - loff[d];
                if (tile != withhold) st[d] = tag | kInc | (excl + cnt_d);
            }
            // where the tile's run of d starts in the output, less its start in
            // the sorted tile (never negative: the tile's counts of the lower
            // digits, loff[d], are at most their totals, which dstart[d] sums)
            tbase[d] = dstart[d] + excl - loff[d];
        }
        __syncthreads();
        // write runs: sorted position p goes to tbase[d] + p (one table read per pair)
        if (col_out == nullptr) {
            for (uint32_t p = threadIdx.x; p < n; p += blockDim.x) {
                const K v = buf[p];
                const uint32_t d = digit_of(v, dg);
                if (PG_CHECK(tbase[d] + p, M)) out[tbase[d] + p] = v;
            }
        } else {
            // the last pass of a CSR: the tile is in (src, dst) order, so each
            // destination goes straight to col, and the last pair of each source
            // in the tile raises row_ptr[src + 1] to its end (the source's last pair
            // overall gives the maximum; the prefix maximum fills empty rows)
            for (uint32_t p = threadIdx.x; p < n; p += blockDim.x) {
                const K v = buf[p];
                const uint32_t d = digit_of(v, dg);
                const uint64_t o = tbase[d] + p;
                if (PG_CHECK_OUT(o, M)) col_out[o] = (Id)v.y;
                const uint64_t src = v.x;
                if (src < N && (p + 1 == n || (uint64_t)buf[p + 1].x != src))
                    atomicMax(reinterpret_cast<unsigned long long*>(row_ptr) + src + 1,
                              (unsigned long long)(o + 1));
            }
        }
        // (a ticket taken before the tile's own work is done would hold up the
        // tiles after it: 0.52 -> 0.59 ms at k = 20)
        if (!kShort && threadIdx.x == 0) s_tile = atomicAdd(words + pass, 1u);
        __syncthreads();   // the next tile reuses the tables
        tile = kShort ? tile + gridDim.x : s_tile;
    }
}

// What comes before the passes: the digits are counted, the status words start
// at zero, and the row ends that the grouped pass wrote before it gave up go:
// all rows, or, where those are many, the rows of the list's sources. (The CTAs
// of a short list are few: 1000 edges on 2^28 vertices, 33.8 ms with all rows, 1.3
// without, of which the memset before and the rows after take nearly all.)
constexpr uint64_t kManyRows = 12;   // per pair: there both cost the same on long lists
template <uint32_t kCopies, typename K, typename P, typename Id, typename In>
__device__ __forceinline__ void prepare_passes(const In in, const SortJob<K, P, Id>& job)
{
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    const uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    count_digits<K, kCopies>(in, job.M, job.pl, job.tot);
    for (uint64_t i = t; i < job.n_status16; i += stride)
        reinterpret_cast<uint4*>(job.status)[i] = make_uint4(0u, 0u, 0u, 0u);
    if (job.n_rows <= kManyRows * job.M) {
        for (uint64_t i = t; i < job.n_rows; i += stride) job.row_ptr[i] = 0;
    } else {
        for (uint64_t i = t; i < job.M; i += stride) {
            const uint64_t src = in[i].x;
            if (src < job.N) job.row_ptr[src + 1] = 0;
        }
    }
}

// After a wait that gave up in a pass the list the next ones read no longer
// has the digit totals the starts are made from, so a scatter could leave the
// output: the remaining passes do nothing.
__device__ __forceinline__ bool pass_can_run(const uint32_t* words, uint32_t pass)
{
    return (*(volatile const uint32_t*)(words + kWordFailed) & ((1u << pass) - 1)) == 0;
}

// A long list: a launch for the digits, then one per pass. (One cooperative
// launch, as below, spills 264 bytes per thread in this shape.)
template <typename K, typename In, typename P, typename Id>
__global__ void __launch_bounds__(256)
    radix_hist_kernel(const In in, const __grid_constant__ SortJob<K, P, Id> job)
{
    if (job.sort_needed && *job.sort_needed == 0) return;
    prepare_passes<kHistCopies>(in, job);
}
// Where each digit's run starts in pass k's output: the exclusive scan of
// that pass's digit totals. grid = passes, block = pl.buckets threads.
__global__ void __launch_bounds__(kMaxBuckets) radix_dstart_kernel(
    const unsigned long long* __restrict__ tot, const __grid_constant__ PassList pl,
    uint64_t* __restrict__ dstart, const uint32_t* __restrict__ sort_needed)
{
    __shared__ uint64_t s_warp[32];
    if (sort_needed && *sort_needed == 0) return;
    const uint32_t k = blockIdx.x, nb = 1u << pl.bits[k], d = threadIdx.x;
    const uint64_t c = d < nb ? tot[(size_t)k * pl.buckets + d] : 0;
    uint64_t total;
    const uint64_t ex = block_exclusive_scan(c, s_warp, total);
    if (d < nb) dstart[(size_t)k * pl.buckets + d] = ex;
}
template <typename K, typename In, typename Id>
__global__ void __launch_bounds__(kSortThreads, 2) radix_scatter_kernel(
    const In in, K* __restrict__ out, Id* __restrict__ col_out, uint64_t* __restrict__ row_ptr,
    const uint64_t M, const uint64_t N, const Digit dg, const uint32_t pass,
    const uint64_t* __restrict__ dstart, unsigned long long* __restrict__ status,
    uint32_t* __restrict__ words, const uint32_t* __restrict__ sort_needed,
    const uint32_t spin_limit, const uint32_t withhold)
{
    if (sort_needed && *sort_needed == 0) return;
    if (!pass_can_run(words, pass)) return;
    scatter_pass<K, In, Id, false>(in, out, col_out, row_ptr, M, N, dg, pass, dstart, status, words, spin_limit,
                                   withhold);
}

// A short list in one cooperative launch, a grid barrier between its parts: a
// launch per part costs more than most parts' work (CSR of 100,003 pairs,
// k = 13: 0.067 -> 0.051 ms, 2^19 pairs: 0.098 -> 0.073), and a list that turned
// out grouped pays one launch (160,000 vertices, m = 4: 0.057 -> 0.034).
template <typename K, typename P, typename Id>
__global__ void __launch_bounds__(kSortThreads, 2)
    radix_sort_kernel(const __grid_constant__ SortJob<K, P, Id> job)
{
    if (job.sort_needed && *job.sort_needed == 0) return;
    if (job.plain) prepare_passes<kHistCopies / 2>((const K*)job.plain, job);
    else prepare_passes<kHistCopies / 2>(job.first, job);
    __shared__ uint32_t s_dstart[kShortPasses][kMaxBuckets];   // a short list's totals fit
    uint32_t epoch = 0;
    for (uint32_t pass = 0; pass < job.pl.n; ++pass) {
        if (!grid_barrier(job.words + kWordBarrier, job.words + kWordBarrier + 1, job.barrier, epoch)) {
            if (threadIdx.x == 0) atomicOr(job.words + kWordErr, 1u);
            return;
        }
        if (!pass_can_run(job.words, pass)) continue;   // the same in every CTA
        if (pass == 0) {   // where each digit's run starts, a warp for every pass
            const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
            if (wid < job.pl.n) {
                constexpr uint32_t kPer = kMaxBuckets / 32;
                const unsigned long long* tot = job.tot + wid * kMaxBuckets + lane * kPer;
                uint32_t c[kPer], sum = 0;
#pragma unroll
                for (uint32_t t = 0; t < kPer; ++t) c[t] = (uint32_t)__ldcg(tot + t);
#pragma unroll
                for (uint32_t t = 0; t < kPer; ++t) sum += c[t];
                uint32_t at = sum;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, at, o);
                    if (lane >= (uint32_t)o) at += y;
                }
                at -= sum;
#pragma unroll
                for (uint32_t t = 0; t < kPer; ++t) {
                    s_dstart[wid][lane * kPer + t] = at;
                    at += c[t];
                }
            }
            __syncthreads();
        }
        auto run = [&](auto in) {
            scatter_pass<K, decltype(in), Id, true>(
                in, job.buf[pass & 1], pass + 1 == job.pl.n ? job.col : nullptr, job.row_ptr, job.M,
                job.N, job.pl.digit(pass), pass, s_dstart[pass], job.status, job.words,
                job.hook.spin_limit, job.hook.withhold);
        };
        if (pass > 0 || job.plain) run((const K*)(pass ? job.buf[(pass - 1) & 1] : job.plain));
        else run(job.first);
    }
}

static_assert(kSortThreads >= (int)kMaxBuckets, "one thread per digit");
static_assert(SortShape<uint2, true>::items % kFly == 0 &&
                  SortShape<ulonglong2, false>::items % kFly == 0,
              "whole groups of items");

template <typename K, bool kShort>
constexpr size_t sort_smem_bytes()
{
    using Shape = SortShape<K, kShort>;
    // the reorder buffer, in which the digit words of the items in flight lie too
    const size_t tile = (size_t)Shape::tile * sizeof(K);
    const size_t words = (size_t)kFly * kSortWarps * Shape::buckets * 4;
    return (size_t)kSortWarps * Shape::buckets * 2 + Shape::buckets * 12 +
           (tile > words ? tile : words);
}

// exclusive scan of n_parts sums in place, one CTA looping over chunks of
// eight neighbouring sums per thread
__global__ void __launch_bounds__(1024) scan_parts_kernel(uint64_t* __restrict__ part,
                                                          uint64_t n_parts)
{
    __shared__ uint64_t s_warp[32];
    constexpr int kPer = 8;
    uint64_t carry = 0;
    for (uint64_t base = 0; base < n_parts; base += kPer * blockDim.x) {
        const uint64_t i = base + kPer * threadIdx.x;
        uint64_t v[kPer], sum = 0;
#pragma unroll
        for (int t = 0; t < kPer; ++t) {
            v[t] = i + t < n_parts ? part[i + t] : 0;
            sum += v[t];
        }
        uint64_t total;
        uint64_t at = carry + block_exclusive_scan(sum, s_warp, total);
#pragma unroll
        for (int t = 0; t < kPer; ++t) {
            if (i + t < n_parts) part[i + t] = at;
            at += v[t];
        }
        carry += total;
    }
}

// ---- lists grouped by source ------------------------------------------------
// One pass over the list, as if it were grouped: every destination goes to its
// row's start + its rank among the row's destinations (ties by position, so
// equal values keep their multiplicity), and the last edge i of row v writes
// row_ptr[v + 1] = i + 1. A tile that finds the list not grouped, or a row of
// more than kGroupedMaxRow edges, sets sort_needed instead; the sort then
// overwrites col, and row_ptr is cleared again. CTAs look at the flag before
// each tile, so an unsorted list costs about one round of tiles.
//
// Bound by instruction issue (0.52 of HBM at m = 5; a row of r edges takes r
// compares per edge), so the work per position is kept small: a tile and 32
// neighbours on each side are staged in shared memory, row starts are one
// ballot per 32 positions, a row's bounds bit searches in three of these
// words, and a rank reads the row once, the lanes of a row the same word.
// Tiles inside the list test no bounds. 2^24 vertices, m = 5: 1.185 -> 0.327 ms
// (64-bit ids 0.48); m = 2: 0.126; 2^22 vertices, m = 30: 6.22 -> 1.12 (each edge
// searched and ranked its row in global memory before, after a pass of its
// own that looked for violations). Six CTAs per SM: five 0.344, eight (spills) 0.37.
constexpr uint32_t kGroupTile = 2048;
template <typename Id>
constexpr int kGroupPlaces = sizeof(Id) == 4 ? 6 : 4;   // CTAs per SM
template <typename Id>
__global__ void __launch_bounds__(256, kGroupPlaces<Id>)
    csr_grouped_kernel(const typename PairOf<Id>::T* __restrict__ s, uint64_t M, uint64_t N,
                       Id* __restrict__ col, uint64_t* __restrict__ row_ptr,
                       uint32_t* __restrict__ sort_needed)
{
    static_assert(kGroupedMaxRow == 32, "a row spans at most two neighbouring words");
    constexpr uint32_t kSpan = kGroupTile + 64;
    __shared__ Id src[kSpan], dst[kSpan];   // edge base + t at 32 + t
    const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    constexpr uint32_t kWords = kGroupTile / 256;   // 32-position words per warp
    // `inner`: every position of the span is an edge of the list
    auto place = [&](uint64_t base, auto inner) -> bool {
        constexpr bool kInner = decltype(inner)::value;
        const uint32_t first = kInner || base ? 0 : 32;
        const uint32_t last = kInner || M - base > kSpan - 32 ? kSpan : (uint32_t)(M - base) + 32;
        const auto* __restrict__ in = s + base - 32;
#pragma unroll
        for (uint32_t t = 0; t < kSpan; t += 256) {
            const uint32_t k = t + threadIdx.x;
            if ((t + 256 <= kSpan || k < kSpan) && (kInner || (k >= first && k < last))) {
                const auto e = in[k];
                src[k] = e.x;
                dst[k] = e.y;
            }
        }
        __syncthreads();
        // bit l of starts[u]: a row starts at position 32 (w0 + u - 1) + l (the
        // end of the list counts as one, and so does the start)
        const uint32_t w0 = 1 + wid * kWords;
        uint32_t starts[kWords + 2];
        bool bad = false;
#pragma unroll
        for (uint32_t u = 0; u < kWords + 2; ++u) {
            const uint32_t k = 32 * (w0 - 1 + u) + lane;
            bool st;
            if (kInner) {
                const Id x = src[k], y = src[k > 0 ? k - 1 : 0];
                st = x != y;
                bad |= y > x;
                if (u <= kWords) bad |= src[k + 32] == x;
            } else {
                st = k == first || k == last;
                if (k > first && k < last) {
                    st = src[k - 1] != src[k];
                    bad |= src[k - 1] > src[k];
                }
                if (k >= first && k + kGroupedMaxRow < last) bad |= src[k + kGroupedMaxRow] == src[k];
            }
            starts[u] = __ballot_sync(0xFFFFFFFFu, st);
        }
        if (__syncthreads_or(bad)) return false;
        Id* __restrict__ out = col + base - 32;
#pragma unroll
        for (uint32_t u = 0; u < kWords; ++u) {
            const uint32_t k0 = 32 * (w0 + u), k = k0 + lane;
            const uint32_t before = starts[u], here = starts[u + 1], after = starts[u + 2];
            if (kInner || k < last) {
                // the last start at or before the lane, the first one after it
                const uint32_t lo = here & (0xFFFFFFFFu >> (31 - lane));
                const uint32_t hi = (here >> lane) >> 1;
                const uint32_t a = lo ? k0 + 31 - __clz(lo) : k0 - 1 - __clz(before);
                const uint32_t b = hi ? k + __ffs(hi) : k0 + 31 + __ffs(after);
                const Id d = dst[k];
                uint32_t at = a;
                // smaller destinations of the row, or equal ones before
#pragma unroll 4
                for (uint32_t j = a; j < b; ++j) {
                    const Id o = dst[j];
                    if constexpr (sizeof(Id) == 4)
                        at += ((uint64_t)o << 32 | j) < ((uint64_t)d << 32 | k) ? 1u : 0u;
                    else
                        at += o < d || (o == d && j < k) ? 1u : 0u;
                }
                if (PG_CHECK_OUT(base + at - 32, M)) out[at] = d;
                if (b == k + 1) {
                    const uint64_t v = src[k];
                    if (v < N) row_ptr[v + 1] = base + (k - 31);
                }
            }
        }
        return true;
    };
    for (uint64_t base = (uint64_t)blockIdx.x * kGroupTile; base < M;
         base += (uint64_t)gridDim.x * kGroupTile) {
        // (a barrier, too: the last tile's readers are done)
        if (__syncthreads_or(threadIdx.x == 0 && *(volatile const uint32_t*)sort_needed != 0)) return;
        const bool inner = base > 0 && M - base >= kGroupTile + 32;
        if (inner ? !place(base, std::true_type{}) : !place(base, std::false_type{})) {
            if (threadIdx.x == 0) atomicOr(sort_needed, 1u);
            return;
        }
    }
}

template <typename V>
__device__ __forceinline__ V warp_inclusive_max(V x, uint32_t lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const V y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= (uint32_t)o && y > x) x = y;
    }
    return x;
}

// In-place inclusive prefix maximum over the n row pointers, in one cooperative
// launch: a CTA takes neighbouring tiles of kScanTile entries, publishes their
// maximum in part[], and after a grid barrier applies what came before to each.
// A CTA with one tile (up to 2.4 million rows) keeps it in registers, one with
// more reads them again. A warp takes kScanTile / 8 neighbouring entries, 32 at
// a time, so that every access is coalesced (row_ptr is aligned to 8 bytes
// only); V is uint32_t when the values, which are positions in the list, fit
// it. Bound by its launch and barrier, then by memory: 160,000 rows 14 -> 8 us,
// 2^20 16.7 -> 10.2, 2^24 75 -> 67, 2^26 259 -> 258 (three launches before).
constexpr int kRowPlaces = 4;   // CTAs per SM
template <typename V>
__global__ void __launch_bounds__(256, kRowPlaces)
    row_max_kernel(uint64_t* data, uint64_t n, uint64_t* part, uint32_t per, uint32_t* words,
                   uint32_t* err, BarrierLimits barrier)
{
    __shared__ V s_warp[8];
    const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    constexpr int kRounds = kScanTile / 256;
    const uint64_t first = (uint64_t)blockIdx.x * per;
    V a[kRounds];
    auto load = [&](uint64_t tile) {
        const uint64_t base = tile * kScanTile + wid * (32 * kRounds) + lane;
#pragma unroll
        for (int r = 0; r < kRounds; ++r) a[r] = base + 32 * r < n ? (V)data[base + 32 * r] : 0;
    };
    // the CTA's maximum of x, in every thread
    auto reduce = [&](V x) {
        x = warp_inclusive_max(x, lane);
        if (lane == 31) s_warp[wid] = x;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < 8; ++w)
            if (s_warp[w] > x) x = s_warp[w];
        __syncthreads();
        return x;
    };
    V carry = 0;
    if (gridDim.x > 1) {
        V m = 0;
        for (uint32_t t = 0; t < per; ++t) {
            load(first + t);
#pragma unroll
            for (int r = 0; r < kRounds; ++r)
                if (a[r] > m) m = a[r];
        }
        m = reduce(m);
        if (threadIdx.x == 0) part[blockIdx.x] = m;
        uint32_t epoch = 0;
        if (!grid_barrier(words, words + 1, barrier, epoch)) {
            if (threadIdx.x == 0) atomicOr(err, 1u);
            return;
        }
        for (uint32_t c = threadIdx.x; c < blockIdx.x; c += blockDim.x) {
            const V x = (V)__ldcg(part + c);
            if (x > carry) carry = x;
        }
        carry = reduce(carry);
    }
    for (uint32_t t = 0; t < per; ++t) {
        if (per > 1 || gridDim.x == 1) load(first + t);
        V run = 0;   // the warp's maximum up to and including round r
#pragma unroll
        for (int r = 0; r < kRounds; ++r) {
            a[r] = warp_inclusive_max(a[r], lane);
            if (run > a[r]) a[r] = run;
            run = __shfl_sync(0xFFFFFFFFu, a[r], 31);
        }
        if (lane == 0) s_warp[wid] = run;
        __syncthreads();
        V before = carry;
#pragma unroll
        for (uint32_t w = 0; w < 8; ++w) {
            const V x = s_warp[w];
            if (w < wid && x > before) before = x;
            if (x > carry) carry = x;
        }
        const uint64_t base = (first + t) * kScanTile + wid * (32 * kRounds) + lane;
#pragma unroll
        for (int r = 0; r < kRounds; ++r)
            if (base + 32 * r < n) data[base + 32 * r] = before > a[r] ? before : a[r];
        __syncthreads();
    }
}

template <typename Id>
__global__ void __launch_bounds__(256) csr_finish_kernel(const typename PairOf<Id>::T* __restrict__ s,
                                                         uint64_t M, uint64_t N, uint64_t* __restrict__ row_ptr,
                                                         Id* __restrict__ col,
                                                         const uint32_t* __restrict__ sort_needed)
{
    if (*sort_needed == 0) return;
    // four grid strides per trip, so each thread has four independent loads
    // in flight
    constexpr int kU = 4;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i0 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i0 < M; i0 += kU * stride) {
        typename PairOf<Id>::T e[kU];
        uint64_t nx[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const uint64_t i = i0 + u * stride;
            if (i < M) {
                e[u] = s[i];
                nx[u] = (i + 1 < M) ? (uint64_t)s[i + 1].x : ~(uint64_t)0;
            }
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const uint64_t i = i0 + u * stride;
            if (i < M) {
                if (PG_CHECK_OUT(i, M)) col[i] = (Id)e[u].y;
                const uint64_t v = e[u].x;
                if (v < N && nx[u] != v) row_ptr[v + 1] = i + 1;
            }
        }
    }
}

// ---- CSR options (symmetrise, dedup, drop loops, odd multiplicity) ---------
// All options act on the list sorted by (src, dst): the sort always runs,
// then a compaction keeps the wanted positions of the sorted pairs, writes
// their destinations to col in order and marks row ends for the prefix max.
constexpr uint32_t kOptSym = 1, kOptDedup = 2, kOptNoLoops = 4, kOptOdd = 8;

template <typename P>
__device__ __forceinline__ bool same_pair(const P& a, const P& b)
{
    return a.x == b.x && a.y == b.y;
}

template <typename P>
__device__ __forceinline__ bool pair_less(const P& a, const P& b)
{
    return a.x < b.x || (a.x == b.x && a.y < b.y);
}

// Where the run of pairs equal to e = s[i] starts. Runs are short in
// practice, so the first steps go back one pair at a time; a longer run is
// found by binary search of the sorted list below. (With ids outside the
// vertex range the list need not be in lexicographic order there, and the
// search only stays within [0, i].)
template <typename L, typename P>
__device__ __forceinline__ uint64_t run_start(const L& s, uint64_t i, const P& e)
{
    uint64_t j = i;
    for (int t = 0; t < 8 && j > 0 && same_pair(s[j - 1], e); ++t) --j;
    if (j == 0 || !same_pair(s[j - 1], e)) return j;
    uint64_t lo = 0, hi = j;   // s[hi] == e: the first index of e lies in [lo, hi]
    while (lo < hi) {
        const uint64_t mid = lo + (hi - lo) / 2;
        if (pair_less(s[mid], e)) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// Which positions of the sorted list survive the options, as one bit per
// position (keep[i / 32]), and how many do in each tile of kScanTile. A warp
// takes kScanTile / 8 neighbouring positions, 32 at a time, with the loads of
// kAhead rounds in flight. The runs of equal pairs come out of one ballot per
// round (bit i: pair i equals pair i - 1), and the rules are bit arithmetic on
// those words, the same in every lane:
//   CSR_DEDUP  the first pair of each run;
//   CSR_ODD    the last pair of each run of odd length: the one whose distance
//              from its run's start is even. The starts' parities are filled
//              forward within the word and carried to the next.
// Bound by reading the list once (8 or 16 bytes per pair). With the apply kernel
// and the row pointers, 1.8 * 10^7 pairs under CSR_ODD: 0.333 -> 0.119 ms; 4 *
// 10^7 under CSR_DEDUP and CSR_NO_LOOPS: 0.439 -> 0.210 ms (every position read
// its neighbours from memory in both kernels, one load in flight, before).
constexpr int kKeepRounds = kScanTile / 256;
constexpr int kAhead = 8;
template <typename L>
__global__ void __launch_bounds__(256) csr_keep_mask_kernel(const L s, uint64_t M, uint32_t flags,
                                                            uint32_t* __restrict__ keep,
                                                            uint64_t* __restrict__ part)
{
    __shared__ uint32_t s_warp[8];
    const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint64_t wbase = (uint64_t)blockIdx.x * kScanTile + (uint64_t)wid * (32 * kKeepRounds);
    uint32_t cnt = 0;
    if (wbase < M) {   // uniform in the warp
        uint32_t eq[kKeepRounds], loop[kKeepRounds];   // ballots
        using P = typename std::decay<decltype(s[0])>::type;
        P prev = s[wbase > 0 ? wbase - 1 : 0];         // the pair before lane 0's
#pragma unroll
        for (int r0 = 0; r0 < kKeepRounds; r0 += kAhead) {
            P e[kAhead];
#pragma unroll
            for (int u = 0; u < kAhead; ++u) {
                const uint64_t i = wbase + (r0 + u) * 32 + lane;
                e[u] = s[i < M ? i : M - 1];
            }
#pragma unroll
            for (int u = 0; u < kAhead; ++u) {
                const uint64_t i = wbase + (r0 + u) * 32 + lane;
                P b;   // the pair before this lane's
                b.x = __shfl_up_sync(0xFFFFFFFFu, e[u].x, 1);
                b.y = __shfl_up_sync(0xFFFFFFFFu, e[u].y, 1);
                if (lane == 0) b = prev;
                eq[r0 + u] = __ballot_sync(0xFFFFFFFFu, i > 0 && i < M && same_pair(b, e[u]));
                loop[r0 + u] = __ballot_sync(0xFFFFFFFFu, e[u].x == e[u].y);
                prev.x = __shfl_sync(0xFFFFFFFFu, e[u].x, 31);
                prev.y = __shfl_sync(0xFFFFFFFFu, e[u].y, 31);
            }
        }
        const uint64_t wend = wbase + 32 * kKeepRounds;
        const bool open = wend < M && same_pair(s[wend], prev);   // the last run goes on
        // parity of the start of the run open before this warp's positions
        uint32_t odd = 0;
        if ((flags & kOptOdd) && (eq[0] & 1u)) odd = (uint32_t)run_start(s, wbase, s[wbase]) & 1u;
        uint32_t mine = 0;
#pragma unroll
        for (int r = 0; r < kKeepRounds; ++r) {
            const uint64_t i0 = wbase + r * 32;
            const uint32_t live = i0 >= M ? 0u : M - i0 >= 32 ? ~0u : (1u << (uint32_t)(M - i0)) - 1u;
            uint32_t k = live;
            if (flags & kOptOdd) {
                // start parities (position parity is the bit's: i0 is even)
                uint32_t known = ~eq[r], par = known & 0xAAAAAAAAu;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    par |= (par << o) & ~known;
                    known |= known << o;
                }
                if (odd) par |= ~known;
                odd = par >> 31;
                const uint32_t more = r + 1 < kKeepRounds ? eq[r + 1 < kKeepRounds ? r + 1 : r] & 1u
                                                          : (open ? 1u : 0u);
                const uint32_t last = ~((eq[r] >> 1) | (more << 31));   // ends of runs
                k &= last & ~(par ^ 0xAAAAAAAAu);
            } else if (flags & kOptDedup) {
                k &= ~eq[r];
            }
            if (flags & kOptNoLoops) k &= ~loop[r];
            cnt += __popc(k);
            if (lane == (uint32_t)r) mine = k;
        }
        if (lane < (uint32_t)kKeepRounds && wbase + 32 * lane < M) keep[wbase / 32 + lane] = mine;
    }
    if (lane == 0) s_warp[wid] = cnt;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint64_t all = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) all += s_warp[w];
        part[blockIdx.x] = all;
    }
}

// The kept destinations to their places, and the row ends: the last position
// of every row writes row_ptr[src + 1] = kept entries up to and including it.
// A warp's positions and loads are those of the mask kernel; a position's
// place is the tile's start, the counts of the warps and rounds before it and
// the kept bits below it in its word.
template <typename Id, typename L>
__global__ void __launch_bounds__(256) csr_keep_apply_kernel(const L s, uint64_t M, uint64_t N,
                                                             const uint32_t* __restrict__ keep,
                                                             const uint64_t* __restrict__ part,
                                                             Id* __restrict__ col,
                                                             uint64_t* __restrict__ row_ptr)
{
    __shared__ uint32_t s_warp[8];
    const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    const uint64_t wbase = (uint64_t)blockIdx.x * kScanTile + (uint64_t)wid * (32 * kKeepRounds);
    // lane r holds round r's word
    const uint32_t word = lane < (uint32_t)kKeepRounds && wbase + 32 * lane < M
                              ? keep[wbase / 32 + lane] : 0u;
    const uint32_t mine = __reduce_add_sync(0xFFFFFFFFu, __popc(word));
    if (lane == 0) s_warp[wid] = mine;
    __syncthreads();
    if (wbase >= M) return;
    uint64_t at = part[blockIdx.x];
    for (uint32_t w = 0; w < wid; ++w) at += s_warp[w];
#pragma unroll
    for (int r0 = 0; r0 < kKeepRounds; r0 += kAhead) {
        typename std::decay<decltype(s[0])>::type e[kAhead];
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            const uint64_t i = wbase + (r0 + u) * 32 + lane;
            e[u] = s[i < M ? i : M - 1];
        }
        // the source after the batch's last position
        const uint64_t inext = wbase + (r0 + kAhead) * 32;
        const auto after = s[inext < M ? inext : M - 1].x;
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            const uint64_t i = wbase + (r0 + u) * 32 + lane;
            const uint32_t m = __shfl_sync(0xFFFFFFFFu, word, r0 + u);
            auto nx = __shfl_down_sync(0xFFFFFFFFu, e[u].x, 1);
            const auto first = u + 1 < kAhead ? __shfl_sync(0xFFFFFFFFu, e[u + 1 < kAhead ? u + 1 : u].x, 0)
                                              : after;
            if (lane == 31) nx = first;
            const uint64_t here = at + __popc(m & lt);
            const uint32_t kept = (m >> lane) & 1u;
            if (i < M) {
                if (kept && PG_CHECK_OUT(here, M)) col[here] = (Id)e[u].y;
                const uint64_t v = e[u].x;
                if (v < N && (i + 1 == M || (uint64_t)nx != v)) row_ptr[v + 1] = here + kept;
            }
            at += __popc(m);
        }
    }
}

}  // namespace

PG_CHECK_UNIT(csr)

namespace {

int bit_length(uint64_t x)
{
    int b = 0;
    while (x) {
        ++b;
        x >>= 1;
    }
    return b;
}

struct CsrLayout {
    size_t off_a, off_b, off_status, off_flag, off_dig, off_rpart, total;
    uint32_t n_tiles, max_nb;
    uint64_t n_status, n_rparts;
};

size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

// Whether the sort moves pairs of 32-bit ids: any list of those, and one of
// 64-bit ids whose vertices leave ~0 free for the ids that don't fit.
bool ids_narrow(uint64_t n_src, uint64_t n_dst, bool id64)
{
    const uint64_t most = ((uint64_t)1 << 32) - (id64 ? 1 : 0);
    return n_src <= most && n_dst <= most;
}

// Whether the sort of M pairs takes the short-list shape.
bool short_list(uint64_t M, uint64_t n_src, uint64_t n_dst, bool id64)
{
    return M <= kShortList && ids_narrow(n_src, n_dst, id64);
}

// The LSD passes that sort pairs by (src, dst): the key (src << nd) | dst,
// nd = the bits of n_dst - 1 and ns those of n_src - 1, cut from its low end
// into ceil((nd + ns) / digit_bits) digits whose widths differ by at most
// one (the wider ones first). A digit inside one id reads that id alone; the
// one that contains the boundary reads both.
PassList make_passes(uint64_t n_src, uint64_t n_dst, uint64_t M, bool id64)
{
    PassList pl;
    std::memset(&pl, 0, sizeof(pl));
    const int nd = bit_length(n_dst > 0 ? n_dst - 1 : 0);
    const int ns = bit_length(n_src > 0 ? n_src - 1 : 0);
    const int total = nd + ns;
    const int digit_bits = short_list(M, n_src, n_dst, id64) ? 9 : 8;
    const int n = (total + digit_bits - 1) / digit_bits;
    pl.buckets = 1u << digit_bits;
    pl.nd = nd;
    int shift = 0;
    for (int k = 0; k < n; ++k) {
        const int b = total / n + (k < total % n ? 1 : 0);
        if (shift + b <= nd) {
            pl.field[k] = 0;
            pl.shift[k] = shift;
        } else if (shift >= nd) {
            pl.field[k] = 1;
            pl.shift[k] = shift - nd;
        } else {
            pl.field[k] = 2;
            pl.shift[k] = shift;
        }
        pl.bits[k] = b;
        shift += b;
    }
    pl.n = (uint32_t)n;
    return pl;
}

CsrLayout csr_layout(uint64_t M, uint64_t N, size_t pair_bytes, uint64_t N_dst = 0)
{
    CsrLayout L;
    const uint64_t nd = N_dst ? N_dst : N;
    const bool id64 = pair_bytes == 16;
    const PassList pl = make_passes(N, nd, M, id64);
    // a list of narrow ids takes half of two copies in the width its caller
    // names; the status words lie in the rest, and what follows behind both
    const size_t lists = 2 * a256(M * pair_bytes);
    if (ids_narrow(N, nd, id64)) pair_bytes = 8;
    int dbits = 0;
    for (uint32_t k = 0; k < pl.n; ++k) dbits = pl.bits[k] > dbits ? pl.bits[k] : dbits;
    const bool is_short = short_list(M, N, nd, id64);
    const uint32_t tile = pair_bytes != 8 ? SortShape<ulonglong2, false>::tile
                          : is_short ? SortShape<uint2, true>::tile : SortShape<uint2, false>::tile;
    L.max_nb = 1u << dbits;
    L.n_tiles = (uint32_t)((M + tile - 1) / tile);
    L.n_status = (uint64_t)L.max_nb * L.n_tiles;
    size_t o = 0;
    L.off_a = o;
    o += a256(M * pair_bytes);
    L.off_b = o;
    o += a256(M * pair_bytes);
    L.off_status = o;   // tile status words of the pass being sorted
    o += a256(L.n_status * 8);
    if (o < lists) o = lists;
    L.off_flag = o;     // +0: sort-needed flag, +64: SortJob's words (+128: wait error),
                        // +192: the row kernel's barrier
    o += 256;
    L.off_dig = o;      // digit totals and, of a long list, digit starts of every pass
    o += is_short ? (size_t)kShortPasses * kMaxBuckets * 8 : 2 * (size_t)kMaxPasses * kLongBuckets * 8;
    L.n_rparts = (N + 1 + kScanTile - 1) / kScanTile;
    L.off_rpart = o;
    o += a256((L.n_rparts + 1) * 8);
    L.total = o;
    return L;
}

// The opt-in shared-memory sizes of the sort kernels, set once per device
// for each id width.
PerDeviceOnce g_csr_attrs[2];
template <typename F>
cudaError_t allow_smem(F* kernel, size_t bytes)
{
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}
template <typename K, typename P, typename Id>
cudaError_t long_sort_attributes()
{
    constexpr size_t smem = sort_smem_bytes<K, false>();
    static_assert(smem <= 113 * 1024, "two CTAs per SM");
    constexpr size_t counters = kMaxPasses * 256 * 4 * kHistCopies;
    return first_error({allow_smem(radix_hist_kernel<K, const K*, P, Id>, counters),
                        allow_smem(radix_hist_kernel<K, PairList<K, P>, P, Id>, counters),
                        allow_smem(radix_scatter_kernel<K, const K*, Id>, smem),
                        allow_smem(radix_scatter_kernel<K, PairList<K, P>, Id>, smem)});
}
template <typename Id>
cudaError_t set_csr_attributes()
{
    using P = typename PairOf<Id>::T;
    return g_csr_attrs[sizeof(Id) == 8].run_current([] {
        constexpr size_t smem = sort_smem_bytes<uint2, true>();
        static_assert(smem + kShortPasses * kMaxBuckets * 4 <= 113 * 1024, "two CTAs per SM");
        static_assert(kShortPasses * kMaxBuckets * 4 * (kHistCopies / 2) <= smem, "the counters");
        static_assert(kShortPasses <= kSortWarps && SortShape<uint2, true>::buckets == kMaxBuckets,
                      "a warp for every pass");
        cudaError_t e = first_error({long_sort_attributes<uint2, P, Id>(),
                                     allow_smem(radix_sort_kernel<uint2, P, Id>, smem)});
        if constexpr (sizeof(Id) == 8)
            if (e == cudaSuccess) e = long_sort_attributes<P, P, Id>();
        return e;
    });
}

int sort_grid(uint64_t work);

// The sort's words and digit totals start at zero on every call that has
// edges; a call without edges has nothing to sort and no wait.
cudaError_t clear_sort_words(unsigned char* ws, const CsrLayout& L, const PassList& pl, uint64_t M,
                             cudaStream_t s)
{
    const size_t bytes = M > 0 ? L.off_dig - L.off_flag + (size_t)pl.n * pl.buckets * 8 : 4;
    return cudaMemsetAsync(ws + L.off_flag, 0, bytes, s);
}

// LSD radix sort of the M pairs of `first` (the digits of the key
// (src << nd) | dst from its low end), unless *sort_needed is 0; K is what the
// passes move. *sorted receives the sorted list (unset when there is no digit
// to sort). With col_final set, the last pass writes the CSR directly instead:
// destinations to col_final, row ends raised into row_ptr.
template <typename K, typename P, typename Id>
cudaError_t radix_sort(const PairList<K, P> first, uint64_t M, uint64_t N, const PassList& pl,
                       const CsrLayout& L, unsigned char* ws, const uint32_t* sort_needed,
                       cudaStream_t s, const K** sorted, Id* col_final, uint64_t* row_ptr)
{
    SortJob<K, P, Id> job;
    job.first = first;
    job.plain = nullptr;
    if constexpr (std::is_same<K, P>::value)
        if (!first.sym) job.plain = first.p;
    job.buf[0] = (K*)(ws + L.off_a);
    job.buf[1] = (K*)(ws + L.off_b);
    *sorted = pl.n ? job.buf[(pl.n - 1) & 1] : job.plain;
    if (M == 0 || pl.n == 0) return cudaSuccess;
    job.M = M;
    job.N = N;
    job.n_status16 = (L.n_status * 8 + 15) / 16;
    job.n_rows = col_final ? N + 1 : 0;   // else no grouped pass ran
    job.status = (unsigned long long*)(ws + L.off_status);
    job.tot = (unsigned long long*)(ws + L.off_dig);
    job.words = (uint32_t*)(ws + L.off_flag + 64);
    job.sort_needed = sort_needed;
    job.col = col_final;
    job.row_ptr = row_ptr;
    job.hook = csr_wait_hook();
    job.barrier = barrier_limits();
    job.pl = pl;
    // Two CTAs per SM, what its registers hold, take tiles until none is left;
    // a long list that turned out grouped pays a launch per pass and not a CTA
    // per tile (five passes over 2^24 x 5 edges: 0.089 -> 0.039 ms)
    const unsigned places = 2 * (unsigned)device_sm_count();
    const unsigned grid = L.n_tiles < places ? L.n_tiles : places;
    if constexpr (sizeof(K) == 8) {
        if (pl.buckets == SortShape<K, true>::buckets) {
            TraceScope trace("csr_sort", s);
            constexpr size_t smem = sort_smem_bytes<K, true>();
            void* args[] = {&job};
            const cudaError_t e = cudaLaunchCooperativeKernel(
                (const void*)radix_sort_kernel<K, P, Id>, dim3(grid), dim3(kSortThreads), args, smem, s);
            note_launch();
            return e;
        }
    }
    {
        TraceScope trace("csr_radix_hist", s);
        const size_t smem = (size_t)pl.n * pl.buckets * 4 * kHistCopies;
        if (job.plain)
            { radix_hist_kernel<K, const K*, P, Id><<<sort_grid(M), 256, smem, s>>>(job.plain, job); note_launch(); }
        else
            { radix_hist_kernel<K, PairList<K, P>, P, Id><<<sort_grid(M), 256, smem, s>>>(first, job); note_launch(); }
    }
    uint64_t* dstart = (uint64_t*)(ws + L.off_dig) + (size_t)kMaxPasses * kLongBuckets;
    {
        TraceScope trace("csr_scan", s);
        { radix_dstart_kernel<<<pl.n, pl.buckets, 0, s>>>(job.tot, pl, dstart, sort_needed); note_launch(); }
    }
    constexpr size_t smem = sort_smem_bytes<K, false>();
    for (uint32_t k = 0; k < pl.n; ++k) {
        TraceScope trace("csr_radix_scatter", s);
        auto launch = [&](auto in) {
            { radix_scatter_kernel<K, decltype(in), Id><<<grid, kSortThreads, smem, s>>>(
                in, job.buf[k & 1], k + 1 == pl.n ? col_final : nullptr, row_ptr, M, N, pl.digit(k), k,
                dstart + (size_t)k * pl.buckets, job.status, job.words, sort_needed,
                job.hook.spin_limit, job.hook.withhold); note_launch(); }
        };
        if (k > 0 || job.plain) launch((const K*)(k ? job.buf[(k - 1) & 1] : job.plain));
        else launch(first);
    }
    return cudaGetLastError();
}

// In-place prefix maximum over the N + 1 row pointers of a list of M > 0 pairs.
template <typename V>
cudaError_t row_max_as(uint64_t* d_row_ptr, uint64_t N, const CsrLayout& L, unsigned char* ws,
                       cudaStream_t s)
{
    const uint64_t places = (uint64_t)kRowPlaces * device_sm_count();
    uint32_t per = (uint32_t)((L.n_rparts + places - 1) / places);
    const unsigned grid = (unsigned)((L.n_rparts + per - 1) / per);
    uint64_t n = N + 1, *part = (uint64_t*)(ws + L.off_rpart);
    uint32_t* words = (uint32_t*)(ws + L.off_flag + 192);
    uint32_t* err = (uint32_t*)(ws + L.off_flag + 64) + kWordErr;
    BarrierLimits barrier = barrier_limits();
    if (grid == 1) {   // nothing to wait for
        { row_max_kernel<V><<<1, 256, 0, s>>>(d_row_ptr, n, part, per, words, err, barrier); note_launch(); }
        return cudaGetLastError();
    }
    void* args[] = {&d_row_ptr, &n, &part, &per, &words, &err, &barrier};
    const cudaError_t e = cudaLaunchCooperativeKernel((const void*)row_max_kernel<V>, dim3(grid),
                                                      dim3(256), args, 0, s);
    note_launch();
    return e;
}
cudaError_t row_max(uint64_t* d_row_ptr, uint64_t N, uint64_t M, const CsrLayout& L,
                    unsigned char* ws, cudaStream_t s)
{
    return M < ((uint64_t)1 << 32) ? row_max_as<uint32_t>(d_row_ptr, N, L, ws, s)
                                   : row_max_as<uint64_t>(d_row_ptr, N, L, ws, s);
}

int sort_grid(uint64_t work)
{
    int grid = (int)((work + 255) / 256);
    const int cap = device_sm_count() * 8;
    if (grid > cap) grid = cap;
    return grid < 1 ? 1 : grid;
}

template <typename Id>
cudaError_t csr_impl(const void* d_edges, uint64_t M, uint64_t N, uint64_t N_dst,
                     uint64_t* d_row_ptr, void* d_col, void* d_ws, cudaStream_t s)
{
    using P = typename PairOf<Id>::T;
    const CsrLayout L = csr_layout(M, N, sizeof(P), N_dst);
    cudaError_t err;
    if ((err = set_csr_attributes<Id>()) != cudaSuccess) return err;
    unsigned char* ws = (unsigned char*)d_ws;
    uint32_t* sort_needed = (uint32_t*)(ws + L.off_flag);
    const int grid = sort_grid(M + 1);
    const PassList pl = make_passes(N, N_dst, M, sizeof(Id) == 8);
    if ((err = clear_sort_words(ws, L, pl, M, s)) != cudaSuccess) return err;
    if (cudaMemsetAsync(d_row_ptr, 0, (N + 1) * 8, s) != cudaSuccess) return cudaErrorUnknown;
    {
        TraceScope trace("csr_grouped", s);
        const uint64_t tiles = (M + kGroupTile - 1) / kGroupTile;
        const uint64_t full = (uint64_t)device_sm_count() * kGroupPlaces<Id>;
        const unsigned places = (unsigned)(tiles < full ? (tiles ? tiles : 1) : full);
        { csr_grouped_kernel<Id><<<places, 256, 0, s>>>((const P*)d_edges, M, N, (Id*)d_col, d_row_ptr,
                                                     sort_needed); note_launch(); }
    }
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
    // with at least one digit to sort, the last pass writes col and the row
    // ends itself; a key without digits (one vertex) leaves the list as it is
    const bool in_sort = M > 0 && pl.n > 0;
    Id* col = in_sort ? (Id*)d_col : nullptr;
    if (ids_narrow(N, N_dst, sizeof(Id) == 8)) {
        const uint2* sorted;
        err = radix_sort<uint2, P, Id>({(const P*)d_edges, 0}, M, N, pl, L, ws, sort_needed, s,
                                         &sorted, col, d_row_ptr);
    } else if constexpr (sizeof(Id) == 8) {   // 32-bit ids are always narrow
        const P* sorted;
        err = radix_sort<P, P, Id>({(const P*)d_edges, 0}, M, N, pl, L, ws, sort_needed, s, &sorted,
                                     col, d_row_ptr);
    }
    if (err != cudaSuccess) return err;
    if (!in_sort) {
        TraceScope trace("csr_finish", s);
        { csr_finish_kernel<Id><<<grid, 256, 0, s>>>((const P*)d_edges, M, N, d_row_ptr, (Id*)d_col, sort_needed); note_launch(); }
    }
    if (M == 0) return cudaSuccess;    // every row is empty, row_ptr all zero
    TraceScope trace("csr_rows", s);   // rows without edges take the previous row's end
    return row_max(d_row_ptr, N, M, L, ws, s);
}

// Workspace of the options path: the sort's layout for the (possibly
// doubled) list, and the parts of the compaction's scan.
struct OptsLayout {
    CsrLayout L;
    size_t off_cpart, off_keep, total;
    uint64_t M2, n_cparts;
};

OptsLayout opts_layout(uint64_t M, uint64_t N, uint32_t flags, size_t pair_bytes)
{
    OptsLayout O;
    O.M2 = (flags & kOptSym) ? 2 * M : M;
    O.L = csr_layout(O.M2, N, pair_bytes);
    size_t o = a256(O.L.total);
    O.n_cparts = (O.M2 + kScanTile - 1) / kScanTile;
    O.off_cpart = o;
    o += a256((O.n_cparts + 1) * 8);
    // (nothing between the lists and the sort's words is needed after the sort)
    const size_t keep = a256((O.M2 + 31) / 32 * 4);
    O.off_keep = O.L.off_flag - O.L.off_status >= keep ? O.L.off_status : o;
    if (O.off_keep == o) o += keep;
    O.total = o;
    return O;
}

// The wanted positions of the sorted list into col, and the row pointers.
template <typename Id, typename List>
cudaError_t csr_compact(const List& list, uint64_t M2, uint64_t N, uint32_t flags,
                        const OptsLayout& O, unsigned char* ws, uint64_t* d_row_ptr, Id* d_col, cudaStream_t s)
{
    if (M2 == 0) return cudaSuccess;   // every row is empty, row_ptr all zero
    cudaError_t err;
    TraceScope trace("csr_compact", s);
    uint64_t* cpart = (uint64_t*)(ws + O.off_cpart);
    uint32_t* keep = (uint32_t*)(ws + O.off_keep);
    { csr_keep_mask_kernel<List><<<(unsigned)O.n_cparts, 256, 0, s>>>(list, M2, flags, keep, cpart); note_launch(); }
    { scan_parts_kernel<<<1, 1024, 0, s>>>(cpart, O.n_cparts); note_launch(); }
    { csr_keep_apply_kernel<Id, List><<<(unsigned)O.n_cparts, 256, 0, s>>>(list, M2, N, keep, cpart,
                                                                          d_col, d_row_ptr); note_launch(); }
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
    return row_max(d_row_ptr, N, M2, O.L, ws, s);
}

template <typename Id>
cudaError_t csr_opts_impl(const void* d_edges, uint64_t M, uint64_t N, uint32_t flags,
                          uint64_t* d_row_ptr, void* d_col, void* d_ws, cudaStream_t s)
{
    using P = typename PairOf<Id>::T;
    const OptsLayout O = opts_layout(M, N, flags, sizeof(P));
    cudaError_t err;
    if ((err = set_csr_attributes<Id>()) != cudaSuccess) return err;
    unsigned char* ws = (unsigned char*)d_ws;
    const uint64_t M2 = O.M2;
    if (cudaMemsetAsync(d_row_ptr, 0, (N + 1) * 8, s) != cudaSuccess) return cudaErrorUnknown;
    const P* in = (const P*)d_edges;
    const uint32_t sym = (flags & kOptSym) ? 1 : 0;
    const PassList pl = make_passes(N, N, M2, sizeof(Id) == 8);
    if ((err = clear_sort_words(ws, O.L, pl, M2, s)) != cudaSuccess) return err;
    // one vertex: the list is sorted as it is (its reverse is the same again)
    if (pl.n == 0)
        return csr_compact<Id>(PairList<P, P>{in, sym}, M2, N, flags, O, ws, d_row_ptr, (Id*)d_col, s);
    // every option needs the sorted list: the sort runs unconditionally
    if (ids_narrow(N, N, sizeof(Id) == 8)) {
        const uint2* sorted;
        if ((err = radix_sort<uint2, P, Id>({in, sym}, M2, N, pl, O.L, ws, nullptr, s, &sorted,
                                              nullptr, nullptr)) != cudaSuccess)
            return err;
        return csr_compact<Id>(sorted, M2, N, flags, O, ws, d_row_ptr, (Id*)d_col, s);
    }
    if constexpr (sizeof(Id) == 8) {
        const P* sorted;
        if ((err = radix_sort<P, P, Id>({in, sym}, M2, N, pl, O.L, ws, nullptr, s, &sorted,
                                          nullptr, nullptr)) != cudaSuccess)
            return err;
        return csr_compact<Id>(sorted, M2, N, flags, O, ws, d_row_ptr, (Id*)d_col, s);
    }
    return cudaErrorInvalidValue;   // 32-bit ids are always narrow
}

}  // namespace

void set_csr_wait_hook(uint32_t spin_limit, uint32_t withhold_tile)
{
    g_hook_spin.store(spin_limit ? spin_limit : kSpinLimit);
    g_hook_withhold.store(withhold_tile);
}

void set_barrier_hook(uint32_t polls, uint32_t withhold_cta)
{
    g_barrier_polls.store(polls ? polls : kBarrierPolls);
    g_barrier_withhold.store(withhold_cta);
}
BarrierLimits barrier_limits()
{
    return BarrierLimits{g_barrier_polls.load(), g_barrier_withhold.load()};
}

size_t csr_workspace_bytes(uint64_t n_edges, uint64_t n_vertices, uint64_t n_dst)
{
    // one size that fits either id width
    const size_t a = csr_layout(n_edges, n_vertices, 16, n_dst).total;
    const size_t b = csr_layout(n_edges, n_vertices, 8, n_dst).total;
    return a > b ? a : b;
}

size_t csr_opts_workspace_bytes(uint64_t n_edges, uint64_t n_vertices, uint32_t flags)
{
    const size_t a = opts_layout(n_edges, n_vertices, flags, 16).total;
    const size_t b = opts_layout(n_edges, n_vertices, flags, 8).total;
    return a > b ? a : b;
}

// Byte offset of the look-back error word in the workspace of a call with
// these arguments (the layout the call itself uses).
size_t csr_wait_error_offset(uint64_t n_edges, uint64_t n_vertices, uint32_t flags, int id64,
                             uint64_t n_dst)
{
    const size_t pair_bytes = id64 ? 16 : 8;
    const CsrLayout L = flags ? opts_layout(n_edges, n_vertices, flags, pair_bytes).L
                              : csr_layout(n_edges, n_vertices, pair_bytes, n_dst);
    return L.off_flag + 128;
}

cudaError_t launch_csr_opts(const void* d_edges, uint64_t n_edges, uint64_t n_vertices, int id64,
                            uint32_t flags, uint64_t* d_row_ptr, void* d_col, void* d_ws,
                            cudaStream_t s)
{
    return id64 ? csr_opts_impl<uint64_t>(d_edges, n_edges, n_vertices, flags, d_row_ptr, d_col,
                                          d_ws, s)
                : csr_opts_impl<uint32_t>(d_edges, n_edges, n_vertices, flags, d_row_ptr, d_col,
                                          d_ws, s);
}

cudaError_t launch_csr(const void* d_edges, uint64_t n_edges, uint64_t n_vertices, int id64,
                       uint64_t* d_row_ptr, void* d_col, void* d_ws, size_t ws_bytes,
                       cudaStream_t s, uint64_t n_dst)
{
    (void)ws_bytes;
    const uint64_t nd = n_dst ? n_dst : n_vertices;
    return id64 ? csr_impl<uint64_t>(d_edges, n_edges, n_vertices, nd, d_row_ptr, d_col, d_ws, s)
                : csr_impl<uint32_t>(d_edges, n_edges, n_vertices, nd, d_row_ptr, d_col, d_ws, s);
}

}  // namespace pgen
