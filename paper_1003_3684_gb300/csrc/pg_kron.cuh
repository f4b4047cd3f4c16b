// The descent of stochastic Kronecker edges for an initiator of order 2,
// shared by the single-graph and the batch kernels.
//
// Level l of edge e consumes word (l mod 4) of the Philox block for counter
// (e_lo, e_hi, l div 4, 3). The kernels are bound by the integer pipes. A
// sub-partition spends 4 FMA-pipe cycles and 2 ALU cycles on a 32x32->64
// multiply, 2 ALU cycles on a three-input logic operation, a compare or a
// select, and 1 on an add (measured with mixes of independent chains), so
// multiplies cost on both pipes, and what blocks share is computed once:
//   - per edge, the first round's product of word 0 and the second round's
//     product of word 2: they depend on e_lo and the constant word 3 alone,
//     so every group of four levels of the edge starts from them;
//   - per group g, the first round's product of word 2 and the second round's
//     of word 0: they depend on (e_hi, g) alone; a CTA keeps them in shared
//     memory (one broadcast load per group and pair of edges).
// A block then costs 16 multiplies instead of 20. A level's bits are
// predicated adds of an immediate to the shifted-up halves (an add is half a
// select), and a thread walks two edges at once, so that the multiplies form
// two independent chains. Per edge of 20 levels that is 82 multiplies, 91
// logic operations, 60 compares and selects and 46 adds: 523 ALU cycles per
// warp at a sub-partition, which is what the kernel takes (508 at 2.02 GHz).
//   2^24 edges, k = 20: 0.272 -> 0.217 ms; 2^26, k = 22: 1.279 -> 1.015 ms;
//   64-bit ids, k = 40, 2^24: 0.608 -> 0.466 ms (GB300).
// Measured and no better: the bits added in the multiply-add pipe (0.220),
// in floating point (0.231), or by selects (0.258); the column bit by three
// chained compares (0.217); 32 registers for full occupancy (0.223).
#pragma once

#include "pg_common.cuh"

namespace pgen {

constexpr uint32_t kKronMaxGroups = 16;   // k <= 64 levels

// What group g contributes to the second round (philox_head's f3, f4, f5).
__device__ __forceinline__ uint4 kron_group_head(uint32_t e_hi, uint32_t g, const Key& key)
{
    const PhiloxHead h = philox_head(e_hi, g, 3u, key);
    return make_uint4(h.f3, h.f4, h.f5, 0u);
}

// What edge e contributes to the second round.
struct KronEdgeHead {
    uint32_t qh, ql, y3;
};
__device__ __forceinline__ KronEdgeHead kron_edge_head(uint32_t e_lo, const Key& key)
{
    const uint64_t p0 = (uint64_t)0xD2511F53u * e_lo;
    const uint32_t y2 = (uint32_t)(p0 >> 32) ^ 3u ^ key.k1[0];
    const uint64_t q1 = (uint64_t)0xCD9E8D57u * y2;
    return KronEdgeHead{(uint32_t)(q1 >> 32), (uint32_t)q1, (uint32_t)p0};
}

// philox((e_lo, e_hi, g, 3), key) from the two heads.
__device__ __forceinline__ uint4 kron_block(const KronEdgeHead& s, const uint4& h, const Key& key)
{
    uint4 c = make_uint4(s.qh ^ h.x, s.ql, s.y3 ^ h.y, h.z);
#pragma unroll
    for (int r = 2; r < 10; ++r) {
        const uint64_t a0 = (uint64_t)0xD2511F53u * c.x;
        const uint64_t a1 = (uint64_t)0xCD9E8D57u * c.z;
        c = make_uint4((uint32_t)(a1 >> 32) ^ c.y ^ key.k0[r], (uint32_t)a1,
                       (uint32_t)(a0 >> 32) ^ c.w ^ key.k1[r], (uint32_t)a0);
    }
    return c;
}

// One level: adds kBit to r and c where the chosen cell's row and column bits
// are set. kFull (n_zero = 0 and three real thresholds u0 <= u1 <= u2): the
// row bit is w > u1 and the column bit w > u2 when that is set, else w > u0.
template <uint32_t kBit, bool kFull>
__device__ __forceinline__ void kron_level(uint32_t w, uint32_t u0, uint32_t u1, uint32_t u2,
                                           uint32_t base, uint32_t& r, uint32_t& c)
{
    if constexpr (kFull) {
        asm("{\n\t"
            ".reg .pred p, q;\n\t"
            ".reg .u32 t;\n\t"
            "setp.gt.u32 p, %2, %4;\n\t"
            "selp.u32 t, %5, %3, p;\n\t"
            "setp.gt.u32 q, %2, t;\n\t"
            "@p add.u32 %0, %0, %6;\n\t"
            "@q add.u32 %1, %1, %6;\n\t"
            "}"
            : "+r"(r), "+r"(c)
            : "r"(w), "r"(u0), "r"(u1), "r"(u2), "n"(kBit));
    } else {
        const uint32_t cell = base + (w > u0) + (w > u1) + (w > u2);
        r += (cell >> 1) * kBit;
        c += (cell & 1) * kBit;
    }
}

// Edges e0 and e1 (low index words; their high word is the one `heads` was
// made with): k levels, most significant first. T is uint32_t for k <= 32.
template <typename T, bool kFull>
__device__ __forceinline__ void kron_two_edges(const uint4* heads, const Key& key, uint32_t k,
                                               uint32_t u0, uint32_t u1, uint32_t u2,
                                               uint32_t base, uint32_t e0, uint32_t e1, T& r0,
                                               T& c0, T& r1, T& c1)
{
    const KronEdgeHead s0 = kron_edge_head(e0, key), s1 = kron_edge_head(e1, key);
    r0 = c0 = r1 = c1 = 0;
    uint32_t g = 0;
#pragma unroll 1
    for (; g < (k >> 2); ++g) {
        const uint4 h = heads[g];
        const uint4 a = kron_block(s0, h, key), b = kron_block(s1, h, key);
        uint32_t x0 = 0, y0 = 0, x1 = 0, y1 = 0;
        if constexpr (sizeof(T) == 4) {
            x0 = (uint32_t)r0 << 4;
            y0 = (uint32_t)c0 << 4;
            x1 = (uint32_t)r1 << 4;
            y1 = (uint32_t)c1 << 4;
        }
        kron_level<8, kFull>(a.x, u0, u1, u2, base, x0, y0);
        kron_level<8, kFull>(b.x, u0, u1, u2, base, x1, y1);
        kron_level<4, kFull>(a.y, u0, u1, u2, base, x0, y0);
        kron_level<4, kFull>(b.y, u0, u1, u2, base, x1, y1);
        kron_level<2, kFull>(a.z, u0, u1, u2, base, x0, y0);
        kron_level<2, kFull>(b.z, u0, u1, u2, base, x1, y1);
        kron_level<1, kFull>(a.w, u0, u1, u2, base, x0, y0);
        kron_level<1, kFull>(b.w, u0, u1, u2, base, x1, y1);
        if constexpr (sizeof(T) == 4) {
            r0 = x0;
            c0 = y0;
            r1 = x1;
            c1 = y1;
        } else {
            r0 = (r0 << 4) | x0;
            c0 = (c0 << 4) | y0;
            r1 = (r1 << 4) | x1;
            c1 = (c1 << 4) | y1;
        }
    }
    const uint32_t rest = k & 3;
    if (rest) {
        const uint4 h = heads[g];
        const uint4 a = kron_block(s0, h, key), b = kron_block(s1, h, key);
        uint32_t x0 = 0, y0 = 0, x1 = 0, y1 = 0;   // the top `rest` of four levels
        kron_level<4, kFull>(a.x, u0, u1, u2, base, x0, y0);
        kron_level<4, kFull>(b.x, u0, u1, u2, base, x1, y1);
        if (rest > 1) {
            kron_level<2, kFull>(a.y, u0, u1, u2, base, x0, y0);
            kron_level<2, kFull>(b.y, u0, u1, u2, base, x1, y1);
        }
        if (rest > 2) {
            kron_level<1, kFull>(a.z, u0, u1, u2, base, x0, y0);
            kron_level<1, kFull>(b.z, u0, u1, u2, base, x1, y1);
        }
        const uint32_t down = 3 - rest;
        r0 = (r0 << rest) | (T)(x0 >> down);
        c0 = (c0 << rest) | (T)(y0 >> down);
        r1 = (r1 << rest) | (T)(x1 >> down);
        c1 = (c1 << rest) | (T)(y1 >> down);
    }
}

}  // namespace pgen
