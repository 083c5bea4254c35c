// pairs.cuh -- two frequency moves per gather: the pair table of the DDMC walk
// and the transition stream it consumes.
//
// Frequency moves dominate a thick line, and two of them in a row visit only
// the states s-1, s and s+1.  The pair of row s is 16 bytes,
//   {T[s-1], T[s], T[s+1], guard},
// T the row's first threshold (w < T: bin - 1) and guard the smallest fast
// threshold of the three rows (0 when one of them has a frequency outcome that
// is not a plain move).  When both words are below the guard, both transitions
// are frequency moves and the pair decides them; otherwise the walk takes the
// rows one by one.  Rows outside the class block are never reached (the end
// bins have no move past them: T = 0 at the bottom, T = the fast threshold at
// the top) and do not enter the guard.
#pragma once
#include <cstdint>

#include "rddmc_internal.cuh"

namespace rddmc {

struct alignas(16) Pair {
    uint32_t m1, z, p1, guard;
};

// The walk keeps a state as the byte offset 16 s of its pair, so that a gather
// takes a uniform base and a 32-bit offset and needs no 64-bit address product
// (kPairRows keeps offsets below 2^31).  Two moves change the offset by -32, 0
// or 32: they add 32 per upward move, and the constant -32 rides on the next
// gather's address, so a move is one predicated add.
//
// Four frequency moves on the words of r from offset o0: two gathers through L1
// (the table is read-only during a walk).  Offsets stay inside the pair region
// and its pads whatever the table and the packet's state hold: o0 comes from
// pair_offset or is at most the last row's, and the second gather lies within two
// rows of it (kPairPad bytes before and after the region).
constexpr int kPairPad = 32;

// Offset of the pair of state s.  A saved state that names a cell in vacuum has
// the class 0xffffffff and an s far past the table: it gets at most `last`, the last row's.
__host__ __device__ __forceinline__ uint32_t pair_offset(uint32_t s, uint32_t last) { return min(16u * s, last); }

__host__ __device__ __forceinline__ Pair load_pair(const Pair* base, uint32_t offset, int shift) {
    const uint4* p = reinterpret_cast<const uint4*>(reinterpret_cast<const char*>(base) + offset + shift);
#ifdef __CUDA_ARCH__
    const uint4 v = __ldg(p);
#else
    const uint4 v = *p;
#endif
    return Pair{v.x, v.y, v.z, v.w};
}

struct FourMoves {
    uint32_t o2, o4;  // offsets after two and four moves, less the constants -32 and -64
    bool ok2, ok4;    // the first two, all four transitions are frequency moves
};

__host__ __device__ __forceinline__ FourMoves walk_four(const Pair* base, const uint4& r, uint32_t o0) {
    FourMoves m;
    const Pair a = load_pair(base, o0, 0);
    const bool d0 = r.x >= a.z;
    const bool d1 = r.y >= (d0 ? a.p1 : a.m1);
    m.o2 = o0;
    if (d0) m.o2 += 32u;
    if (d1) m.o2 += 32u;
    const Pair b = load_pair(base, m.o2, -32);
    const bool d2 = r.z >= b.z;
    const bool d3 = r.w >= (d2 ? b.p1 : b.m1);
    m.o4 = m.o2;
    if (d2) m.o4 += 32u;
    if (d3) m.o4 += 32u;
    m.ok2 = max(r.x, r.y) < a.guard;
    m.ok4 = m.ok2 && max(r.z, r.w) < b.guard;
    return m;
}

// Four transitions of any plain moves on the rows, without a branch on their
// outcomes.  In a cell at least four moves inside its class (P.inside) a spatial
// move leaves the row as it is, so a transition is one row's thresholds against
// its word, and the rows' flags say that every outcome is a plain move
// (FLAG_FASTX, FLAG_FASTZ); nearer the class's edge the outcome's own action is
// looked at and the class follows the cell.  s is a row of the table, and inside a
// class it moves by one row at a time: rows up to three beyond the ends are read
// there without a clamp, and they lie in the table buffer's neighbouring blocks of
// 256 bytes or more (the profile before the rows, the heads after them).  The
// clamps cost 2 % of the wide-core slab.  Moves s, cell and cls and returns
// true; returns false with all as they were when a transition is not a plain
// move, and on moving grids, which the caller walks outcome by outcome.
// Such groups took 520 of 650 cycles per warp on the wide-core slab when every
// transition branched.
template <int NDIM, bool INSIDE, bool DUST, class K>
__device__ __forceinline__ bool walk_rows(const K& P, unsigned nr1, unsigned J, const uint4& r, unsigned& s,
                                          unsigned& cell, unsigned& cls) {
    unsigned s1 = s, c1 = cell, k1 = cls, flags = FLAG_FASTX | FLAG_FASTZ;
    bool plain = true;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const unsigned w = q == 0 ? r.x : (q == 1 ? r.y : (q == 2 ? r.z : r.w));
        const int row = INSIDE ? (int)s1 : (int)min(s1, nr1);
        const uint4 a = __ldg(&P.rows[NDIM == 1 ? row : 2 * row]);
        const bool spatial = w >= a.y;  // thresholds of j-1 | j+1 | -x | +x ...
        unsigned move, outcome;
        if (NDIM == 1) {
            const bool up = w >= (spatial ? a.z : a.x);
            move = up ? 1u : 0xffffffffu;
            outcome = (spatial ? 2u : 0u) + (up ? 1u : 0u);
        } else {
            const uint4 b = __ldg(&P.rows[2 * row + 1]);  // ... | -y | +y | -z | +z
            const bool y = w >= b.x, z = w >= b.z;
            const bool up = w >= (spatial ? (z ? b.w : (y ? b.y : a.z)) : a.x);
            const unsigned stride = !spatial ? 1u : (z ? (unsigned)P.n01 : (y ? (unsigned)P.n0 : 1u));
            move = up ? stride : 0u - stride;
            outcome = (spatial ? (z ? 6u : (y ? 4u : 2u)) : 0u) + (up ? 1u : 0u);
        }
        if constexpr (DUST) plain = plain && w < __ldg(&P.abs_thr[row]);  // not absorbed
        if (INSIDE) flags &= a.w;
        else plain = plain && ((a.w >> (2u * outcome)) & 3u) == ACT_MOVE;
        if (!spatial) {
            s1 += move;
        } else {
            c1 += move;
            if (!INSIDE) {
                c1 = min(c1, (unsigned)P.ncell - 1u);
                const unsigned k = __ldg(&P.cell_class[c1]);
                s1 += (k - k1) * J;
                k1 = k;
            }
        }
    }
    if (!plain || flags != (FLAG_FASTX | FLAG_FASTZ)) return false;
    s = s1;
    cell = c1;
    cls = k1;
    return true;
}

template <int NDIM, class K>
__device__ __forceinline__ bool walk_four_rows(const K& P, unsigned nr1, unsigned J, const uint4& r, unsigned& s,
                                               unsigned& cell, unsigned& cls) {
    if (!P.inside) return false;
    if constexpr (K::kDust)
        if (P.dust) return walk_rows<NDIM, false, true>(P, nr1, J, r, s, cell, cls);
    return __ldg(&P.inside[cell]) ? walk_rows<NDIM, true, false>(P, nr1, J, r, s, cell, cls)
                                        : walk_rows<NDIM, false, false>(P, nr1, J, r, s, cell, cls);
}

// Consecutive transition blocks of one packet for a fixed high word of the
// block index: Philox4x32-10 of (b, b_hi, p_lo, p_hi) with what the first three
// rounds owe to the packet and b_hi alone computed once, and the first product
// of the block index carried from block to block as a sum.  Three of the twenty
// 32x32->64 products and three of the xors leave the loop that way (a wide
// product takes the multiply pipe twice as long as any other instruction takes
// its pipe, and that pipe is what the loop saturates).  K: a kernel's
// parameter block with the round keys rk0[10], rk1[10], read from the constant
// bank at fixed offsets (through a pointer they would be copied to local memory).
struct TransitionStream {
    uint32_t e0, e1, e2, e3;
    unsigned long long w0;  // first product of the next block

    template <class K>
    __device__ __forceinline__ void init(uint32_t b, uint32_t b_hi, uint32_t p_lo, uint32_t p_hi, const K& P) {
        const unsigned long long w1 = mul_wide(0xCD9E8D57u, p_lo);
        const unsigned long long w2 = mul_wide(0xD2511F53u, hi(w1) ^ b_hi ^ P.rk0[0]);
        e0 = p_hi ^ P.rk1[0];
        e1 = lo(w1) ^ P.rk0[1];
        e2 = hi(w2) ^ P.rk1[1];
        e3 = lo(w2) ^ P.rk1[2];
        w0 = mul_wide(0xD2511F53u, b);
    }

    template <class K>
    __device__ __forceinline__ uint4 next(const K& P) {
        const unsigned long long w1 = mul_wide(0xCD9E8D57u, hi(w0) ^ e0);
        const unsigned long long w2 = mul_wide(0xD2511F53u, hi(w1) ^ e1), w3 = mul_wide(0xCD9E8D57u, lo(w0) ^ e2);
        w0 += 0xD2511F53u;
        uint4 c = make_uint4(hi(w3) ^ lo(w1) ^ P.rk0[2], lo(w3), hi(w2) ^ e3, lo(w2));
#pragma unroll
        for (int r = 3; r < 10; ++r) {
            const unsigned long long a0 = mul_wide(0xD2511F53u, c.x), a1 = mul_wide(0xCD9E8D57u, c.z);
            c = make_uint4(hi(a1) ^ c.y ^ P.rk0[r], lo(a1), hi(a0) ^ c.w ^ P.rk1[r], lo(a0));
        }
        return c;
    }

private:
    static __device__ __forceinline__ uint32_t hi(unsigned long long v) { return (uint32_t)(v >> 32); }
    static __device__ __forceinline__ uint32_t lo(unsigned long long v) { return (uint32_t)v; }
};

}  // namespace rddmc
