// The sequential looping algorithm on sub-blocks of 2^8 outputs and less with 8-bit successors: one lane has one
// sub-block.  Nothing here but these loops: no type of the library, so that they also run on a host that plays a warp's
// lanes in any order between two votes.
#pragma once

namespace benes {
namespace {

// Bytes from the marks of a sub-block of 2^8 to the next one's: the lanes of a warp look at the same place of theirs.
constexpr uint32_t kMarkStride = 128 + 8;

// The looping algorithm: ascending start switches, every output it stands on goes up.  In sub-blocks of 2^8 hops come in
// rounds, and only at the end of one a lane whose loop has closed goes on with the next (it went round its loop again
// meanwhile and noted what it had noted): what is done once a round need not be done with every hop.
constexpr int kLoopHops = 3;

// Marks the switches on loops of one or two.
__device__ __forceinline__ uint32_t mark_short_loops(const unsigned char *N, unsigned char *marks) {
    uint32_t seen = 0;
    for (uint32_t i = 0; i < 32; ++i) {
        const uint32_t t0 = 4u * ((i + threadIdx.x) & 31u);    // (lanes side by side would meet in a bank)
        const uint2 n = *reinterpret_cast<const uint2 *>(N + 2u * t0);
        const uint32_t f[4] = {n.x & 255u, (n.x >> 16) & 255u, n.y & 255u, (n.y >> 16) & 255u};
        uint32_t m = *reinterpret_cast<const uint32_t *>(marks + t0);
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) {
            const uint32_t j = 2u * (t0 + k);
            if (N[f[k]] == j) m |= (2u + (min(j, f[k]) & 1u)) << (8u * k);
        }
        *reinterpret_cast<uint32_t *>(marks + t0) = m;
        seen += uint32_t(__popc(m & 0x02020202u));
    }
    return seen;
}

// The 2^8 outputs whose successors start at N.  The mark of a switch, 2 + the colour of its even output, says that it has
// been seen; marks are clear at first.  The next start, the smallest switch without a mark, is looked up eight marks at a
// time beside the hops of a round, and not taken if this round has seen it.  A hop is a load, a store and
// eight instructions (with the set of seen switches and its smallest gap in registers it was 36, and they, not the
// load, were what a hop took: 114 cycles alone and 186 with two warps on a scheduler, now 88).
// `mine`: the lane has a sub-block.  The others vote as finished and store nothing: only a vote keeps lanes together, and one
// that repeated another's walk could show it marks that it is not to know yet, and so a start that is not the smallest of
// its loop; and one that walked padding, the identity, would take three times as long as those beside it.
__device__ __forceinline__ void loop_marks(const unsigned char *N, unsigned char *marks, bool mine) {
    constexpr uint32_t kSw = 128;
    uint32_t j = 0, start = 0, from = 0, seen = mine ? 0u : kSw;
    bool idle = !mine;                         // the loop has closed, and there was no next one to take
    for (uint32_t round = 0; round < 3u * kSw; ++round) {
        uint32_t t[kLoopHops];
        bool closed = idle;
        uint2 x;
#pragma unroll
        for (int k = 0; k < kLoopHops; ++k) {
            const uint32_t next = N[j];
            t[k] = j >> 1;
            if (mine) marks[t[k]] = uint8_t(2u + (j & 1u));
            if (k == 0) x = *reinterpret_cast<const uint2 *>(marks + from);
            seen += closed ? 0u : 1u;
            closed |= next == start;
            j = next;
        }
        const uint32_t y0 = ~x.x & 0x02020202u, y1 = ~x.y & 0x02020202u, y = y0 ? y0 : y1;
        const uint32_t fresh = from + (y0 ? 0u : 4u) + (uint32_t(__ffs(int(y))) >> 3);
        bool take = mine && closed && y != 0u;
#pragma unroll
        for (int k = 1; k < kLoopHops; ++k) take = take && t[k] != fresh;
        idle = closed && !take;
        from = y ? from : min(from + 8u, kSw - 8u);
        start = take ? 2u * fresh : start;
        j = take ? 2u * fresh : j;
        if (__all_sync(~0u, seen >= kSw)) break;
        // Loop after loop that ends within a round: the short ones together first, which adds 2 us to the walk of the others,
        // where 128 loops of one take 11 us longer than a long one.  Loops of one in any lane do (when most lanes had to
        // have short ones, 12000 x 2^8 took 46 us instead of 36 with a quarter of them the identity, 9741 x 2^9 shift 105
        // instead of 81), loops of two, 70 rounds instead of 48 to 60, in most.  (A lane has seen 7 of 12 switches or
        // less in no random permutation of 200000, 8 in one of 5000; in any lane 8 and less made 128 x 2^13 50.3 us
        // instead of 48.6.  What is left of the loop at hand is then not short, unless it has not been begun.)
        if (round == 3u && (__any_sync(~0u, seen <= 7u) ||
                            2 * __popc(__ballot_sync(~0u, seen <= 8u)) > __popc(__ballot_sync(~0u, mine)))) {
            if (mine) seen = mark_short_loops(N, marks);
            idle = idle || (j == start && marks[j >> 1] != 0);
        }
    }
}

// A sub-block of 2^7.  Bit sets run from the top bit down, so that the smallest gap is one count of leading ones.
__device__ __forceinline__ uint2 loop_128(const unsigned char *N) {
    uint32_t seen0 = 0, seen1 = 0, col0 = 0, col1 = 0, j = 0, start = 0;
#pragma unroll 4
    for (uint32_t it = 0; it < 64u; ++it) {
        const uint32_t next = N[j] & 127u;                     // (places that nobody has written)
        const uint32_t bit = 0x80000000u >> ((j >> 1) & 31u), odd = (j & 1u) ? bit : 0u;
        if (j >= 64u) {
            seen1 |= bit;
            col1 |= odd;
        } else {
            seen0 |= bit;
            col0 |= odd;
        }
        const bool full0 = seen0 == ~0u, closed = next == start;
        const uint32_t fresh = ((full0 ? 64u : 0u) + 2u * uint32_t(__clz(int(~(full0 ? seen1 : seen0))))) & 127u;
        start = closed ? fresh : start;
        j = closed ? fresh : next;
    }
    return make_uint2(__brev(col0), __brev(col1));
}

// The 2^LOGREG outputs whose successors start at N: a sub-block of 2^6 or 2^5, or the two sub-blocks of 16 of a region
// of 32.  One visit per switch: a look for the next start with every hop costs less than the hops that rounds waste here.
template <int LOGREG>
__device__ __forceinline__ uint32_t loop_region(const unsigned char *N, uint32_t smask) {
    constexpr uint32_t kReg = 1u << LOGREG, kSw = kReg / 2;
    uint32_t seen = 0, col = 0, j = 0, start = 0;
#pragma unroll 4
    for (uint32_t it = 0; it < kSw; ++it) {
        uint32_t next = N[j] & smask;
        if (LOGREG == 5) next |= j & ~smask;                   // (entries are local to sub-blocks of 16 or 32)
        const uint32_t bit = 0x80000000u >> (j >> 1);
        seen |= bit;
        col |= (j & 1u) ? bit : 0u;
        const bool closed = next == start;
        start = closed ? (2u * uint32_t(__clz(int(~seen)))) & (kReg - 1u) : start;
        j = closed ? start : next;
    }
    return __brev(col);
}

}  // namespace
}  // namespace benes
