// Fused path: one CTA finishes every remaining level of 2^LOGC consecutive
// outputs entirely in shared memory (inverse, loop labelling, colouring, stage
// bits, compaction, middle stage).  It serves the tail of a large permutation
// (blocks of 2^logs outputs of the flat level array) and batches of small
// permutations; a CTA holds one block, or several when the blocks are smaller
// than 2^LOGC.
//
// A level works on sub-blocks of S = 2^logs outputs.  The kernel is bound by the
// shared-memory wavefronts of its random 16-bit accesses (3-4 per warp access; about
// 25 thousand per level of 2^15 outputs, of 34 thousand cycles) and by instruction
// issue, hardly by memory, so the labelling changes with S:
//
//   S >= 256   16-bit entries.  One ruler switch per 8 switches; a walker per
//              ruler output follows g, claims the switches it passes and stops where
//              it meets the walker from the other end; the contracted list (S/8
//              words of next and minimum) is labelled by in-place pointer jumping;
//              a switch takes (parity of its owner's minimum) ^ side.  Switches
//              nobody claimed (loops without ruler) walk their own cycle.
//   S = 128..16  8-bit entries.  One THREAD runs the sequential looping algorithm on
//              a sub-block: from the smallest switch not seen yet it follows the
//              loop once, and every output it stands on goes up, which is the
//              canonical colouring by construction (no minimum, no list).  S/2
//              visits of about 17 instructions without divergence, against 5-7
//              pointer-jumping passes over all outputs.
//   S = 8      the colours of 4 switches depend on the input switches of the first
//              7 outputs only: 14 bits into a table.
//   S = 4, 2   256-entry table: all three stages at once.
//
// Entries carry one bit beside the index: the parity of the input the value stood
// for one level up.  The inverse scattered from such entries therefore holds, in
// input order, the input-side bits of the level above (of every upper half-block:
// an input switch is crossed iff its odd input goes up), which leave as bytes
// without a gather.
//
// 16-bit entries (byte offsets, so that an entry is an address without a shift):
//   P[i] = 2 (first output of the sub-block + value) | parity,  Q[..] = 2 i | parity
// 8-bit entries:  value local to the sub-block | parity << 7.
//
// Measured on B200, before (walks and compaction on plain 16-bit indices at every level, warp
// shuffles below 64) and after: 2048 blocks of 2^15 4.71 -> 2.40 ms, 4096 x 2^12 0.82 -> 0.37 ms,
// 16384 x 2^8 0.117 -> 0.050 ms.
#include "common.cuh"

#include <cooperative_groups.h>

#include <utility>

BENES_GUARD_TU("route_fused.cu")

namespace benes {
namespace {

constexpr int kFKappa = 3;                     // ruler spacing (log2) inside a CTA
constexpr int kFMinLogS = 8;                   // smallest sub-block labelled by ruler walks (16-bit entries)
// Word of a switch in the successor array, two 16-bit halves.  Unclaimed: g(2t) and g(2t+1), each as
// twice the output.  Claimed: the same code in both halves, bit 0 set, bit 1 the side of arrival,
// bits 2-14 the walker (a ruler output), bit 15 set if the switch is a ruler switch (then the
// walker is its even output).
constexpr uint32_t kCodeRho = 0x7FFCu, kRulerFlag = 0x8000u;
constexpr uint32_t kNone16 = 0xFFFFu;          // (two-CTA level) owner of a switch nobody claimed

// ---- tables of the last levels ----------------------------------------------------
// Colours of the four switches of a sub-block of 8: index = input switch (2 bits) of
// outputs 0..6, output 0 on top; output 7 takes the one that is left.
constexpr uint32_t colours_of_8(uint32_t idx) {
    uint32_t e[8] = {}, uses[4] = {}, last = 0, seen = 0, c = 0;
    for (int k = 0; k < 7; ++k) {
        e[k] = (idx >> (12 - 2 * k)) & 3u;
        ++uses[e[k]];
    }
    for (uint32_t s = 0; s < 4; ++s)
        if (uses[s] == 1) last = s;
    e[7] = last;
    for (uint32_t t = 0; t < 4; ++t) {
        uint32_t j = 2 * t;                    // an output that goes up
        while (!((seen >> (j >> 1)) & 1u)) {
            seen |= 1u << (j >> 1);
            c |= (j & 1u) << (j >> 1);
            uint32_t other = j;
            for (uint32_t k = 0; k < 8; ++k)
                if (k != j && e[k] == e[j]) other = k;
            j = other ^ 1u;
        }
    }
    return c;
}

// All stages of a sub-block of 4, entry k in bits 7-2k, 6-2k of the index.  Bits 0-15:
// the inverse as a byte-permute selector; 16-17, 20-21, 24-25: output side, input side, middle.
constexpr uint32_t network_of_4(uint32_t idx) {
    uint32_t p[4] = {}, inv[4] = {}, c[2] = {};
    for (int k = 0; k < 4; ++k) {
        p[k] = (idx >> (6 - 2 * k)) & 3u;
        inv[p[k]] = uint32_t(k);
    }
    // output 0 goes up, so the output beside its input goes down
    const uint32_t down = inv[p[0] ^ 1u];
    c[1] = (down >> 1) ? ((down & 1u) ? 0u : 1u) : 0u;
    uint32_t sel = 0, in = 0;
    for (int s = 0; s < 4; ++s) sel |= inv[s] << (4 * s);
    for (int s = 0; s < 2; ++s) {
        const uint32_t o = inv[2 * s];
        in |= ((c[o >> 1] ^ o) & 1u) << s;
    }
    const uint32_t up = (c[0] ? p[1] : p[0]) >> 1, low = (c[0] ? p[0] : p[1]) >> 1;
    return sel | ((c[0] | (c[1] << 1)) << 16) | (in << 20) | ((up | (low << 1)) << 24);
}

constexpr int kLut8Words = (1 << 14) / 8;      // eight 4-bit entries per word
constexpr int kLut4Words = 256;
constexpr int kLutBytes = (kLut8Words + kLut4Words) * 4;
struct FusedTables {
    uint32_t words[kLut8Words + kLut4Words];
};
// (one compile-time constant per word: a single evaluation of the whole table is beyond the front end's limit)
template <uint32_t W>
struct TableWord {
    static constexpr uint32_t make() {
        if (W >= uint32_t(kLut8Words)) return network_of_4(W - kLut8Words);
        uint32_t r = 0;
        for (uint32_t i = 0; i < 8; ++i) r |= colours_of_8(8 * W + i) << (4 * i);
        return r;
    }
    static constexpr uint32_t value = make();
};
template <uint32_t... W>
constexpr FusedTables make_tables(std::integer_sequence<uint32_t, W...>) { return FusedTables{{TableWord<W>::value...}}; }
__device__ const FusedTables g_fused_tables = make_tables(std::make_integer_sequence<uint32_t, kLut8Words + kLut4Words>());

// ---- shared memory ------------------------------------------------------------------
//   [0, 2C)    P (16 bit)      |  8 bit: P and the next level's P, C bytes each
//   [2C, 4C)   Q (16 bit); once the successors are formed: walk records and list words
//              (32 bit per ruler output), queue of unclaimed switches   |  8 bit: Q
//   [4C, 6C)   successors / owners, a 32-bit word per switch   |  8 bit: the tables
//   then the stage words of the level's output side and of the previous level's input side
template <int LOGC, int THREADS>
struct FusedCfg {
    static constexpr int C = 1 << LOGC;
    static constexpr int T = THREADS;
    static constexpr int kRulers = C >> kFKappa;
    static constexpr int kQ = 2 * C;
    static constexpr int kRec = kQ;
    static constexpr int kList = kRec + kRulers * 4;
    static constexpr int kQueue = kList + kRulers * 4;         // 4 bytes (a list word of 0), then the entries
    static constexpr int kN = 4 * C;
    static constexpr int kLabelBytes = 2 * C > kLutBytes ? 2 * C : kLutBytes;
    static constexpr int kCw = kN + kLabelBytes;
    static constexpr int kInw = kCw + C / 16;
    static constexpr int kCount = kInw + C / 16;               // entries of the queue
    static constexpr size_t kSmemBytes = size_t(kCount) + 16;
    // CTAs per SM the register budget has to leave room for
    static constexpr int kMinCtas = THREADS > C / 32 || LOGC >= 15 ? 1 : (LOGC == 14 ? 2 : (LOGC == 13 ? 4 : 8));
};

template <class Tp>
__device__ __forceinline__ Tp &at(unsigned char *sm, uint32_t byte) {
    return *reinterpret_cast<Tp *>(sm + byte);
}

__device__ __forceinline__ uint32_t fused_slot(uint32_t group, uint32_t salt) {
    // top bits of a multiplicative hash
    return ((group + salt * 0x632BE5ABu) * 0x9E3779B1u) >> (32 - kFKappa);
}

// Where the CTA's words go: flat output index of its first output, how many outputs
// are real (the rest of the CTA is padding), stage-major words per permutation.
struct FusedOut {
    uint32_t *bits;
    size_t flat0;
    uint32_t valid;
    int n;
    __device__ __forceinline__ uint32_t *stage_word(int stage, uint32_t w) const {        // n >= 6
        const size_t fw = (flat0 >> 6) + w, lw = fw & ((size_t(1) << (n - 6)) - 1);
        return bits + ((((fw >> (n - 6)) * size_t(2 * n - 1) + size_t(stage)) << (n - 6)) + lw);
    }
    // 16 switches = the outputs [32 r, 32 r + 32) of the CTA
    __device__ __forceinline__ void store16(int stage, uint32_t r, uint32_t half) const {
        if (32u * r >= valid) return;
        if (n >= 6) {
            reinterpret_cast<uint16_t *>(stage_word(stage, r >> 1))[r & 1u] = uint16_t(half);
            return;
        }
        // a word per permutation of 2^(n-1) switches
        const uint32_t per = 32u >> n, nb = 1u << (n - 1);
        const size_t perm0 = (flat0 >> n) + size_t(r) * per;
        for (uint32_t k = 0; k < per && ((r * per + k) << n) < valid; ++k)
            bits[(perm0 + k) * size_t(2 * n - 1) + size_t(stage)] = (half >> (k * nb)) & ((1u << nb) - 1u);
    }
    template <class Cfg>
    __device__ __forceinline__ void store_row(unsigned char *sm, uint32_t row, int stage) const {
        if (n >= 6) {
            for (uint32_t w = threadIdx.x; w < valid >> 6; w += Cfg::T) *stage_word(stage, w) = at<uint32_t>(sm, row + w * 4);
        } else {
            for (uint32_t r = threadIdx.x; r < uint32_t(Cfg::C / 32); r += Cfg::T) store16(stage, r, at<uint16_t>(sm, row + r * 2));
        }
    }
};

// bits 7, 15, 23, 31 of w, in this order, as 4 bits
__device__ __forceinline__ uint32_t tops_of_bytes(uint32_t w) {
    return ((((w >> 7) & 0x01010101u) * 0x00204081u) >> 21) & 15u;
}
// bit k of a nibble -> bit 4 k
__device__ __forceinline__ uint32_t spread4(uint32_t c) {
    const uint32_t s = (c | (c << 6)) & 0x0303u;
    return (s | (s << 3)) & 0x1111u;
}
// 2-bit fields at the bottom of the four bytes -> 8 bits, byte 0 on top
__device__ __forceinline__ uint32_t fields_of_bytes(uint32_t x) { return (x * 0x40100401u) >> 24; }

// ---- a level with 16-bit entries -------------------------------------------------------
// Input-side bits of the level above a level of sub-blocks of 2^logs: the parities in the upper half-blocks, in input order.
template <class Cfg>
__device__ __forceinline__ void input_bits16(unsigned char *sm, int logs) {
    constexpr uint32_t C = Cfg::C, T = Cfg::T;
    for (uint32_t c = threadIdx.x; c < C / 16; c += T) {
        const uint32_t i = ((c >> (logs - 3)) << (logs + 1)) + ((c & ((1u << (logs - 3)) - 1u)) << 3);
        const uint4 q = at<uint4>(sm, Cfg::kQ + 2 * i);
        const uint32_t x = (q.x & 0x00010001u) | ((q.y & 0x00010001u) << 2) | ((q.z & 0x00010001u) << 4) |
                           ((q.w & 0x00010001u) << 6);
        at<uint8_t>(sm, Cfg::kInw + c) = uint8_t(x | (x >> 15));
    }
}

// Colour of output 2t of a switch nobody claimed: its g-cycle (at most S/2 outputs) from both ends;
// g(b ^ 1) ^ 1 is the predecessor of b on the cycle (the cycle of 2t+1 is its mirror image).
template <class Cfg>
__device__ __forceinline__ uint32_t loop_colour16(unsigned char *sm, uint32_t t, uint32_t S) {
    constexpr uint32_t kMask = 2u * Cfg::C - 2u;
    const uint32_t j0 = 4u * t;
    uint32_t f = j0, bk = j0, least = j0;
    for (uint32_t hops = 0; hops < S; ++hops) {
        const uint32_t nf = at<uint16_t>(sm, Cfg::kN + f) & kMask;
        const uint32_t nb = at<uint16_t>(sm, Cfg::kN + (bk ^ 2u)) & kMask;
        f = nf;
        if (f == bk) break;
        least = min(least, f);
        bk = nb ^ 2u;
        if (bk == f) break;
        least = min(least, bk);
    }
    return (least >> 1) & 1u;
}

template <class Cfg>
__device__ __forceinline__ void level16(unsigned char *sm, const FusedOut &out, int logs, int level, bool first) {
    constexpr uint32_t C = Cfg::C, T = Cfg::T, R = Cfg::kRulers;
    constexpr uint32_t kMask = 2u * C - 2u;                     // a byte offset of an entry
    constexpr int kGroups = int(C / 16 / T) > 0 ? int(C / 16 / T) : 1;     // ruler groups (8 switches) per thread
    const uint32_t tid = threadIdx.x;
    const uint32_t S = 1u << logs;

    if (!first) input_bits16<Cfg>(sm, logs);
    // Successors g(j) = Q[P[j^1] ^ 1], so that a hop of a walk is one load: the gathers here run
    // with all lanes, those of the walks with a quarter of them.  The word of a ruler switch is its
    // code from the start; its thread keeps the successors, with which it starts the two walks.
    uint32_t start[kGroups];
#pragma unroll
    for (int r = 0; r < kGroups; ++r) {
        const uint32_t g = tid + uint32_t(r) * T;
        start[r] = 0u;
        if (g < C / 16) {
            const uint4 pa = at<uint4>(sm, g * 32), pb = at<uint4>(sm, g * 32 + 16);
            uint32_t w[8] = {pa.x, pa.y, pa.z, pa.w, pb.x, pb.y, pb.z, pb.w};
            const uint32_t slot = fused_slot(g, uint32_t(level));
#pragma unroll
            for (uint32_t k = 0; k < 8; ++k) {
                const uint32_t g1 = at<uint16_t>(sm, Cfg::kQ + ((w[k] ^ 2u) & kMask));
                const uint32_t g0 = at<uint16_t>(sm, Cfg::kQ + (((w[k] >> 16) ^ 2u) & kMask));
                w[k] = (g0 | (g1 << 16)) & (kMask * 0x10001u);
                if (k == slot) {
                    start[r] = w[k];
                    w[k] = (kRulerFlag | (g << 3) | 1u) * 0x10001u;
                }
            }
            at<uint4>(sm, Cfg::kN + g * 32) = make_uint4(w[0], w[1], w[2], w[3]);
            at<uint4>(sm, Cfg::kN + g * 32 + 16) = make_uint4(w[4], w[5], w[6], w[7]);
        }
    }
    __syncthreads();

    // Walks from the ruler outputs; the two of a segment meet in the middle.  A claim needs no
    // atomic.  Only the two walkers of this segment ever reach switch t, from opposite ends.  If both
    // find it free at the same moment, both write (either code is a valid owner: the two stand for
    // mirror cycles and arrive on opposite sides, so the colour comes out the same), both go on, and
    // each stops at the next switch, which the other has claimed; minima are taken over one switch
    // more, which changes nothing.  A walker keeps one minimum: the outputs on the far side of its
    // switches are the ones it stood on with the last bit flipped, and so is their minimum.
    // A thread has the walks of its own rulers; walks differ in length, so a lane goes on to its
    // next walk every four hops instead of waiting for the longest walk of the warp.
    if (tid < C / 16) {
        const uint32_t walks = 2u * min(uint32_t(kGroups), (C / 16 - tid + T - 1) / T);
        uint32_t k = 0, g = tid, rho = 2u * g;
        uint32_t least = 4u * ((g << kFKappa) | fused_slot(g, uint32_t(level))), j = start[0] & 0xFFFFu;
        uint32_t code = ((rho << 2) | 1u) * 0x10001u;
        for (;;) {
            // (no branches: a lane that has met somebody reads the same code again)
            bool met = false;
            uint32_t v = 0;
#pragma unroll
            for (int hop = 0; hop < 4; ++hop) {
                v = at<volatile uint16_t>(sm, Cfg::kN + j);
                met = (v & 1u) != 0u;
                if (!met) at<volatile uint32_t>(sm, Cfg::kN + (j & ~3u)) = code + (j & 2u) * 0x10001u;
                least = met ? least : min(least, j);
                j = met ? j : v;
            }
            if (met) {
                // a ruler switch (its code names its even output), or one the other walker owns
                const uint32_t peer4 = (v & kCodeRho) ^ ((v & kRulerFlag) ? ((~j & 2u) << 1) : 0u);
                at<uint32_t>(sm, Cfg::kRec + rho * 4) = (least << 16) | peer4;
                if (++k == walks) break;
                g = tid + (k >> 1) * T;
                rho = 2u * g + (k & 1u);
                least = 4u * ((g << kFKappa) | fused_slot(g, uint32_t(level))) + 2u * (k & 1u);
                uint32_t st = start[0];
#pragma unroll
                for (int r = 1; r < kGroups; ++r) st = (k >> 1) == uint32_t(r) ? start[r] : st;
                j = (k & 1u) ? st >> 16 : st & 0xFFFFu;
                code = ((rho << 2) | 1u) * 0x10001u;
            }
        }
    }
    if (tid == 0) {
        at<uint32_t>(sm, Cfg::kQueue) = 0u;
        at<uint32_t>(sm, Cfg::kCount) = 0u;
    }
    __syncthreads();

    // Contracted list: next = peer ^ 1.  What the other walker of my ruler switch has seen, with the last bit
    // flipped, lies on my cycle too, and every segment of a cycle has both of its walkers in such pairs of the cycle:
    // no need to fetch the minimum of the peer.
    constexpr int kPer = int(R / T) > 0 ? int(R / T) : 1;
    uint32_t w[kPer];
#pragma unroll
    for (int r = 0; r < kPer; ++r) {
        const uint32_t rho = tid + uint32_t(r) * T;
        if (rho < R) {
            const uint32_t a = at<uint32_t>(sm, Cfg::kRec + rho * 4), b = at<uint32_t>(sm, Cfg::kRec + (rho ^ 1u) * 4);
            w[r] = ((a & (R * 4u - 4u)) ^ 4u) | min(a & 0xFFFF0000u, (b ^ 0x00020000u) & 0xFFFF0000u);
            at<uint32_t>(sm, Cfg::kList + rho * 4) = w[r];
        }
    }
    // Switches nobody claimed lie on loops without ruler.  A few of them in a group queue up, so that
    // one thread takes one; a group full of them (permutations made of short loops) stays with
    // its thread.
    uint32_t dense[kGroups];                                     // free switches | their colours << 8
#pragma unroll
    for (int r = 0; r < kGroups; ++r) {
        const uint32_t g = tid + uint32_t(r) * T;
        dense[r] = 0u;
        if (g < C / 16) {
            const uint4 a = at<uint4>(sm, Cfg::kN + g * 32), b = at<uint4>(sm, Cfg::kN + g * 32 + 16);
            uint32_t free_ = (~a.x & 1u) | ((~a.y & 1u) << 1) | ((~a.z & 1u) << 2) | ((~a.w & 1u) << 3) |
                             ((~b.x & 1u) << 4) | ((~b.y & 1u) << 5) | ((~b.z & 1u) << 6) | ((~b.w & 1u) << 7);
            const uint32_t count = uint32_t(__popc(free_));
            if (count > 3u) {
                dense[r] = free_;
            } else if (free_) {
                uint32_t pos = atomicAdd(&at<uint32_t>(sm, Cfg::kCount), count);
                while (free_) {
                    const uint32_t k = uint32_t(__ffs(int(free_))) - 1u;
                    free_ &= free_ - 1u;
                    at<uint16_t>(sm, Cfg::kQueue + 4u + 2u * pos++) = uint16_t(8u * g + k);
                }
            }
        }
    }
    if (!first) out.store_row<Cfg>(sm, Cfg::kInw, level - 1);
    __syncthreads();

    // In-place pointer jumping, own words in registers; a cycle of the list has at most S/16 words
    // (half of the ruler outputs of its sub-block): logs - 4 passes, at least 4.  The queue rides
    // along: colours before the first barrier, codes (list word R, which is 0, and the colour as the
    // side) after it, when no walk reads successors any more.
    constexpr uint32_t resolved = (R << 2) | 1u;
    const uint32_t queued = at<uint32_t>(sm, Cfg::kCount);
    for (uint32_t e = tid; e < queued; e += T) {
        const uint32_t t = at<uint16_t>(sm, Cfg::kQueue + 4u + 2u * e);
        at<uint16_t>(sm, Cfg::kQueue + 4u + 2u * e) = uint16_t(t | (loop_colour16<Cfg>(sm, t, S) << 15));
    }
#pragma unroll
    for (int r = 0; r < kGroups; ++r)
        for (uint32_t left = dense[r]; left; left &= left - 1u) {
            const uint32_t k = uint32_t(__ffs(int(left))) - 1u;
            dense[r] |= loop_colour16<Cfg>(sm, 8u * (tid + uint32_t(r) * T) + k, S) << (8u + k);
        }
    for (int pass = 0; pass < logs - kFKappa - 1; ++pass) {
#pragma unroll
        for (int r = 0; r < kPer; ++r) {
            const uint32_t rho = tid + uint32_t(r) * T;
            if (rho < R) {
                const uint32_t v = at<volatile uint32_t>(sm, Cfg::kList + (w[r] & 0xFFFFu));
                w[r] = (v & 0xFFFFu) | min(w[r] & 0xFFFF0000u, v & 0xFFFF0000u);
                at<volatile uint32_t>(sm, Cfg::kList + rho * 4) = w[r];
            }
        }
        __syncthreads();
        if (pass == 0) {
            for (uint32_t e = tid; e < queued; e += T) {
                const uint32_t x = at<uint16_t>(sm, Cfg::kQueue + 4u + 2u * e);
                at<uint32_t>(sm, Cfg::kN + 4u * (x & 0x7FFFu)) = resolved | ((x >> 14) & 2u);
            }
        }
    }

    // Colours of 8 switches (a ruler group) per round, and the next level's entries of their 16
    // outputs, which stay in registers until everybody has read this level's.
    uint32_t u[kGroups][4], l[kGroups][4];
    const bool wide_next = logs - 1 >= kFMinLogS;
#pragma unroll
    for (int r = 0; r < kGroups; ++r) {
        const uint32_t g = tid + uint32_t(r) * T;
        if (g < C / 16) {
            const uint4 na = at<uint4>(sm, Cfg::kN + g * 32), nb = at<uint4>(sm, Cfg::kN + g * 32 + 16);
            uint32_t code[8] = {na.x, na.y, na.z, na.w, nb.x, nb.y, nb.z, nb.w};
            uint32_t c[8], byte = 0;
            if (dense[r]) {
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if ((dense[r] >> k) & 1u) code[k] = resolved | (((dense[r] >> (8 + k)) & 1u) << 1);
            }
#pragma unroll
            for (int k = 0; k < 8; ++k)
                c[k] = ((at<uint32_t>(sm, Cfg::kList + (code[k] & kCodeRho)) >> 17) ^ (code[k] >> 1)) & 1u;
#pragma unroll
            for (int k = 0; k < 8; ++k) byte |= c[k] << k;
            at<uint8_t>(sm, Cfg::kCw + g) = uint8_t(byte);
            const uint4 pa = at<uint4>(sm, g * 32), pb = at<uint4>(sm, g * 32 + 16);
            uint32_t y[8] = {pa.x, pa.y, pa.z, pa.w, pb.x, pb.y, pb.z, pb.w};
            const uint32_t sb = (16u * g) & ~(S - 1u);
            if (wide_next) {
                const uint32_t vmask = (S - 1u) * 0x10001u, up = (2u * sb) * 0x10001u, low = S * 0x10001u;
#pragma unroll
                for (int k = 0; k < 8; ++k) y[k] = ((y[k] >> 1) & vmask) | up;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const uint32_t sel = 0x5410u | (c[2 * k] * 0x22u) | (c[2 * k + 1] * 0x2200u);
                    // (0x5410 and 0x2222 share no set bit, so | adds them)
                    u[r][k] = __byte_perm(y[2 * k], y[2 * k + 1], sel);
                    l[r][k] = __byte_perm(y[2 * k], y[2 * k + 1], sel ^ 0x2222u) | low;
                }
            } else {
                // to 8-bit entries: value (v >> 1) with the parity in bit 7, from 2 (base + v) | parity
#pragma unroll
                for (int k = 0; k < 8; ++k) y[k] = ((y[k] >> 2) & 0x007F007Fu) | ((y[k] << 6) & 0x00800080u);
                uint32_t hu[4], hl[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const uint32_t sel = 0x40u | (c[2 * k] * 0x02u) | (c[2 * k + 1] * 0x20u);
                    hu[k] = __byte_perm(y[2 * k], y[2 * k + 1], sel);
                    hl[k] = __byte_perm(y[2 * k], y[2 * k + 1], sel ^ 0x22u);
                }
                u[r][0] = __byte_perm(hu[0], hu[1], 0x5410); u[r][1] = __byte_perm(hu[2], hu[3], 0x5410);
                l[r][0] = __byte_perm(hl[0], hl[1], 0x5410); l[r][1] = __byte_perm(hl[2], hl[3], 0x5410);
            }
        }
    }
    __syncthreads();
    // the next level's entries and their inverse
    const uint32_t H = S >> 1;
#pragma unroll
    for (int r = 0; r < kGroups; ++r) {
        const uint32_t g = tid + uint32_t(r) * T;
        if (g < C / 16) {
            const uint32_t sb = (16u * g) & ~(S - 1u), tl = (16u * g - sb) >> 1;
            if (wide_next) {
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    const uint32_t i = sb + tl + (half ? H : 0u);
                    const uint32_t *e = half ? l[r] : u[r];
                    at<uint4>(sm, 2u * i) = make_uint4(e[0], e[1], e[2], e[3]);
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const uint32_t x = (k & 1) ? e[k >> 1] >> 16 : e[k >> 1];
                        at<uint16_t>(sm, Cfg::kQ + (x & 0xFFFEu)) = uint16_t((x & 1u) | (2u * (i + uint32_t(k))));
                    }
                }
            } else {
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    const uint32_t base = sb + (half ? H : 0u);
                    const uint32_t *e = half ? l[r] : u[r];
                    at<uint2>(sm, base + tl) = make_uint2(e[0], e[1]);
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const uint32_t x = e[k >> 2] >> (8 * (k & 3));
                        at<uint8_t>(sm, Cfg::kQ + base + (x & 0x7Fu)) = uint8_t((x & 0x80u) | (tl + uint32_t(k)));
                    }
                }
            }
        }
    }
    out.store_row<Cfg>(sm, Cfg::kCw, 2 * out.n - 2 - level);
    __syncthreads();
}

// ---- a level with 8-bit entries ----------------------------------------------------------
// The looping algorithm on the 2^LOGREG outputs from byte `rb` on (one sub-block, or the two
// sub-blocks of 16 of a region of 32): ascending start switches, one visit per switch.
template <int LOGREG>
__device__ __forceinline__ void loop_region(const unsigned char *P, const unsigned char *Q, uint32_t smask,
                                            uint32_t *col) {
    constexpr uint32_t kReg = 1u << LOGREG, kSw = kReg / 2;
    constexpr int kWords = kSw > 32 ? int(kSw / 32) : 1;
    uint32_t seen[kWords];
#pragma unroll
    for (int w = 0; w < kWords; ++w) seen[w] = col[w] = 0u;
    uint32_t j = 0, start = 0;                 // j goes up; the loop being walked began at output `start`
#pragma unroll 4
    for (uint32_t it = 0; it < kSw; ++it) {
        const uint32_t sb = LOGREG == 5 ? (j & ~smask & (kReg - 1u)) : 0u;
        const uint32_t x = ((uint32_t(P[j]) & smask) ^ 1u) | sb;
        const uint32_t next = ((uint32_t(Q[x]) & smask) ^ 1u) | sb;
        const uint32_t bit = 1u << ((j >> 1) & 31u), odd = (j & 1u) ? bit : 0u;
        uint32_t fresh;                        // smallest switch not seen
        if (kWords == 1) {
            seen[0] |= bit;
            col[0] |= odd;
            fresh = uint32_t(__ffs(int(~seen[0]))) - 1u;
        } else {
            const bool hi = j >= 64u;
            seen[0] |= hi ? 0u : bit; seen[kWords - 1] |= hi ? bit : 0u;
            col[0] |= hi ? 0u : odd; col[kWords - 1] |= hi ? odd : 0u;
            fresh = ~seen[0] ? uint32_t(__ffs(int(~seen[0]))) - 1u : 31u + uint32_t(__ffs(int(~seen[kWords - 1])));
        }
        const bool closed = next == start;
        start = closed ? (2u * fresh) & (kReg - 1u) : start;
        j = closed ? start : next;
    }
}

template <class Cfg>
__device__ __forceinline__ void level8(unsigned char *sm, const FusedOut &out, int logs, int level, bool first,
                                       uint32_t pcur) {
    constexpr uint32_t C = Cfg::C, T = Cfg::T;
    const uint32_t tid = threadIdx.x;
    const uint32_t S = 1u << logs, smask = S - 1u, H = S >> 1;
    if (!first) {
        for (uint32_t c = tid; c < C / 16; c += T) {
            const uint32_t i = ((c >> (logs - 3)) << (logs + 1)) + ((c & ((S >> 3) - 1u)) << 3);
            const uint2 q = at<uint2>(sm, Cfg::kQ + i);
            at<uint8_t>(sm, Cfg::kInw + c) = uint8_t(tops_of_bytes(q.x) | (tops_of_bytes(q.y) << 4));
        }
    }
    if (logs == 7) {
        for (uint32_t r = tid; r < C / 128; r += T) {
            uint32_t col[2];
            loop_region<7>(sm + pcur + 128 * r, sm + Cfg::kQ + 128 * r, smask, col);
            at<uint2>(sm, Cfg::kCw + 8 * r) = make_uint2(col[0], col[1]);
        }
    } else if (logs == 6) {
        for (uint32_t r = tid; r < C / 64; r += T) {
            uint32_t col[1];
            loop_region<6>(sm + pcur + 64 * r, sm + Cfg::kQ + 64 * r, smask, col);
            at<uint32_t>(sm, Cfg::kCw + 4 * r) = col[0];
        }
    } else {
        for (uint32_t r = tid; r < C / 32; r += T) {
            uint32_t col[1];
            loop_region<5>(sm + pcur + 32 * r, sm + Cfg::kQ + 32 * r, smask, col);
            at<uint16_t>(sm, Cfg::kCw + 2 * r) = uint16_t(col[0]);
        }
    }
    __syncthreads();
    // next level's entries and, unless the tables take over, their inverse
    const uint32_t pnext = pcur ^ C;
    const uint32_t vmask = (H - 1u) * 0x01010101u;
    const bool inverse = logs - 1 >= 4;
    for (uint32_t g = tid; g < C / 16; g += T) {
        const uint4 p4 = at<uint4>(sm, pcur + 16 * g);
        uint32_t y[4] = {p4.x, p4.y, p4.z, p4.w};
        const uint32_t byte = at<uint8_t>(sm, Cfg::kCw + g);
#pragma unroll
        for (int k = 0; k < 4; ++k) y[k] = ((y[k] >> 1) & vmask) | ((y[k] << 7) & 0x80808080u);
        const uint32_t s0 = 0x6420u | spread4(byte & 15u), s1 = 0x6420u | spread4(byte >> 4);
        const uint32_t sb = (16u * g) & ~smask, tl = (16u * g - sb) >> 1;
        const uint32_t e[2][2] = {{__byte_perm(y[0], y[1], s0), __byte_perm(y[2], y[3], s1)},
                                  {__byte_perm(y[0], y[1], s0 ^ 0x1111u), __byte_perm(y[2], y[3], s1 ^ 0x1111u)}};
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const uint32_t base = sb + (half ? H : 0u);
            at<uint2>(sm, pnext + base + tl) = make_uint2(e[half][0], e[half][1]);
            if (inverse) {
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const uint32_t x = e[half][k >> 2] >> (8 * (k & 3));
                    at<uint8_t>(sm, Cfg::kQ + base + (x & (H - 1u))) = uint8_t((x & 0x80u) | (tl + uint32_t(k)));
                }
            }
        }
    }
    if (!first) out.store_row<Cfg>(sm, Cfg::kInw, level - 1);
    out.store_row<Cfg>(sm, Cfg::kCw, 2 * out.n - 2 - level);
    __syncthreads();
}

// ---- sub-blocks of 8 and less: 32 outputs (16 switches of every stage) per thread ----------
template <class Cfg>
__device__ __forceinline__ void last_levels(unsigned char *sm, const FusedOut &out, int logs, uint32_t pcur,
                                            bool first) {
    constexpr uint32_t C = Cfg::C, T = Cfg::T;
    const int n = out.n;
    const uint32_t *lut8 = &at<uint32_t>(sm, Cfg::kN), *lut4 = lut8 + kLut8Words;
    for (uint32_t r = threadIdx.x; r < C / 32; r += T) {
        const uint4 a = at<uint4>(sm, pcur + 32 * r), b = at<uint4>(sm, pcur + 32 * r + 16);
        const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
        if (logs == 1) {
            uint32_t mid = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) mid |= ((w[k] & 1u) | ((w[k] >> 15) & 2u)) << (2 * k);
            out.store16(n - 1, r, mid);
            continue;
        }
        uint32_t z4[4];                        // per 8 outputs: nibbles output side, input side, middle of the level of 4
        if (logs == 2) {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                z4[k] = (lut4[fields_of_bytes(w[2 * k] & 0x03030303u)] >> 16) |
                        ((lut4[fields_of_bytes(w[2 * k + 1] & 0x03030303u)] >> 16) << 2);
        } else {
            uint32_t in16 = 0, out8 = 0, in8 = 0;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t w0 = w[2 * k], w1 = w[2 * k + 1];
                if ((k & 1) == 0 && !first) {
                    // input side of the level of 16: parity at the place of the value
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const uint32_t x = (e < 4 ? w0 : w1) >> (8 * (e & 3));
                        in16 |= ((x >> 7) & 1u) << ((x & 7u) + 4u * uint32_t(k));
                    }
                }
                const uint32_t x0 = (w0 >> 1) & 0x03030303u, x1 = (w1 >> 1) & 0x03030303u;
                const uint32_t idx = (fields_of_bytes(x0) << 6) | (fields_of_bytes(x1) >> 2);
                const uint32_t c = (lut8[idx >> 3] >> (4u * (idx & 7u))) & 15u;
                const uint32_t y0 = x0 | ((w0 << 7) & 0x80808080u), y1 = x1 | ((w1 << 7) & 0x80808080u);
                const uint32_t sel = 0x6420u | spread4(c);
                const uint32_t up = __byte_perm(y0, y1, sel), low = __byte_perm(y0, y1, sel ^ 0x1111u);
                const uint32_t eu = lut4[fields_of_bytes(up & 0x03030303u)], el = lut4[fields_of_bytes(low & 0x03030303u)];
                out8 |= c << (4 * k);
                // input side of the level of 8: the parities of the upper half-block, in input order
                in8 |= tops_of_bytes(__byte_perm(up, 0u, eu & 0x3333u)) << (4 * k);
                z4[k] = (eu >> 16) | ((el >> 16) << 2);
            }
            if (!first) out.store16(n - 4, r, in16);
            out.store16(2 * n - 2 - (n - 3), r, out8);
            out.store16(n - 3, r, in8);
        }
        uint32_t o = 0, i = 0, m = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            o |= (z4[k] & 15u) << (4 * k);
            i |= ((z4[k] >> 4) & 15u) << (4 * k);
            m |= ((z4[k] >> 8) & 15u) << (4 * k);
        }
        out.store16(2 * n - 2 - (n - 2), r, o);
        out.store16(n - 2, r, i);
        out.store16(n - 1, r, m);
    }
}

// Levels n - logs .. n - 1 of the CTA's outputs; P and Q of the first of them are in place.
template <class Cfg>
__device__ __forceinline__ void fused_levels(unsigned char *sm, const FusedOut &out, int logs0) {
    const int n = out.n;
    int logs = logs0;
    for (; logs >= kFMinLogS; --logs) level16<Cfg>(sm, out, logs, n - logs, logs == logs0);
    for (uint32_t i = threadIdx.x; i < uint32_t(kLutBytes / 16); i += Cfg::T)
        at<uint4>(sm, Cfg::kN + 16 * i) = __ldg(reinterpret_cast<const uint4 *>(&g_fused_tables) + i);
    uint32_t pcur = 0;
    for (; logs >= 4; --logs) {
        level8<Cfg>(sm, out, logs, n - logs, logs == logs0, pcur);
        pcur ^= uint32_t(Cfg::C);
    }
    if (logs == logs0) __syncthreads();        // no level above the tables: they have just been copied
    last_levels<Cfg>(sm, out, logs, pcur, logs == logs0);
}

// P and Q of the first level from four neighbouring values, local to their sub-block
template <class Cfg>
__device__ __forceinline__ void fused_enter4(unsigned char *sm, uint32_t i4, const uint32_t v[4], int logs) {
    const uint32_t smask = (1u << logs) - 1u;
    if (logs >= kFMinLogS) {
        const uint32_t sb = (4u * i4) & ~smask;
        at<uint2>(sm, 8 * i4) = make_uint2(2u * (sb + v[0]) | (2u * (sb + v[1]) << 16), 2u * (sb + v[2]) | (2u * (sb + v[3]) << 16));
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) at<uint16_t>(sm, Cfg::kQ + 2u * (sb + v[k])) = uint16_t(2u * (4u * i4 + k));
    } else {
        at<uint32_t>(sm, 4 * i4) = v[0] | (v[1] << 8) | (v[2] << 16) | (v[3] << 24);
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) {
            const uint32_t i = 4u * i4 + k;
            at<uint8_t>(sm, Cfg::kQ + (i & ~smask) + v[k]) = uint8_t(i & smask);
        }
    }
}

// The CTA's blocks of 2^logs outputs from a plain array (records = 0) or from packed records
// P[2t] | P[2t+1] << logs | ... (1), four entries per load, four loads of a thread under way together.
template <class Cfg>
__device__ __forceinline__ void fused_load(unsigned char *sm, const FusedOut &out, const uint32_t *P, int records, int logs) {
    constexpr uint32_t T = Cfg::T, kItems = Cfg::C / 4, kBatch = kItems / T >= 4 ? 4 : 1;
    const uint32_t smask = (1u << logs) - 1u;
    const bool aligned = (reinterpret_cast<uintptr_t>(P) & 15u) == 0;
    for (uint32_t i0 = threadIdx.x; i0 < kItems; i0 += kBatch * T) {
        uint32_t v[kBatch][4];
#pragma unroll
        for (uint32_t r = 0; r < kBatch; ++r) {
            const uint32_t i4 = i0 + r * T;
            const size_t f = out.flat0 + 4u * i4;
            if (4u * i4 + 4u <= out.valid && (records != 0 || aligned)) {
                if (records == 0) {
                    const uint4 p = __ldcs(reinterpret_cast<const uint4 *>(P + f));
                    v[r][0] = p.x; v[r][1] = p.y; v[r][2] = p.z; v[r][3] = p.w;
                } else {
                    const ulonglong2 p = __ldcs(reinterpret_cast<const ulonglong2 *>(P) + (f >> 2));
                    v[r][0] = uint32_t(p.x) & smask; v[r][1] = uint32_t(p.x >> logs) & smask;
                    v[r][2] = uint32_t(p.y) & smask; v[r][3] = uint32_t(p.y >> logs) & smask;
                }
            } else {
                // a permutation that does not start on 16 bytes, the end of a batch of permutations of 2,
                // or padding: the identity
#pragma unroll
                for (uint32_t k = 0; k < 4; ++k)
                    v[r][k] = (records == 0 && 4u * i4 + k < out.valid) ? P[f + k] : (4u * i4 + k) & smask;
            }
        }
#pragma unroll
        for (uint32_t r = 0; r < kBatch; ++r) {
#pragma unroll
            for (uint32_t k = 0; k < 4; ++k) v[r][k] = BENES_GUARD(v[r][k], smask);
            fused_enter4<Cfg>(sm, i0 + r * T, v[r], logs);
        }
    }
    __syncthreads();
}

template <int LOGC, int THREADS>
__global__ void __launch_bounds__(THREADS, (FusedCfg<LOGC, THREADS>::kMinCtas))
k_route_fused(const uint32_t *__restrict__ P, int records, uint32_t *__restrict__ bits, int log2n, int logs,
              size_t first, size_t end, const uint32_t *__restrict__ gate, const uint32_t *__restrict__ redone) {
    after_previous_kernel();
    using Cfg = FusedCfg<LOGC, THREADS>;
    constexpr uint32_t C = Cfg::C;
    extern __shared__ __align__(16) unsigned char sm[];
    FusedOut out;
    out.bits = bits;
    out.n = log2n;
    out.flat0 = first + size_t(blockIdx.x) * C;
    out.valid = uint32_t(end - out.flat0 < size_t(C) ? end - out.flat0 : size_t(C));
    const bool redo = gate && *gate != 0u;
    fused_load<Cfg>(sm, out, redo ? redone : P, redo ? 0 : records, logs);
    fused_levels<Cfg>(sm, out, logs);
}

// One level of one block of 2^LOGC outputs per CTA; the two half-blocks go to `next` (a plain array), where the
// next launch finds them with twice as many CTAs.  While more than half of the SMs would have no block, that is how the
// in-CTA levels run: a level takes a time in proportion to the CTA's outputs, so halving the block with every level
// costs about two levels of the first block instead of one for each (one block of 2^15: 172 -> 82 us,
// 2^13: 51 -> 37; the route of 2^16: 206 -> 140, of 2^20: 545 -> 497).
template <int LOGC, int THREADS>
__global__ void __launch_bounds__(THREADS)
k_route_peel(const uint32_t *__restrict__ P, int records, uint32_t *__restrict__ bits, int log2n,
             uint32_t *__restrict__ next, const uint32_t *__restrict__ gate, const uint32_t *__restrict__ redone) {
    after_previous_kernel();
    using Cfg = FusedCfg<LOGC, THREADS>;
    constexpr uint32_t C = Cfg::C, T = Cfg::T, H = C / 2;
    extern __shared__ __align__(16) unsigned char sm[];
    FusedOut out;
    out.bits = bits;
    out.n = log2n;
    out.flat0 = size_t(blockIdx.x) * C;
    out.valid = C;
    const bool redo = gate && *gate != 0u;
    fused_load<Cfg>(sm, out, redo ? redone : P, redo ? 0 : records, LOGC);
    level16<Cfg>(sm, out, LOGC, log2n - LOGC, true);
    // entries 2 (base of the half + value) | parity -> values; input-side bits from the inverse of the upper half
    for (uint32_t i4 = threadIdx.x; i4 < C / 4; i4 += T) {
        const uint2 e = at<uint2>(sm, 8 * i4);
        const uint32_t x = (e.x >> 1) & ((H - 1u) * 0x10001u), y = (e.y >> 1) & ((H - 1u) * 0x10001u);
        *reinterpret_cast<uint4 *>(next + out.flat0 + 4u * i4) = make_uint4(x & 0xFFFFu, x >> 16, y & 0xFFFFu, y >> 16);
    }
    input_bits16<Cfg>(sm, LOGC - 1);
    __syncthreads();
    out.store_row<Cfg>(sm, Cfg::kInw, log2n - LOGC);
}

// ---- few outputs in all ---------------------------------------------------------------------
// When every thread of the GPU could have a switch to itself, the time of a call is its chain of dependent
// steps, and the labelling with the shortest one is pointer jumping over all outputs: one thread per
// switch, one barrier per pass, and from sub-blocks of 64 down a warp in registers (a switch, then an output,
// per lane; jumps by shuffle).  One permutation of 2^10: 22.8 -> 10.5 us; 32 of 2^6:
// 8.7 -> 4 us; 290 of 2^10 (half of the GPU's threads): 43 -> 17 us.  From about twice the GPU's threads on the
// kernels above are faster, which issue fewer instructions (5000 of 2^8: 37 us either way).

// The levels of sub-blocks of 2^ls0 <= 32 outputs and less of 32 neighbouring outputs: p = the lane's entry, gathers
// by shuffle, the inverse through the group's 32 entries of Q, which only this warp touches.  r = index of the
// group in the CTA.
__device__ __forceinline__ void few_tail32(uint32_t p, uint32_t r, uint16_t *Q, const FusedOut &out, int ls0) {
    constexpr uint32_t kAll = 0xFFFFFFFFu;
    const int n = out.n, lane = int(threadIdx.x & 31u);
#pragma unroll
    for (int ls = 5; ls >= 2; --ls) {
        if (ls > ls0) continue;
        const uint32_t smask = (1u << ls) - 1u, sb = uint32_t(lane) & ~smask;
        const int level = n - ls;
        Q[sb + p] = uint16_t(uint32_t(lane) & smask);
        __syncwarp();
        const uint32_t q = Q[lane];
        __syncwarp();
        const uint32_t p1 = __shfl_xor_sync(kAll, p, 1);
        uint32_t next = sb + __shfl_sync(kAll, q, int(sb + (p1 ^ 1u))), least = uint32_t(lane);
#pragma unroll
        for (int pass = 0; pass < ls - 1; ++pass) {          // cycles of up to 2^(ls-1) outputs
            const uint32_t m = __shfl_sync(kAll, least, int(next));
            next = __shfl_sync(kAll, next, int(next));
            least = min(least, m);
        }
        const uint32_t c = least & 1u;
        // switch `lane` (< 16): colour of its even output; of the output its even input feeds
        const uint32_t ce = __shfl_sync(kAll, c, (lane & 15) * 2);
        const uint32_t out_half = __ballot_sync(kAll, int(ce)) & 0xFFFFu;
        const uint32_t qe = __shfl_sync(kAll, q, (lane & 15) * 2);
        const uint32_t ci = __shfl_sync(kAll, c, int((uint32_t((lane & 15) * 2) & ~smask) + qe));
        const uint32_t in_half = __ballot_sync(kAll, int(ci)) & 0xFFFFu;
        if (lane == 0) {
            out.store16(2 * n - 2 - level, r, out_half);
            out.store16(level, r, in_half);
        }
        // position dl of the upper (lower) half takes the colour-0 (1) output of switch tl
        const uint32_t H = 1u << (ls - 1), dl = uint32_t(lane) & smask, tl = dl & (H - 1u), lower = dl >> (ls - 1);
        const uint32_t c2 = __shfl_sync(kAll, c, int(sb + 2u * tl));
        p = __shfl_sync(kAll, p, int(sb + 2u * tl + (c2 ^ lower))) >> 1;
    }
    const uint32_t mid = __ballot_sync(kAll, int(__shfl_sync(kAll, p, (lane & 15) * 2) & 1u)) & 0xFFFFu;
    if (lane == 0) out.store16(n - 1, r, mid);
}

template <int LOGC>
__global__ void __launch_bounds__((1 << LOGC) / 2)
k_route_few(const uint32_t *__restrict__ P, uint32_t *__restrict__ bits, int n, int logs, size_t total) {
    after_previous_kernel();
    constexpr uint32_t C = 1u << LOGC, kAll = 0xFFFFFFFFu;
    __shared__ uint32_t W[C];                  // (minimum << 16 | next) of every output
    __shared__ uint32_t Q32[C / 2], Pn32[C / 2];
    uint16_t *Q = reinterpret_cast<uint16_t *>(Q32), *Pn = reinterpret_cast<uint16_t *>(Pn32);
    __shared__ uint32_t cw[C / 64];
    FusedOut out;
    out.bits = bits;
    out.n = n;
    out.flat0 = size_t(blockIdx.x) << LOGC;
    out.valid = uint32_t(total - out.flat0 < size_t(C) ? total - out.flat0 : size_t(C));
    const uint32_t t = threadIdx.x, lane = t & 31u, warp = t >> 5, j = 2u * t;
    const uint32_t block = (1u << logs) - 1u;
    uint32_t p0 = j & block, p1 = (j + 1u) & block;            // padding: the identity
    if (j < out.valid) {                                       // (valid is even)
        p0 = BENES_GUARD(P[out.flat0 + j], block);
        p1 = BENES_GUARD(P[out.flat0 + j + 1], block);
    }
    for (; logs > 6; --logs) {
        const int level = n - logs;
        const uint32_t smask = (1u << logs) - 1u, sb = j & ~smask, H = (smask + 1u) >> 1;
        Q[sb + p0] = uint16_t(j);
        Q[sb + p1] = uint16_t(j + 1u);
        __syncthreads();
        const uint32_t q0 = BENES_GUARD(uint32_t(Q[j]), C - 1u);
        uint32_t w0 = (j << 16) | BENES_GUARD(uint32_t(Q[sb + (p1 ^ 1u)]), C - 1u);
        uint32_t w1 = ((j + 1u) << 16) | BENES_GUARD(uint32_t(Q[sb + (p0 ^ 1u)]), C - 1u);
        *reinterpret_cast<uint2 *>(W + j) = make_uint2(w0, w1);
        __syncthreads();
        // in place: a word always holds the minimum of the path up to, but excluding, its next; a cycle has
        // at most S/2 outputs
        volatile uint32_t *Wv = W;
        for (int pass = 1; pass < logs; ++pass) {
            const uint32_t v0 = Wv[w0 & 0xFFFFu], v1 = Wv[w1 & 0xFFFFu];
            w0 = (v0 & 0xFFFFu) | min(w0 & 0xFFFF0000u, v0 & 0xFFFF0000u);
            w1 = (v1 & 0xFFFFu) | min(w1 & 0xFFFF0000u, v1 & 0xFFFF0000u);
            Wv[j] = w0;
            Wv[j + 1u] = w1;
            __syncthreads();
        }
        const uint32_t c = (w0 >> 16) & 1u;
        const uint32_t word = __ballot_sync(kAll, int(c));
        if (lane == 0) cw[warp] = word;
        const uint32_t at0 = sb + ((j - sb) >> 1);
        Pn[at0] = uint16_t((c ? p1 : p0) >> 1);
        Pn[at0 + H] = uint16_t((c ? p0 : p1) >> 1);
        __syncthreads();
        const uint32_t in = __ballot_sync(kAll, int(((cw[q0 >> 6] >> ((q0 >> 1) & 31u)) ^ q0) & 1u));
        if (lane == 0 && 64u * warp < out.valid) {
            *out.stage_word(2 * n - 2 - level, warp) = word;
            *out.stage_word(level, warp) = in;
        }
        const uint32_t pp = Pn32[t];
        p0 = pp & 0xFFFFu;
        p1 = pp >> 16;
    }
    uint16_t *Qw = Q + 64u * warp;             // the warp's 64 outputs
    __syncwarp();
    if (logs == 6) {
        // a lane has one of the sub-block's 32 switches; the (next, minimum) words of its two outputs share a register
        const int level = n - 6;
        Qw[p0] = uint16_t(2u * lane);
        Qw[p1] = uint16_t(2u * lane + 1u);
        __syncwarp();
        const uint32_t q0 = BENES_GUARD(uint32_t(Qw[2u * lane]), 63u);
        const uint32_t n0 = BENES_GUARD(uint32_t(Qw[p1 ^ 1u]), 63u), n1 = BENES_GUARD(uint32_t(Qw[p0 ^ 1u]), 63u);
        __syncwarp();
        uint32_t w = (n0 | ((2u * lane) << 8)) | ((n1 | ((2u * lane + 1u) << 8)) << 16);
#pragma unroll
        for (int pass = 0; pass < 5; ++pass) {
            const uint32_t a0 = w & 0xFFu, a1 = (w >> 16) & 0xFFu;
            const uint32_t v0 = (__shfl_sync(kAll, w, int(a0 >> 1)) >> ((a0 & 1u) * 16u)) & 0xFFFFu;
            const uint32_t v1 = (__shfl_sync(kAll, w, int(a1 >> 1)) >> ((a1 & 1u) * 16u)) & 0xFFFFu;
            w = ((v0 & 0xFFu) | min(w & 0xFF00u, v0 & 0xFF00u)) | (((v1 & 0xFFu) | min((w >> 16) & 0xFF00u, v1 & 0xFF00u)) << 16);
        }
        const uint32_t c = (w >> 8) & 1u;
        const uint32_t word = __ballot_sync(kAll, int(c));
        const uint32_t in = __ballot_sync(kAll, int((__shfl_sync(kAll, c, int(q0 >> 1)) ^ q0) & 1u));
        if (lane == 0 && 64u * warp < out.valid) {
            *out.stage_word(2 * n - 2 - level, warp) = word;
            *out.stage_word(level, warp) = in;
        }
        few_tail32((c ? p1 : p0) >> 1, 2u * warp, Qw, out, 5);
        few_tail32((c ? p0 : p1) >> 1, 2u * warp + 1u, Qw + 32, out, 5);
    } else {
        // several permutations of 2^n <= 32: from a switch to an output per lane
        const uint32_t a0 = __shfl_sync(kAll, p0, int(lane >> 1)), a1 = __shfl_sync(kAll, p1, int(lane >> 1));
        const uint32_t b0 = __shfl_sync(kAll, p0, int(16u + (lane >> 1))), b1 = __shfl_sync(kAll, p1, int(16u + (lane >> 1)));
        few_tail32((lane & 1u) ? a1 : a0, 2u * warp, Qw, out, logs);
        few_tail32((lane & 1u) ? b1 : b0, 2u * warp + 1u, Qw + 32, out, logs);
    }
}

template <int LOGC>
int launch_few(const uint32_t *P, size_t total, uint32_t *bits, int n, int logs, cudaStream_t s) {
    launch_kernel(k_route_few<LOGC>, unsigned((total + (size_t(1) << LOGC) - 1) >> LOGC), (1 << LOGC) / 2, 0, s, P, bits, n, logs, total);
    return launch_status();
}

// ---- a block of 2^16 outputs in a thread-block cluster of two CTAs ----------------
// The level whose sub-block spans both CTAs runs on distributed shared memory:
// CTA r keeps outputs / inputs [r 2^15, (r+1) 2^15) of P and Q, the owners of
// switches [r 2^14, (r+1) 2^14), the records of ruler outputs [r 2^12, (r+1) 2^12)
// and colour words [512 r, 512 (r+1)), in the same layout the one-CTA kernel uses
// for a block of 2^15; an index picks the CTA with its top bit.  Walkers hop
// between the two shared memories with ordinary loads and a 16-bit
// compare-and-swap on the owner (no multicast, no bulk copies).  The compaction
// sends the upper half-block to CTA 0 and the lower one to CTA 1, after which
// each CTA finishes its half exactly like the one-CTA kernel.  All values of this
// level fit 16 bits (indices < 2^16, owner codes < 2^14, 0xFFFF = none).
constexpr int kClusterLog2M = kFusedLog2M + 1;

template <class Tp>
struct Pair2 {                       // the same array in the two CTAs of the cluster
    Tp *a, *b;
    __device__ __forceinline__ Tp *of(uint32_t rank) const { return rank ? b : a; }
};

// The layout of the level that spans both CTAs (P 2M, Q 2M, colour words, the next P 2M + the
// part of the scratch that does not fit there); the levels below use FusedCfg's.
using ClusterTailCfg = FusedCfg<kFusedLog2M, 1024>;
constexpr size_t kClusterTopBytes = size_t(ClusterTailCfg::C) * 6 + ClusterTailCfg::C / 16 + size_t(ClusterTailCfg::kRulers) * 2 + 16;
constexpr size_t kClusterSmemBytes = kClusterTopBytes > ClusterTailCfg::kSmemBytes ? kClusterTopBytes : ClusterTailCfg::kSmemBytes;

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(ClusterTailCfg::T)
k_route_cluster2(const uint32_t *__restrict__ P, int records, uint32_t *__restrict__ bits, int log2n,
                 uint32_t block0, const uint32_t *__restrict__ gate, const uint32_t *__restrict__ redone) {
    after_previous_kernel();
    if (gate && *gate != 0u) {
        P = redone;
        records = 0;
    }
    constexpr int LOGM = kFusedLog2M;           // per CTA
    using Cfg = ClusterTailCfg;
    constexpr int M = Cfg::C;                      // outputs per CTA
    constexpr int T = Cfg::T;
    constexpr int R = Cfg::kRulers;                // ruler outputs per CTA
    constexpr int LOGR = LOGM - kFKappa;
    constexpr uint32_t kInCta = uint32_t(M) - 1u, kSwInCta = uint32_t(M / 2) - 1u, kRInCta = uint32_t(R) - 1u;
    constexpr uint32_t kWordsPerCta = M / 64;    // colour words per CTA
    constexpr uint32_t kBoth = 2u * uint32_t(M) - 1u;
    static_assert(size_t(M) + size_t(R) * 10 > size_t(2 * M), "peers live in the tail");

    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    const uint32_t rank = cluster.block_rank();

    extern __shared__ __align__(16) unsigned char smem_raw[];
    uint16_t *Pa = reinterpret_cast<uint16_t *>(smem_raw);
    uint16_t *Q = Pa + M;
    uint32_t *cw = reinterpret_cast<uint32_t *>(Q + M);
    uint16_t *Pb = reinterpret_cast<uint16_t *>(cw + M / 64);
    unsigned char *tail = reinterpret_cast<unsigned char *>(Pb + M);
    // scratch of the labelling, over the buffer the next level's P' goes to
    uint16_t *own = Pb;
    uint32_t *recm = reinterpret_cast<uint32_t *>(reinterpret_cast<unsigned char *>(Pb) + M);
    uint32_t *list = recm + R;
    uint16_t *peer = reinterpret_cast<uint16_t *>(tail);

    const Pair2<uint16_t> Pa2{cluster.map_shared_rank(Pa, 0), cluster.map_shared_rank(Pa, 1)};
    const Pair2<uint16_t> Q2{cluster.map_shared_rank(Q, 0), cluster.map_shared_rank(Q, 1)};
    const Pair2<uint16_t> Pb2{cluster.map_shared_rank(Pb, 0), cluster.map_shared_rank(Pb, 1)};
    const Pair2<uint16_t> own2{cluster.map_shared_rank(own, 0), cluster.map_shared_rank(own, 1)};
    const Pair2<uint32_t> recm2{cluster.map_shared_rank(recm, 0), cluster.map_shared_rank(recm, 1)};
    const Pair2<uint32_t> list2{cluster.map_shared_rank(list, 0), cluster.map_shared_rank(list, 1)};
    const Pair2<uint32_t> cw2{cluster.map_shared_rank(cw, 0), cluster.map_shared_rank(cw, 1)};

    const int tid = threadIdx.x;
    const int lane = tid & 31;
    const int n = log2n;
    const int level = n - kClusterLog2M;         // recursion level of the cluster's block
    const size_t flat0 = size_t((blockIdx.x >> 1) + block0) << kClusterLog2M;
    const size_t N = size_t(1) << n;
    const size_t stage_w = N / 64;
    const size_t perm = flat0 >> n;
    const size_t local_first_switch = (flat0 & (N - 1)) >> 1;
    // this CTA's half of the block's words of a stage
    uint32_t *my_bits = bits + perm * size_t(2 * n - 1) * stage_w + (local_first_switch >> 5) + rank * kWordsPerCta;

    for (int j = tid; j < M; j += T) {
        const size_t f = flat0 + rank * uint32_t(M) + j;
        uint32_t v;
        if (records) {
            const unsigned long long w = reinterpret_cast<const unsigned long long *>(P)[f >> 1];
            v = uint32_t(w >> ((f & 1) ? kClusterLog2M : 0)) & kBoth;
        } else {
            v = P[f];
        }
        Pa[j] = uint16_t(BENES_GUARD(v, kBoth));
    }
    for (int t = tid; t < M / 2; t += T) own[t] = uint16_t(kNone16);
    cluster.sync();           // both CTAs are running (and loaded) before either touches the other's memory
    // a1: the inverse goes to the CTA that keeps that input
    for (int j = tid; j < M; j += T) {
        const uint32_t v = Pa[j];
        Q2.of(v >> LOGM)[v & kInCta] = uint16_t(rank * uint32_t(M) + j);
    }
    cluster.sync();

    // walks from this CTA's ruler outputs (its ruler switches are its own); about half of
    // the switches and inverse entries a walker reaches are in the other CTA
    for (int rl = tid; rl < R; rl += T) {
        const uint32_t rho = rank * uint32_t(R) + rl;
        const uint32_t group = rho >> 1, side0 = rho & 1u;
        const uint32_t t0 = (group << kFKappa) | fused_slot(group, uint32_t(level));
        uint32_t j = 2u * t0 + side0;
        uint32_t fwd = j, part = kNone16, pr = rho ^ 1u;
        if (!side0) own[t0 & kSwInCta] = uint16_t(rho << 1);
        uint32_t pp = *reinterpret_cast<const uint32_t *>(Pa + 2u * (t0 & kSwInCta));
        uint32_t p = (side0 ? pp : (pp >> 16)) & kBoth;                // P[j^1]
        uint32_t q = Q2.of((p ^ 1u) >> LOGM)[(p ^ 1u) & kInCta];
        for (uint32_t hops = 0; hops <= kBoth; ++hops) {                 // a walk claims < 2^15 switches
            j = q;
            const uint32_t t = j >> 1, side = j & 1u, g = t >> kFKappa;
            if ((t & ((1u << kFKappa) - 1u)) == fused_slot(g, uint32_t(level))) {
                pr = (2u * g + side) ^ 1u;                               // reached the next ruler
                break;
            }
            const uint32_t c = t >> (LOGM - 1), tl = t & kSwInCta;
            pp = *reinterpret_cast<const uint32_t *>(Pa2.of(c) + 2u * tl);
            p = (side ? pp : (pp >> 16)) & kBoth;
            const uint32_t qn = Q2.of((p ^ 1u) >> LOGM)[(p ^ 1u) & kInCta];
            const uint32_t prev = atomicCAS(reinterpret_cast<unsigned short *>(own2.of(c) + tl),
                                            static_cast<unsigned short>(kNone16),
                                            static_cast<unsigned short>((rho << 1) | side));
            if (prev != kNone16) {                                       // met the other walker
                pr = prev >> 1;
                break;
            }
            fwd = min(fwd, j);
            part = min(part, j ^ 1u);
            q = qn;
        }
        recm[rl] = fwd | (part << 16);
        peer[rl] = uint16_t(pr < 2u * uint32_t(R) ? pr : rho);
    }
    cluster.sync();
    // contracted list: next = peer ^ 1, minimum = own side of mine, far side of the peer's
    for (int rl = tid; rl < R; rl += T) {
        const uint32_t pr = peer[rl];
        const uint32_t mn = min(recm[rl] & 0xFFFFu, recm2.of(pr >> LOGR)[pr & kRInCta] >> 16);
        list[rl] = (pr ^ 1u) | (mn << 16);
    }
    cluster.sync();
    // in-place pointer jumping; a cycle of the list has at most 2^12 words (half of the ruler outputs)
    for (int r = 0; r < kClusterLog2M - kFKappa - 1; ++r) {
        for (int e = tid; e < R; e += T) {
            const uint32_t w = list[e], nx = w & 0xFFFFu;
            const uint32_t v = list2.of((nx >> LOGR) & 1u)[nx & kRInCta];
            const uint32_t hw = w & 0xFFFF0000u, hv = v & 0xFFFF0000u;
            list[e] = (hw < hv ? hw : hv) | (v & 0xFFFFu);
        }
        cluster.sync();
    }
    // a4 + output side of a5 for this CTA's switches
    for (int tl = tid; tl < M / 2; tl += T) {
        uint32_t c;
        const uint32_t code = own[tl];
        if (code != kNone16) {
            const uint32_t rr = code >> 1;
            c = ((list2.of((rr >> LOGR) & 1u)[rr & kRInCta] >> 16) ^ code) & 1u;
        } else {
            // loop without ruler: walk the cycle of output 2t from both ends
            const uint32_t j0 = 2u * (rank * uint32_t(M / 2) + tl);
            uint32_t f = j0, bk = j0, mn = j0;
            for (uint32_t hops = 0; hops <= kBoth; ++hops) {
                const uint32_t pf = Pa2.of((f ^ 1u) >> LOGM)[(f ^ 1u) & kInCta], pb = Pa2.of(bk >> LOGM)[bk & kInCta];
                const uint32_t qf = Q2.of((pf ^ 1u) >> LOGM)[(pf ^ 1u) & kInCta];
                const uint32_t qb = Q2.of((pb ^ 1u) >> LOGM)[(pb ^ 1u) & kInCta];
                f = qf;
                if (f == bk) break;
                mn = min(mn, f);
                bk = qb ^ 1u;
                if (bk == f) break;
                mn = min(mn, bk);
            }
            c = mn & 1u;
        }
        const uint32_t word = __ballot_sync(0xFFFFFFFFu, c);
        if (lane == 0) {
            cw[tl >> 5] = word;
            my_bits[size_t(2 * n - 2 - level) * stage_w + (tl >> 5)] = word;
        }
    }
    cluster.sync();
    // input side of a5 + a6: the upper half-block goes to CTA 0, the lower one to CTA 1
    for (int tl = tid; tl < M / 2; tl += T) {
        const uint32_t t = rank * uint32_t(M / 2) + tl;                  // position of the switch in either half-block
        const uint32_t c = (cw[tl >> 5] >> (tl & 31)) & 1u;
        const uint32_t pp = *reinterpret_cast<const uint32_t *>(Pa + 2 * tl);
        Pb2.of(c)[t] = uint16_t((pp & 0xFFFFu) >> 1);
        Pb2.of(c ^ 1u)[t] = uint16_t(pp >> 17);
        const uint32_t q0 = Q[2 * tl];                                   // output fed by input 2t of the block
        const uint32_t wq = q0 >> 6;
        const uint32_t cin = ((cw2.of(wq / kWordsPerCta)[wq % kWordsPerCta] >> ((q0 >> 1) & 31u)) ^ q0) & 1u;
        const uint32_t word = __ballot_sync(0xFFFFFFFFu, cin);
        if (lane == 0) my_bits[size_t(level) * stage_w + (tl >> 5)] = word;
    }
    cluster.sync();
    // from here on nothing leaves the CTA
    constexpr int kEnter = M / 4 / T;
    uint32_t v[kEnter][4];
#pragma unroll
    for (int r = 0; r < kEnter; ++r) {
        const uint2 p = *reinterpret_cast<const uint2 *>(Pb + 4 * (tid + r * T));
        v[r][0] = p.x & kInCta; v[r][1] = (p.x >> 16) & kInCta; v[r][2] = p.y & kInCta; v[r][3] = (p.y >> 16) & kInCta;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kEnter; ++r) fused_enter4<Cfg>(smem_raw, uint32_t(tid + r * T), v[r], LOGM);
    __syncthreads();
    FusedOut out;
    out.bits = bits;
    out.n = n;
    out.flat0 = flat0 + rank * uint32_t(M);
    out.valid = uint32_t(M);
    fused_levels<Cfg>(smem_raw, out, LOGM);
}

template <int LOGC, int THREADS>
int configure_one() {
    using Cfg = FusedCfg<LOGC, THREADS>;
    static OncePerDevice configured;
    return configured.run([]() -> int {
        BENES_CUDA_TRY(cudaFuncSetAttribute(k_route_fused<LOGC, THREADS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            int(Cfg::kSmemBytes)));
        BENES_CUDA_TRY(cudaFuncSetAttribute(k_route_fused<LOGC, THREADS>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                            cudaSharedmemCarveoutMaxShared));
        cudaFuncAttributes loaded;                             // (asking for them loads the kernel)
        BENES_CUDA_TRY(cudaFuncGetAttributes(&loaded, k_route_fused<LOGC, THREADS>));
        return BENES_OK;
    });
}

template <int LOGC, int THREADS>
int launch_one(const uint32_t *P, int records, size_t first, size_t end, uint32_t *bits, int log2n, int logs,
               cudaStream_t s, const uint32_t *gate, const uint32_t *redone) {
    using Cfg = FusedCfg<LOGC, THREADS>;
    const int rc = configure_one<LOGC, THREADS>();
    if (rc) return rc;
    const size_t ctas = (end - first + Cfg::C - 1) >> LOGC;
    launch_kernel(k_route_fused<LOGC, THREADS>, unsigned(ctas), THREADS, Cfg::kSmemBytes, s, P, records, bits, log2n, logs, first, end,
                  gate, redone);
    return launch_status();
}

template <int LOGC>
int launch_peel(const uint32_t *P, int records, size_t total, uint32_t *bits, int log2n, uint32_t *next, cudaStream_t s,
                const uint32_t *gate, const uint32_t *redone) {
    constexpr int T = 1024;
    using Cfg = FusedCfg<LOGC, T>;
    static OncePerDevice configured;
    const int rc = configured.run([]() -> int {
        BENES_CUDA_TRY(cudaFuncSetAttribute(k_route_peel<LOGC, T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            int(Cfg::kSmemBytes)));
        return BENES_OK;
    });
    if (rc) return rc;
    launch_kernel(k_route_peel<LOGC, T>, unsigned(total >> LOGC), T, Cfg::kSmemBytes, s, P, records, bits, log2n, next, gate, redone);
    return launch_status();
}

int launch_cluster2(const uint32_t *P, int records, size_t first_block, size_t blocks, uint32_t *bits,
                    int log2n, cudaStream_t s, const uint32_t *gate, const uint32_t *redone) {
    static OncePerDevice configured;
    const int rc = configured.run([]() -> int {
        BENES_CUDA_TRY(cudaFuncSetAttribute(k_route_cluster2, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            int(kClusterSmemBytes)));
        BENES_CUDA_TRY(cudaFuncSetAttribute(k_route_cluster2, cudaFuncAttributePreferredSharedMemoryCarveout,
                                            cudaSharedmemCarveoutMaxShared));
        return BENES_OK;
    });
    if (rc) return rc;
    // two CTAs per block (the cluster size is part of the kernel)
    launch_kernel(k_route_cluster2, unsigned(2 * blocks), ClusterTailCfg::T, kClusterSmemBytes, s, P, records, bits, log2n,
                  uint32_t(first_block), gate, redone);
    return launch_status();
}

}  // namespace

int launch_fused(const void *Pv, int records, size_t total, int log2m, uint32_t *bits, int log2n,
                 cudaStream_t s, size_t first_block, size_t blocks, const uint32_t *gate, const uint32_t *redone,
                 uint32_t *const spare[2]) {
    const uint32_t *P = static_cast<const uint32_t *>(Pv);
    if (log2m < 1 || log2m > kClusterLog2M) return BENES_ERR_BADARG;
    if (blocks == 0) blocks = (total >> log2m) - first_block;        // all the rest
    if (first_block + blocks > (total >> log2m)) return BENES_ERR_BADARG;
    if (log2m == kClusterLog2M) return launch_cluster2(P, records, first_block, blocks, bits, log2n, s, gate, redone);
    const size_t first = first_block << log2m, end = first + (blocks << log2m);
    int m = log2m;
    if (spare && first == 0 && end == total) {
        // A call that splits whole permutations readies the kernel of a call that may not (a captured one) too, so that
        // one ordinary call is enough before a capture.
        if (log2m == log2n && m >= kPeelLog2 && 2 * (total >> m) <= size_t(sm_count())) {
            const int rc = m == 15 ? configure_one<15, 1024>() : m == 14 ? configure_one<14, 1024>()
                         : m == 13 ? configure_one<13, 1024>() : configure_one<12, 1024>();
            if (rc) return rc;
        }
        for (int i = 0; m >= kPeelLog2 && 2 * (total >> m) <= size_t(sm_count()); --m, i ^= 1) {
            const int rc = m == 15 ? launch_peel<15>(P, records, total, bits, log2n, spare[i], s, gate, redone)
                         : m == 14 ? launch_peel<14>(P, records, total, bits, log2n, spare[i], s, gate, redone)
                         : m == 13 ? launch_peel<13>(P, records, total, bits, log2n, spare[i], s, gate, redone)
                                   : launch_peel<12>(P, records, total, bits, log2n, spare[i], s, gate, redone);
            if (rc) return rc;
            P = spare[i];
            records = 0;
            gate = nullptr;
        }
    }
    // blocks of up to 2^11 in a plain array, and not more switches than the GPU has threads
    if (records == 0 && !gate && m <= 11 && first == 0 && end / 2 <= size_t(sm_count()) * 2048) {
        const int logc = m > 8 ? m : 8;
        return logc == 8 ? launch_few<8>(P, end, bits, log2n, m, s) : logc == 9 ? launch_few<9>(P, end, bits, log2n, m, s)
             : logc == 10 ? launch_few<10>(P, end, bits, log2n, m, s) : launch_few<11>(P, end, bits, log2n, m, s);
    }
    // Small blocks share a CTA: a thread of the 8-bit levels takes a whole sub-block, so the more
    // sub-blocks a CTA holds, the fuller its warps.  Up to 2^13 outputs per CTA, as long as
    // every SM still gets a few CTAs.
    int logc = m > 10 ? m : 10;
    while (logc < 13 && ((end - first) >> logc) > 4 * size_t(sm_count())) ++logc;
    // CTAs that have an SM to themselves get more threads: their time is a chain of short
    // phases, not the instructions they issue.
    const bool alone = ((end - first + (size_t(1) << logc) - 1) >> logc) <= size_t(sm_count());
#define BENES_FUSED(LC, T) return launch_one<LC, T>(P, records, first, end, bits, log2n, m, s, gate, redone)
    switch (logc) {
        case 10: if (alone) BENES_FUSED(10, 256); BENES_FUSED(10, 32);
        case 11: if (alone) BENES_FUSED(11, 512); BENES_FUSED(11, 64);
        case 12: if (alone) BENES_FUSED(12, 1024); BENES_FUSED(12, 128);
        case 13: if (alone) BENES_FUSED(13, 1024); BENES_FUSED(13, 256);
        case 14: if (alone) BENES_FUSED(14, 1024); BENES_FUSED(14, 512);
        default: BENES_FUSED(15, 1024);
    }
#undef BENES_FUSED
}

}  // namespace benes
