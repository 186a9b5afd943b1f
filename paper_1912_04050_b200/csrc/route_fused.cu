// Fused path: one CTA finishes every remaining level of 2^LOGC consecutive
// outputs entirely in shared memory (inverse, loop labelling, colouring, stage
// bits, compaction, middle stage).  It serves the tail of a large permutation
// (blocks of 2^logs outputs of the flat level array) and batches of small
// permutations; a CTA holds one block, or several when the blocks are smaller
// than 2^LOGC.
//
// A level works on sub-blocks of S = 2^logs outputs, and from its inverse Q alone.  The outputs a = Q[2s] and
// b = Q[2s+1] of an input switch are each other's partners on the loop, so one pass over the input switches
// scatters the successors, g(a ^ 1) = b and g(b ^ 1) = a: no gather forms them and no P is kept.  Behind the
// colouring the same pass takes the colour of every input switch (a bit gathered through Q[2s]: the input-side
// stage), forms the two half-blocks' inverses from pairs of neighbouring switches, and scatters their successors.
// What bounds the kernel: the shared-memory wavefronts of these random accesses (3.5 per warp access) and, as close, the
// integer pipe (64 lanes per clock and SM, so that two cycles go by with every instruction of a warp).  Hence one
// scatter of all outputs and two gathers per switch in a level, nothing else at random but the walks, and little
// arithmetic beside them.
//
//   S >= 512   16-bit entries (byte offsets in the CTA, so that an entry is an address).  One ruler INPUT switch
//              per 8 G; a walker leaves it from either output, follows g, claims the output switches it stands on
//              and stops where it meets the walker from the other end.  In place of the two successors that lead
//              across a ruler switch lie the codes of the walkers beyond, so that a walker meets a ruler as it
//              meets a walker.  The contracted list (next and minimum) is labelled by in-place pointer jumping; a
//              switch takes (parity of its owner's minimum) ^ side.  Switches nobody claimed (loops without
//              ruler) walk their own cycle.
//   S = 256..16  8-bit entries.  One THREAD runs the sequential looping algorithm on a sub-block: from the
//              smallest switch not seen yet it follows the loop; the output it started from goes up, which
//              is the canonical colouring by construction (no minimum, no list).
//   S = 8      the colours of 4 switches depend on the input switches of the first
//              7 outputs only: 14 bits into a table.
//   S = 4, 2   256-entry table: all three stages at once.
//
// Measured on B200, before (P and Q kept, successors gathered through both; twice as many rulers; a look for
// the next start with every hop in sub-blocks of 2^8 too, by register sets from the low bit up) and after: 2048 blocks of 2^15 2.38 -> 1.87 ms, 4096 x 2^14
// 1.96 -> 1.61 ms, 4096 x 2^12 374 -> 316 us, 16384 x 2^8 53 -> 38 us.  Units of 8192 outputs inside a larger CTA with
// barriers of their own, meant to fall out of step, took 2.04 and 1.90 ms for the first two: the CTA waits for
// its last unit.
#include "common.cuh"
#include "loops8.cuh"

#include <cooperative_groups.h>

#include <utility>

BENES_GUARD_TU("route_fused.cu")

namespace benes {
namespace {

constexpr int kFMinLogS = 9;                   // smallest sub-block labelled by ruler walks (16-bit entries)
// A half of the word of an output switch t in the successor array, at the place of output j = 2t or 2t + 1: the
// successor of j as twice the output; or, bit 0 set, the walker (a ruler output, from bit 2 on: its byte offset in
// the list) that owns the switch and stood on the OTHER output of it.
constexpr uint32_t kCodeRho = 0xFFFCu;

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
// A thread has 16 G inputs (8 G switches) of every level.
//   [0, 2C)     successors / owners, 16 bit       |  8 bit: successors, the first half; then the tables
//   kRec        walk records, contracted list, 32 bit per walker each  |  marks of the sub-blocks of 2^8, behind the tables
//   kQ (2C)     inverse: pairs of 16-bit entries per input switch, as uint4 of four switches at a place of
//               their thread's that makes reads and writes free of bank conflicts  |  8 bit: two buffers
//   kCw (C/16)  colours of the level
template <int LOGC, int GROUPS>
struct FusedCfg {
    static constexpr int LOG = LOGC;
    static constexpr uint32_t C = 1u << LOGC;
    static constexpr uint32_t G = GROUPS;
    static constexpr uint32_t T = C / (16 * G);
    static constexpr int kSpacing = G == 2 ? 4 : 3;              // log2(input switches per ruler): one ruler per thread
    static constexpr uint32_t R = C / (8 * G);                   // walkers = words of the contracted list, 2 per thread
    static constexpr uint32_t kRec = 2 * C;
    static constexpr uint32_t kList = kRec + 4 * R;
    static constexpr uint32_t kLevelBytes = kList + 4 * R;
    static constexpr uint32_t kTables = C;
    static constexpr uint32_t kTablesEnd = kTables + uint32_t(kLutBytes);
    static constexpr uint32_t kMarks = kTablesEnd;                 // marks of the sub-blocks of 2^8
    static constexpr uint32_t kMarkBytes = C / 256 * kMarkStride;
    static constexpr uint32_t kMarksEnd = kMarks + kMarkBytes;
    static constexpr uint32_t kQ = ((kMarksEnd > kLevelBytes ? kMarksEnd : kLevelBytes) + 15u) & ~15u;
    static constexpr uint32_t kCw = kQ + 2 * C;
    static constexpr uint32_t kCount = kCw + C / 16;            // queued switches
    static constexpr size_t kSmemBytes = size_t(kCount) + 16;
    // CTAs per SM the register budget has to leave room for
    static constexpr int kMinCtas = G == 1 || T > 512 ? 1 : int(1024 / T) < 8 ? int(1024 / T) : 8;
};

template <class Tp>
__device__ __forceinline__ Tp &at(unsigned char *sm, uint32_t byte) {
    return *reinterpret_cast<Tp *>(sm + byte);
}

// The ruler switch of a group: top bits of a multiplicative hash
template <int SPACING>
__device__ __forceinline__ uint32_t fused_slot(uint32_t group, uint32_t salt) {
    return ((group + salt * 0x632BE5ABu) * 0x9E3779B1u) >> (32 - SPACING);
}

// Place of the pair word of input switch s (the four from a multiple of 4 on are 16 bytes): the four switches `c` of
// every thread side by side; the odd ones shifted by half of the banks, because neighbouring threads write them
// together.
template <class Cfg>
__device__ __forceinline__ uint32_t q_place(uint32_t s) {
    constexpr uint32_t G = Cfg::G;
    const uint32_t i = s / (8 * G), c = (s / 4) % (2 * G);
    return Cfg::kQ + (c * Cfg::T + (i ^ (c >= G ? 4u : 0u))) * 16u + (s & 3u) * 4u;
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

// Byte `g` of a stage: the 8 switches of the CTA's outputs [16 g, 16 g + 16) (n >= 6).
__device__ __forceinline__ uint8_t *stage_byte(const FusedOut &out, int stage, uint32_t g) {
    return reinterpret_cast<uint8_t *>(out.stage_word(stage, g >> 2)) + (g & 3u);
}

// ---- a level with 16-bit entries -------------------------------------------------------
// Pair words x = Q[2s] | Q[2s+1] << 16 scatter the successors of the outputs beside theirs.
template <class Cfg>
__device__ __forceinline__ void scatter_successors(unsigned char *sm, uint32_t x) {
    const uint32_t y = x ^ 0x00020002u;
    at<uint16_t>(sm, y & 0xFFFFu) = uint16_t(x >> 16);
    at<uint16_t>(sm, y >> 16) = uint16_t(x);
}

// The ruler of a thread: its group, and the pair of outputs its walkers start from.
struct Ruler {
    uint32_t group, pair;
};

// Puts the codes of the two walkers of ruler switch s in place of the successors across it; the calling thread
// has written the pair word and those successors itself.
template <class Cfg>
__device__ __forceinline__ Ruler place_ruler(unsigned char *sm, uint32_t s) {
    Ruler r;
    r.group = s >> Cfg::kSpacing;
    r.pair = at<uint32_t>(sm, q_place<Cfg>(s));
    const uint32_t y = r.pair ^ 0x00020002u, code = (r.group << 3) | 1u;
    at<uint16_t>(sm, y & 0xFFFFu) = uint16_t(code);
    at<uint16_t>(sm, y >> 16) = uint16_t(code + 4u);
    return r;
}

// Colour of output 2t of a switch nobody claimed: its g-cycle (at most S/2 outputs) from both ends;
// g(b ^ 1) ^ 1 is the predecessor of b on the cycle (the cycle of 2t+1 is its mirror image).
template <class Cfg>
__device__ __forceinline__ uint32_t loop_colour16(unsigned char *sm, uint32_t t, uint32_t S) {
    constexpr uint32_t kMask = 2u * Cfg::C - 2u;
    const uint32_t j0 = 4u * t;
    uint32_t f = at<uint16_t>(sm, j0) & kMask, bk = (at<uint16_t>(sm, j0 ^ 2u) & kMask) ^ 2u, least = min(j0, f);
    if (f == bk) return (least >> 1) & 1u;     // (one switch or two)
    least = min(least, bk);
    // (four hops per look at whether the two have met: on the way past each other they see what they know already)
    for (uint32_t hops = 0; hops < S; hops += 4) {
        bool met = false;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t nf = at<uint16_t>(sm, f) & kMask, nb = (at<uint16_t>(sm, bk ^ 2u) & kMask) ^ 2u;
            met |= nf == bk || nf == nb;
            f = nf;
            bk = nb;
            least = min(least, min(f, bk));
        }
        if (met) break;
    }
    return (least >> 1) & 1u;
}

// Labelling and colouring of a level; the colours go to kCw.
template <class Cfg>
__device__ __forceinline__ void colours16(unsigned char *sm, int logs, const Ruler &ruler) {
    constexpr uint32_t T = Cfg::T, R = Cfg::R, G = Cfg::G;
    const uint32_t tid = threadIdx.x;
    const uint32_t S = 1u << logs;

    // Walks from the ruler outputs; the two of a segment meet in the middle.  A claim needs no atomic.  Only the
    // two walkers of this segment ever reach a switch, from opposite ends, and each looks at the half the
    // other one writes.  If both find it free at the same moment, both write (either code is a valid owner: the two
    // stand for mirror cycles and on opposite outputs, so the colour comes out the same), both go on, and
    // each stops at the next switch, which the other has claimed; minima are taken over one switch
    // more, which changes nothing.  A walker keeps one minimum: the outputs on the far side of its
    // switches are the ones it stood on with the last bit flipped, and so is their minimum.
    // Walks differ in length, so a lane goes on to its next one every few hops instead of waiting for the longest walk of
    // the warp.  (Successors that form no cycles, of an input that is no permutation, end with the rounds.)
    {
        uint32_t rounds = S + 8u;
        uint32_t code = (ruler.group << 3) | 1u, j = ruler.pair & 0xFFFFu, least = j;
        for (;;) {
            // (no branches: a lane that has met somebody reads the same code again)
            bool met = false;
            uint32_t v = 0;
#pragma unroll
            for (int hop = 0; hop < 4; ++hop) {
                v = at<volatile uint16_t>(sm, j);
                met = (v & 1u) != 0u;
                if (!met) at<volatile uint16_t>(sm, j ^ 2u) = uint16_t(code);
                least = met ? least : min(least, j);
                j = met ? j : v;
            }
            if (met || --rounds == 0u) {
                at<uint32_t>(sm, Cfg::kRec + code - 1u) = (least << 16) | (v & kCodeRho);
                if ((code & 4u) || rounds == 0u) break;
                code += 4u;
                j = ruler.pair >> 16;
                least = j;
            }
        }
    }
    __syncthreads();

    // Contracted list: next = peer ^ 1.  What the other walker of my ruler switch has seen, with the last bit
    // flipped, lies on my cycle too, and every segment of a cycle has both of its walkers in such pairs of the cycle:
    // no need to fetch the minimum of the peer.  In-place pointer jumping, own words in registers; a cycle of the list
    // has at most half of the walkers of its sub-block.
    uint32_t w[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const uint32_t o = (tid + uint32_t(r) * T) * 4u;
        const uint32_t a = at<uint32_t>(sm, Cfg::kRec + o), b = at<uint32_t>(sm, Cfg::kRec + (o ^ 4u));
        w[r] = ((a & (R * 4u - 4u)) ^ 4u) | (min(a, b ^ 0x00020000u) & 0xFFFF0000u);
        at<uint32_t>(sm, Cfg::kList + o) = w[r];
    }
    if (tid == 0u) at<uint32_t>(sm, Cfg::kCount) = 0u;
    __syncthreads();
    for (int pass = 0; pass < logs - Cfg::kSpacing - 1; ++pass) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const uint32_t v = at<volatile uint32_t>(sm, Cfg::kList + (w[r] & 0xFFFFu));
            w[r] = (v & 0xFFFFu) | (min(w[r], v) & 0xFFFF0000u);
            at<volatile uint32_t>(sm, Cfg::kList + (tid + uint32_t(r) * T) * 4u) = w[r];
        }
        __syncthreads();
    }

    // Switches nobody claimed lie on loops without ruler.  They queue up over the walk records, so that one thread takes
    // one; where the queue is full (permutations made of short loops) they stay with their thread.
    // Colours of 8 switches per round.  A half with a code names the owner, who stood on the output of the other half.
    constexpr uint32_t kQueue = 2u * R;
    const uint32_t h = (tid >> 2) & 1u;                             // (lanes 4 apart would meet in a bank)
#pragma unroll
    for (uint32_t r = 0; r < G; ++r) {
        const uint32_t g = tid + r * T;
        const uint4 first = at<uint4>(sm, g * 32u + h * 16u), second = at<uint4>(sm, g * 32u + (h ^ 1u) * 16u);
        const uint32_t n8[8] = {first.x, first.y, first.z, first.w, second.x, second.y, second.z, second.w};
        uint32_t bits = 0, free_ = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const uint32_t lo = n8[k] & 1u, code = lo ? n8[k] : n8[k] >> 16;
            const uint32_t c = (at<uint32_t>(sm, Cfg::kList + (code & (R * 4u - 4u))) >> 17) ^ lo;
            bits |= (c & 1u) << k;
            free_ |= (~code & 1u) << k;
        }
        bits &= ~free_;
        if (__popc(free_) > 4) {
            // a permutation made of short loops: those of one switch or two at once, by one load each
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const uint32_t j = 4u * (8u * g + (uint32_t(k) ^ (h << 2))), f = n8[k] & (2u * Cfg::C - 2u);
                if (((free_ >> k) & 1u) && (at<uint16_t>(sm, f) & (2u * Cfg::C - 2u)) == j) {
                    free_ &= ~(1u << k);
                    bits |= ((min(j, f) >> 1) & 1u) << k;
                }
            }
        }
        if (free_) {
            uint32_t pos = atomicAdd(&at<uint32_t>(sm, Cfg::kCount), uint32_t(__popc(free_)));
            for (uint32_t left = free_; left; left &= left - 1u, ++pos) {
                const uint32_t k = uint32_t(__ffs(int(left))) - 1u, t = 8u * g + (k ^ (h << 2));
                if (pos < kQueue) at<uint16_t>(sm, Cfg::kRec + 2u * pos) = uint16_t(t);
                else bits |= loop_colour16<Cfg>(sm, t, S) << k;
            }
        }
        at<uint8_t>(sm, Cfg::kCw + g) = uint8_t(h ? (bits >> 4) | (bits << 4) : bits);
    }
    __syncthreads();
    const uint32_t queued = min(at<uint32_t>(sm, Cfg::kCount), kQueue);
    if (queued) {                                                   // (same value for all threads)
        for (uint32_t e = tid; e < queued; e += T) {
            const uint32_t t = at<uint16_t>(sm, Cfg::kRec + 2u * e);
            if (loop_colour16<Cfg>(sm, t, S)) atomicOr(&at<uint32_t>(sm, Cfg::kCw + ((t >> 3) & ~3u)), 1u << (t & 31u));
        }
        __syncthreads();
    }
}

// Input side of the thread's 8 G switches and the next level's entries: u[], l[] = pairs of the upper and the lower
// half-block, as they are stored (16-bit entries), or, if the next level has 8-bit entries, words of four of them.
template <class Cfg>
__device__ __forceinline__ void split16(unsigned char *sm, const FusedOut &out, int logs, int level, bool wide_next,
                                        uint32_t u[4 * Cfg::G], uint32_t l[4 * Cfg::G]) {
    constexpr uint32_t G = Cfg::G;
    const uint32_t tid = threadIdx.x;
    const uint32_t S = 1u << logs, sb = (16u * G * tid) & ~(S - 1u);
    const uint32_t vmask = (S - 1u) * 0x10001u, up = (2u * sb) * 0x10001u, low = S * 0x10001u;
    uint32_t in = 0;
#pragma unroll
    for (uint32_t q = 0; q < 2 * G; ++q) {
        const uint4 w4 = at<uint4>(sm, q_place<Cfg>(8u * G * tid + 4u * q));
        uint32_t y[4] = {w4.x, w4.y, w4.z, w4.w}, c[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            // output 2 t + side is entry 4 t + 2 side; its switch is bit t
            const uint32_t word = at<uint32_t>(sm, Cfg::kCw + ((y[k] >> 5) & (Cfg::C / 16 - 4)));
            c[k] = (__funnelshift_r(word, word, y[k] >> 2) ^ (y[k] >> 1)) & 1u;
            in |= c[k] << (4u * q + uint32_t(k));
        }
        if (wide_next) {
#pragma unroll
            for (int k = 0; k < 4; ++k) y[k] = ((y[k] >> 1) & vmask & 0xFFFEFFFEu) | up;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                // (0x5410 and 0x2222 share no set bit, so | adds them)
                const uint32_t sel = 0x5410u | (c[2 * k] * 0x22u) | (c[2 * k + 1] * 0x2200u);
                u[2 * q + k] = __byte_perm(y[2 * k], y[2 * k + 1], sel);
                l[2 * q + k] = __byte_perm(y[2 * k], y[2 * k + 1], sel ^ 0x2222u) | low;
            }
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) y[k] = (y[k] >> 2) & 0x00FF00FFu;
            uint32_t hu[2], hl[2];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const uint32_t sel = 0x40u | (c[2 * k] * 0x02u) | (c[2 * k + 1] * 0x20u);
                hu[k] = __byte_perm(y[2 * k], y[2 * k + 1], sel);
                hl[k] = __byte_perm(y[2 * k], y[2 * k + 1], sel ^ 0x22u);
            }
            u[q] = __byte_perm(hu[0], hu[1], 0x5410);
            l[q] = __byte_perm(hl[0], hl[1], 0x5410);
        }
    }
    if (16u * G * tid < out.valid) {
        uint8_t *to_in = stage_byte(out, level, G * tid), *to_out = stage_byte(out, 2 * out.n - 2 - level, G * tid);
        if (G == 1) {
            *to_in = uint8_t(in);
            *to_out = at<uint8_t>(sm, Cfg::kCw + tid);
        } else {
            *reinterpret_cast<uint16_t *>(to_in) = uint16_t(in);
            *reinterpret_cast<uint16_t *>(to_out) = at<uint16_t>(sm, Cfg::kCw + 2u * tid);
        }
    }
}

// Successors of four 8-bit pairs (words e0, e1 = eight entries in input order), local to a sub-block that starts at byte n8
__device__ __forceinline__ void scatter_successors8(unsigned char *sm, uint32_t n8, uint32_t e0, uint32_t e1) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t e = (k < 2 ? e0 : e1) >> (16 * (k & 1)), a = e & 0xFFu, b = (e >> 8) & 0xFFu;
        at<uint8_t>(sm, n8 + a) = uint8_t(b ^ 1u);
        at<uint8_t>(sm, n8 + b) = uint8_t(a ^ 1u);
    }
}

template <class Cfg>
__device__ __forceinline__ void clear_marks(unsigned char *sm) {
    for (uint32_t o = 8u * threadIdx.x; o < Cfg::kMarkBytes; o += 8u * Cfg::T) at<uint2>(sm, Cfg::kMarks + o) = make_uint2(0, 0);
}

// One level of 16-bit entries after another, down to sub-blocks of 2^8 (whose entries are then in place).
template <class Cfg>
__device__ __forceinline__ void levels16(unsigned char *sm, const FusedOut &out, int logs, Ruler &ruler) {
    constexpr uint32_t G = Cfg::G;
    const uint32_t tid = threadIdx.x;
    for (;; --logs) {
        const int level = out.n - logs;
        const uint32_t S = 1u << logs;
        colours16<Cfg>(sm, logs, ruler);
        uint32_t u[4 * G], l[4 * G];
        const bool wide_next = logs - 1 >= kFMinLogS;
        split16<Cfg>(sm, out, logs, level, wide_next, u, l);
        __syncthreads();
        const uint32_t sb = (16u * G * tid) & ~(S - 1u), tl = (16u * G * tid - sb) >> 1, H = S >> 1;
        if (!wide_next) {
            clear_marks<Cfg>(sm);
#pragma unroll
            for (uint32_t q = 0; q < G; ++q) {
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    const uint32_t *e = half ? l : u;
                    const uint32_t base = sb + (half ? H : 0u);
                    at<uint2>(sm, Cfg::kQ + base + tl + 8u * q) = make_uint2(e[2 * q], e[2 * q + 1]);
                    scatter_successors8(sm, base, e[2 * q], e[2 * q + 1]);
                }
            }
            __syncthreads();
            return;
        }
        // positions (in switches) of the thread's first pair in either half-block
        const uint32_t su = (sb + tl) >> 1, sl = su + (H >> 1);
#pragma unroll
        for (uint32_t q = 0; q < G; ++q) {
            at<uint4>(sm, q_place<Cfg>(su + 4u * q)) = make_uint4(u[4 * q], u[4 * q + 1], u[4 * q + 2], u[4 * q + 3]);
            at<uint4>(sm, q_place<Cfg>(sl + 4u * q)) = make_uint4(l[4 * q], l[4 * q + 1], l[4 * q + 2], l[4 * q + 3]);
        }
#pragma unroll
        for (uint32_t k = 0; k < 4 * G; ++k) {
            scatter_successors<Cfg>(sm, u[k]);
            scatter_successors<Cfg>(sm, l[k]);
        }
        // a group is the upper or the lower switches of two threads: one of them takes its ruler in the upper one,
        // the other in the lower one
        const uint32_t slot = fused_slot<Cfg::kSpacing>(tid >> 1, uint32_t(level) + 1u);
        ruler = place_ruler<Cfg>(sm, (((slot / (4 * G)) ^ tid) & 1u ? sl : su) + slot % (4 * G));
        __syncthreads();
    }
}

// ---- a level with 8-bit entries ----------------------------------------------------------
// `q8` is the buffer (0 or 1) of the inverse; the next level's goes to the other one, or, below 16, its P.
template <class Cfg, int LOGS>
__device__ __forceinline__ void level8(unsigned char *sm, const FusedOut &out, uint32_t q8) {
    constexpr uint32_t C = Cfg::C, T = Cfg::T, S = 1u << LOGS, H = S >> 1;
    constexpr int kReg = LOGS > 5 ? LOGS : 5;
    const uint32_t tid = threadIdx.x;
    const int level = out.n - LOGS;
    constexpr uint32_t kRegions = C >> kReg;
    const uint32_t q_from = Cfg::kQ + q8 * C, q_to = Cfg::kQ + (q8 ^ 1u) * C;
    // (whole warps: lanes without a sub-block follow the last one's successors and store nothing.  With few sub-blocks it
    // is the first warps that have one: an SM's warps are bound to its four schedulers, warp w of its k-th CTA to
    // scheduler (w + k) % 4)
    for (uint32_t r0 = tid & ~31u; r0 < kRegions; r0 += T) {
        const uint32_t r = min(r0 + tid % 32u, kRegions - 1u);
        const bool mine = kRegions >= 32u || r == r0 + tid % 32u;
        if (LOGS == 8) {
            // (sub-blocks of padding, the identity, are coloured as they are: all marks clear.  Loop after loop of one switch
            // takes three times as long as one loop, so the last CTA kept the call waiting: 9741 x 2^8 42 -> 31 us, 2435 x 2^8
            // 35 -> 23, 1722 x 2^10 50 -> 39.  CTAs above 2^13 have no padding)
            loop_marks(sm + (r << kReg), sm + Cfg::kMarks + r * kMarkStride, mine && (Cfg::LOG > 13 || (r << kReg) < out.valid));
            continue;
        }
        if (LOGS == 7) {
            const uint2 col = loop_128(sm + (r << kReg));
            if (mine) at<uint2>(sm, Cfg::kCw + 8u * r) = col;
            continue;
        }
        const uint32_t col = loop_region<LOGS == 6 ? 6 : 5>(sm + (r << kReg), S - 1u);
        if (!mine) continue;
        if (LOGS == 6) at<uint32_t>(sm, Cfg::kCw + 4u * r) = col;
        else at<uint16_t>(sm, Cfg::kCw + 2u * r) = uint16_t(col);
    }
    __syncthreads();
    for (uint32_t g = tid; g < C / 16; g += T) {
        const uint4 q4 = at<uint4>(sm, q_from + 16u * g);
        const uint32_t q[4] = {q4.x, q4.y, q4.z, q4.w};
        const uint32_t sb = (16u * g) & ~(S - 1u), tl = (16u * g - sb) >> 1;
        const uint32_t own = Cfg::kMarks + (g >> 4) * kMarkStride;
        uint32_t in = 0, out8, y[4], word = 0;
        if (LOGS <= 6) word = at<uint32_t>(sm, Cfg::kCw + ((sb >> 4) & ~3u)) >> ((sb >> 1) & 31u);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const uint32_t v = q[k >> 1] >> (16 * (k & 1));              // Q[2 s] in the low byte
            if (LOGS == 8) {
                in |= ((at<uint8_t>(sm, own + ((v >> 1) & 127u)) ^ v) & 1u) << k;
            } else {
                if (LOGS > 6) word = at<uint32_t>(sm, Cfg::kCw + (sb >> 4) + ((v >> 4) & (S / 16 - 4)));
                in |= ((__funnelshift_r(word, word, v >> 1) ^ v) & 1u) << k;
            }
        }
        if (LOGS == 8) {
            const uint2 m8 = at<uint2>(sm, own + tl);
            out8 = tops_of_bytes(m8.x << 7) | (tops_of_bytes(m8.y << 7) << 4);
        } else {
            out8 = at<uint8_t>(sm, Cfg::kCw + g);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) y[k] = (q[k] >> 1) & ((H - 1u) * 0x01010101u);
        const uint32_t s0 = 0x6420u | spread4(in & 15u), s1 = 0x6420u | spread4(in >> 4);
        const uint32_t e[2][2] = {{__byte_perm(y[0], y[1], s0), __byte_perm(y[2], y[3], s1)},
                                  {__byte_perm(y[0], y[1], s0 ^ 0x1111u), __byte_perm(y[2], y[3], s1 ^ 0x1111u)}};
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const uint32_t base = sb + (half ? H : 0u);
            if (LOGS > 4) {
                at<uint2>(sm, q_to + base + tl) = make_uint2(e[half][0], e[half][1]);
                scatter_successors8(sm, base, e[half][0], e[half][1]);
            } else {
                // the tables want P
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    at<uint8_t>(sm, q_to + base + ((e[half][k >> 2] >> (8 * (k & 3))) & 7u)) = uint8_t(k);
            }
        }
        if (out.n >= 6) {
            if (16u * g < out.valid) {
                *stage_byte(out, level, g) = uint8_t(in);
                *stage_byte(out, 2 * out.n - 2 - level, g) = uint8_t(out8);
            }
        } else {
            // permutations of 2^5 (two threads) or 2^4: a word per stage
            const uint32_t in2 = __shfl_xor_sync(~0u, in, 1), out2 = __shfl_xor_sync(~0u, out8, 1);
            uint32_t *row = out.bits + ((out.flat0 + 16u * g) >> out.n) * size_t(2 * out.n - 1);
            const bool first = !(g & 1u);
            if (16u * g < out.valid) {
                if (out.n == 4 || first) row[level] = out.n == 4 ? in : in | (in2 << 8);
                if (out.n == 4 || !first) row[2 * out.n - 2 - level] = out.n == 4 ? out8 : out2 | (out8 << 8);
            }
        }
    }
    __syncthreads();
}

// ---- sub-blocks of 8 and less: 32 outputs (16 switches of every stage) per thread ----------
template <class Cfg>
__device__ __forceinline__ void last_levels(unsigned char *sm, const FusedOut &out, int logs, uint32_t q8) {
    const int n = out.n;
    const uint32_t p8 = Cfg::kQ + q8 * Cfg::C;
    const uint32_t *lut8 = &at<uint32_t>(sm, Cfg::kTables), *lut4 = lut8 + kLut8Words;
    for (uint32_t r = threadIdx.x; r < Cfg::C / 32; r += Cfg::T) {
        const uint4 a = at<uint4>(sm, p8 + 32 * r), b = at<uint4>(sm, p8 + 32 * r + 16);
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
            uint32_t out8 = 0, in8 = 0;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t w0 = w[2 * k], w1 = w[2 * k + 1];
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

// The 8-bit levels from sub-blocks of 2^logs on; their entries (P, for sub-blocks of 8 and less) are in place.
template <class Cfg>
__device__ __forceinline__ void levels8(unsigned char *sm, const FusedOut &out, int logs) {
    uint32_t q8 = 0;
    if (logs == 8) { level8<Cfg, 8>(sm, out, q8); q8 ^= 1u; --logs; }
    if (logs == 7) { level8<Cfg, 7>(sm, out, q8); q8 ^= 1u; --logs; }
    if (logs == 6) { level8<Cfg, 6>(sm, out, q8); q8 ^= 1u; --logs; }
    if (logs == 5) { level8<Cfg, 5>(sm, out, q8); q8 ^= 1u; --logs; }
    if (logs == 4) { level8<Cfg, 4>(sm, out, q8); q8 ^= 1u; --logs; }
    last_levels<Cfg>(sm, out, logs, q8);
}

template <class Cfg>
__device__ __forceinline__ void copy_tables(unsigned char *sm) {
    for (uint32_t i = threadIdx.x; i < uint32_t(kLutBytes / 16); i += Cfg::T)
        at<uint4>(sm, Cfg::kTables + 16 * i) = __ldg(reinterpret_cast<const uint4 *>(&g_fused_tables) + i);
}

// Four neighbouring values: 16-bit entries of the inverse in input order at the start of the shared memory, 8-bit ones
// in the first buffer (of the permutation, for sub-blocks of 8 and less).
template <class Cfg>
__device__ __forceinline__ void enter4(unsigned char *sm, uint32_t i4, const uint32_t v[4], bool inverse, int logs) {
    const uint32_t smask = (1u << logs) - 1u, sb = (4u * i4) & ~smask;
    if (logs >= kFMinLogS) {
        if (inverse) {
            at<uint2>(sm, 8u * i4) = make_uint2(2u * (sb + v[0]) | (2u * (sb + v[1]) << 16), 2u * (sb + v[2]) | (2u * (sb + v[3]) << 16));
        } else {
#pragma unroll
            for (uint32_t k = 0; k < 4; ++k) at<uint16_t>(sm, 2u * (sb + v[k])) = uint16_t(2u * (4u * i4 + k));
        }
        return;
    }
    if (logs < 4) {
        at<uint32_t>(sm, Cfg::kQ + 4u * i4) = v[0] | (v[1] << 8) | (v[2] << 16) | (v[3] << 24);
    } else {
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) {
            const uint32_t i = 4u * i4 + k;
            at<uint8_t>(sm, Cfg::kQ + (i & ~smask) + v[k]) = uint8_t(i & smask);
        }
    }
}

// The first level's entries from an array of 32-bit values of the CTA's blocks, local to their blocks of 2^logs: the
// permutation, or its inverse.  Four values per load, four loads of a thread under way together.
template <class Cfg>
__device__ __forceinline__ void fused_load(unsigned char *sm, const FusedOut &out, const uint32_t *src, bool inverse, int logs) {
    constexpr uint32_t T = Cfg::T, kItems = Cfg::C / 4, kBatch = 4;
    const uint32_t smask = (1u << logs) - 1u;
    const bool aligned = (reinterpret_cast<uintptr_t>(src) & 15u) == 0;
    if (!inverse && logs >= kFMinLogS) {
        // (an input that is no permutation leaves places nobody writes; from here on the successor array holds
        // nothing but places in it and codes)
        for (uint32_t i = threadIdx.x; i < Cfg::C / 8; i += T) at<uint4>(sm, 16u * i) = make_uint4(0, 0, 0, 0);
        __syncthreads();
    }
    for (uint32_t i0 = threadIdx.x; i0 < kItems; i0 += kBatch * T) {
        uint32_t v[kBatch][4];
#pragma unroll
        for (uint32_t r = 0; r < kBatch; ++r) {
            const uint32_t i4 = i0 + r * T;
            const size_t f = out.flat0 + 4u * i4;
            if (4u * i4 + 4u <= out.valid && aligned) {
                const uint4 p = __ldcs(reinterpret_cast<const uint4 *>(src + f));
                v[r][0] = p.x; v[r][1] = p.y; v[r][2] = p.z; v[r][3] = p.w;
            } else {
                // a permutation that does not start on 16 bytes, the end of a batch of permutations of 2,
                // or padding: the identity
#pragma unroll
                for (uint32_t k = 0; k < 4; ++k) v[r][k] = 4u * i4 + k < out.valid ? src[f + k] : (4u * i4 + k) & smask;
            }
        }
#pragma unroll
        for (uint32_t r = 0; r < kBatch; ++r) {
#pragma unroll
            for (uint32_t k = 0; k < 4; ++k) v[r][k] = BENES_GUARD(v[r][k], smask);
            enter4<Cfg>(sm, i0 + r * T, v[r], inverse, logs);
        }
    }
    __syncthreads();
}

// From the entries of enter4 (complete: a barrier lies between) to the places and successors of the first level.
template <class Cfg>
__device__ __forceinline__ void start16(unsigned char *sm, int logs, int level, Ruler &ruler) {
    constexpr uint32_t G = Cfg::G;
    const uint32_t tid = threadIdx.x, first = 8u * G * tid;
    // (whatever the entries of an input that is no permutation hold: they stay in their block)
    const uint32_t local = (2u << logs) - 2u, keep = local * 0x10001u, base = ((32u * G * tid) & ~(local + 1u)) * 0x10001u;
    uint32_t x[8 * G];
#pragma unroll
    for (uint32_t q = 0; q < 2 * G; ++q) {
        const uint4 w = at<uint4>(sm, 4u * first + 16u * q);
        x[4 * q] = w.x; x[4 * q + 1] = w.y; x[4 * q + 2] = w.z; x[4 * q + 3] = w.w;
    }
    __syncthreads();
#pragma unroll
    for (uint32_t k = 0; k < 8 * G; ++k) x[k] = (x[k] & keep) | base;
#pragma unroll
    for (uint32_t q = 0; q < 2 * G; ++q)
        at<uint4>(sm, q_place<Cfg>(first + 4u * q)) = make_uint4(x[4 * q], x[4 * q + 1], x[4 * q + 2], x[4 * q + 3]);
#pragma unroll
    for (uint32_t k = 0; k < 8 * G; ++k) scatter_successors<Cfg>(sm, x[k]);
    ruler = place_ruler<Cfg>(sm, first + fused_slot<Cfg::kSpacing>(tid, uint32_t(level)));
    __syncthreads();
}
template <class Cfg>
__device__ __forceinline__ void start8(unsigned char *sm, int logs) {
    const uint32_t smask = (1u << logs) - 1u;
    if (logs == 8) clear_marks<Cfg>(sm);
    for (uint32_t g = threadIdx.x; g < Cfg::C / 16; g += Cfg::T) {
        uint4 q = at<uint4>(sm, Cfg::kQ + 16u * g);
        const uint32_t keep = smask * 0x01010101u;
        q.x &= keep; q.y &= keep; q.z &= keep; q.w &= keep;
        at<uint4>(sm, Cfg::kQ + 16u * g) = q;
        const uint32_t n8 = (16u * g) & ~smask;
        scatter_successors8(sm, n8, q.x, q.y);
        scatter_successors8(sm, n8, q.z, q.w);
    }
    __syncthreads();
}

// All levels of the CTA's blocks of 2^logs outputs; enter4 has been called for every entry, and a barrier passed.
template <class Cfg>
__device__ __forceinline__ void fused_levels(unsigned char *sm, const FusedOut &out, int logs) {
    if (logs >= kFMinLogS) {
        Ruler ruler;
        start16<Cfg>(sm, logs, out.n - logs, ruler);
        levels16<Cfg>(sm, out, logs, ruler);
        logs = kFMinLogS - 1;
    } else if (logs >= 4) {
        start8<Cfg>(sm, logs);
    }
    copy_tables<Cfg>(sm);
    if (logs < 4) __syncthreads();
    levels8<Cfg>(sm, out, logs);
}

template <class Cfg>
__global__ void __launch_bounds__(Cfg::T, Cfg::kMinCtas)
k_route_fused(const uint32_t *__restrict__ src, bool inverse, uint32_t *__restrict__ bits, int log2n, int logs,
              size_t first, size_t end) {
    after_previous_kernel();
    constexpr uint32_t C = Cfg::C;
    extern __shared__ __align__(16) unsigned char sm[];
    FusedOut out;
    out.bits = bits;
    out.n = log2n;
    out.flat0 = first + size_t(blockIdx.x) * C;
    out.valid = uint32_t(end - out.flat0 < size_t(C) ? end - out.flat0 : size_t(C));
    fused_load<Cfg>(sm, out, src, inverse, logs);
    fused_levels<Cfg>(sm, out, logs);
}

// One level of one block of 2^LOGC outputs per CTA; the inverses of the two half-blocks go to `next`, where the
// next launch finds them with twice as many CTAs.  While more than half of the SMs would have no block, that is how the
// in-CTA levels run: a level takes a time in proportion to the CTA's outputs, so halving the block with every level
// costs about two levels of the first block instead of one for each (all levels in one launch -> this: one block of 2^15
// 134 -> 68 us, 2^13 47 -> 32, 37 of 2^12 34 -> 24; the route of 2^16 175 -> 109, of 2^20 441 -> 388).
template <class Cfg>
__global__ void __launch_bounds__(Cfg::T, 1)
k_route_peel(const uint32_t *__restrict__ src, bool inverse, uint32_t *__restrict__ bits, int log2n, uint32_t *__restrict__ next) {
    after_previous_kernel();
    constexpr uint32_t C = Cfg::C, G = Cfg::G, H = C / 2;
    constexpr int logs = Cfg::LOG;
    extern __shared__ __align__(16) unsigned char sm[];
    FusedOut out;
    out.bits = bits;
    out.n = log2n;
    out.flat0 = size_t(blockIdx.x) * C;
    out.valid = C;
    fused_load<Cfg>(sm, out, src, inverse, logs);
    Ruler ruler;
    start16<Cfg>(sm, logs, log2n - logs, ruler);
    colours16<Cfg>(sm, logs, ruler);
    uint32_t u[4 * G], l[4 * G];
    split16<Cfg>(sm, out, logs, log2n - logs, true, u, l);
    // pairs of entries 2 (half-block + value) -> values
#pragma unroll
    for (uint32_t q = 0; q < 2 * G; ++q) {
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const uint32_t *e = half ? l : u;
            const uint32_t x = (e[2 * q] >> 1) & ((H - 1u) * 0x10001u), y = (e[2 * q + 1] >> 1) & ((H - 1u) * 0x10001u);
            *reinterpret_cast<uint4 *>(next + out.flat0 + half * H + 8u * G * threadIdx.x + 4u * q) =
                make_uint4(x & 0xFFFFu, x >> 16, y & 0xFFFFu, y >> 16);
        }
    }
}

// ---- few outputs in all ---------------------------------------------------------------------
// When every thread of the GPU could have a switch to itself, the time of a call is its chain of dependent
// steps, and the labelling with the shortest one is pointer jumping over all outputs: one thread per
// switch, one barrier per pass, and from sub-blocks of 64 down a warp in registers (a switch, then an output,
// per lane; jumps by shuffle).  Up to 64 of 2^10: 23.9 -> 8.6 us; 32 of
// 2^6: 6.6 -> 3.3; 290 of 2^10 (half of the GPU's threads): 30 -> 14.  Where the kernels above take over, because they
// issue fewer instructions: see launch_fused.

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
k_route_few(const uint32_t *__restrict__ src, bool inverse, uint32_t *__restrict__ bits, int n, int logs, size_t total) {
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
        p0 = BENES_GUARD(src[out.flat0 + j], block);
        p1 = BENES_GUARD(src[out.flat0 + j + 1], block);
    }
    if (LOGC == 11 && inverse) {               // (blocks of 2^11 that k_route_peel has made)
        const uint32_t sb = j & ~block;
        Pn[sb + p0] = uint16_t(j & block);
        Pn[sb + p1] = uint16_t((j + 1u) & block);
        __syncthreads();
        const uint32_t pp = Pn32[t];
        p0 = pp & block;
        p1 = (pp >> 16) & block;
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

constexpr int kMinInverseLog2 = 11;            // (see k_route_few: from the inverse in blocks of 2^11 only)

template <int LOGC>
int launch_few(const uint32_t *src, bool inverse, size_t total, uint32_t *bits, int n, int logs, cudaStream_t s) {
    launch_kernel(k_route_few<LOGC>, unsigned((total + (size_t(1) << LOGC) - 1) >> LOGC), (1 << LOGC) / 2, 0, s, src, inverse, bits, n, logs, total);
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
using ClusterTailCfg = FusedCfg<kFusedLog2M, 2>;
constexpr int kClusterKappa = 3;                // ruler spacing (log2) of that level
constexpr uint32_t kNone16 = 0xFFFFu;          // owner of a switch nobody claimed
constexpr size_t kClusterTopBytes = size_t(ClusterTailCfg::C) * 6 + ClusterTailCfg::C / 16 + (size_t(ClusterTailCfg::C) >> kClusterKappa) * 2 + 16;
constexpr size_t kClusterSmemBytes = kClusterTopBytes > ClusterTailCfg::kSmemBytes ? kClusterTopBytes : ClusterTailCfg::kSmemBytes;

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(ClusterTailCfg::T)
k_route_cluster2(const uint32_t *__restrict__ src, bool inverse, uint32_t *__restrict__ bits, int log2n, uint32_t block0) {
    after_previous_kernel();
    constexpr int LOGM = kFusedLog2M;           // per CTA
    using Cfg = ClusterTailCfg;
    constexpr int M = int(Cfg::C);                      // outputs per CTA
    constexpr int T = int(Cfg::T);
    constexpr int R = M >> kClusterKappa;        // ruler outputs per CTA
    constexpr int LOGR = LOGM - kClusterKappa;
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

    // what is given stays with the CTA: the permutation, or its inverse
    uint16_t *const given = inverse ? Q : Pa;
    const Pair2<uint16_t> &other = inverse ? Pa2 : Q2;
    for (int j = tid; j < M; j += T) given[j] = uint16_t(BENES_GUARD(src[flat0 + rank * uint32_t(M) + j], kBoth));
    for (int t = tid; t < M / 2; t += T) own[t] = uint16_t(kNone16);
    cluster.sync();           // both CTAs are running (and loaded) before either touches the other's memory
    // a1: its inverse goes to the CTA that keeps that place
    for (int j = tid; j < M; j += T) {
        const uint32_t v = given[j];
        other.of(v >> LOGM)[v & kInCta] = uint16_t(rank * uint32_t(M) + j);
    }
    cluster.sync();

    // walks from this CTA's ruler outputs (its ruler switches are its own); about half of
    // the switches and inverse entries a walker reaches are in the other CTA
    for (int rl = tid; rl < R; rl += T) {
        const uint32_t rho = rank * uint32_t(R) + rl;
        const uint32_t group = rho >> 1, side0 = rho & 1u;
        const uint32_t t0 = (group << kClusterKappa) | fused_slot<kClusterKappa>(group, uint32_t(level));
        uint32_t j = 2u * t0 + side0;
        uint32_t fwd = j, part = kNone16, pr = rho ^ 1u;
        if (!side0) own[t0 & kSwInCta] = uint16_t(rho << 1);
        uint32_t pp = *reinterpret_cast<const uint32_t *>(Pa + 2u * (t0 & kSwInCta));
        uint32_t p = (side0 ? pp : (pp >> 16)) & kBoth;                // P[j^1]
        uint32_t q = Q2.of((p ^ 1u) >> LOGM)[(p ^ 1u) & kInCta];
        for (uint32_t hops = 0; hops <= kBoth; ++hops) {                 // a walk claims < 2^15 switches
            j = q;
            const uint32_t t = j >> 1, side = j & 1u, g = t >> kClusterKappa;
            if ((t & ((1u << kClusterKappa) - 1u)) == fused_slot<kClusterKappa>(g, uint32_t(level))) {
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
    for (int r = 0; r < kClusterLog2M - kClusterKappa - 1; ++r) {
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
    for (int r = 0; r < kEnter; ++r) enter4<Cfg>(smem_raw, uint32_t(tid + r * T), v[r], false, LOGM);
    __syncthreads();
    FusedOut out;
    out.bits = bits;
    out.n = n;
    out.flat0 = flat0 + rank * uint32_t(M);
    out.valid = uint32_t(M);
    fused_levels<Cfg>(smem_raw, out, LOGM);
}

template <class Cfg>
int configure_fused() {
    static OncePerDevice configured;
    return configured.run([]() -> int {
        BENES_CUDA_TRY(cudaFuncSetAttribute(k_route_fused<Cfg>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(Cfg::kSmemBytes)));
        BENES_CUDA_TRY(cudaFuncSetAttribute(k_route_fused<Cfg>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                            cudaSharedmemCarveoutMaxShared));
        cudaFuncAttributes loaded;                             // (asking for them loads the kernel)
        BENES_CUDA_TRY(cudaFuncGetAttributes(&loaded, k_route_fused<Cfg>));
        return BENES_OK;
    });
}

template <class Cfg>
int launch_one(const uint32_t *src, bool inverse, size_t first, size_t end, uint32_t *bits, int log2n, int logs, cudaStream_t s) {
    const int rc = configure_fused<Cfg>();
    if (rc) return rc;
    const size_t ctas = (end - first + Cfg::C - 1) >> Cfg::LOG;
    launch_kernel(k_route_fused<Cfg>, unsigned(ctas), Cfg::T, Cfg::kSmemBytes, s, src, inverse, bits, log2n, logs, first, end);
    return launch_status();
}

template <class Cfg>
int launch_peel(const uint32_t *src, bool inverse, size_t total, uint32_t *bits, int log2n, uint32_t *next, cudaStream_t s) {
    static OncePerDevice configured;
    const int rc = configured.run([]() -> int {
        BENES_CUDA_TRY(cudaFuncSetAttribute(k_route_peel<Cfg>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(Cfg::kSmemBytes)));
        return BENES_OK;
    });
    if (rc) return rc;
    launch_kernel(k_route_peel<Cfg>, unsigned(total >> Cfg::LOG), Cfg::T, Cfg::kSmemBytes, s, src, inverse, bits, log2n, next);
    return launch_status();
}

int launch_cluster2(const uint32_t *src, bool inverse, size_t first_block, size_t blocks, uint32_t *bits, int log2n, cudaStream_t s) {
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
    launch_kernel(k_route_cluster2, unsigned(2 * blocks), ClusterTailCfg::T, kClusterSmemBytes, s, src, inverse, bits, log2n,
                  uint32_t(first_block));
    return launch_status();
}

}  // namespace

int launch_fused(const uint32_t *src, bool inverse, size_t total, int log2m, uint32_t *bits, int log2n,
                 cudaStream_t s, size_t first_block, size_t blocks, uint32_t *const spare[2]) {
    if (log2m < 1 || log2m > kClusterLog2M) return BENES_ERR_BADARG;
    // Inverses are taken where every kernel below does (and k_route_peel leaves them): k_route_few of 2^11, 16-bit entries.
    static_assert(kPeelLog2 - 1 >= kMinInverseLog2 && kMinInverseLog2 >= kFMinLogS, "");
    if (inverse && log2m < kMinInverseLog2) return BENES_ERR_BADARG;
    if (blocks == 0) blocks = (total >> log2m) - first_block;        // all the rest
    if (first_block + blocks > (total >> log2m)) return BENES_ERR_BADARG;
    if (log2m == kClusterLog2M) return launch_cluster2(src, inverse, first_block, blocks, bits, log2n, s);
    const size_t first = first_block << log2m, end = first + (blocks << log2m);
    int m = log2m;
    if (spare && first == 0 && end == total) {
        // A call that splits whole permutations readies the kernel of a call that may not (a captured one) too, so that
        // one ordinary call is enough before a capture.
        if (log2m == log2n && m >= kPeelLog2 && 2 * (total >> m) <= size_t(sm_count())) {
            const int rc = m == 15 ? configure_fused<FusedCfg<15, 2>>() : m == 14 ? configure_fused<FusedCfg<14, 1>>()
                         : m == 13 ? configure_fused<FusedCfg<13, 1>>() : configure_fused<FusedCfg<12, 1>>();
            if (rc) return rc;
        }
        for (int i = 0; m >= kPeelLog2 && 2 * (total >> m) <= size_t(sm_count()); --m, i ^= 1) {
            const int rc = m == 15 ? launch_peel<FusedCfg<15, 2>>(src, inverse, total, bits, log2n, spare[i], s)
                         : m == 14 ? launch_peel<FusedCfg<14, 1>>(src, inverse, total, bits, log2n, spare[i], s)
                         : m == 13 ? launch_peel<FusedCfg<13, 1>>(src, inverse, total, bits, log2n, spare[i], s)
                                   : launch_peel<FusedCfg<12, 1>>(src, inverse, total, bits, log2n, spare[i], s);
            if (rc) return rc;
            src = spare[i];
            inverse = true;
        }
    }
    // Blocks of up to 2^11 and few switches: k_route_few.  A thread of it goes through every level of its switch, which costs
    // the same at every size; the kernels below have tables and one thread per sub-block for the last levels, so
    // the smaller the blocks, the earlier they are faster.  Limits in outputs per SM (a GPU full of threads has 4096), either
    // side of the line: 2^5 2^17.0 outputs 4.8 and 5.7 us, 2^17.5 5.3 and 5.0; 2^6 2^18 6.2 and 6.4, 2^18.5 8.0 and 6.6;
    // 2^7 2^18.75 11.5 and 13.0, 2^19 13.0 and 11.4; 2^8 2^19 15.8 and 19.2, 2^20 29 and 21; 2^11 2^19 33 and 36, 2^19.25 49 and 38.
    // (Up to 4096 for all of them, 17912 x 2^5 took 12.4 us and 25171 x 2^5 7.6.)
    const size_t few_per_sm = 1024 * size_t(m <= 5 ? 1 : m <= 8 ? m - 4 : 4);
    if (m <= 11 && first == 0 && end <= few_per_sm * size_t(sm_count())) {
        const int logc = m > 8 ? m : 8;
        return logc == 8 ? launch_few<8>(src, inverse, end, bits, log2n, m, s) : logc == 9 ? launch_few<9>(src, inverse, end, bits, log2n, m, s)
             : logc == 10 ? launch_few<10>(src, inverse, end, bits, log2n, m, s) : launch_few<11>(src, inverse, end, bits, log2n, m, s);
    }
    // Small blocks share a CTA: a thread of the 8-bit levels takes a whole sub-block, so the more sub-blocks a CTA holds, the
    // fuller its warps, and every CTA copies 9 KiB of tables; but it takes its phases one after the other, and smaller ones
    // run side by side.  Up to CTAs of 2^12, of which an SM holds eight: as soon as there are more CTAs than SMs for
    // blocks of 2^6 and less (against up to five per SM 22708 x 2^5 9.2 -> 7.1 us, 9741 x 2^6 10.6 -> 8.9), above three per SM
    // up to 2^9 (4915 x 2^8 27.6 -> 25.2, 2896 x 2^9 34.4 -> 32.2; as soon as there are more than SMs 6888 x 2^7 shift 13.4 ->
    // 14.1), above four from there on (1448 x 2^10 40.9 -> 38.7; above three 1024 x 2^10 34.2 -> 35.3).  CTAs of 2^13 pay
    // where those of 2^12 do not run all at once (1024 x 2^12 84 us in CTAs of 2^12 and 95 in larger ones, 2048 x 2^11 72 and
    // 82; blocks of 2^3 and less already above five per SM: 440871 x 2^3 14.6 and 13.4), and never for blocks of 2^4 to 2^9
    // (22230 x 2^8 61 and 72, 32768 x 2^7 28 and 32; CTAs of 2^11 98 and 36).
    int logc = m > 10 ? m : 10;
    const int most = m >= 4 && m <= 9 ? 12 : 13;
    auto per_sm = [m](int lc) { return size_t(lc < 12 ? (m <= 6 ? 1 : m <= 9 ? 3 : 4) : (m <= 3 ? 5 : 8)); };
    while (logc < most && ((end - first) >> logc) > per_sm(logc) * size_t(sm_count())) ++logc;
    // CTAs that have an SM to themselves get more threads: their time is a chain of short
    // phases, not the instructions they issue.
    const bool alone = ((end - first + (size_t(1) << logc) - 1) >> logc) <= size_t(sm_count());
#define BENES_FUSED(LC, G) return launch_one<FusedCfg<LC, G>>(src, inverse, first, end, bits, log2n, m, s)
    switch (logc) {
        case 10: if (alone) BENES_FUSED(10, 1); BENES_FUSED(10, 2);
        case 11: if (alone) BENES_FUSED(11, 1); BENES_FUSED(11, 2);
        case 12: if (alone) BENES_FUSED(12, 1); BENES_FUSED(12, 2);
        case 13: if (alone) BENES_FUSED(13, 1); BENES_FUSED(13, 2);
        case 14: if (alone) BENES_FUSED(14, 1); BENES_FUSED(14, 2);
        default: BENES_FUSED(15, 2);
    }
#undef BENES_FUSED
}

}  // namespace benes
