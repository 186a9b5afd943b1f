// Payload apply over several stages per pass.
//
// One stage per kernel moves the whole payload through HBM 2n-1 times.  Here a
// CTA takes 2^C elements and runs many stages on them:
//
//   inner kernel : every block of 2^b elements (b = min(n, C)) of level n-b
//                  is closed under the 2b-1 innermost stages (input side of
//                  levels n-b .. n-2, middle, output side back up to n-b); a CTA has
//                  one block, or 2^(C-b) of them;
//   outer kernels: k consecutive input-side stages of levels l0..l0+k-1
//                  send a contiguous chunk of 2^k * T elements of a level-l0
//                  block to 2^k runs of T consecutive positions (one run per
//                  path through the k switches), so a CTA reads one chunk,
//                  runs k stages and writes 2^k runs; the output-side kernel is the mirror
//                  image.
//
// The payload itself does not move through the stages: 16-bit PLACES do, and at the end
// every output position fetches its element from the place it ended up with.  The
// elements arrive in shared memory by asynchronous copies while the places are routed.
// "Slot" u of a chunk keeps, in its low bits, the outcomes of the stages done so far
// (bit i = 1 if the element left stage l0+i through the lower output) and in
// its high bits the part of its position the remaining stages still act on:
// stage l0+i pairs slots u and u | (1 << i), and a crossed switch swaps them.
// The true position after i stages is
//     (bit-reversed low i bits of u) << (m0 - i)  +  (X0 >> i) + (u >> i),
// m0 = log2 of the level-l0 block size, X0 = offset of the chunk in that
// block; this gives both the switch index of a pair and where a slot is
// written at the end.  The output side reads the same relation backwards.
//
// A 32-bit word holds two slots that differ in the top slot bit, so one
// exchange (t = (a ^ b) & mask; a ^= t; b ^= t) serves two switches: 6 instructions per
// two switches with the mask, where 64-bit selects took 8 per switch and moved 8 bytes per
// element through shared memory in every round.  The switch words of a pass are staged in
// shared memory in the order that makes the masks cheap: a staged word has the bits of 16
// switches in its low half and those of their partners (top slot bit set) in its high half.
// A thread holds 2^R words (R <= 4 slot bits) and runs all the stages of a pass on those slot bits
// between two barriers.
//
// Measured on B200: 2^26 elements of 8 bytes (5 passes) 2.10 -> 1.13 ms, 4 x 2^22 of 8 bytes (5 passes -> 3)
// 0.54 -> 0.27 ms, 16384 x 2^8 of 4 bytes 84 -> 19 us.
#include "common.cuh"

namespace benes {
namespace {

constexpr int kChunkLog2 = 13;               // slots per CTA
constexpr int kSmallLog2 = 10;               // ... of a pass with too few elements to go round the SMs
constexpr int kMaxOuter = 10;                // stages of an outer pass at most
template <typename E> constexpr int kOuterLog2 = sizeof(E) == 8 ? 12 : 13;     // slots per CTA of an outer pass
template <int C> constexpr int kApplyThreads = 1 << (C - 5);
template <int C> constexpr int kRowWords = 1 << (C - 6);        // staged words per stage

__device__ __forceinline__ uint32_t rev_bits(uint32_t v, int i) {
    return i ? (__brev(v) >> (32 - i)) : 0u;
}

// Word w of the places lives at shared-memory index swz(w): an XOR of the low five bits, chosen so that the
// 16-word groups of a round and the columns of the outer kernels' transposition spread over the banks.
__device__ __forceinline__ constexpr uint32_t swz(uint32_t w) { return w ^ ((w >> 5) & 31u) ^ (w >> 10); }

// Element e of the payload lives at place(e): whole 16-byte units move (the copies write them), by an XOR of the
// unit's low three bits, so that power-of-two strides do not meet in one bank.  Linear over XOR.
template <typename E>
__device__ __forceinline__ constexpr uint32_t place(uint32_t e) {
    const int lg = sizeof(E) == 8 ? 1 : 2;   // log2(elements per unit)
    const uint32_t u = e >> lg;
    return ((u ^ (((u >> 3) ^ (u >> 6) ^ (u >> 9)) & 7u)) << lg) | (e & ((1u << lg) - 1u));
}

template <int BYTES>
__device__ __forceinline__ void copy_async(void *smem, const void *global) {
    const uint32_t d = uint32_t(__cvta_generic_to_shared(smem));
    if (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(d), "l"(global) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" :: "r"(d), "l"(global), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// What a pass needs to know about its switch words.
struct Geometry {
    const uint32_t *bits;     // outer: the words of this permutation; inner: of the batch
    size_t stage_w;           // words per stage
    size_t first_sw;          // outer: first switch of the level-l0 block (within the permutation);
                              // inner: first switch of the chunk (within the batch)
    size_t end_sw;            // inner: switches of the batch
    uint32_t x0;              // outer: offset of the chunk inside that block
    int m0;                   // outer: log2 of the level-l0 block size
    int n;
};

// Switch bits [32 w, 32 w + 32) of one stage of the chunk.  The inner kernel's are consecutive in the
// stage (of several permutations for small n).
__device__ __forceinline__ uint32_t bits32_inner(const Geometry &g, int stage, uint32_t w) {
    const size_t sw = g.first_sw + 32u * w;
    if (sw >= g.end_sw) return 0u;
    if (g.n >= 6) {
        const size_t fw = sw >> 5, perm = fw >> (g.n - 6), lw = fw & (g.stage_w - 1);
        return __ldg(g.bits + ((perm * size_t(2 * g.n - 1) + size_t(stage)) << (g.n - 6)) + lw);
    }
    // a word per permutation of 2^(n-1) switches
    const int lg = g.n - 1;
    const uint32_t per = 32u >> lg, mask = (1u << (1u << lg)) - 1u;
    uint32_t v = 0;
    for (uint32_t r = 0; r < per && sw + (size_t(r) << lg) < g.end_sw; ++r)
        v |= (__ldg(g.bits + ((sw >> lg) + r) * size_t(2 * g.n - 1) + size_t(stage)) & mask) << (r << lg);
    return v;
}

// ... the outer kernels' come in runs of 2^(C-1-i), one per path through the i stages before.
template <int C>
__device__ __forceinline__ uint32_t bits32_outer(const Geometry &g, int stage, int i, uint32_t w) {
    const int lg = C - 1 - i;
    const uint32_t *row = g.bits + size_t(stage) * g.stage_w;
    const uint32_t first = uint32_t(g.first_sw) + (g.x0 >> (i + 1)), idx = 32u * w;
    if (lg >= 5) {
        const uint32_t sw = first + ((idx >> lg) << (g.m0 - 1 - i)) + (idx & ((1u << lg) - 1u));
        return __ldg(row + (sw >> 5));
    }
    // 2, 4 or 8 runs of 2^lg >= 4 switches (k <= kMaxOuter); their loads are under way together
    static_assert(C - kMaxOuter >= 2, "a run has at least four switches");
    uint32_t v = 0;
#pragma unroll
    for (uint32_t r = 0; r < 8; ++r) {
        if ((r << lg) >= 32u) continue;
        const uint32_t sw = first + (((idx >> lg) + r) << (g.m0 - 1 - i));
        v |= ((__ldg(row + (sw >> 5)) >> (sw & 31u)) & ((1u << (1u << lg)) - 1u)) << (r << lg);
    }
    return v;
}

// Staged rows: bit k of the low half of word q of a row is the switch whose index has q, k and a 0 put in at
// bit e (where the packed slot bit is), bit k of the high half the one with a 1 there.  A thread makes two words
// of a row at a time; the loads of four such items are under way together.
// row_of(r) = e of row r; bits32(r, w) = switch bits [32 w, 32 w + 32) of row r.
template <int C, class RowE, class Bits32>
__device__ __forceinline__ void stage_rows(uint32_t *rows, int count, const RowE &row_e, const Bits32 &bits32) {
    constexpr uint32_t T = kApplyThreads<C>, kItems = kRowWords<C> / 2;
    const uint32_t items = uint32_t(count) * kItems;
    for (uint32_t base = threadIdx.x; base < items; base += 4 * T) {
        uint32_t x[4], y[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint32_t idx = base + uint32_t(q) * T;
            x[q] = y[q] = 0u;
            if (idx < items) {
                const int r = int(idx / kItems), e = row_e(r);
                const uint32_t t = idx & (kItems - 1u);
                if (e >= 5) {
                    const uint32_t w = ((t >> (e - 5)) << (e - 4)) | (t & ((1u << (e - 5)) - 1u));
                    x[q] = bits32(r, w);
                    y[q] = bits32(r, w | (1u << (e - 5)));
                } else {
                    x[q] = bits32(r, 2u * t);
                    y[q] = bits32(r, 2u * t + 1u);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint32_t idx = base + uint32_t(q) * T;
            if (idx < items) {
                const int r = int(idx / kItems), e = row_e(r);
                const uint32_t t = idx & (kItems - 1u);
                uint32_t a = x[q], b = y[q];
                if (e >= 5) {
                    a = __byte_perm(x[q], y[q], 0x5410);
                    b = __byte_perm(x[q], y[q], 0x7632);
                } else {
                    // the two kinds alternate inside a word: bit-index e moves up to 4
                    auto swap = [&](int s, uint32_t mask) {             // bit-indices s and s + 1
                        const uint32_t da = ((a >> (1 << s)) ^ a) & mask, db = ((b >> (1 << s)) ^ b) & mask;
                        a ^= da ^ (da << (1 << s));
                        b ^= db ^ (db << (1 << s));
                    };
                    if (e <= 0) swap(0, 0x22222222u);
                    if (e <= 1) swap(1, 0x0C0C0C0Cu);
                    if (e <= 2) swap(2, 0x00F000F0u);
                    if (e <= 3) swap(3, 0x0000FF00u);
                }
                *reinterpret_cast<uint2 *>(rows + r * int(kRowWords<C>) + 2u * t) = make_uint2(a, b);
            }
        }
    }
}

// One exchange of two packed switches.
__device__ __forceinline__ void exchange(uint32_t &a, uint32_t &b, uint32_t bits) {
    const uint32_t t = (a ^ b) & ((bits & 0x00010001u) * 0xFFFFu);
    a ^= t;
    b ^= t;
}

// The stages of one pass on slot bits [ILO, ILO + R): ascending on the input side (IN), descending on
// the output side (OUT); with both, the highest of them is the middle stage.  The packed slot bit is the top one, so the
// switches of the words u0 | q << ILO are, in a chunk of 2^beff-slot blocks with that bit taken out, at
//     (block << (beff - 1)) + (rev_i(low i bits of the slot) << (beff - 1 - i)) + (slot >> (i + 1)):
// the bits of q below the stage's move the run, those above it are neighbouring switches of one staged word.
// rows_in / rows_out: staged words of slot bit 0.
// FULL: beff = C - 1, known at compile time (all passes above 2^C elements).
template <int C, int ILO, int R, bool IN, bool OUT, bool FULL>
__device__ __forceinline__ void run_round(uint32_t *words, const uint32_t *rows_in, const uint32_t *rows_out, int beff_) {
    const int beff = FULL ? C - 1 : beff_;
    for (uint32_t g = threadIdx.x; g < (1u << (C - 1 - R)); g += kApplyThreads<C>) {
        const uint32_t u0 = ((g >> ILO) << (ILO + R)) | (g & ((1u << ILO) - 1u));
        uint32_t *mine = words;
        const uint32_t p0 = swz(u0);
        uint32_t v[1 << R];
#pragma unroll
        for (int q = 0; q < (1 << R); ++q) v[q] = mine[p0 ^ swz(uint32_t(q) << ILO)];
        const uint32_t block = (u0 >> beff) << (beff - 1), in_block = u0 & ((1u << beff) - 1u);
        auto stage = [&](int j, const uint32_t *rows) {
            const int i = ILO + j, sh = beff - 1 - i;
            const uint32_t pos0 = block + (rev_bits(u0 & ((1u << i) - 1u), i) << sh) + (in_block >> (i + 1));
            const uint32_t *row = rows + i * kRowWords<C>;
#pragma unroll
            for (int lo = 0; lo < (1 << R); ++lo) {
                if (lo >= (1 << j)) continue;
                uint32_t crev = 0;                        // lo with its j bits reversed
#pragma unroll
                for (int t = 0; t < R; ++t)
                    if (t < j) crev |= ((uint32_t(lo) >> t) & 1u) << (j - 1 - t);
                // (the low four bits of pos0 are clear where crev puts any)
                const uint32_t off = crev << sh;
                const uint32_t w = row[(pos0 >> 4) + (off >> 4)] >> ((pos0 & 15u) + (off & 15u));
#pragma unroll
                for (int hi = 0; hi < (1 << R); ++hi) {
                    if (hi >= (1 << (R - 1 - j))) continue;
                    const int q = lo | (hi << (j + 1));
                    exchange(v[q], v[q | (1 << j)], w >> hi);
                }
            }
        };
        if (IN) {
#pragma unroll
            for (int j = 0; j < R; ++j) stage(j, rows_in);
        }
        if (OUT) {
#pragma unroll
            for (int j = R - 1; j >= 0; --j)
                if (!IN || j < R - 1) stage(j, rows_out);
        }
#pragma unroll
        for (int q = 0; q < (1 << R); ++q) mine[p0 ^ swz(uint32_t(q) << ILO)] = v[q];
    }
}

template <int C, int ILO, bool IN, bool OUT, bool FULL>
__device__ __forceinline__ void run_round_r(uint32_t *words, const uint32_t *rows_in, const uint32_t *rows_out, int beff, int r) {
    if (r == 4) run_round<C, ILO, 4, IN, OUT, FULL>(words, rows_in, rows_out, beff);
    else if (r == 3) run_round<C, ILO, 3, IN, OUT, FULL>(words, rows_in, rows_out, beff);
    else if (r == 2) run_round<C, ILO, 2, IN, OUT, FULL>(words, rows_in, rows_out, beff);
    else run_round<C, ILO, 1, IN, OUT, FULL>(words, rows_in, rows_out, beff);
}

template <int C, bool IN, bool OUT, bool FULL>
__device__ __forceinline__ void run_group(uint32_t *words, const uint32_t *rows_in, const uint32_t *rows_out, int beff, int ilo, int r) {
    if (ilo == 0) run_round_r<C, 0, IN, OUT, FULL>(words, rows_in, rows_out, beff, r);
    else if (ilo == 4) run_round_r<C, 4, IN, OUT, FULL>(words, rows_in, rows_out, beff, r);
    else run_round_r<C, 8, IN, OUT, FULL>(words, rows_in, rows_out, beff, r);
    __syncthreads();
}

// Block of 2^C: the middle stage and the output stages on slot bits C-2, C-3, C-4.  The top slot bit takes
// part, so the words are packed on slot bit C-5 meanwhile.
template <int C>
__device__ __forceinline__ void run_middle(uint32_t *words, const uint32_t *rows_in, const uint32_t *rows_out) {
    const uint32_t u0 = threadIdx.x, p0 = swz(u0);              // slot bits 0 .. C-6
    uint32_t v[16];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const uint32_t a = words[p0 ^ swz(uint32_t(q) << (C - 4))], b = words[p0 ^ swz((uint32_t(q) << (C - 4)) | (1u << (C - 5)))];
        v[q] = __byte_perm(a, b, 0x5410);
        v[q | 8] = __byte_perm(a, b, 0x7632);
    }
    const uint32_t pos0 = rev_bits(u0, C - 5) << 3;
#pragma unroll
    for (int jj = 0; jj < 4; ++jj) {
        const int j = 3 - jj;
        const uint32_t w = (j == 3 ? rows_in : rows_out)[(C - 4 + j) * kRowWords<C> + (pos0 >> 4)] >> (pos0 & 15u);
#pragma unroll
        for (int lo = 0; lo < 8; ++lo) {
            if (lo >= (1 << j)) continue;
            uint32_t crev = 0;
#pragma unroll
            for (int t = 0; t < 3; ++t)
                if (t < j) crev |= ((uint32_t(lo) >> t) & 1u) << (j - 1 - t);
#pragma unroll
            for (int hi = 0; hi < 8; ++hi) {
                if (hi >= (1 << (3 - j))) continue;
                const int q = lo | (hi << (j + 1));
                exchange(v[q], v[q | (1 << j)], w >> ((crev << (3 - j)) + hi));
            }
        }
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        words[p0 ^ swz(uint32_t(q) << (C - 4))] = __byte_perm(v[q], v[q | 8], 0x5410);
        words[p0 ^ swz((uint32_t(q) << (C - 4)) | (1u << (C - 5)))] = __byte_perm(v[q], v[q | 8], 0x7632);
    }
    __syncthreads();
}

// shared memory: payload, places, staged switch words
template <typename E, int C>
constexpr size_t apply_smem(int rows) {
    return (sizeof(E) << C) + (size_t(4) << (C - 1)) + size_t(rows) * kRowWords<C> * 4;
}

// Inner kernel: all 2b-1 stages of the blocks of 2^b elements of level n-b in the CTA's chunk.
// (In this kernel and the next a thread's items are tid + r T: every index map is linear over XOR,
// so the part of r is a constant and the part of tid is formed once.)
template <typename E, int C>
__global__ void __launch_bounds__(kApplyThreads<C>, (C == kChunkLog2 ? (sizeof(E) == 8 ? 2 : 3) : 8))
k_apply_inner(const uint32_t *__restrict__ bits, const E *__restrict__ x, E *__restrict__ y, int n, int b,
              size_t total, uint32_t cta0) {
    after_previous_kernel();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr uint32_t T = kApplyThreads<C>, kHalf = 1u << (C - 1);
    E *sm = reinterpret_cast<E *>(smem_raw);
    uint32_t *words = reinterpret_cast<uint32_t *>(smem_raw + (sizeof(E) << C));
    uint32_t *rows = words + kHalf;
    const uint32_t tid = threadIdx.x;
    const size_t flat0 = size_t(blockIdx.x + cta0) << C;
    const uint32_t valid = uint32_t(total - flat0 < (size_t(1) << C) ? total - flat0 : size_t(1) << C);
    constexpr uint32_t kUnit = 16 / uint32_t(sizeof(E)), kUnits = (1u << C) / kUnit;
    x += flat0;
    y += flat0;
    if (((reinterpret_cast<uintptr_t>(x) | (valid * sizeof(E))) & 15u) == 0) {
        const uint32_t p0 = place<E>(tid * kUnit);
#pragma unroll
        for (uint32_t r = 0; r < kUnits / T; ++r)
            if (tid + r * T < valid / kUnit) copy_async<16>(sm + (p0 ^ place<E>(r * T * kUnit)), x + tid * kUnit + r * T * kUnit);
    } else {
        for (uint32_t u = tid; u < valid; u += T) copy_async<int(sizeof(E))>(sm + place<E>(u), x + u);
    }
    Geometry g;
    g.bits = bits; g.n = n;
    g.stage_w = n >= 6 ? size_t(1) << (n - 6) : 1;
    g.first_sw = flat0 >> 1; g.end_sw = total >> 1;
    g.x0 = 0; g.m0 = b;
    // words of the b input-side + middle stages in rows 0..b-1, of the b-1 output-side stages in rows
    // b..2b-2 (row b+i for slot bit i); bit of the index the packed slot bit is at
    auto row_e = [&](int r) {
        const int i = r < b ? r : r - b;
        const bool middle = b == C && (r < b ? i == C - 1 : i >= C - 4);
        return b < C ? C - 2 : (middle ? 3 : C - 2 - i);
    };
    auto stage_of = [&](int r) { return r < b ? n - b + r : 2 * n - 2 - (n - b + (r - b)); };
    if (n >= C) {
        // one permutation
        const uint32_t *p = bits + (flat0 >> n) * size_t(2 * n - 1) * g.stage_w + ((flat0 & ((size_t(1) << n) - 1)) >> 6);
        stage_rows<C>(rows, 2 * b - 1, row_e, [&](int r, uint32_t w) { return __ldg(p + size_t(stage_of(r)) * g.stage_w + w); });
    } else {
        stage_rows<C>(rows, 2 * b - 1, row_e, [&](int r, uint32_t w) { return bits32_inner(g, stage_of(r), w); });
    }
    const uint32_t s0 = swz(tid), w0 = place<E>(tid) | (place<E>(tid | kHalf) << 16);
#pragma unroll
    for (uint32_t r = 0; r < kHalf / T; ++r) words[s0 ^ swz(r * T)] = w0 ^ (place<E>(r * T) * 0x10001u);
    __syncthreads();
    const uint32_t *rows_out = rows + b * int(kRowWords<C>);
    if (b == C) {
        run_group<C, true, false, true>(words, rows, rows_out, C - 1, 0, 4);
        run_group<C, true, false, true>(words, rows, rows_out, C - 1, 4, 4);
        run_group<C, true, false, true>(words, rows, rows_out, C - 1, 8, C - 9);
        run_middle<C>(words, rows, rows_out);
        if (C - 5 >= 8) run_group<C, false, true, true>(words, rows, rows_out, C - 1, 8, C - 12 > 0 ? C - 12 : 1);
        run_group<C, false, true, true>(words, rows, rows_out, C - 1, 4, C - 5 >= 8 ? 4 : C - 8);
        run_group<C, false, true, true>(words, rows, rows_out, C - 1, 0, 4);
    } else {
        const int last = (b - 1) & ~3;
        for (int ilo = 0; ilo < last; ilo += 4) run_group<C, true, false, false>(words, rows, rows_out, b, ilo, 4);
        run_group<C, true, true, false>(words, rows, rows_out, b, last, b - last);
        for (int ilo = last - 4; ilo >= 0; ilo -= 4) run_group<C, false, true, false>(words, rows, rows_out, b, ilo, 4);
    }
    copies_done();
    __syncthreads();
#pragma unroll
    for (uint32_t r = 0; r < kHalf / T; ++r) {
        const uint32_t v = words[s0 ^ swz(r * T)];
        if (tid + r * T < valid) y[tid + r * T] = sm[v & 0xFFFFu];
        if (tid + r * T + kHalf < valid) y[tid + r * T + kHalf] = sm[v >> 16];
    }
}

// Outer kernel, input side (OUT = false): stages l0 .. l0+k-1 on a contiguous
// chunk; output side (OUT = true): stages 2n-2-(l0+k-1) .. 2n-2-l0, chunk
// gathered from its 2^k runs and written contiguously.
template <typename E, int C, bool OUT>
__global__ void __launch_bounds__(kApplyThreads<C>, (sizeof(E) == 8 ? 5 : 4))
k_apply_outer(const uint32_t *__restrict__ bits, const E *__restrict__ x, E *__restrict__ y, int n,
              int l0, int k, uint32_t cta0) {
    after_previous_kernel();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr uint32_t T = kApplyThreads<C>, kHalf = 1u << (C - 1);
    E *sm = reinterpret_cast<E *>(smem_raw);
    uint32_t *words = reinterpret_cast<uint32_t *>(smem_raw + (sizeof(E) << C));
    uint32_t *rows = words + kHalf;
    const uint32_t tid = threadIdx.x;
    const size_t flat0 = size_t(blockIdx.x + cta0) << C;
    const int m0 = n - l0, tbits = C - k;                           // log2 of the run length
    Geometry g;
    g.n = n; g.m0 = m0;
    g.stage_w = size_t(1) << (n - 6);
    g.bits = bits + (flat0 >> n) * size_t(2 * n - 1) * g.stage_w;
    const uint32_t local = uint32_t(flat0 & ((size_t(1) << n) - 1));
    const uint32_t block = local & ~((1u << m0) - 1u);
    g.first_sw = block >> 1; g.end_sw = 0; g.x0 = local - block;
    // the runs' first element in memory, and where element e of the chunk (run e >> tbits, position
    // e & (2^tbits - 1)) lies from there on; like every map below it is linear over disjoint bits
    const size_t runs = flat0 - g.x0 + (g.x0 >> k);
    auto in_runs = [&](uint32_t e) { return (rev_bits(e >> tbits, k) << (m0 - k)) + (e & ((1u << tbits) - 1u)); };
    constexpr uint32_t kUnit = 16 / uint32_t(sizeof(E)), kUnits = (1u << C) / kUnit;
    const E *src = x + (OUT ? runs : flat0);
    auto source = [&](uint32_t e) { return OUT ? in_runs(e) : e; };
    if ((reinterpret_cast<uintptr_t>(x) & 15u) == 0) {
        const uint32_t p0 = place<E>(tid * kUnit);
        src += source(tid * kUnit);
#pragma unroll
        for (uint32_t r = 0; r < kUnits / T; ++r)
            copy_async<16>(sm + (p0 ^ place<E>(r * T * kUnit)), src + source(r * T * kUnit));
    } else {
        for (uint32_t u = tid; u < (1u << C); u += T) copy_async<int(sizeof(E))>(sm + place<E>(u), src + source(u));
    }
    stage_rows<C>(rows, k, [&](int i) { return C - 2 - i; },
                  [&](int i, uint32_t w) { return bits32_outer<C>(g, OUT ? 2 * n - 2 - (l0 + i) : l0 + i, i, w); });
    // slot u is element (u's low k bits on top) of the chunk on the output side
    auto start = [&](uint32_t u) { return place<E>(OUT ? ((u & ((1u << k) - 1u)) << tbits) | (u >> k) : u); };
    const uint32_t s0 = swz(tid), w0 = start(tid) | (start(tid | kHalf) << 16);
#pragma unroll
    for (uint32_t r = 0; r < kHalf / T; ++r) words[s0 ^ swz(r * T)] = w0 ^ (start(r * T) * 0x10001u);
    __syncthreads();
    if (!OUT) {
        for (int ilo = 0; ilo < k; ilo += 4) run_group<C, true, false, true>(words, rows, rows, C - 1, ilo, min(4, k - ilo));
    } else {
        for (int ilo = (k - 1) & ~3; ilo >= 0; ilo -= 4) run_group<C, false, true, true>(words, rows, rows, C - 1, ilo, min(4, k - ilo));
    }
    copies_done();
    __syncthreads();
    if (OUT) {
        y += flat0 + tid;
#pragma unroll
        for (uint32_t r = 0; r < kHalf / T; ++r) {
            const uint32_t v = words[s0 ^ swz(r * T)];
            y[r * T] = sm[v & 0xFFFFu];
            y[r * T + kHalf] = sm[v >> 16];
        }
    } else if (tbits > 5) {
        // item t: position yy = t's low bits of the first half of run c; that half comes from the low
        // halves of its words, the second from the high halves
        const int hbits = tbits - 1;
        auto word = [&](uint32_t t) { return swz(((t & ((1u << hbits) - 1u)) << k) | (t >> hbits)); };
        auto out = [&](uint32_t t) { return (rev_bits(t >> hbits, k) << (m0 - k)) + (t & ((1u << hbits) - 1u)); };
        y += runs + out(tid);
        const uint32_t q0 = word(tid);
#pragma unroll
        for (uint32_t r = 0; r < kHalf / T; ++r) {
            const uint32_t v = words[q0 ^ word(r * T)];
            E *p = y + out(r * T);
            p[0] = sm[v & 0xFFFFu];
            p[size_t(1) << hbits] = sm[v >> 16];
        }
    } else {
        // short runs: neighbouring lanes take neighbouring positions of a whole run, so that sectors leave complete
        const uint32_t hbit = 1u << (tbits - 1), shift = (tid & hbit) ? 16u : 0u;
        auto word = [&](uint32_t e) { return swz(((e & (hbit - 1u)) << k) | (e >> tbits)); };
        y += runs + in_runs(tid);
        const uint32_t q0 = word(tid);
#pragma unroll
        for (uint32_t r = 0; r < (1u << C) / T; ++r)
            y[in_runs(r * T)] = sm[(words[q0 ^ word(r * T)] >> shift) & 0xFFFFu];
    }
}

// Few outputs in all: when every thread of the GPU can have one to itself, the shortest chain of steps is to
// trace it back through the network: from output j, stage by stage, to the input its element came from.  A
// CTA keeps the switch words of its permutations in shared memory; a stage is one load and a rotation of the low m
// bits of the position (2^m = size of the level's blocks).
//   output side of level l: position B + 2t + s came from B + t of the upper (lower) half-block if s ^ bit is 0 (1)
//   input side:             position s of the upper (lower) half came from B + 2s + (lower ^ bit)
// (The chunk kernels' long unrolled code runs once there and waits for its instructions: one network of 2^11
// 10.4 -> 6 us; with more outputs than threads they are faster: 300 networks of 2^12 14.5 against 30 us.)
constexpr int kTraceLog2 = 12;
constexpr int kTraceThreads = 1024;

template <typename E>
__global__ void __launch_bounds__(kTraceThreads)
k_apply_trace(const uint32_t *__restrict__ bits, const E *__restrict__ x, E *__restrict__ y, int n, size_t total) {
    after_previous_kernel();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    uint32_t *sb = reinterpret_cast<uint32_t *>(smem_raw);
    const uint32_t N = 1u << n, W = n >= 6 ? N >> 6 : 1u, per = uint32_t(2 * n - 1) * W;     // words per permutation
    const size_t j0 = size_t(blockIdx.x) * blockDim.x;                // a CTA has whole permutations, or part of one
    const uint32_t perms = blockDim.x > N ? blockDim.x >> n : 1u;
    const size_t perm0 = j0 >> n, left = (total >> n) - perm0;
    const uint32_t words = uint32_t(left < perms ? left : perms) * per;
    for (uint32_t i = threadIdx.x; i < words; i += blockDim.x) sb[i] = __ldg(bits + perm0 * per + i);
    __syncthreads();
    const size_t j = j0 + threadIdx.x;
    if (j >= total) return;
    const uint32_t *row = sb + uint32_t((j >> n) - perm0) * per + (uint32_t(2 * n - 2)) * W;
    uint32_t pos = uint32_t(j) & (N - 1u);
    for (int m = n; m > 1; --m, row -= W) {
        const uint32_t bit = (row[pos >> 6] >> ((pos >> 1) & 31u)) & 1u, mask = (1u << m) - 1u, low = pos & mask;
        pos = (pos & ~mask) | (low >> 1) | (((low ^ bit) & 1u) << (m - 1));
    }
    pos ^= (row[pos >> 6] >> ((pos >> 1) & 31u)) & 1u;
    row -= W;
    for (int m = 2; m <= n; ++m, row -= W) {
        const uint32_t half = (1u << (m - 1)) - 1u, mask = 2u * half + 1u;
        const uint32_t s = pos & half, sw = ((pos & ~mask) >> 1) + s;
        const uint32_t bit = (row[sw >> 5] >> (sw & 31u)) & 1u;
        pos = (pos & ~mask) | (2u * s) | (((pos >> (m - 1)) ^ bit) & 1u);
    }
    y[j] = x[(j & ~size_t(N - 1u)) + pos];
}

template <typename K>
int opt_in_smem(K kernel, size_t bytes) {
    if (bytes > 48 * 1024)
        BENES_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(bytes)));
    // room for two CTAs per SM
    BENES_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                        cudaSharedmemCarveoutMaxShared));
    return BENES_OK;
}

// Passes per side above the inner kernel's blocks.  A run of an outer pass is at least a 32-byte sector, so
// up to 10 levels go in one pass; more are split.
template <typename E>
int outer_passes(int n) {
    const int outer = n > kChunkLog2 ? n - kChunkLog2 : 0;
    return (outer + kMaxOuter - 1) / kMaxOuter;
}

template <typename E>
int apply_fused_typed(const uint32_t *bits, const E *in, E *out, E *scratch, int n, size_t batch,
                      cudaStream_t s, const ApplyHostPipe *pipe) {
    const size_t total = batch << n;
    if (n <= kTraceLog2 && total <= size_t(sm_count()) * 2048) {
        const unsigned threads = n < 7 ? 128u : n < 10 ? 1u << n : unsigned(kTraceThreads);
        const size_t words = size_t(2 * n - 1) * (n >= 6 ? size_t(1) << (n - 6) : 1);
        const size_t perms = (threads >> n) > 1 ? threads >> n : 1;
        launch_kernel(k_apply_trace<E>, unsigned((total + threads - 1) / threads), threads, words * perms * 4, s, bits, in, out, n, total);
        return launch_status();
    }
    static OncePerDevice configured;
    {
        const int rc0 = configured.run([&]() -> int {
            int rc;
            if ((rc = opt_in_smem(k_apply_inner<E, kChunkLog2>, apply_smem<E, kChunkLog2>(2 * kChunkLog2 - 1)))) return rc;
            if ((rc = opt_in_smem(k_apply_inner<E, kSmallLog2>, apply_smem<E, kSmallLog2>(2 * kSmallLog2 - 1)))) return rc;
            if ((rc = opt_in_smem(k_apply_outer<E, kOuterLog2<E>, false>, apply_smem<E, kOuterLog2<E>>(kMaxOuter)))) return rc;
            return opt_in_smem(k_apply_outer<E, kOuterLog2<E>, true>, apply_smem<E, kOuterLog2<E>>(kMaxOuter));
        });
        if (rc0) return rc0;
    }
    const int b = n < kChunkLog2 ? n : kChunkLog2;
    const int outer = n - b;                       // levels handled by the outer kernels, per side
    const int per_side = outer_passes<E>(n);       // passes per side
    const int passes = 2 * per_side + 1;
    // split `outer` levels evenly over the passes of a side
    int ks[8] = {0};
    for (int i = 0; i < per_side; ++i) ks[i] = outer / per_side + (i < outer % per_side ? 1 : 0);

    // ping-pong between `out` and the scratch buffer so that the last pass lands in `out`
    const E *src = in;
    int pass = 0;
    auto next_dst = [&]() { ++pass; return ((passes - pass) % 2 == 0) ? out : scratch; };
    const unsigned chunks = unsigned(total >> kOuterLog2<E>);
    // A pass is one launch, or `parts` launches over equal ranges of CTAs: the
    // first pass of a piped call waits for each part of `in`, its last pass
    // hands each finished part of `out` to the side stream.  CTA c of the first
    // (last) pass reads (writes) elements [c, c+1) * 2^13 (2^b in the inner pass).
    const int total_passes = passes;
    auto run_pass = [&](int index, unsigned ctas, size_t elems_per_cta, auto &&launch) -> int {
        const bool first = pipe && index == 0, last = pipe && index == total_passes - 1;
        const unsigned parts = (first || last) ? unsigned(pipe->parts) : 1u;
        const unsigned per = ctas / parts;
        for (unsigned p = 0; p < parts; ++p) {
            if (first) BENES_CUDA_TRY(cudaStreamWaitEvent(s, pipe->in_ready[p], 0));
            launch(per, p * per);
            int rc = launch_status();
            if (rc) return rc;
            if (last) {
                BENES_CUDA_TRY(cudaEventRecord(pipe->out_done[p], s));
                BENES_CUDA_TRY(cudaStreamWaitEvent(pipe->side, pipe->out_done[p], 0));
                const size_t off = size_t(p) * per * elems_per_cta * sizeof(E), bytes = size_t(per) * elems_per_cta * sizeof(E);
                BENES_CUDA_TRY(cudaMemcpyAsync(static_cast<char *>(pipe->out_host) + off,
                                               reinterpret_cast<const char *>(out) + off, bytes,
                                               cudaMemcpyDeviceToHost, pipe->side));
            }
        }
        return BENES_OK;
    };
    int l0 = 0, index = 0, rc;
    for (int i = 0; i < per_side; ++i) {
        E *dst = next_dst();
        const int k = ks[i], lvl = l0;
        if ((rc = run_pass(index++, chunks, size_t(1) << kOuterLog2<E>, [&](unsigned ctas, unsigned cta0) {
                 launch_kernel(k_apply_outer<E, kOuterLog2<E>, false>, ctas, kApplyThreads<kOuterLog2<E>>, apply_smem<E, kOuterLog2<E>>(k), s, bits, src, dst, n, lvl, k, cta0);
             })))
            return rc;
        src = dst;
        l0 += ks[i];
    }
    {
        E *dst = next_dst();
        // chunks of 2^13, or of 2^10 while those do not give every SM one
        const bool small = b <= kSmallLog2 && (total >> kChunkLog2) < size_t(sm_count());
        const int c = small ? kSmallLog2 : kChunkLog2;
        const unsigned blocks = unsigned((total + (size_t(1) << c) - 1) >> c);
        if ((rc = run_pass(index++, blocks, size_t(1) << c, [&](unsigned ctas, unsigned cta0) {
                 if (small)
                     launch_kernel(k_apply_inner<E, kSmallLog2>, ctas, kApplyThreads<kSmallLog2>, apply_smem<E, kSmallLog2>(2 * b - 1), s,
                         bits, src, dst, n, b, total, cta0);
                 else
                     launch_kernel(k_apply_inner<E, kChunkLog2>, ctas, kApplyThreads<kChunkLog2>, apply_smem<E, kChunkLog2>(2 * b - 1), s,
                         bits, src, dst, n, b, total, cta0);
             })))
            return rc;
        src = dst;
    }
    for (int i = per_side - 1; i >= 0; --i) {
        E *dst = next_dst();
        l0 -= ks[i];
        const int k = ks[i], lvl = l0;
        if ((rc = run_pass(index++, chunks, size_t(1) << kOuterLog2<E>, [&](unsigned ctas, unsigned cta0) {
                 launch_kernel(k_apply_outer<E, kOuterLog2<E>, true>, ctas, kApplyThreads<kOuterLog2<E>>, apply_smem<E, kOuterLog2<E>>(k), s, bits, src, dst, n, lvl, k, cta0);
             })))
            return rc;
        src = dst;
    }
    return BENES_OK;
}

}  // namespace

size_t apply_fused_chunks(int log2n, size_t batch) {
    return log2n > kChunkLog2 ? (batch << log2n) >> kChunkLog2 : 0;
}

int launch_apply_fused(const uint32_t *bits, const void *in, void *out, void *scratch, int elem_bytes,
                       int log2n, size_t batch, cudaStream_t s, const ApplyHostPipe *pipe) {
    if (pipe && (pipe->parts < 1 || pipe->parts > kApplyMaxParts ||
                 apply_fused_chunks(log2n, batch) % size_t(pipe->parts) != 0 || apply_fused_chunks(log2n, batch) == 0))
        return BENES_ERR_BADARG;
    if (elem_bytes == 4)
        return apply_fused_typed<uint32_t>(bits, static_cast<const uint32_t *>(in),
                                           static_cast<uint32_t *>(out), static_cast<uint32_t *>(scratch),
                                           log2n, batch, s, pipe);
    if (elem_bytes == 8)
        return apply_fused_typed<unsigned long long>(bits, static_cast<const unsigned long long *>(in),
                                                     static_cast<unsigned long long *>(out),
                                                     static_cast<unsigned long long *>(scratch), log2n,
                                                     batch, s, pipe);
    return BENES_ERR_BADARG;
}

}  // namespace benes
