// Work-efficient loop labelling for the HBM levels: ruler sampling.
//
// Pointer jumping over all outputs costs O(M log M) random accesses per level.
// Here every output switch is visited ONCE per level:
//
//   1. Switches are cut into groups of k = 2^kappa consecutive switches; a hash
//      of the group number picks one RULER switch per group.  Both outputs of
//      a ruler switch are ruler outputs; ruler output rho = 2*group + (j & 1).
//   2. k_walk: one thread per ruler output follows the successor
//      g(j) = base + Q[base + (P[j^1] ^ 1)].  The g-cycle through output j
//      and the g-cycle through j^1 are mirror images (g(g(j)^1) = j^1), so the
//      walker that leaves ruler switch T forwards and the walker that leaves
//      the next ruler switch T' backwards run over the same switches from the
//      two ends.  Each claims the switches it reaches with one atomic operation
//      on the switch's record and stops at the first switch the other one
//      owns: together they touch every switch of the segment once.  A walker
//      keeps the smallest output index on its own side of the switches it
//      claimed (on the far side it is the same with the last bit flipped) and its partner
//      (peer).  The claim stores (walker, side of arrival).
//   3. The segment of walker rho ends at ruler output peer^1: the walk records are the
//      contracted list as they are (see pair_least for the minima).
//   4. The contracted list is labelled with the parity of every cycle's minimum:
//      lists of up to 2^14 words per block in one CTA's shared memory, longer
//      ones by sampling again: the list is mirror symmetric like the loops, so
//      it is sampled the same way (one ruler pair per 4 to 16 pairs of words, walks
//      that meet in the middle).
//   5. k_colour: output 2t lies on its owner's cycle if the owner arrived on
//      the even side, else on the mirror cycle, which has the other colour:
//      colour = (cycle minimum of the owner & 1) ^ side.  A switch nobody
//      claimed lies on a loop without ruler; such loops are short
//      (probability (1-1/k)^length) and the thread walks the cycle itself.
//
// Every walk gives up after `cap` hops and raises the gate, one word for the whole route.  What the
// kernels after it then compute is discarded (they only have to stay in bounds and to end): behind the
// last of these levels the gate opens the pointer-jumping kernel of route_levels.cu, which does all of
// them again from the caller's permutation.  So the result never depends on the sampling.
#include "common.cuh"

BENES_GUARD_TU("route_sampled.cu")

namespace benes {


namespace {

constexpr int kThreads = 256;
constexpr int kWalkThreads = 128;             // a CTA's slots are free again when its longest walk ends
constexpr int kListThreads = 1024;

__device__ __forceinline__ bool gate_raised(const uint32_t *gate) {
    return *reinterpret_cast<const volatile uint32_t *>(gate) != 0u;
}

// Step 2.  W walks per thread, one after another, launched in index order so that the blocks being
// walked at any moment are neighbours in memory.
//
// Wide records: one 64-bit exchange of the claim record for my code returns the
// two P values, or the code of the walker that was here first.  Packed records: one
// 64-bit atomic AND with (my code << 2m | ones) returns the two P values and the
// previous owner and, if the switch was free (owner all ones), leaves my code
// there.  If the switch was taken, the other walker's code is gone, and since nobody
// but the two of us ever touches this switch, writing the old word back repairs it.
//
// What bounds a launch is the latency of a hop, a chain of two dependent accesses (0.7 us with the
// GPU full of them), times the longest walk of a warp: walks have all lengths, with one walk per
// thread 9 of 32 lanes are active on average.  With W = 2 a thread has both walks of a ruler
// switch, fetches the first hop of the two at once, and a lane whose walk ends goes on with its
// second one in the same round.
template <bool PACKED, int W>
__global__ void __launch_bounds__(kWalkThreads)
k_walk(unsigned long long *__restrict__ S8, const uint32_t *__restrict__ P, const uint32_t *__restrict__ Q,
       uint2 *__restrict__ rec, uint32_t rulers, int m, int kappa, uint32_t salt, uint32_t cap,
       uint32_t *__restrict__ gate) {
    after_previous_kernel();
    uint32_t rho = (blockIdx.x * kWalkThreads + threadIdx.x) * W;
    if (rho >= rulers) return;                                       // rulers is a multiple of W
    const uint32_t mmask = (1u << m) - 1u;
    const uint32_t kmask = (1u << kappa) - 1u;
    // the rulers of a thread lie in one block (a block has at least 2^7 ruler outputs)
    const uint32_t base = ((rho >> 1) << (kappa + 1)) & ~mmask;
    // packed owners are local to the block: its first ruler output is base >> kappa
    const uint32_t rho_base = base >> kappa;
    const int cshift = 2 * m;
    const unsigned long long low_ones = PACKED ? ((1ull << cshift) - 1ull) : 0ull;
    const uint32_t none8 = PACKED ? uint32_t(~0ull >> cshift) : 0u;

    // where each walk goes first: g(j) of its ruler output j needs P[j^1]
    uint32_t q[W];
#pragma unroll
    for (int i = 0; i < (W > 1 ? W / 2 : 1); ++i) {
        const uint32_t group = (rho >> 1) + uint32_t(i);
        const uint32_t t0 = (group << kappa) | ruler_slot(group, salt, kmask);
        uint32_t pe, po;
        if (PACKED) {
            // the ruler switch belongs to its even-side walker (nobody else claims it)
            const unsigned long long w = (W > 1 || !(rho & 1u))
                ? atomicAnd(S8 + t0, ((unsigned long long)((2u * group - rho_base) << 1) << cshift) | low_ones)
                : __ldcg(S8 + t0);
            pe = uint32_t(w) & mmask;
            po = uint32_t(w >> m) & mmask;
        } else {
            // (the ruler switch carries its even-side walker's code from the start)
            const uint2 p = __ldcs(reinterpret_cast<const uint2 *>(P) + t0);
            pe = BENES_GUARD(p.x, mmask);
            po = BENES_GUARD(p.y, mmask);
        }
        if (W > 1) {
            q[2 * i] = BENES_GUARD(__ldcg(Q + base + (po ^ 1u)), mmask);
            q[(2 * i + 1) % W] = BENES_GUARD(__ldcg(Q + base + (pe ^ 1u)), mmask);
        } else {
            q[0] = BENES_GUARD(__ldcg(Q + base + (((rho & 1u) ? pe : po) ^ 1u)), mmask);
        }
    }
    uint32_t walk = 0, hops = 0, rounds = 0;
    uint32_t j = base + q[0];
    uint32_t least = 2u * (((rho >> 1) << kappa) | ruler_slot(rho >> 1, salt, kmask)) + (rho & 1u);
    for (;;) {
        const uint32_t t = j >> 1, side = j & 1u, g = t >> kappa;
        uint32_t peer = rho ^ 1u;
        bool ends = true;
        if ((t & kmask) == ruler_slot(g, salt, kmask)) {             // reached the next ruler
            peer = (2u * g + side) ^ 1u;
        } else if (++hops > cap) {
            *gate = 1u;
        } else {
            uint32_t p, prev;
            unsigned long long w;
            bool met;
            if (PACKED) {
                w = atomicAnd(S8 + t, ((unsigned long long)(((rho - rho_base) << 1) | side) << cshift) | low_ones);
                p = uint32_t(w >> (side ? 0 : m)) & mmask;
                prev = rho_base + (uint32_t(w >> cshift) >> 1);
                met = uint32_t(w >> cshift) != none8;
            } else {
                w = atomicExch(S8 + t, kClaimed | (unsigned long long)((rho << 1) | side));
                p = uint32_t(side ? w : (w >> 32)) & mmask;          // (of a claimed record: some code, harmless)
                prev = uint32_t(w) >> 1;
                met = (w & kClaimed) != 0ull;
            }
            // next hop's gather, issued before the claim is looked at (harmless if we stop)
            const uint32_t qn = BENES_GUARD(__ldcg(Q + base + (p ^ 1u)), mmask);
            if (met) {                                               // the walker from the other end was here
                __stcg(S8 + t, w);                                   // put its code back
                peer = prev;
            } else {
                least = min(least, j);
                j = base + qn;
                ends = false;
            }
        }
        if (W == 1 || (++rounds & 63u) == 0u) {
            if (((W == 1 ? hops : rounds) & 63u) == 0u && gate_raised(gate)) {           // the route is redone anyway
                // (what an earlier route left in the records could name words beyond this one's lists)
                do rec[rho] = make_uint2(least, rho ^ 1u), ++rho; while (W > 1 && ++walk < uint32_t(W));
                break;
            }
        }
        if (ends) {
            rec[rho] = make_uint2(least, peer);
            if (W == 1 || ++walk == uint32_t(W)) break;
            ++rho;
            hops = 0;
            uint32_t qk = q[0];
#pragma unroll
            for (int i = 1; i < W; ++i) qk = walk == uint32_t(i) ? q[i] : qk;
            j = base + qk;
            least = 2u * (((rho >> 1) << kappa) | ruler_slot(rho >> 1, salt, kmask)) + (rho & 1u);
        }
    }
}

// ---- chained levels ---------------------------------------------------------------------
// Where a level lasts as long as its longest walk, what counts is what a hop waits for.  Here that is one access: the
// successor G[j] and the claim of its switch (a compare-and-swap on the owner's word) are under way together.  On
// records a hop waits for an atomic and then for a gather.  One permutation, on
// records and chained, with the same rulers: 2^20 walks of a level 30.5 -> 22.5 us, route 417 -> 394; 2^18 route 231 ->
// 203.  A switch that the two walkers of a segment claim at the same time may be counted by both.
// (Behind a raised gate, or an input that is no permutation, some successors are left over from other levels: they are
// masked into the block.)
__global__ void __launch_bounds__(kWalkThreads)
k_chain_walk(const uint32_t *__restrict__ G, uint32_t *__restrict__ owner, uint2 *__restrict__ rec, uint32_t rulers, int m,
             int kappa, uint32_t salt, uint32_t cap, uint32_t *__restrict__ gate) {
    after_previous_kernel();
    const uint32_t rho = blockIdx.x * kWalkThreads + threadIdx.x;
    if (rho >= rulers) return;
    const uint32_t mmask = (1u << m) - 1u, kmask = (1u << kappa) - 1u;
    const uint32_t t0 = ((rho >> 1) << kappa) | ruler_slot(rho >> 1, salt, kmask);
    const uint32_t base = (2u * t0) & ~mmask;
    if (!(rho & 1u)) owner[t0] = ~(rho << 1);                       // the ruler switch belongs to its even walker
    uint32_t least = 2u * t0 + (rho & 1u), peer = rho ^ 1u, hops = 0;
    uint32_t j = base + (__ldcg(G + least) & mmask);
    for (;;) {
        const uint32_t t = j >> 1, side = j & 1u, g = t >> kappa;
        if ((t & kmask) == ruler_slot(g, salt, kmask)) {
            peer = (2u * g + side) ^ 1u;
            break;
        }
        if (++hops > cap) *gate = 1u;
        if (hops > cap || ((hops & 63u) == 0u && gate_raised(gate))) break;
        const uint32_t next = __ldcg(G + j);
        const uint32_t met = atomicCAS(owner + t, kUnowned, ~((rho << 1) | side));
        least = min(least, j);
        if (met != kUnowned) {
            peer = ~met >> 1;
            break;
        }
        j = base + (next & mmask);
    }
    rec[rho] = make_uint2(least, peer);
}

// The successors of the first level: g(j) = Q[P[j ^ 1] ^ 1].  Two switches per thread.
__global__ void __launch_bounds__(kThreads)
k_chain_start(const uint4 *__restrict__ P4, const uint32_t *__restrict__ Q, uint4 *__restrict__ G4, uint2 *__restrict__ owner2,
              uint32_t quads, int m) {
    after_previous_kernel();
    const uint32_t i = blockIdx.x * kThreads + threadIdx.x;
    if (i >= quads) return;
    const uint32_t mmask = (1u << m) - 1u;
    const uint32_t *Qb = Q + ((4u * i) & ~mmask);
    const uint4 p = __ldcs(P4 + i);
    G4[i] = make_uint4(Qb[BENES_GUARD(p.y, mmask) ^ 1u], Qb[BENES_GUARD(p.x, mmask) ^ 1u], Qb[BENES_GUARD(p.w, mmask) ^ 1u],
                       Qb[BENES_GUARD(p.z, mmask) ^ 1u]);
    owner2[i] = make_uint2(kUnowned, kUnowned);
}

// A switch on a loop without ruler: the minimum of the g-cycle of output 2t, from both ends (see loop_colour).
__device__ __forceinline__ uint32_t chain_loop_colour(const uint32_t *G, uint32_t t, uint32_t base, uint32_t mmask, uint32_t cap,
                                                      uint32_t *gate) {
    const uint32_t j0 = 2u * t;
    uint32_t f = j0, bk = j0, mn = j0, hops = 0;
    for (;;) {
        const uint32_t nf = base + (__ldg(G + f) & mmask), nb = (base + (__ldg(G + (bk ^ 1u)) & mmask)) ^ 1u;
        f = nf;
        if (f == bk) break;
        mn = min(mn, f);
        bk = nb;
        if (bk == f) break;
        mn = min(mn, bk);
        if (++hops > cap) {
            *gate = 1u;
            break;
        }
        if ((hops & 63u) == 0u && gate_raised(gate)) break;
    }
    return mn & 1u;
}

// Output side of a chained level; hands the owners back as kUnowned.  Two switches per thread.
__global__ void __launch_bounds__(kThreads)
k_chain_colour(const uint32_t *__restrict__ G, uint2 *__restrict__ owner2, const uint32_t *__restrict__ cb, uint32_t pairs,
               uint32_t rulers, int m, BitsLayout L, int out_stage, uint32_t cap, uint32_t *__restrict__ gate) {
    after_previous_kernel();
    const uint32_t i = blockIdx.x * kThreads + threadIdx.x;         // pairs is a multiple of 32
    if (i >= pairs) return;
    const uint32_t mmask = (1u << m) - 1u, t = 2u * i, base = (2u * t) & ~mmask;
    const uint2 o = owner2[i];
    owner2[i] = make_uint2(kUnowned, kUnowned);
    // (the gathers of the two switches are under way together)
    const uint32_t r0 = o.x != kUnowned ? BENES_GUARD_BELOW(~o.x >> 1, rulers, 0u) : 0u;
    const uint32_t r1 = o.y != kUnowned ? BENES_GUARD_BELOW(~o.y >> 1, rulers, 0u) : 0u;
    const uint32_t w0 = __ldg(cb + (r0 >> 5)), w1 = __ldg(cb + (r1 >> 5));
    uint32_t c0 = ((w0 >> (r0 & 31u)) ^ ~o.x) & 1u, c1 = ((w1 >> (r1 & 31u)) ^ ~o.y) & 1u;
    if (o.x == kUnowned) c0 = chain_loop_colour(G, t, base, mmask, cap, gate);
    if (o.y == kUnowned) c1 = chain_loop_colour(G, t + 1u, base, mmask, cap, gate);
    store_stage_bits64(L.bits + L.word32(out_stage, (t - 2u * (threadIdx.x & 31u)) >> 5), c0, c1);
}

// Step 3, the contracted list.  It needs no pass of its own.  The segment of walker rho ends at ruler output
// peer ^ 1, so that is the word after rho.  Words 2q and 2q + 1 (the two outputs of a ruler switch) form a pair; the
// cycle through one and the cycle through the other are mirror images, so what walker 2q + 1 has seen, with
// the last bit flipped, lies on the cycle of word 2q, and every segment of a cycle has both of its walkers in
// pairs of the cycle: the minimum over a cycle is the minimum over its pairs of
//     min(least[2q], least[2q + 1] ^ 1)          (on the side of word 2q; on the other side, that ^ 1).
__device__ __forceinline__ uint32_t pair_least(uint32_t least0, uint32_t least1) { return min(least0, least1 ^ 1u); }

// Step 4, sampling a list.  The contracted list inherits the mirror symmetry
// of the loops (next[rho] = sigma implies next[sigma ^ 1] = rho ^ 1), and so does
// every list sampled from it this way: a list is sampled the way the switches are.  One pair per 2^spacing
// pairs is a ruler pair, both of its words start a walker; the walker from the
// even word runs along its cycle, the walker from the odd word of the NEXT
// ruler pair runs along the mirror cycle, i.e. over the same pairs from the
// other end; each claims pairs (owner[q] = walker, side of arrival) and stops
// where the other one has been.  A walker's record is (minimum, peer) again.
__global__ void __launch_bounds__(kWalkThreads)
k_list_walk_pairs(const uint4 *__restrict__ pair, uint32_t *__restrict__ owner, uint2 *__restrict__ rec,
                  uint32_t rulers, uint32_t pairs, int spacing, uint32_t salt, uint32_t cap, uint32_t *__restrict__ gate) {
    after_previous_kernel();
    const uint32_t sigma = blockIdx.x * kWalkThreads + threadIdx.x;
    if (sigma >= rulers) return;
    const uint32_t kmask = (1u << spacing) - 1u;
    const uint32_t group = sigma >> 1, side0 = sigma & 1u;
    const uint32_t q0 = (group << spacing) | ruler_slot(group, salt, kmask);
    uint4 w = __ldcg(pair + q0);
    if (!side0) owner[q0] = ~(sigma << 1);                          // the ruler pair belongs to its even walker
    uint32_t least = pair_least(w.x, w.z) ^ side0, next = (side0 ? w.w : w.y) ^ 1u, peer = sigma ^ 1u, hops = 0;
    for (;;) {
        // (a batch need not be a power of two: an index a raised gate left undefined is clamped, not masked)
        const uint32_t q = BENES_GUARD_BELOW(next >> 1, pairs, 0u), side = next & 1u, g = q >> spacing;
        if ((q & kmask) == ruler_slot(g, salt, kmask)) {           // reached the next ruler pair
            peer = (2u * g + side) ^ 1u;
            break;
        }
        if (++hops > cap) {
            *gate = 1u;
            break;
        }
        if ((hops & 63u) == 0u && gate_raised(gate)) break;
        w = __ldcg(pair + q);
        const uint32_t prev = atomicCAS(owner + q, kUnowned, ~((sigma << 1) | side));
        if (prev != kUnowned) {                                    // met the walker from the other end
            peer = ~prev >> 1;
            break;
        }
        least = min(least, pair_least(w.x, w.z) ^ side);
        next = (side ? w.w : w.y) ^ 1u;
    }
    rec[sigma] = make_uint2(least, peer);
}

// Back from a sampled list: a thread takes the pair 2q, 2q+1 (and hands the
// owner slot back as kUnowned).  Word 2q lies on its owner's cycle if the
// owner arrived on side 0, else on the mirror cycle, whose minimum has the other
// parity, and so does word 2q+1's: one bit of the sampled list (`cb2`) gives the two bits of
// the pair (`cb`).  A pair nobody claimed lies on a cycle without ruler pair: the thread walks the
// cycle of word 2q.
__global__ void __launch_bounds__(kThreads)
k_list_resolve_pairs(const uint4 *__restrict__ pair, uint32_t *__restrict__ owner,
                     const uint32_t *__restrict__ cb2, uint32_t pairs,
                     uint32_t cap, uint32_t *__restrict__ gate, uint32_t *__restrict__ cb) {
    after_previous_kernel();
    const uint32_t q = blockIdx.x * kThreads + threadIdx.x;       // pairs is a multiple of 32
    if (q >= pairs) return;
    const uint32_t code = owner[q];
    uint32_t bit0;
    if (code != kUnowned) {
        const uint32_t sigma = ~code >> 1;
        bit0 = ((__ldg(cb2 + (sigma >> 5)) >> (sigma & 31u)) ^ ~code) & 1u;
        owner[q] = kUnowned;
    } else {
        uint4 w = __ldg(pair + q);
        uint32_t least = pair_least(w.x, w.z), next = w.y ^ 1u, hops = 0;
        while (next != 2u * q) {
            if (++hops > cap) {
                *gate = 1u;
                break;
            }
            if ((hops & 63u) == 0u && gate_raised(gate)) break;
            w = __ldg(pair + BENES_GUARD_BELOW(next >> 1, pairs, 0u));
            least = min(least, pair_least(w.x, w.z) ^ (next & 1u));
            next = ((next & 1u) ? w.w : w.y) ^ 1u;
        }
        bit0 = least & 1u;
    }
    // a warp covers 64 words: two words of cb
    store_stage_bits64(cb + ((q - (threadIdx.x & 31u)) >> 4), bit0, bit0 ^ 1u);
}

// Step 4, the end of the recursion: one CTA labels one block's list of B = 2^log2b words in shared memory, by
// the same sampling once more: one ruler pair per 8 pairs, walks that meet in the middle over 16-bit
// successors (claims go into the successor words, which nobody reads again), pointer jumping over the B/8 words
// that are left, and a queue for the pairs of cycles without ruler pair.  Pointer jumping over the whole list
// took log2b - 1 passes of random shared-memory reads (2^14 words: 25 us, now 16).
// Only the parities of the minima are needed from here on (a cycle and its mirror image differ in it): they
// go to `cb`, one bit per word.  Indices a raised gate may have left undefined are masked into the block.
constexpr int kLGroup = 3;                            // pairs per ruler pair (log2)
constexpr uint32_t kLRho = 0x7FFCu, kLRuler = 0x8000u;

constexpr size_t list_label_smem(int log2b) { return (size_t(6) << log2b) + 16; }

__global__ void __launch_bounds__(kListThreads)
k_list_label(const uint4 *__restrict__ src, uint16_t *__restrict__ cb, int log2b, uint32_t salt) {
    after_previous_kernel();
    extern __shared__ __align__(16) unsigned char lsm[];
    const uint32_t B = 1u << log2b, bmask = B - 1u, R = B >> kLGroup, groups = B >> (kLGroup + 1);
    const size_t base = size_t(blockIdx.x) << log2b;
    const uint32_t T = blockDim.x, tid = threadIdx.x;
    uint32_t *M = reinterpret_cast<uint32_t *>(lsm);                            // minimum of every pair
    unsigned char *N = lsm + 2 * B;                                             // successors / claims, 16 bit
    uint32_t *own = reinterpret_cast<uint32_t *>(N + 2 * B), *peer = own + R;   // walk records
    unsigned long long *L = reinterpret_cast<unsigned long long *>(peer + R);   // list of the ruler words (+ a 0)
    uint16_t *queue = reinterpret_cast<uint16_t *>(own);                        // after `own` and `peer`
    __shared__ uint32_t queued;
    // eight pairs per thread (fewer than 512 words: a warp takes turns), all their loads under way together
    for (uint32_t e0 = tid; e0 < B / 2; e0 += 8 * T) {
        uint4 w[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uint32_t q = e0 + uint32_t(i) * T;
            w[i] = q < B / 2 ? __ldcs(src + base / 2 + q) : make_uint4(0, 0, 0, 0);
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uint32_t q = e0 + uint32_t(i) * T;
            if (q >= B / 2) continue;
            M[q] = pair_least(w[i].x, w[i].z);
            *reinterpret_cast<uint32_t *>(N + 4 * q) = 2u * ((w[i].y & bmask) ^ 1u) | (2u * ((w[i].w & bmask) ^ 1u)) << 16;
        }
    }
    if (tid == 0) queued = 0u;
    __syncthreads();
    const uint32_t g = tid;                              // a thread has one group of 8 pairs
    uint32_t start = 0, q0 = 0;
    if (g < groups) {
        q0 = (g << kLGroup) | ruler_slot(g, salt, (1u << kLGroup) - 1u);
        uint32_t *word = reinterpret_cast<uint32_t *>(N + 4 * q0);
        start = *word;
        *word = (kLRuler | (g << 3) | 1u) * 0x10001u;
    }
    __syncthreads();
    if (g < groups) {
        uint32_t rho = 2u * g, j = start & 0xFFFFu, code = ((rho << 2) | 1u) * 0x10001u;
        uint32_t least = M[q0];
        for (uint32_t k = 0;;) {
            // (no branches: a lane that has met somebody reads the same code again)
            bool met = false;
            uint32_t v = 0;
#pragma unroll
            for (int hop = 0; hop < 4; ++hop) {
                v = *reinterpret_cast<volatile uint16_t *>(N + j);
                met = (v & 1u) != 0u;
                const uint32_t mm = M[j >> 2] ^ ((j >> 1) & 1u);
                if (!met) *reinterpret_cast<volatile uint32_t *>(N + (j & ~3u)) = code + (j & 2u) * 0x10001u;
                least = met ? least : min(least, mm);
                j = met ? j : v;
            }
            if (met) {
                // a ruler pair (its code names its even word), or one the other walker owns
                own[rho] = least;
                peer[rho] = ((v & kLRho) >> 2) ^ ((v & kLRuler) ? ((~j & 2u) >> 1) : 0u);
                if (++k == 2u) break;
                ++rho;
                j = start >> 16;
                code = ((rho << 2) | 1u) * 0x10001u;
                least = M[q0] ^ 1u;
            }
        }
    }
    __syncthreads();
    for (uint32_t rho = tid; rho < R; rho += T) {
        L[rho] = make_word((peer[rho] & (R - 1u)) ^ 1u, min(own[rho], own[rho ^ 1u] ^ 1u));
    }
    if (tid == 0) L[R] = 0ull;
    __syncthreads();
    // pairs of cycles without ruler pair queue up; pointer jumping over the ruler words meanwhile: a cycle of
    // theirs has at most R/2 words (it and its mirror image share the block)
    uint4 n0 = make_uint4(1, 1, 1, 1), n1 = n0;
    if (g < groups) {
        n0 = *reinterpret_cast<const uint4 *>(N + 32 * g);
        n1 = *reinterpret_cast<const uint4 *>(N + 32 * g + 16);
        uint32_t free_ = (~n0.x & 1u) | ((~n0.y & 1u) << 1) | ((~n0.z & 1u) << 2) | ((~n0.w & 1u) << 3) |
                         ((~n1.x & 1u) << 4) | ((~n1.y & 1u) << 5) | ((~n1.z & 1u) << 6) | ((~n1.w & 1u) << 7);
        if (free_) {
            uint32_t pos = atomicAdd(&queued, uint32_t(__popc(free_)));
            for (; free_; free_ &= free_ - 1u) queue[pos++] = uint16_t(8u * g + uint32_t(__ffs(int(free_))) - 1u);
        }
    }
    volatile unsigned long long *Lv = L;
    for (int pass = 0; pass < log2b - kLGroup - 1; ++pass) {
        for (uint32_t rho = tid; rho < R; rho += T) {
            const unsigned long long w = Lv[rho], t = Lv[uint32_t(w)];
            Lv[rho] = make_word(uint32_t(t), min(uint32_t(w >> 32), uint32_t(t >> 32)));
        }
        __syncthreads();
        if (pass == 0) {
            // (the queue is complete, and the walks below only read unclaimed words until the next barrier)
            for (uint32_t i = tid; i < queued; i += T) {
                const uint32_t q = queue[i];
                uint32_t f = 4u * q, mn = M[q];
                for (uint32_t hops = 0; hops < B; ++hops) {
                    f = *reinterpret_cast<volatile uint16_t *>(N + f) & (2u * bmask);
                    if (f == 4u * q) break;
                    mn = min(mn, M[f >> 2] ^ ((f >> 1) & 1u));
                }
                queue[i] = uint16_t(q | (mn << 15));
            }
        } else if (pass == 1) {
            for (uint32_t i = tid; i < queued; i += T) {
                const uint32_t x = queue[i];
                *reinterpret_cast<uint32_t *>(N + 4 * (x & 0x7FFFu)) = (R << 2) | 1u | ((x >> 14) & 2u);
            }
        }
    }
    __syncthreads();
    if (g < groups) {
        n0 = *reinterpret_cast<const uint4 *>(N + 32 * g);
        n1 = *reinterpret_cast<const uint4 *>(N + 32 * g + 16);
        const uint32_t code[8] = {n0.x, n0.y, n0.z, n0.w, n1.x, n1.y, n1.z, n1.w};
        uint32_t bits = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const uint32_t b = (uint32_t(L[(code[k] & kLRho) >> 2] >> 32) ^ (code[k] >> 1)) & 1u;
            bits |= (b | ((b ^ 1u) << 1)) << (2 * k);
        }
        cb[(base >> 4) + g] = uint16_t(bits);
    }
}

int launch_list_label(const uint2 *rec, uint32_t *cb, uint32_t count, int beta, uint32_t salt, cudaStream_t s) {
    static OncePerDevice configured;
    {
        const int rc = configured.run([]() -> int {
            BENES_CUDA_TRY(cudaFuncSetAttribute(k_list_label, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                int(list_label_smem(kListSmemLog2))));
            return BENES_OK;
        });
        if (rc) return rc;
    }
    const unsigned threads = beta > 9 ? 1u << (beta - 4) : 32u;
    launch_kernel(k_list_label, count >> beta, threads, list_label_smem(beta), s, reinterpret_cast<const uint4 *>(rec),
                  reinterpret_cast<uint16_t *>(cb), beta, salt);
    return launch_status();
}

// Step 5 for a switch on a loop without ruler: the minimum of the g-cycle C of
// output 2t, walked from both ends.  The cycle of output 2t+1 is the mirror
// image of C (g(g(j)^1) = j^1), so g(b^1)^1 is the predecessor of b on C: one
// chain follows C forwards, the other backwards, their gathers overlap, and
// they stop where they meet.  The caller has fetched their first steps, qf = g(2t) and qb = g(2t ^ 1).
template <bool PACKED>
__device__ __forceinline__ uint32_t loop_colour(const void *S, const uint32_t *P, const uint32_t *Q, uint32_t t, uint32_t base,
                                                uint32_t qf, uint32_t qb, int m, uint32_t mmask,
                                                uint32_t cap, uint32_t *gate) {
    const uint32_t j0 = 2u * t;
    uint32_t f = j0, bk = j0, mn = j0, hops = 0;
    for (;;) {
        f = base + qf;
        if (f == bk) break;                                             // forwards reached the part walked backwards
        mn = min(mn, f);
        bk = (base + qb) ^ 1u;
        if (bk == f) break;                                             // both ends on the same output
        mn = min(mn, bk);
        if (++hops > cap) {
            *gate = 1u;
            break;
        }
        if ((hops & 63u) == 0u && gate_raised(gate)) break;
        const uint32_t pf = rec_p<PACKED>(S, P, f ^ 1u, m), pb = rec_p<PACKED>(S, P, bk, m);
        qf = BENES_GUARD(__ldg(Q + base + (pf ^ 1u)), mmask);
        qb = BENES_GUARD(__ldg(Q + base + (pb ^ 1u)), mmask);
    }
    return mn & 1u;
}

// Step 5 + output side of the level's switches + the next level's records
// (owner reset).  A thread owns the neighbouring switches 2i and 2i+1: their
// colour-0 outputs are neighbours in the upper half-block of the next level and
// their colour-1 outputs in the lower one, i.e. the thread writes one whole
// record of each.  (With the gate raised what it writes is never used.)  The last level writes none: the in-CTA levels
// start from the inverses (256 x 2^16: 921 -> 907 us, 2^24: 3.40 -> 3.38 ms).
enum NextRecords { kNextWide, kNextPacked, kNextNone };
template <bool PACKED, NextRecords NEXT>
__global__ void __launch_bounds__(kThreads)
k_colour(const void *__restrict__ S, const uint32_t *__restrict__ P, const uint32_t *__restrict__ Q,
         const uint32_t *__restrict__ cb, void *__restrict__ Sn, uint32_t *__restrict__ Pn, uint32_t salt_next, uint32_t pairs,
         uint32_t rulers, int m, int kappa, BitsLayout L, int out_stage, uint32_t cap,
         uint32_t *__restrict__ gate, uint32_t rounds) {
    after_previous_kernel();
    // a CTA takes `rounds` consecutive groups of blockDim.x pairs: the ruler bits
    // it gathers belong to one block of the level for a long time (L1 hits)
    const uint32_t stride = blockDim.x;
    const uint32_t last = min(pairs, (blockIdx.x + 1u) * rounds * stride);
    const uint32_t mmask = (1u << m) - 1u;
    const uint32_t H = (mmask + 1) >> 1;
    const uint32_t none = PACKED ? uint32_t(~0ull >> (2 * m)) : 0u;
    // packed fields with 32-bit operations (m < 32): the owner starts at bit 2m of
    // the word, the next level's owner (all ones) at bit 2(m-1)
    const int s_own = 2 * m, s_next = 2 * (m - 1);
    const uint32_t ones_lo = s_next < 32 ? ~0u << s_next : 0u;
    const uint32_t ones_hi = s_next < 32 ? ~0u : ~0u << (s_next - 32);
    // the records of the next round are on their way while this one is coloured
    // (pairs is a multiple of 32: a warp stays together)
    uint32_t i = blockIdx.x * rounds * stride + threadIdx.x;
    ulonglong2 w = make_ulonglong2(0, 0);                       // packed records, or claim records
    uint4 p4 = make_uint4(0, 0, 0, 0);                          // wide: the P values beside them
    if (i < last) {
        w = __ldcs(static_cast<const ulonglong2 *>(S) + i);
        if (!PACKED) p4 = __ldcs(reinterpret_cast<const uint4 *>(P) + i);
    }
    while (i < last) {
        const uint32_t inext = i + stride;
        ulonglong2 wn = make_ulonglong2(0, 0);
        uint4 p4n = make_uint4(0, 0, 0, 0);
        if (inext < last) {
            wn = __ldcs(static_cast<const ulonglong2 *>(S) + inext);
            if (!PACKED) p4n = __ldcs(reinterpret_cast<const uint4 *>(P) + inext);
        }
        const uint32_t t = 2u * i;                              // first switch of the pair
        const uint32_t base = (2u * t) & ~mmask;
        uint32_t px0, py0, px1, py1, code0, code1;
        bool own0, own1;
        if (PACKED) {
            const uint32_t rb = (base >> kappa) << 1;
            const uint32_t lo0 = uint32_t(w.x), hi0 = uint32_t(w.x >> 32);
            const uint32_t lo1 = uint32_t(w.y), hi1 = uint32_t(w.y >> 32);
            px0 = lo0 & mmask; py0 = __funnelshift_r(lo0, hi0, m) & mmask;
            px1 = lo1 & mmask; py1 = __funnelshift_r(lo1, hi1, m) & mmask;
            const uint32_t l0 = s_own >= 32 ? hi0 >> (s_own - 32) : __funnelshift_r(lo0, hi0, s_own);
            const uint32_t l1 = s_own >= 32 ? hi1 >> (s_own - 32) : __funnelshift_r(lo1, hi1, s_own);
            own0 = l0 != none; own1 = l1 != none;
            code0 = rb + l0; code1 = rb + l1;                    // owner local to the block -> global
        } else {
            px0 = BENES_GUARD(p4.x, mmask); py0 = BENES_GUARD(p4.y, mmask); code0 = uint32_t(w.x); own0 = (w.x & kClaimed) != 0ull;
            px1 = BENES_GUARD(p4.z, mmask); py1 = BENES_GUARD(p4.w, mmask); code1 = uint32_t(w.y); own1 = (w.y & kClaimed) != 0ull;
        }
        // all but the switches of loops without ruler are owned; the gathers of the two switches, and the first steps along
        // their loops, are under way together (2^24 3.37 -> 3.34 ms, transposed 2.12 -> 2.05)
        const uint32_t r0 = own0 ? BENES_GUARD_BELOW(code0 >> 1, rulers, 0u) : 0u, r1 = own1 ? BENES_GUARD_BELOW(code1 >> 1, rulers, 0u) : 0u;
        const uint32_t w0 = __ldg(cb + (r0 >> 5)), w1 = __ldg(cb + (r1 >> 5));
        uint32_t c0 = ((w0 >> (r0 & 31u)) ^ code0) & 1u, c1 = ((w1 >> (r1 & 31u)) ^ code1) & 1u;
        if (!(own0 && own1)) {
            const uint32_t *Qb = Q + base;
            uint32_t f0 = 0, b0 = 0, f1 = 0, b1 = 0;
            if (!own0) { f0 = BENES_GUARD(__ldg(Qb + (py0 ^ 1u)), mmask); b0 = BENES_GUARD(__ldg(Qb + (px0 ^ 1u)), mmask); }
            if (!own1) { f1 = BENES_GUARD(__ldg(Qb + (py1 ^ 1u)), mmask); b1 = BENES_GUARD(__ldg(Qb + (px1 ^ 1u)), mmask); }
            if (!own0) c0 = loop_colour<PACKED>(S, P, Q, t, base, f0, b0, m, mmask, cap, gate);
            if (!own1) c1 = loop_colour<PACKED>(S, P, Q, t + 1u, base, f1, b1, m, mmask, cap, gate);
        }
        // a warp covers 64 switches: two words of the output-side stage
        store_stage_bits64(L.bits + L.word32(out_stage, (t - 2u * (threadIdx.x & 31u)) >> 5), c0, c1);
        const uint32_t r = (base >> 1) + (((t - (base >> 1)) >> 1));   // record of the upper half
        const uint32_t u0 = (c0 ? py0 : px0) >> 1, u1 = (c1 ? py1 : px1) >> 1;     // upper half-block
        const uint32_t d0 = (c0 ? px0 : py0) >> 1, d1 = (c1 ? px1 : py1) >> 1;     // lower half-block
        if (NEXT == kNextPacked) {
            uint2 *Sn8 = static_cast<uint2 *>(Sn);
            Sn8[r] = make_uint2(u0 | (u1 << (m - 1)) | ones_lo, (u1 >> (33 - m)) | ones_hi);
            Sn8[r + (H >> 1)] = make_uint2(d0 | (d1 << (m - 1)) | ones_lo, (d1 >> (33 - m)) | ones_hi);
        } else if (NEXT == kNextWide) {
            rec_write<false>(Sn, Pn, r, m - 1, u0, u1, kappa, salt_next);
            rec_write<false>(Sn, Pn, r + (H >> 1), m - 1, d0, d1, kappa, salt_next);
        }
        w = wn; p4 = p4n;
        i = inext;
    }
}

inline size_t align256(size_t v) { return (v + 255) & ~size_t(255); }
constexpr int kMaxLists = 5;

// Spacing at which a block's list of 2^beta words is sampled again: 2^4 while it is far from what one CTA labels, just
// enough at the end (short walks are quick, and the CTA's labelling does not mind a full list).  0: fits.
inline int list_spacing(int beta) {
    const int over = beta - kListSmemLog2;
    return over <= 0 ? 0 : over < 2 ? 2 : over > 4 ? 4 : over;
}

}  // namespace

// Scratch: walk records (each a list), and the owners and parity bits of their words.
// A list that is sampled again shrinks to a quarter at least.
size_t sampled_scratch_bytes(size_t total, int kappa) {
    size_t R = total >> kappa, bytes = 0;
    for (int i = 0; i < kMaxLists; ++i) {
        size_t c = R >> (2 * i);
        if (c < 32) c = 32;
        bytes += align256(c * 2) + align256(c * 8) + align256(c / 8);
    }
    return bytes;
}

void sampled_scratch_carve(char *base, size_t total, int kappa, SampledScratch *out) {
    size_t R = total >> kappa, off = 0;
    for (int i = 0; i < kMaxLists; ++i) {                      // the owners of all lists lie together
        size_t c = R >> (2 * i);
        if (c < 32) c = 32;
        out->owner[i] = reinterpret_cast<uint32_t *>(base + off);
        off += align256(c * 2);
    }
    for (int i = 0; i < kMaxLists; ++i) {
        size_t c = R >> (2 * i);
        if (c < 32) c = 32;
        out->rec[i] = reinterpret_cast<uint2 *>(base + off);
        off += align256(c * 8);
        out->bits[i] = reinterpret_cast<uint32_t *>(base + off);
        off += align256(c / 8);
    }
}

// From the start of the scratch to the end of the owners of the lists that the first level (which has the longest)
// samples again.
size_t sampled_owner_bytes(const SampledScratch &sc, size_t total, int log2m, int kappa) {
    size_t c = total >> kappa, bytes = 0;
    int beta = log2m - kappa;
    for (int i = 0, sp; (sp = list_spacing(beta)) != 0; ++i) {
        bytes = size_t(reinterpret_cast<char *>(sc.owner[i]) - reinterpret_cast<char *>(sc.owner[0])) + c * 2;
        c >>= sp;
        beta -= sp;
    }
    return bytes;
}

// The parities of the minima of the walk records in sc.rec[0] (R words, 2^beta per block), to sc.bits[0].
static int label_lists(const SampledScratch &sc, uint32_t R, int beta, uint32_t salt, uint32_t cap, uint32_t *gate, cudaStream_t s) {
    // label the contracted list: sample it until a block's list fits one CTA
    int depth = 0;
    if (beta < 7) return BENES_ERR_BADARG;                     // (a CTA labels 2^7 words at least)
    uint32_t counts[kMaxLists + 1] = {R};
    for (int sp; (sp = list_spacing(beta)) != 0; ++depth) {
        // walks from both ends
        if (depth + 1 >= kMaxLists) return BENES_ERR_BADARG;
        const uint32_t count = counts[depth], next = count >> sp;
        ProfileScope ps(kListWalk, s);
        launch_kernel(k_list_walk_pairs, (next + kWalkThreads - 1) / kWalkThreads, kWalkThreads, 0, s,
            reinterpret_cast<const uint4 *>(sc.rec[depth]), sc.owner[depth], sc.rec[depth + 1], next, count >> 1, sp,
            salt * 7u + uint32_t(depth) + 1u, cap, gate);
        int rc = launch_status();
        if (rc) return rc;
        counts[depth + 1] = next;
        beta -= sp;
    }
    {
        ProfileScope ps(kListLabel, s);
        int rc = launch_list_label(sc.rec[depth], sc.bits[depth], counts[depth], beta, salt + 77u, s);
        if (rc) return rc;
    }
    for (int d = depth - 1; d >= 0; --d) {
        ProfileScope ps(kListResolve, s);
        const uint32_t c = counts[d];
        launch_kernel(k_list_resolve_pairs, (c / 2 + kThreads - 1) / kThreads, kThreads, 0, s,
            reinterpret_cast<const uint4 *>(sc.rec[d]), sc.owner[d], sc.bits[d + 1], c / 2, cap, gate, sc.bits[d]);
        int rc = launch_status();
        if (rc) return rc;
    }
    return BENES_OK;
}

int sampled_label(LevelRecords S, const uint32_t *Q, LevelRecords Sn, const SampledScratch &sc, size_t total,
                  int log2m, int kappa, uint32_t salt, uint32_t cap, int walk_pairs, BitsLayout L, int out_stage,
                  uint32_t *gate, cudaStream_t s) {
    if (!S.packed && !Sn.S) return BENES_ERR_BADARG;           // (no k_colour for a last level on wide records)
    const uint32_t R = uint32_t(total >> kappa);
    {
        ProfileScope ps(kWalk, s);
        // Two walks per thread pay once half of the threads still fills the GPU (2^26, levels 0-3:
        // 2.05 / 1.70 / 1.20 / 0.70 -> 1.98 / 1.62 / 1.08 / 0.67 ms, cache-resident levels 0.62 -> 0.53);
        // below that the launch lasts as long as its longest thread and one walk per thread is
        // faster.  More are slower: the rulers that are being walked at any moment then
        // spread over more blocks than the L2 holds (four: 0.95 ms per cache-resident level, eight: 1.6).
        const bool two = walk_pairs == 2 || (walk_pairs == 1 && size_t(R >> 1) >= size_t(sm_count()) * 2048);
#define BENES_WALK(PACKED, W)                                                                            \
    launch_kernel(k_walk<PACKED, W>, (R / W + kWalkThreads - 1) / kWalkThreads, kWalkThreads, 0, s, \
        static_cast<unsigned long long *>(S.S), S.P, Q, sc.rec[0], R, log2m, kappa, salt, cap, gate)
        if (S.packed) { if (two) BENES_WALK(true, 2); else BENES_WALK(true, 1); }
        else { if (two) BENES_WALK(false, 2); else BENES_WALK(false, 1); }
#undef BENES_WALK
        int rc = launch_status();
        if (rc) return rc;
    }
    const uint32_t *cb = sc.bits[0];
    if (const int rc = label_lists(sc, R, log2m - kappa, salt, cap, gate, s)) return rc;
    {
        ProfileScope ps(kColour, s);
        const uint32_t switches = uint32_t(total / 4);           // pairs of switches, one per thread
        const uint32_t rounds = stream_rounds(switches, kThreads);
        const unsigned grid = unsigned((size_t(switches) + size_t(kThreads) * rounds - 1) / (size_t(kThreads) * rounds));
#define BENES_COLOUR(PACKED, NEXT)                                                                                        \
    launch_kernel(k_colour<PACKED, NEXT>, grid, kThreads, 0, s, S.S, S.P, Q, cb, Sn.S, Sn.P, salt + 1u, switches, R, log2m, kappa, L, \
                  out_stage, cap, gate, rounds)
        // (a packed level is followed by packed levels only, and so is the last one)
        if (S.packed) { if (Sn.S) BENES_COLOUR(true, kNextPacked); else BENES_COLOUR(true, kNextNone); }
        else if (Sn.packed) BENES_COLOUR(false, kNextPacked);
        else BENES_COLOUR(false, kNextWide);
#undef BENES_COLOUR
        return launch_status();
    }
}

int launch_chain_start(const uint32_t *perm, const uint32_t *Q, uint32_t *G, uint32_t *owner, size_t total, int log2m, cudaStream_t s) {
    const uint32_t quads = uint32_t(total / 4);
    launch_kernel(k_chain_start, (quads + kThreads - 1) / kThreads, kThreads, 0, s, reinterpret_cast<const uint4 *>(perm), Q,
                  reinterpret_cast<uint4 *>(G), reinterpret_cast<uint2 *>(owner), quads, log2m);
    return launch_status();
}

int chain_label(const uint32_t *G, uint32_t *owner, const SampledScratch &sc, size_t total, int log2m, int kappa, uint32_t salt,
                uint32_t cap, BitsLayout L, int out_stage, uint32_t *gate, cudaStream_t s) {
    const uint32_t R = uint32_t(total >> kappa), pairs = uint32_t(total / 4);
    int rc;
    {
        ProfileScope ps(kWalk, s);
        launch_kernel(k_chain_walk, (R + kWalkThreads - 1) / kWalkThreads, kWalkThreads, 0, s, G, owner, sc.rec[0], R, log2m, kappa,
                      salt, cap, gate);
        if ((rc = launch_status())) return rc;
    }
    if ((rc = label_lists(sc, R, log2m - kappa, salt, cap, gate, s))) return rc;
    ProfileScope ps(kColour, s);
    launch_kernel(k_chain_colour, (pairs + kThreads - 1) / kThreads, kThreads, 0, s, G, reinterpret_cast<uint2 *>(owner), sc.bits[0],
                  pairs, R, log2m, L, out_stage, cap, gate);
    return launch_status();
}

}  // namespace benes
