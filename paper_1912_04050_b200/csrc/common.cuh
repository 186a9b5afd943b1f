// Shared declarations of the Benes routing library (CUDA side only).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <stddef.h>

#include <atomic>
#include <mutex>

#include "benes.h"

namespace benes {

// Largest block finished inside one CTA (log2).  Blocks above it go through
// the per-level HBM kernels.
constexpr int kFusedLog2M = 15;

// Largest list (log2 of its 64-bit words) that one CTA labels in shared memory.
constexpr int kListSmemLog2 = 14;

// Owner of a pair of list words nobody has claimed; a claim is ~(walker << 1 | side of arrival).  Zero, so that one
// memset clears it with the gate and the bucket counters.
constexpr uint32_t kUnowned = 0u;

// Every kernel launch of the library goes through this counter.
extern std::atomic<unsigned long long> g_launches;

#define BENES_CUDA_TRY(expr)                                   \
    do {                                                       \
        cudaError_t e_ = (expr);                               \
        if (e_ != cudaSuccess) {                               \
            cudaGetLastError(); /* reported here, not by a later launch */ \
            return BENES_ERR_CUDA;                             \
        }                                                      \
    } while (0)

// Result of the launch just issued; a launch error is taken off the runtime's
// error state so that it is reported once, by the call that caused it.
inline int launch_status() {
    ++g_launches;
    return cudaGetLastError() == cudaSuccess ? BENES_OK : BENES_ERR_CUDA;
}

// Launches `kernel` so that its CTAs may take their places while the last CTAs of the kernel before it in the stream
// are ending (programmatic dependent launch).  Every kernel of the library begins with after_previous_kernel(), so none
// of it runs before that kernel has finished and its memory operations are visible; what overlaps is the launch itself
// and the start of the CTAs.  A route above 2^15 is a chain of 10 to 60 launches, most of them of 5 to 60 us: 2^18 272
// -> 230 us, 2^20 499 -> 434, 2^24 3.71 -> 3.59 ms, 2^20 apply 24.8 -> 18.3 us.
template <class... P, class... A>
inline void launch_kernel(void (*kernel)(P...), size_t grid, size_t threads, size_t smem, cudaStream_t s, A &&...args) {
    cudaLaunchAttribute overlap = {};
    overlap.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    overlap.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned(grid));
    cfg.blockDim = dim3(unsigned(threads));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &overlap;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, P(args)...);               // launch_status() has the result
}
// Waits for the previous grid.  The wait comes before any access, so that a kernel that has ended implies that all
// kernels before it in the stream have.  (No explicit trigger, which would let the next grid's CTAs in as soon as all of this
// grid have started: they fill the SMs that happen to have room, two and three on one SM, and are slower for it: 2^20
// apply 39 us, route 442.)
__device__ __forceinline__ void after_previous_kernel() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Kernel attributes (opt-in shared memory) belong to a device: a launcher sets
// them the first time it runs on each device of the process.
constexpr int kMaxDevices = 64;
struct OncePerDevice {
    std::mutex mu;
    bool done[kMaxDevices] = {};
    // Runs `configure` (returns a status) the first time on each device; a second
    // thread that arrives meanwhile waits until the attributes are set.
    template <class F>
    int run(F &&configure) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) { cudaGetLastError(); return BENES_ERR_CUDA; }
        std::lock_guard<std::mutex> lk(mu);
        if (done[dev]) return BENES_OK;
        const int rc = configure();
        if (rc == BENES_OK) done[dev] = true;
        return rc;
    }
};

// ---- index guards ---------------------------------------------------------------
// Every index a kernel forms from data stays in range, so that an input that is not a permutation cannot cause an access
// out of bounds.  What comes from global memory (permutations, inverses, owners, next words) passes a guard, a mask or a
// clamp that on a permutation never changes its value.  A build with -DBENES_DEBUG checks exactly that: a guard that has to
// change its value counts the event in a device word of its translation unit and keeps the source line (no trap, no
// printf; the access itself is still the guarded one).  benes_debug_guard_hits adds the words up.  It stands in for a
// memory checker where none can be run.  What it does not see: the fields of packed records, which cannot exceed their
// mask; the successors of chained levels, masked without a count, because behind a raised gate some are left over from
// other levels, rightly out of range; and successors, codes and list words in shared memory (k_list_label, in-CTA levels),
// which have plain masks, or none where everything that writes them keeps them in their array.
//   BENES_GUARD(v, mask)          v & mask, v expected to be <= mask already
//   BENES_GUARD_BELOW(v, n, alt)  v < n ? v : alt, v expected to be < n
#ifdef BENES_DEBUG
static __device__ unsigned int t_guard_words[2];         // hits, line of the last one
__device__ __forceinline__ uint32_t guard_mask(uint32_t v, uint32_t mask, unsigned line) {
    if (v & ~mask) {
        atomicAdd(&t_guard_words[0], 1u);
        t_guard_words[1] = line;
    }
    return v & mask;
}
__device__ __forceinline__ uint32_t guard_below(uint32_t v, uint32_t n, uint32_t alt, unsigned line) {
    if (v >= n) {
        atomicAdd(&t_guard_words[0], 1u);
        t_guard_words[1] = line;
        return alt;
    }
    return v;
}
#define BENES_GUARD(v, mask) ::benes::guard_mask((v), (mask), __LINE__)
#define BENES_GUARD_BELOW(v, n, alt) ::benes::guard_below((v), (n), (alt), __LINE__)
// Every translation unit with kernels registers a reader of its own words.
using GuardReader = int (*)(unsigned int out[2], int clear);
void guard_register(GuardReader reader, const char *file);
#define BENES_GUARD_TU(name)                                                                     \
    namespace {                                                                                  \
    int guard_read_tu(unsigned int out[2], int clear) {                                          \
        if (cudaMemcpyFromSymbol(out, ::benes::t_guard_words, 8) != cudaSuccess) { cudaGetLastError(); return BENES_ERR_CUDA; } \
        if (clear) {                                                                             \
            const unsigned int zero[2] = {0u, 0u};                                               \
            if (cudaMemcpyToSymbol(::benes::t_guard_words, zero, 8) != cudaSuccess) { cudaGetLastError(); return BENES_ERR_CUDA; } \
        }                                                                                        \
        return BENES_OK;                                                                         \
    }                                                                                            \
    struct GuardRegistrar { GuardRegistrar() { ::benes::guard_register(&guard_read_tu, name); } } t_guard_registrar; \
    }
#else
#define BENES_GUARD(v, mask) ((v) & (mask))
#define BENES_GUARD_BELOW(v, n, alt) ((v) < (n) ? (v) : (alt))
#define BENES_GUARD_TU(name)
#endif

// Multiprocessors of the current device (read once per device).
int sm_count();

// Optional event timing of a group of launches of one kind (see benes.h).
enum ProfileKind {
    kInverse = 0, kFullLabel, kSplit, kFused, kApply, kWalk, kListWalk = 7, kListLabel,    // 6: no kernel any more
    kListResolve, kColour, kApplyFused
};
struct ProfileScope {
    ProfileScope(int kind, cudaStream_t s);
    ~ProfileScope();
    int kind_;
    cudaStream_t s_;
    int slot_;
    unsigned long long launches0_;
};

// Where the words of one stage live.  T = flat switch-word index over the
// whole batch (flat switch index >> 5); valid when N >= 64, so that a word
// never straddles two permutations.
struct BitsLayout {
    uint32_t *bits;        // batch x (2n-1) x W words
    int log2n;             // n
    int log2w;             // log2(W), W = N/64
    __host__ __device__ size_t word(int stage, size_t flat_word) const {
        size_t perm = flat_word >> log2w;
        size_t lw = flat_word & ((size_t(1) << log2w) - 1);
        return ((perm * size_t(2 * log2n - 1) + size_t(stage)) << log2w) + lw;
    }
    // the same in 32 bits: a chunk has at most 2^30 elements, i.e. fewer than
    // 2^24 * (2n-1) < 2^30 words
    __host__ __device__ uint32_t word32(int stage, uint32_t flat_word) const {
        const uint32_t perm = flat_word >> log2w;
        const uint32_t lw = flat_word & ((1u << log2w) - 1u);
        return ((perm * uint32_t(2 * log2n - 1) + uint32_t(stage)) << log2w) + lw;
    }
};

// ---- layout of a level in HBM ------------------------------------------------
// A level of the per-level path keeps its sub-permutations (P, block-local values) and the claims
// of the walks per output switch t of the flat array, and the inverses Q as a plain uint32 array
// (read at random, never claimed).  Two formats of the first part:
//
//   wide   P is a plain uint32 array (level 0: the caller's permutation itself), and S holds an
//          8-byte claim record per switch: { P[2t], P[2t+1] } until a walk of the sampled labelling
//          claims the switch, kClaimed | owner afterwards.  One 64-bit exchange returns the two P
//          values and claims the switch.  What a claim costs is the random sector it dirties
//          (2^25 of them: 1.30 ms in a 512 MiB table, 1.07 in 256, 0.62 in 128, 0.25 in 64 and
//          less), so the records are as small as they can be and what the later kernels
//          need in order stays apart from them.  The ruler switches are claimed from the start.
//   packed (8 B)   P[2t] | P[2t+1] << m | owner << 2m for blocks of 2^m outputs,
//                  owner local to the block, all ones = unowned.  One 64-bit
//                  atomic AND both returns the two P values and claims the
//                  switch, and there is no second copy of P.  Used when the owner fits
//                  with room for the all-ones value: 2m + (m - kappa + 1) < 64.
//
// Owner = (ruler output that claimed the switch) << 1 | side of arrival.
constexpr unsigned long long kClaimed = 1ull << 63;
__host__ __device__ inline bool rec_is_packed(int m, int kappa) {
    return kappa != 0 && 3 * m - kappa + 1 < 64;
}

// The ruler switch of a group of 2^kappa switches (kmask = 2^kappa - 1); salt = level.
__device__ __forceinline__ uint32_t ruler_slot(uint32_t group, uint32_t salt, uint32_t kmask) {
    uint32_t h = group * 0x9E3779B1u + salt;
    h ^= h >> 15;
    h *= 0x85EBCA6Bu;
    h ^= h >> 13;
    return h & kmask;
}

// one P value, P[j], read at random
template <bool PACKED>
__device__ __forceinline__ uint32_t rec_p(const void *S, const uint32_t *P, uint32_t j, int m) {
    if (PACKED) {
        const unsigned long long w = __ldg(static_cast<const unsigned long long *>(S) + (j >> 1));
        return uint32_t(w >> ((j & 1u) ? m : 0)) & ((1u << m) - 1u);
    }
    return BENES_GUARD(P[j], (1u << m) - 1u);
}

// A thread of the streaming kernels owns the two neighbouring switches 2i and
// 2i+1; a warp therefore covers 64 switches = two stage words.  c0 / c1 = the
// bit of the thread's first / second switch.  Lane l fetches the bits of
// switches l and 32 + l (held by threads l/2 and 16 + l/2), so that two
// ballots give the two words.
__device__ __forceinline__ void store_stage_bits64(uint32_t *row_words, uint32_t c0, uint32_t c1) {
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t both = c0 | (c1 << 1);
    const uint32_t lo = __shfl_sync(0xFFFFFFFFu, both, int(lane >> 1));
    const uint32_t hi = __shfl_sync(0xFFFFFFFFu, both, int(16u + (lane >> 1)));
    const uint32_t w0 = __ballot_sync(0xFFFFFFFFu, (lo >> (lane & 1u)) & 1u);
    const uint32_t w1 = __ballot_sync(0xFFFFFFFFu, (hi >> (lane & 1u)) & 1u);
    if (lane < 2) row_words[lane] = lane ? w1 : w0;
}

// the packed record of a switch nobody owns, in a level with blocks of 2^m outputs
__device__ __forceinline__ unsigned long long packed_record(int m, uint32_t p0, uint32_t p1) {
    return (unsigned long long)p0 | ((unsigned long long)p1 << m) | (~0ull << (2 * m));
}
// the claim record of switch t of a level whose rulers are drawn with `salt`
__device__ __forceinline__ unsigned long long claim_record(uint32_t t, uint32_t p0, uint32_t p1, int kappa, uint32_t salt) {
    const uint32_t group = t >> kappa, kmask = (1u << kappa) - 1u;
    return (t & kmask) == ruler_slot(group, salt, kmask) ? (kClaimed | (unsigned long long)(group << 2))
                                                         : ((unsigned long long)p0 | ((unsigned long long)p1 << 32));
}
// Two neighbouring switches t, t + 1 (t even) of a level: 16-byte stores.  A wide level gets its P
// here too, unless P is null (level 0).
template <bool PACKED>
__device__ __forceinline__ void rec_write2(void *S, uint32_t *P, size_t t, int m, uint4 p, int kappa, uint32_t salt) {
    if (PACKED) {
        static_cast<ulonglong2 *>(S)[t >> 1] = make_ulonglong2(packed_record(m, p.x, p.y), packed_record(m, p.z, p.w));
    } else {
        if (P) reinterpret_cast<uint4 *>(P)[t >> 1] = p;
        static_cast<ulonglong2 *>(S)[t >> 1] = make_ulonglong2(claim_record(uint32_t(t), p.x, p.y, kappa, salt),
                                                               claim_record(uint32_t(t) + 1u, p.z, p.w, kappa, salt));
    }
}
template <bool PACKED>
__device__ __forceinline__ void rec_write(void *S, uint32_t *P, size_t t, int m, uint32_t p0, uint32_t p1, int kappa, uint32_t salt) {
    if (PACKED) {
        static_cast<unsigned long long *>(S)[t] = packed_record(m, p0, p1);
    } else {
        if (P) reinterpret_cast<uint2 *>(P)[t] = make_uint2(p0, p1);
        static_cast<unsigned long long *>(S)[t] = claim_record(uint32_t(t), p0, p1, kappa, salt);
    }
}

__device__ __forceinline__ unsigned long long make_word(uint32_t nxt, uint32_t mn) {
    return (static_cast<unsigned long long>(mn) << 32) | nxt;
}

// The streaming kernels of a level give every CTA `rounds` consecutive groups of
// `threads` items: as many as keep 8 CTAs per SM busy, at most 4.  More than one, because the next group's loads
// are under way while one is worked on and the words a CTA gathers stay in the L1; few, because with 16 the last wave of
// the 1184 CTAs that run together was nearly as long as the others (2^24: 1.7 waves) and the CTAs whose loops have no
// ruler ended late.  Colouring + split, 16 -> 4 (2: the same, 1: slower at 2^26): 2^24 0.82 -> 0.70 ms, transposed 1.33
// -> 1.09, 2^26 3.16 -> 2.97, 256 x 2^16 0.101 -> 0.079.
inline uint32_t stream_rounds(size_t items, int threads) {
    const size_t r = items / (size_t(threads) * size_t(sm_count()) * 8);
    return uint32_t(r < 1 ? 1 : (r > 4 ? 4 : r));
}

// ---- per-level HBM path (route_levels.cu) ----------------------------------
// total = batch * N flat elements (<= 2^30), all blocks of one level per launch.
// The records of a level: packed, or wide (S = claim records, P = plain array).
struct LevelRecords {
    void *S;
    uint32_t *P;
    bool packed;
};
// Level 0: records from the caller's permutation (rulers of salt 0; none if S.S is null), and Q[P[j]] = j.
int launch_inverse(const uint32_t *perm, LevelRecords S, uint32_t *Q, size_t total, int log2m, int kappa,
                   cudaStream_t s);
// The same for total >= 2^kInversePartitionMinLog2 in two streaming passes:
// `pairs` = total x 8 bytes of scratch, `fill` = kInverseMaxBuckets zero-initialised counters, one
// per bucket (total >> 15 of them are used, or total >> 18 where that would be too many).
constexpr int kInversePartitionMinLog2 = 22;
constexpr int kInverseMaxBuckets = 4096;
int launch_inverse_partitioned(const uint32_t *perm, LevelRecords S, uint32_t *Q, void *pairs,
                               uint32_t *fill, size_t total, int log2m, int kappa, cudaStream_t s);
int launch_inverse_partition_piece(const uint32_t *perm, LevelRecords S, void *pairs, uint32_t *fill,
                                   size_t total, size_t j_first, size_t count, int log2m, int kappa,
                                   cudaStream_t s);
int launch_inverse_scatter(const void *pairs, uint32_t *Q, size_t total, int log2m, cudaStream_t s);
// Levels of blocks of 2^log2n .. 2^(last_m + 1) by pointer jumping over all outputs, in ONE cooperative launch;
// `gate` (may be null) is a device word: the kernel returns at once while it is 0.  P[], Q[]: total words each; the
// blocks of 2^last_m are left in P[(log2n - last_m) & 1], their inverses, where the in-CTA levels start, in Q[ditto].
int launch_route_jump(const uint32_t *perm, uint32_t *const P[2], uint32_t *const Q[2], unsigned long long *Wd,
                      size_t total, int log2n, int last_m, BitsLayout L, const uint32_t *gate, cudaStream_t s);
// Input-side bits + next level's inverses; its successors too, if G is not null (chained levels).
int launch_split(const uint32_t *Q, uint32_t *Qn, size_t total, int log2m, BitsLayout L, int in_stage, int out_stage,
                 cudaStream_t s, uint32_t *G = nullptr);

// ---- ruler-sampled loop labelling (route_sampled.cu) --------------------------
struct SampledScratch {
    uint2 *rec[5];               // walk records (minimum, peer), which are contracted lists: at most
                                 // total >> (kappa + 2 i) words
    uint32_t *owner[5];          // owners of the pairs of words of rec[i] (all kUnowned between uses)
    uint32_t *bits[5];           // parity of every word's cycle minimum, one bit each
};
size_t sampled_scratch_bytes(size_t total, int kappa);
void sampled_scratch_carve(char *base, size_t total, int kappa, SampledScratch *out);
// Labels every loop of the level, writes the output-side stage and the next
// level's records Sn (none if Sn.S is null, behind packed records S only); raises *gate if some walk exceeded `cap` hops (the route must then be
// redone by launch_route_jump).
int sampled_label(LevelRecords S, const uint32_t *Q, LevelRecords Sn, const SampledScratch &sc, size_t total,
                  int log2m, int kappa, uint32_t salt, uint32_t cap, int walk_pairs, BitsLayout L, int out_stage, uint32_t *gate, cudaStream_t s);
// Chained levels: the successors themselves in an array, G[j] = g(j), local to the block (two per 8 bytes), and the owners
// of the switches beside them (`owner`, one word per switch, all kUnowned between levels).  A hop then waits for one load,
// G[j], and its claim, which are under way together.  Total elements up to which the sampled levels run that way: where a
// level lasts as long as its longest chain, not where the GPU is full of them, because a successor costs the level above a
// random store and the walks a second table (records -> chained: 2^20 417 -> 394 us, 2^21 593 -> 597, 3 x 2^20 612 -> 625,
// 2^22 946 -> 981, 2^24 3.35 -> 3.76 ms).
constexpr size_t kChainMaxTotal = size_t(1) << 20;
int launch_chain_start(const uint32_t *perm, const uint32_t *Q, uint32_t *G, uint32_t *owner, size_t total, int log2m, cudaStream_t s);
// Labels every loop of a chained level and writes the output-side stage.
int chain_label(const uint32_t *G, uint32_t *owner, const SampledScratch &sc, size_t total, int log2m, int kappa, uint32_t salt,
                uint32_t cap, BitsLayout L, int out_stage, uint32_t *gate, cudaStream_t s);
// The bytes from the start of the scratch that have to be zero (owners kUnowned) before the first sampled_label of a
// route (log2m of the first level).
size_t sampled_owner_bytes(const SampledScratch &sc, size_t total, int log2m, int kappa);

// ---- fused path (route_fused.cu) -------------------------------------------
// Finishes levels (n - log2m) .. n-1 of every block of size 2^log2m of the flat
// level array (total elements), one CTA per block for log2m <= kFusedLog2M, one
// cluster of two CTAs per block for log2m = kFusedLog2M + 1.
// `src`: the blocks' values, local to their block: the permutation, or its inverse if `inverse` (blocks of 2^11 and more).
// `blocks` blocks from `first_block` on (blocks = 0: all from first_block).
int launch_fused(const uint32_t *src, bool inverse, size_t total, int log2m, uint32_t *bits, int log2n,
                 cudaStream_t s, size_t first_block = 0, size_t blocks = 0, uint32_t *const spare[2] = nullptr);
// With `spare` (two arrays of total words), blocks of 2^kPeelLog2 and more that leave at least half of the SMs without
// one run a level at a time, on twice as many SMs each time.
constexpr int kPeelLog2 = 12;

// ---- payload apply (apply.cu) ----------------------------------------------
int launch_apply_stage(const uint32_t *bits, const void *x, void *y, int elem_bytes, int stage,
                       int log2n, size_t batch, cudaStream_t s);

// ---- payload apply, several stages per pass (apply_fused.cu) -----------------
// `scratch` (batch * N elements) is needed above 2^13 elements per permutation.
// With a pipe the first pass runs part by part as the parts of `in` arrive
// (in_ready[i], recorded on another stream), and the parts of `out` the last
// pass has finished are copied to out_host on the side stream.
constexpr int kApplyMaxParts = 8;
struct ApplyHostPipe {
    int parts;                              // divides the number of 2^13-element chunks
    cudaEvent_t in_ready[kApplyMaxParts];
    cudaEvent_t out_done[kApplyMaxParts];
    cudaStream_t side;
    void *out_host;
};
int launch_apply_fused(const uint32_t *bits, const void *in, void *out, void *scratch, int elem_bytes,
                       int log2n, size_t batch, cudaStream_t s, const ApplyHostPipe *pipe = nullptr);
// chunks (CTAs) of the first and of the last pass, 0 if the size is too small to pipe
size_t apply_fused_chunks(int log2n, size_t batch);

// ---- sizes that are not a power of two (pad.cu) ------------------------------
int launch_pad_perm(const uint32_t *src, uint32_t *dst, size_t n_elems, int log2n, size_t batch,
                    cudaStream_t s);
int launch_pad_rows(const void *src, void *dst, int elem_bytes, bool pad, size_t n_elems, int log2n,
                    size_t batch, cudaStream_t s);

int launch_export_butterfly(const uint32_t *bits, uint32_t *out, int log2n, size_t batch, cudaStream_t s);

// ---- validation (route_levels.cu) -------------------------------------------
int launch_validate(const uint32_t *perm, size_t total, int log2n, uint32_t *seen_words,
                    uint32_t *flag, cudaStream_t s);

}  // namespace benes
