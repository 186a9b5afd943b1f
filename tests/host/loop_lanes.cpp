// Plays the lanes of a warp through the loops of loops8.cuh, one lane after the other between two votes.  Lanes of a
// warp run in lockstep only where they vote, so every order of them in between has to give the same marks.
#include <stdint.h>
#include <string.h>
#include <ucontext.h>

#include <algorithm>
#include <random>
#include <vector>

#define __device__
#define __forceinline__ inline
struct uint2 {
    uint32_t x, y;
};
static inline uint2 make_uint2(uint32_t x, uint32_t y) { return uint2{x, y}; }
static inline int __ffs(int v) { return __builtin_ffs(v); }
static inline int __clz(int v) { return v ? __builtin_clz(unsigned(v)) : 32; }
static inline int __popc(uint32_t v) { return __builtin_popcount(v); }
static inline uint32_t __brev(uint32_t v) {
    uint32_t r = 0;
    for (int i = 0; i < 32; ++i) r |= ((v >> i) & 1u) << (31 - i);
    return r;
}
using std::min;

static struct {
    uint32_t x;
} threadIdx;

namespace {
constexpr int kWarp = 32;
ucontext_t g_scheduler, g_lane[kWarp];
uint32_t g_vote[kWarp];        // what each lane has brought to the vote at hand
uint32_t g_ballot;             // the last vote's result
bool g_done[kWarp];

uint32_t vote(bool v) {
    const uint32_t lane = threadIdx.x;
    g_vote[lane] = v;
    swapcontext(&g_lane[lane], &g_scheduler);
    return g_ballot;
}
}  // namespace
static inline int __all_sync(uint32_t, bool v) { return vote(v) == ~0u; }
static inline uint32_t __ballot_sync(uint32_t, bool v) { return vote(v); }
static inline int __any_sync(uint32_t, bool v) { return vote(v) != 0u; }

#include "loops8.cuh"

namespace {
struct Job {
    const unsigned char *N;
    unsigned char *marks;
    uint32_t regions, valid;
} g_job;

void lane_main() {
    // (the pointers level8 gives: a lane behind the CTA's last sub-block has that one's)
    const uint32_t lane = threadIdx.x, r = min(lane, g_job.regions - 1u);
    benes::loop_marks(g_job.N + 256u * r, g_job.marks + benes::kMarkStride * r, lane < g_job.valid);
    g_done[lane] = true;
    swapcontext(&g_lane[lane], &g_scheduler);
}
}  // namespace

// `regions` sub-blocks, of which those from `valid` on are padding.  `order`: 0 = lanes ascending, 1 = descending, otherwise
// the seed of an order drawn anew after every vote.  Returns the number of votes, or -1 where some lanes ended while others
// wait for one.
extern "C" int play_loop_marks(uint32_t regions, uint32_t valid, const unsigned char *N, unsigned char *marks, uint32_t order) {
    g_job = Job{N, marks, regions, valid};
    std::vector<std::vector<char>> stacks(kWarp, std::vector<char>(1 << 16));
    std::vector<int> turn(kWarp);
    for (int i = 0; i < kWarp; ++i) {
        turn[i] = order == 1 ? kWarp - 1 - i : i;
        g_done[i] = false;
        getcontext(&g_lane[i]);
        g_lane[i].uc_stack.ss_sp = stacks[i].data();
        g_lane[i].uc_stack.ss_size = stacks[i].size();
        g_lane[i].uc_link = &g_scheduler;
        makecontext(&g_lane[i], lane_main, 0);
    }
    std::mt19937 rng(order);
    for (int votes = 0;; ++votes) {
        if (order > 1) std::shuffle(turn.begin(), turn.end(), rng);
        for (int lane : turn) {
            threadIdx.x = uint32_t(lane);
            swapcontext(&g_scheduler, &g_lane[lane]);
        }
        uint32_t ballot = 0;
        int done = 0;
        for (int i = 0; i < kWarp; ++i) {
            ballot |= g_vote[i] << i;
            done += g_done[i];
        }
        if (done == kWarp) return votes;
        if (done) return -1;
        g_ballot = ballot;
    }
}
