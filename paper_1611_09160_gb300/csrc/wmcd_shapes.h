// Launch shapes of a colour phase: plain host arithmetic on sizes, no CUDA.
#pragma once
#include <algorithm>
#include <cstdint>

namespace wmcd {

constexpr int kMaxStageWarps = 4;  // most queues of ordinary regions a block serves, one warp each
// ordinary regions: at most this many beads
constexpr int kLightCap = 80;

struct PhaseShape {
    int slots;                     // a queue with more slots than this goes to a block though its region is light
    bool wide;                     // the dense regions up to the middle size take eight warps, not four
};

// The shape of a phase of nq queues in each of S simulations (maxN beads in the largest) on n_sm SMs.
// Blocks hurry the longest queues of a phase: their warps run a queue's moves ahead. Where the phase has
// fewer queues than the light launch has warps in flight, its longest queue is its time; where it has many,
// their number is (a block costs a short queue more). 16k dilute beads (512 queues) with the line at 4 and
// eight warps: 5.33 -> 4.80 ms a sweep; 79k suspension 13.3 -> 11.4. Twice the warps for a dense region
// where its queue is the phase's time (16k dilute beads: 5.05 -> 4.84 ms a sweep), not where the phase has
// more queues than blocks of either kind hold at once (FENE chains, 3,375 queues: 5.76 with four warps, 5.97
// with eight) or every region is dense. The queues of a batch's phase are those of all its members: 64 of
// 4,096 dilute beads 8.1 -> 7.0 ms a sweep (binary64 15.9 -> 11.8), 256 of 3,072 17.3 -> 14.3, against one
// member's count. (A lone simulation of 1,331-2,197 queues: 2% faster with eight warps, 6% slower in binary64;
// a batch of 16 with 2,000 queues 4% faster, so its line is twice as high.)
inline PhaseShape phase_shape(int nq, int S, int64_t maxN, int n_sm) {
    const int64_t all = (int64_t)nq * S;
    PhaseShape p;
    p.slots = all <= 32 * n_sm ? 4 : 24;
    p.wide = nq <= 8 * n_sm && all <= 16 * n_sm && ((double)maxN / nq <= kLightCap || all <= 3 * n_sm);
    return p;
}

// queues of ordinary regions per block for a choice of stage_warps
inline int light_queues(int stage_warps) { return std::min(kMaxStageWarps, 2 * std::max(1, stage_warps)); }

}  // namespace wmcd
