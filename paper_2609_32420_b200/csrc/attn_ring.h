// The steps of a block of the tcgen05 attention kernels: which barrier says that the scores of a step are there (or that its
// P V has completed), in which phase, and when a producer may fill a ring slot again.
//
// attn_tcgen05_kernel: there is a barrier per softmax group, so a barrier stands for every second step.  The softmax groups wait for each phase of
// theirs in turn.  The producers wait for step u = i - kStages before they fill its slot with tile i, and that wait needs
// care: step u + 2 is on the same barrier, and its tile is loaded already.  A producer that looks late finds the barrier two
// phases on, whose parity reads as if step u were still to come; tile i is then never asked for and the block runs into its
// time limit.  Steps complete in order, so "step u + 1 has completed" will do as well, and that barrier cannot run ahead:
// the next step on it is u + 3 = i, which needs the tile.  Either barrier read alone is wrong or late, the two together are
// exact, however late the producer looks.
//
// attn_tcgen05_b64_kernel: a barrier per group again, of which there are three, and rings of at most three slots (Ring below).  A
// producer that waits for step u = i - slots watches the one barrier: the next step on it is u + 3 >= i, which needs the tile.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define CARNATOR_HD __host__ __device__
#else
#define CARNATOR_HD
#endif

namespace carnator {
namespace tc {

constexpr int kStages = 3;             // ring slots for K tiles and for V tiles
static_assert(kStages == 3, "slot_is_free: step u + 3 is the one that needs the slot of step u");

CARNATOR_HD constexpr int step_bar(int i) { return i & 1; }
CARNATOR_HD constexpr uint32_t step_parity(int i) { return uint32_t(i >> 1) & 1u; }

// Has step u completed, asked by the producer of tile u + kStages (which knows that step u - 1 has)?
// done(bar, parity): whether the phase of that parity has completed on barrier `bar` (an mbarrier parity test).
template <typename Done>
CARNATOR_HD inline bool slot_is_free(int u, Done done) {
    return done(step_bar(u), step_parity(u)) || done(step_bar(u + 1), step_parity(u + 1));
}

// Counts the steps of a ring of N slots: slot and phase of step i without a division.
template <int N>
struct Ring {
    int slot = 0;
    uint32_t phase = 0;
    CARNATOR_HD inline void next() { if (++slot == N) { slot = 0; phase ^= 1u; } }
};

}  // namespace tc
}  // namespace carnator
