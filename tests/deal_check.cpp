// Host-side check of dealing blocks to kinds of members (spg::deal_blocks):
// every kind with work has a block while there are enough, none more than it can
// use, all blocks are dealt while a kind can use one, and no kind with room has
// more work per block left than the one that got the last block.  And members
// of about the same work are scheduled side by side, and a population's launches
// are cut.
#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <random>
#include <vector>

#include "spegg_engine.h"

static int fail(int c, const char *what) {
    std::printf("FAIL case %d: %s\n", c, what);
    return 1;
}

int main() {
    std::mt19937 rng(7u);
    for (int c = 0; c < 2000; ++c) {
        const size_t K = 1 + rng() % 6;
        const uint32_t blocks = c % 3 ? 152u : rng() % 153u;
        std::vector<double> work(K);
        std::vector<uint32_t> most(K);
        uint32_t kinds = 0;
        for (size_t k = 0; k < K; ++k) {
            work[k] = rng() % 4 == 0 ? 0.0 : (double)(1u + rng() % 1000000u);
            most[k] = work[k] > 0.0 ? 1u + rng() % 152u : 0u;
            kinds += work[k] > 0.0;
        }
        const std::vector<uint32_t> got = spg::deal_blocks(work, most, blocks);
        uint32_t sum = 0, room = 0;
        for (size_t k = 0; k < K; ++k) {
            sum += got[k];
            if (got[k] > most[k]) return fail(c, "more than a kind can use");
            if (work[k] > 0.0 && !got[k] && kinds <= blocks) return fail(c, "a kind without a block");
            if (work[k] == 0.0 && got[k]) return fail(c, "a block without work");
            if (got[k] && got[k] < most[k]) ++room;
        }
        if (sum > blocks || (sum < blocks && room && kinds <= blocks)) return fail(c, "blocks left over or invented");
        for (size_t k = 0; k < K; ++k)  // taking one block back would not have been better
            for (size_t j = 0; j < K; ++j)
                if (got[k] > 1u && got[j] && got[j] < most[j] && work[j] / got[j] > work[k] / (got[k] - 1u) * (1.0 + 1e-12))
                    return fail(c, "not by work");
    }
    // members of about the same work, no more of them than blocks, are formed side
    // by side: no block has two, and the schedule takes little longer than one of
    // them on its part of the blocks
    for (int c = 0; c < 200; ++c) {
        const uint32_t M = 2 + rng() % 15;
        std::vector<spg::TeamMember> members(M);
        double alone = 0.0;
        for (auto &m : members) {
            m.n = 150000u + rng() % 100000u;
            m.words = 1u;
            m.general = rng() % 2 == 0;
        }
        std::vector<spg::TeamPlace> places;
        std::vector<uint32_t> start;
        for (auto &m : members) alone = std::max(alone, spg::schedule_teams({m}, 152u / M, places, start));
        const double cycles = spg::schedule_teams(members, 152u, places, start);
        for (uint32_t b = 0; b < 152u; ++b)
            if (start[b + 1] - start[b] > 1u) return fail(c, "two members on a block");
        if (cycles > 1.25 * alone) return fail(c, "members one after the other");
    }
    // a population's launches: whole for small ones, short for large ones
    uint32_t last = 512u;
    for (uint32_t n = 100u; n < 100000000u; n *= 2u) {
        spg::TeamMember m;
        m.n = n;
        m.words = 4u;
        const uint32_t gens = spg::launch_generations(m, spg::solo_grid(n, m.words, 152u), 152u);
        if (gens > last + 16u || gens < 8u || gens > 512u) return fail((int)n, "launch length");
        if (n > 900000u && n < 4000000u && gens > 80u) return fail((int)n, "a launch of several milliseconds");
        last = gens;
    }
    std::printf("ok\n");
    return 0;
}
