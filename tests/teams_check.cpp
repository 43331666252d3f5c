// Host-side check of the team schedule (spg::schedule_teams): seeded batches
// of members over 1..152 blocks.  Every member has ranks 0 .. team - 1 once, on
// different blocks; replaying the blocks' lists with teams that start only
// when all their blocks are at them finishes (no block waits for ever).
#include <cmath>
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
    std::mt19937 rng(31u);
    for (int c = 0; c < 200; ++c) {
        const uint32_t M = 1 + rng() % (c % 4 == 0 ? 600 : 40), blocks = c % 3 == 0 ? 152u : 1 + rng() % 152;
        std::vector<spg::TeamMember> members(M);
        for (auto &m : members) {
            const double u = (double)(rng() % 1000000u) / 1e6;
            m.n = 1 + (uint32_t)std::exp(u * std::log(c % 5 == 0 ? 1e9 : 2e6));
            m.words = 1u << (rng() % 4);
            m.linked = rng() % 5 == 0;
            m.weighted = rng() % 5 == 0;
        }
        std::vector<spg::TeamPlace> places;
        std::vector<uint32_t> start;
        const double cycles = spg::schedule_teams(members, blocks, places, start);
        if (!(cycles > 0) || start.size() != blocks + 1u || start[0] != 0 || start[blocks] != places.size())
            return fail(c, "block offsets");
        std::vector<std::vector<uint8_t>> seen(M);
        std::vector<uint32_t> team(M, 0), at(start.begin(), start.end() - 1);
        for (uint32_t b = 0; b < blocks; ++b)
            for (uint32_t p = start[b]; p < start[b + 1]; ++p) {
                const spg::TeamPlace &x = places[p];
                if (x.member >= M || x.team == 0 || x.team > blocks || x.rank >= x.team) return fail(c, "place bounds");
                if (team[x.member] && team[x.member] != x.team) return fail(c, "team sizes differ");
                team[x.member] = x.team;
                seen[x.member].resize(x.team);
                if (seen[x.member][x.rank]++) return fail(c, "a rank twice");
                if (p > start[b] && members[places[p - 1].member].words < members[x.member].words)
                    return fail(c, "locus counts not in order");
                for (uint32_t q = start[b]; q < p; ++q)
                    if (places[q].member == x.member) return fail(c, "a block twice in a team");
            }
        for (uint32_t m = 0; m < M; ++m) {
            if (!team[m]) return fail(c, "member without a team");
            for (uint8_t s : seen[m])
                if (s != 1) return fail(c, "rank missing");
        }
        for (size_t done = 0; done < M;) {  // teams whose blocks are all at them
            std::vector<uint32_t> here(M, 0);
            for (uint32_t b = 0; b < blocks; ++b)
                if (at[b] < start[b + 1]) ++here[places[at[b]].member];
            size_t ran = 0;
            std::vector<uint8_t> runs(M, 0);
            for (uint32_t m = 0; m < M; ++m)
                if (here[m] && here[m] == team[m]) {
                    runs[m] = 1;
                    ++ran;
                }
            if (!ran) return fail(c, "every block waits");
            for (uint32_t b = 0; b < blocks; ++b)
                if (at[b] < start[b + 1] && runs[places[at[b]].member]) ++at[b];
            done += ran;
        }
    }
    std::printf("ok\n");
    return 0;
}
