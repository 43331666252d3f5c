// Closing a generation of a biallelic population: its totals, its statistics
// record and state, and the ordered survivor list.  Shared by the generation
// kernel (generations.cuh) and the kernel that closes a call of one generation
// (kernels.cu).
#pragma once

#include "device_common.cuh"
#include "ecology.cuh"

namespace spg {
namespace {

// The generation's totals over the accumulator's copies, by one warp: x is word
// l % 8 of copy l / 8 in lane l, which returns the total of that word (words
// 0-5 sums, 6 the minimum below the maximum).
__device__ __forceinline__ unsigned long long total_stats(unsigned long long x, uint32_t lane) {
    static_assert(sizeof(GenAcc) == 64 && kGenAccCopies == 4, "a lane per word");
#pragma unroll
    for (int o = 8; o <= 16; o <<= 1) {
        const unsigned long long y = __shfl_xor_sync(0xFFFFFFFFu, x, o);
        if ((lane & 7u) == 6u)
            x = (unsigned long long)(uint32_t)min((int)(uint32_t)x, (int)(uint32_t)y) |
                (unsigned long long)(uint32_t)max((int)(x >> 32), (int)(y >> 32)) << 32;
        else x += y;
    }
    return x;
}

// Generation g's statistics record and the population's new state, by one warp
// (sum: total_stats; R and f: the resource and factor after it), and empty sums
// for the generation after next: every block has read what they held, and none
// adds to them before that generation.
__device__ __forceinline__ void write_state(const SoloArgs &a, uint32_t lane, uint32_t g, unsigned long long sum,
                                            uint32_t S, double R, uint32_t f) {
    const bool eco = a.has_eco != 0u;
    const int32_t status = S == 0u ? SPG_EXTINCT : SPG_OK;
    spg_stats *rec = a.ring + (g - 1u) % a.stats_cap;
    DevState *st = a.state;
    if (lane == 0u) {
        rec->gen = g;
        rec->n = a.n;
        rec->s = S;
        rec->status = (uint32_t)status;
        rec->R = eco ? R : 0.0;
        rec->f = f;
        rec->pad = 0;
        rec->sum_raw = (long long)sum;
        st->gen = g;
        st->S = S;
        st->f = f;
        st->R = R;
        st->status = status;
    } else if (lane < 7u) {
        if (lane == 1u) rec->sum_raw_surv = (long long)sum;
        if (lane == 2u) rec->sum_raw2 = sum;
        if (lane == 3u) rec->consumption = eco ? sum : 0ull;
        if (lane == 4u) rec->het = sum;
        if (lane == 5u) rec->allele = sum;
        if (lane == 6u) {
            rec->min_raw = (int)(uint32_t)sum;
            rec->max_raw = (int)(sum >> 32);
        }
    }
    reinterpret_cast<unsigned long long *>(a.acc + (size_t)((g + 2u) % 3u) * kGenAccCopies)[lane] =
        (lane & 7u) == 6u ? kEmptyMinMax : 0ull;
}

// The survivors of slots slot0 .. slot1 - 1 in the ordered list, from the bitmap
// and the rank of each slot's first survivor, by warp `warp` of `warps`.  A warp
// takes the bitmap words of several slots at once, a word per lane: a word and
// its load at a time, a wait for L2 each, calls of one generation took 45.1 us
// at N = 10^6 (43.1 now) and 4.43 ms for 4,096 members (3.83 now).
// ready() runs once, before the first rank is asked for, with the first words on
// their way; false: nothing to list.
template <class Ready, class First>
__device__ __forceinline__ void list_survivors(const SoloArgs &a, uint32_t slot0, uint32_t slot1, uint32_t warp,
                                               uint32_t warps, uint32_t lane, Ready ready, First first_rank) {
    const uint32_t len = a.slot_len, words = (a.n + 31u) >> 5, share = (slot1 - slot0 + warps - 1u) / warps;
    const uint32_t per = len > 32u ? 1u : min(32u / len, max(share, 1u));  // slots a pass
    const uint32_t seg = len > 32u ? 0u : min(lane / len, per), in = len > 32u ? lane : lane - seg * len;
    auto load = [&](uint32_t slot, uint32_t c) {
        const uint32_t q = slot * len + c + in;
        return seg < per && slot < slot1 && c + in < len && q < words ? __ldcg(a.alive + q) : 0u;
    };
    uint32_t s = slot0 + warp * per, bits = load(s + seg, 0u);
    if (!ready()) return;
    for (; s < slot1; s += warps * per) {
        const uint32_t slot = s + seg;
        uint32_t before = seg < per && slot < slot1 ? first_rank(slot) : 0u;
        for (uint32_t c = 0; c < len; c += 32u) {  // once, but for slots of more than 32 words
            const uint32_t own = __popc(bits);
            uint32_t at = own;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, at, o);
                if ((int)lane >= o) at += y;
            }
            const uint32_t all = __shfl_sync(0xFFFFFFFFu, at, 31);
            at -= own;
            at += before - __shfl_sync(0xFFFFFFFFu, at, (int)min(lane - in, 31u));
            before += all;
            // the words of lanes 0, 1, ..., four at a time (one at a time waits for each)
            const uint32_t q0 = s * len + c, m = q0 < words ? min(min(32u, per * len), words - q0) : 0u;
            for (uint32_t b = 0; b < m; b += 4u) {
#pragma unroll
                for (uint32_t i = 0; i < 4u; ++i) {
                    const uint32_t w = __shfl_sync(0xFFFFFFFFu, bits, (int)(b + i)),
                                   r = __shfl_sync(0xFFFFFFFFu, at, (int)(b + i));
                    if ((w >> lane) & 1u) a.surv[r + __popc(w & ((1u << lane) - 1u))] = (q0 + b + i) * 32u + lane;
                }
            }
            bits = c + 32u < len ? load(slot, c + 32u) : load(slot + warps * per, 0u);
        }
    }
}

}  // namespace
}  // namespace spg
