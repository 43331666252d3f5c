// Device kernels of the per-generation update (sm_103a) other than the
// biallelic generation kernel (generations.cuh) and the allocation-free
// call's (offspring.cu): the continuous-allele generation kernel, the
// compaction kernel that closes a generation for both of the two-launch
// forms, and the set-up kernels (founders, the slot layout of biallelic
// populations, state resets).
//
// A generation of continuous-allele populations, or of the allocation-free
// call, is two launches (Fig. 1 A-F of the paper):
//   offspring    draws both parents of every offspring from the previous
//                survivors (A), forms the gametes (B), sums the genetic value
//                (C) and decides survival from the threshold table (D); it
//                writes the child records, the alive bitmap, per-bucket
//                survivor counts and exact integer statistics;
//   k_compact    one block per bucket of kBucket offspring: turns the bitmap
//                into the ordered survivor list (E) with a two-level scan
//                (earlier buckets' counts + a block scan), and the block that
//                finishes a population's last bucket closes its generation:
//                statistics header, resource update in IEEE double with
//                explicitly rounded basic operations (F), new state.
// No block ever waits on another block.
//
// All random numbers are Philox4x32-10 lanes at counters that name
// (individual, generation, replicate, purpose<<24 | sub); see spegg.h.
#include <cuda_runtime.h>

#include <climits>
#include <cstdint>

#include "closing.cuh"
#include "spegg_internal.h"

namespace spg {
namespace {

__device__ __forceinline__ void clear_acc(StatAcc *a) {
    a->s = 0;
    a->sum_raw = 0;
    a->sum_raw_s = 0;
    a->sum_raw2 = 0;
    a->cons = 0;
    a->het = 0;
    a->allele = 0;
    a->mn = INT_MAX;
    a->mx = INT_MIN;
}

// Close generation g of one population (run by one full warp while the
// population's survivors are being compacted; everything it reads was final
// when the offspring launch ended).  The statistics accumulators (kAccCopies
// copies) are summed, the resource is updated, the statistics record is
// written, the accumulators are reset for the next generation, and the new
// survivor count, factor, resource and status are left in the state's next_*
// fields for commit_state.
__device__ void finalize_warp(const Segment &sg, const PopParams *P, uint32_t g, uint32_t f_used) {
    const uint32_t lane = threadIdx.x & 31u;
    DevState *st = sg.state;
    // state loads issued together with the accumulator loads
    const double R_prev = ld_relaxed_f64(&st->R);
    StatAcc mine;
    clear_acc(&mine);
    if (lane < (uint32_t)kAccCopies) {
        StatAcc *src = sg.acc + lane;
        mine.s = __ldcg(&src->s);
        mine.sum_raw = __ldcg(&src->sum_raw);
        mine.sum_raw_s = __ldcg(&src->sum_raw_s);
        mine.sum_raw2 = __ldcg(&src->sum_raw2);
        mine.cons = __ldcg(&src->cons);
        mine.het = __ldcg(&src->het);
        mine.allele = __ldcg(&src->allele);
        mine.mn = __ldcg(&src->mn);
        mine.mx = __ldcg(&src->mx);
        clear_acc(src);
    }
    const unsigned long long S_new = shfl_sum_u64(mine.s);
    const unsigned long long sum_raw = shfl_sum_u64((unsigned long long)mine.sum_raw);
    const unsigned long long sum_raw_s = shfl_sum_u64((unsigned long long)mine.sum_raw_s);
    const unsigned long long sum_raw2 = shfl_sum_u64(mine.sum_raw2);
    const unsigned long long cons = shfl_sum_u64(mine.cons);
    const unsigned long long het = shfl_sum_u64(mine.het);
    const unsigned long long allele = shfl_sum_u64(mine.allele);
    const int mn = __reduce_min_sync(0xFFFFFFFFu, mine.mn), mx = __reduce_max_sync(0xFFFFFFFFu, mine.mx);
    if (lane == 0) {
        spg_stats *rec = sg.ring + (g - 1) % P->stats_cap;
        uint32_t f_next = f_used;
        double R = 0.0;
        if (P->has_eco) {
            R = resource_eaten(P->eco_model == 1u ? resource_grown_bh(R_prev, growth_rate(P->r, P->r_sd, g, P->rep, P->key0, P->key1),
                                                                     P->K)
                                                  : resource_grown(R_prev, P->r, P->K),
                               cons);
            f_next = factor_q32(R, P->R_half);
        }
        const int32_t status = (S_new == 0ull) ? SPG_EXTINCT : SPG_OK;
        rec->gen = g;
        rec->n = sg.n;
        rec->s = (uint32_t)S_new;
        rec->status = (uint32_t)status;
        rec->sum_raw = (long long)sum_raw;
        rec->sum_raw2 = sum_raw2;
        rec->sum_raw_surv = (long long)sum_raw_s;
        rec->min_raw = mn;
        rec->max_raw = mx;
        rec->het = het;
        rec->allele = allele;
        rec->consumption = P->has_eco ? cons : 0ull;
        rec->R = R;
        rec->f = f_next;
        rec->pad = 0;
        st->next_S = (uint32_t)S_new;
        st->next_f = f_next;
        st->next_R = P->has_eco ? R : R_prev;
        st->next_status = status;
    }
}

// Make generation g the population's current one (one thread of the block
// that finished the last compaction bucket, after every block has read the
// state and the closing warp's next_* values are visible).
__device__ void commit_state(DevState *st, uint32_t g) {
    const uint32_t S = ld_relaxed_u32(&st->next_S), f = ld_relaxed_u32(&st->next_f);
    const int32_t status = (int32_t)ld_relaxed_u32(reinterpret_cast<const uint32_t *>(&st->next_status));
    const double R = ld_relaxed_f64(&st->next_R);
    if (st->status == SPG_OK) st->status = status;
    st->f = f;
    st->S = S;
    st->R = R;
    st->done = 0;
    st->gen = g;
}

// ------------------------------------------------ continuous allelic values
// A normal step in raw units from twelve Philox lanes (Irwin-Hall(12)): the
// lanes of subs sub0..sub0+2 summed, t = sum - 6 * 2^32, step =
// ((t >> 8) * s) >> 40 for a Q16 scale s (see spegg.h).
__device__ __forceinline__ int32_t irwin_hall_step(uint32_t j, uint32_t g, uint32_t rep, uint32_t purpose,
                                                   uint32_t sub0, long long s, uint32_t k0, uint32_t k1) {
    unsigned long long sum = 0;
#pragma unroll
    for (uint32_t q = 0; q < 3; ++q) {
        const uint4 d = philox(make_uint4(j, g, rep, (purpose << 24) | (sub0 + q)), k0, k1);
        sum += (unsigned long long)d.x + d.y + d.z + d.w;
    }
    const long long t = (long long)sum - 6LL * 4294967296LL;
    return (int32_t)(((t >> 8) * s) >> 40);
}

// Eight packed int16 values (one 16-byte access) per lane and haplotype.
// val16: value `half` (0 low, 1 high) of a packed word, sign-extended.
__device__ __forceinline__ int32_t val16(uint32_t w, uint32_t half) {
    return half ? (int32_t)w >> 16 : (int32_t)(int16_t)(w & 0xFFFFu);
}
__device__ __forceinline__ uint32_t word_of(const uint4 &c, uint32_t q) {
    return q == 0u ? c.x : q == 1u ? c.y : q == 2u ? c.z : c.w;
}
__device__ __forceinline__ void set_word(uint4 &c, uint32_t q, uint32_t v) {
    if (q == 0u) c.x = v;
    else if (q == 1u) c.y = v;
    else if (q == 2u) c.z = v;
    else c.w = v;
}
// the values of b where bit k (k = 0..7, value k of the eight) of `bits` is set, of a elsewhere
__device__ __forceinline__ uint4 pick8(const uint4 &a, const uint4 &b, uint32_t bits) {
    auto sel = [](uint32_t x, uint32_t y, uint32_t two) {  // a byte permutation of (x, y): selectors 0-3 or 4-7
        return __byte_perm(x, y, (((two & 3u) * 0x2244u) & 0x4444u) | 0x3210u);
    };
    return make_uint4(sel(a.x, b.x, bits), sel(a.y, b.y, bits >> 2), sel(a.z, b.z, bits >> 4),
                      sel(a.w, b.w, bits >> 6));
}
// Sums over eight values v = 256 h + l (h signed, l unsigned): of v, and for
// their squares 65536 h^2 + 512 hl + l^2 of h^2, hl and l^2, by byte dot
// products.
__device__ __forceinline__ int32_t sum8(const uint4 &c, int32_t acc) {
    const int one = 0x0101;
    acc = __dp2a_lo((int)c.x, one, acc);
    acc = __dp2a_lo((int)c.y, one, acc);
    acc = __dp2a_lo((int)c.z, one, acc);
    return __dp2a_lo((int)c.w, one, acc);
}
__device__ __forceinline__ void squares8(const uint4 &c, int32_t &hh, int32_t &hl, uint32_t &ll) {
    const uint32_t h0 = __byte_perm(c.x, c.y, 0x7531), l0 = __byte_perm(c.x, c.y, 0x6420);
    const uint32_t h1 = __byte_perm(c.z, c.w, 0x7531), l1 = __byte_perm(c.z, c.w, 0x6420);
    hh = __dp4a((int)h1, (int)h1, __dp4a((int)h0, (int)h0, hh));
    ll = __dp4a(l1, l1, __dp4a(l0, l0, ll));
    asm("dp4a.s32.u32 %0, %1, %2, %0;" : "+r"(hl) : "r"(h0), "r"(l0));
    asm("dp4a.s32.u32 %0, %1, %2, %0;" : "+r"(hl) : "r"(h1), "r"(l1));
}
// How many of the eight values of a and b differ.
__device__ __forceinline__ uint32_t differ8(const uint4 &a, const uint4 &b) {
    auto top = [](uint32_t x) { return ((x & 0x7FFF7FFFu) + 0x7FFF7FFFu) | x; };  // a half's top bit: half != 0
    uint32_t d = top(a.x ^ b.x) & 0x80008000u;
    d |= (top(a.y ^ b.y) & 0x80008000u) >> 1;
    d |= (top(a.z ^ b.z) & 0x80008000u) >> 2;
    d |= (top(a.w ^ b.w) & 0x80008000u) >> 3;
    return (uint32_t)__popc(d);
}
// value k of the eight moved by `step`, clamped to the int16 range
__device__ __forceinline__ void add_step(uint4 &c, uint32_t k, int32_t step) {
    const uint32_t q = k >> 1, half = k & 1u, w = word_of(c, q);
    const int32_t nv = min(max(val16(w, half) + step, -32768), 32767);
    set_word(c, q, half ? (w & 0xFFFFu) | ((uint32_t)nv << 16) : (w & 0xFFFF0000u) | ((uint32_t)nv & 0xFFFFu));
}

// Generation kernel of a continuous-allele population (S2 "Genetics").  A
// group of G = L/8 lanes forms one offspring, lane li owning loci
// 8li .. 8li+7 of both haplotypes, so parent and child records (2L int16)
// move in coalesced 16-byte accesses; a warp holds 32/G groups, each forming
// U offspring at a time with all their parent loads issued before any is
// used.  The per-offspring draws (parents, survival and mutation uniforms,
// environmental step, gamete-mask streams, mutations) are made once per warp,
// one offspring or mutation per lane, and read by the groups from shared
// memory.  Parents, gamete bits, mutation counts and positions follow the
// biallelic model's draws; mutated values take Irwin-Hall steps; the phenotype
// is the group sum of the values plus the environmental step.  Survivors, statistics and the bitmap
// feed the compaction kernel.
//
// Bound by DRAM at L >= 128 (1,548 bytes an offspring at L = 128: 234 us at N =
// 10^6, 6.6 TB/s) and by instructions below.  L = 32 / 64 / 128 at N = 10^6 and
// L = 256 at 5 x 10^5, us per generation (mu = 10^-3): 107 / 176 / 327 / 349
// with every mutation drawn by its group, the draws handed over by shuffles
// and no prefetch; 93 / 145 / 255 / 254 with the list and shared memory; 92 /
// 143 / 234 / 236 with the prefetch and the byte dot products.
constexpr int kContInFlight = 1;  // offspring a group of lanes forms at a time (four blocks per SM)
constexpr uint32_t kContMutations = 128;  // mutations of a warp's 32 offspring listed before the offspring are formed
// Steps of the warp a parent's record is prefetched into L2 ahead of its use.
// N = 10^6 (L = 256: 5 x 10^5), us per generation with 0 / 1 / 2 / 3 steps: L =
// 128 254 / 234 / 236 / 245, L = 256 255 / 236 / 244 / 260 (further ahead, the
// records leave L2 again before they are used); with 0 / 2 / 4: L = 64 145 /
// 149 / 152, L = 32 93 / 106 / 106 (their steps take more records of less
// memory each, and are bound by instructions).
template <int G>
constexpr uint32_t kContAhead = G >= 16 ? 1u : 0u;

template <int G, int U, bool GROUP>
__global__ void __launch_bounds__(kBlock, 4) k_offspring_cont(const __grid_constant__ GenArgs a) {
    constexpr uint32_t L = 8u * G;
    constexpr int NW = kBlock / 32, NO = 32 / G;
    constexpr int NST = G >= 8 ? G / 8 : 1;  // gamete-mask streams per offspring (2 words per parent each)
    constexpr uint32_t AHEAD = kContAhead<G>;
    static_assert(G >= 4 && G <= 32 && (G & (G - 1)) == 0 && G % U == 0, "group of 4..32 lanes");
    __shared__ uint32_t s_cdf[kMaxKmax];
    __shared__ uint32_t s_mpos[NW * NO][kMaxKmax];
    __shared__ uint4 s_draw[NW][32];        // the warp's offspring: mother, father, survival draw, mutations
    __shared__ int32_t s_envs[NW][32];
    __shared__ uint4 s_mask[NW][32 * NST];  // their gamete-mask streams
    __shared__ uint16_t s_lpos[NW][kContMutations];
    __shared__ int32_t s_lstep[NW][kContMutations];
    __shared__ long long s_ll[2][NW];
    __shared__ unsigned long long s_ull[4][NW];
    __shared__ uint32_t s_u32[2][NW];
    __shared__ int s_mm[2][NW];
    // the block's population and its tile there (GROUP: a launch group of
    // several populations, from the tile map, one block per launch-wide tile of
    // 256 offspring; otherwise the segment in the kernel parameters)
    const Segment *sgp = &a.one;
    uint32_t tile = blockIdx.x;
    if constexpr (GROUP) {
        sgp = a.segs + __ldg(a.tile_seg + tile);
        tile -= sgp->tile_begin;
    }
    const Segment &sg = *sgp;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const PopNow now = read_state(sg.state);
    if (!now.active) return;
    const PopParams *P = sg.prm;
    const uint32_t n = sg.n, S = now.S, g = now.gen + 1u, f = now.f;
    const uint32_t rep = P->rep, k0 = P->key0, k1 = P->key1, kmax = P->kmax, shift_bin = P->shift;
    const int32_t bias = P->bias;
    const long long s_mut = P->s_mut, s_env = P->s_env;
    const bool has_eco = P->has_eco != 0u;
    const uint4 *par = reinterpret_cast<const uint4 *>(sg.geno[now.gen & 1u]);
    uint4 *chi = reinterpret_cast<uint4 *>(sg.geno[g & 1u]);
    const uint32_t *sin = sg.surv[now.gen & 1u];
    uint32_t *bucket_now = sg.bucket_sum + (g & 1u) * sg.nbuckets;
    uint32_t *bucket_next = sg.bucket_sum + ((g + 1u) & 1u) * sg.nbuckets;
    if (tid < kMaxKmax) s_cdf[tid] = (uint32_t)tid < kmax ? P->cdf[tid] : 0u;
    __syncthreads();
    const uint32_t base = tile * (uint32_t)kBlock;
    if (tid == 0 && base % kBucket == 0u) bucket_next[base / kBucket] = 0u;
    const uint32_t wbase = base + (uint32_t)warp * 32u;
    const uint32_t grp = (uint32_t)lane / G, li = (uint32_t)lane % G;
    const uint32_t gmask = G == 32 ? 0xFFFFFFFFu : ((1u << G) - 1u) << (grp * G);
    const uint32_t wv = li >> 2, sh = (li & 3u) * 8u;  // this lane's mask word and first bit
    uint32_t *mpos = s_mpos[warp * NO + grp];
    constexpr uint32_t R4 = L / 4;  // 16-byte units per record

    // (A) the draws of offspring wbase + lane and its parents' indices
    const uint32_t jl = wbase + (uint32_t)lane;
    const uint4 rl = philox(make_uint4(jl, g, rep, kMate << 24), k0, k1);
    const uint32_t mom_l = jl < n ? __ldcg(sin + __umulhi(rl.x, S)) : 0u;
    const uint32_t dad_l = jl < n ? __ldcg(sin + __umulhi(rl.y, S)) : 0u;
    auto prefetch = [&](uint32_t rec) {
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(par + (size_t)rec * R4), "n"(16u * R4)
                     : "memory");
    };
    if ((uint32_t)lane < AHEAD * NO && jl < n) {
        prefetch(mom_l);
        prefetch(dad_l);
    }
    s_envs[warp][lane] = s_env != 0 ? irwin_hall_step(jl, g, rep, kEnv, 0u, s_env, k0, k1) : 0;
    // (B) gamete-mask streams: entry NST * o + q holds stream q of offspring o
#pragma unroll
    for (int q = 0; q < NST; ++q) {
        const uint32_t e = 32u * (uint32_t)q + (uint32_t)lane;
        s_mask[warp][e] = philox(make_uint4(wbase + e / NST, g, rep, (kRecomb << 24) | (e % NST)), k0, k1);
    }

    // (B) mutations: each lane counts its offspring's and draws their distinct
    // positions, then the warp's lanes draw the Irwin-Hall steps, one
    // mutation each.  (Drawn where they are applied, a mutation in one
    // offspring made the whole warp draw four Philox blocks.)  A warp with more
    // than kContMutations draws them there after all.
    uint32_t K_l = 0;
    if (jl < n && kmax != 0u && rl.w >= s_cdf[0])
        for (uint32_t qk = 0; qk < kmax; ++qk) K_l += rl.w >= s_cdf[qk] ? 1u : 0u;
    uint32_t off_l = K_l;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, off_l, o);
        if (lane >= o) off_l += y;
    }
    const uint32_t nmut = __shfl_sync(0xFFFFFFFFu, off_l, 31);
    off_l -= K_l;  // the offspring's first entry in the warp's list
    const bool listed = nmut <= kContMutations;
    if (listed && nmut != 0u) {
        uint16_t *lpos = s_lpos[warp] + off_l;
        uint32_t chosen = 0;
        uint4 dp = make_uint4(0u, 0u, 0u, 0u);
        for (uint32_t d = 0; d < (uint32_t)kMutDraws && chosen < K_l; ++d) {
            if ((d & 3u) == 0u) dp = philox(make_uint4(jl, g, rep, (kMutPos << 24) | (d >> 2)), k0, k1);
            const uint32_t pos = __umulhi(lane_of(dp, (int)(d & 3u)), 2u * L);
            bool dup = false;
            for (uint32_t qk = 0; qk < chosen; ++qk) dup |= lpos[qk] == pos;
            if (!dup) lpos[chosen++] = (uint16_t)pos;
        }
        for (uint32_t e0 = 0; e0 < nmut; e0 += 32u) {
            const uint32_t e = e0 + (uint32_t)lane;
            uint32_t o = 0;  // the owner: the last lane whose first entry is <= e
#pragma unroll
            for (uint32_t step = 16u; step > 0u; step >>= 1)
                if (__shfl_sync(0xFFFFFFFFu, off_l, (int)(o + step)) <= e) o += step;
            const uint32_t ooff = __shfl_sync(0xFFFFFFFFu, off_l, (int)o);
            if (e < nmut)
                s_lstep[warp][e] = irwin_hall_step(wbase + o, g, rep, kMutSize, 3u * (e - ooff), s_mut, k0, k1);
        }
        K_l = chosen;
    }
    s_draw[warp][lane] = make_uint4(mom_l, dad_l, rl.z, K_l | (off_l << 16));
    __syncwarp();

    long long sum_raw = 0, sum_raw_s = 0;
    unsigned long long sum_raw2 = 0, cons = 0;
    uint32_t lane_het = 0, alive_bits = 0, nsurv = 0;
    uint32_t sq_ll = 0;  // squares of at most 16 * 32 values a lane: each part below 2^25
    int32_t sq_hh = 0, sq_hl = 0;
    int mn = INT_MAX, mx = INT_MIN;
    for (uint32_t it = 0; it < (uint32_t)(G / U); ++it) {
        uint32_t bit[U], rz[U], mut[U];
        uint4 m0[U], m1[U], f0[U], f1[U];
        // the group's U offspring: parents and draws from their lanes, then all the records
#pragma unroll
        for (int u = 0; u < U; ++u) {
            bit[u] = (it * U + (uint32_t)u) * NO + grp;
            const uint4 dr = s_draw[warp][bit[u]];
            const uint32_t mom = dr.x, dad = dr.y;
            rz[u] = dr.z;
            mut[u] = dr.w;
            const uint4 z = make_uint4(0u, 0u, 0u, 0u);
            const bool ok = wbase + bit[u] < n;
            const uint4 *pm = par + (size_t)mom * R4, *pf = par + (size_t)dad * R4;
            m0[u] = ok ? __ldg(pm + li) : z;
            m1[u] = ok ? __ldg(pm + G + li) : z;
            f0[u] = ok ? __ldg(pf + li) : z;
            f1[u] = ok ? __ldg(pf + G + li) : z;
            const uint32_t ahead = bit[u] + AHEAD * NO;
            if (AHEAD != 0u && li < 2u && ahead < 32u && wbase + ahead < n)  // a parent for each of two lanes
                prefetch(reinterpret_cast<const uint32_t *>(&s_draw[warp][ahead])[li]);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint32_t j = wbase + bit[u];
            const bool ok = j < n;
            // (B) gametes: mask word wv of the mother (stream 2wv) and father (2wv + 1)
            const uint2 mk = reinterpret_cast<const uint2 *>(&s_mask[warp][NST * bit[u]])[wv];
            const uint32_t mm = mk.x, mf = mk.y;
            uint4 c0 = pick8(m0[u], m1[u], (mm >> sh) & 0xFFu), c1 = pick8(f0[u], f1[u], (mf >> sh) & 0xFFu);
            // (B) mutation: the listed values moved by the lanes that own them
            auto move = [&](uint32_t pos, int32_t step) {
                if (pos >= L) add_step(c1, pos & 7u, step);
                else add_step(c0, pos & 7u, step);
            };
            if (listed) {
                for (uint32_t m = 0; m < (mut[u] & 0xFFFFu); ++m) {  // the same in the whole group
                    const uint32_t e = (mut[u] >> 16) + m, pos = s_lpos[warp][e];
                    if (((pos & (L - 1u)) >> 3) == li) move(pos, s_lstep[warp][e]);
                }
            } else {
                const uint32_t K = mut[u] & 0xFFFFu;
                uint32_t chosen = 0;
                uint4 dp = make_uint4(0u, 0u, 0u, 0u);
                for (uint32_t d = 0; d < (uint32_t)kMutDraws && chosen < K; ++d) {
                    if ((d & 3u) == 0u) dp = philox(make_uint4(j, g, rep, (kMutPos << 24) | (d >> 2)), k0, k1);
                    const uint32_t pos = __umulhi(lane_of(dp, (int)(d & 3u)), 2u * L);
                    bool dup = false;
                    for (uint32_t qk = 0; qk < chosen; ++qk) dup |= mpos[qk] == pos;
                    if (!dup) {
                        if (li == 0u) mpos[chosen] = pos;
                        __syncwarp(gmask);
                        ++chosen;
                    }
                }
                for (uint32_t m = 0; m < chosen; ++m) {
                    const uint32_t pos = mpos[m];
                    if (((pos & (L - 1u)) >> 3) == li)
                        move(pos, irwin_hall_step(j, g, rep, kMutSize, 3u * m, s_mut, k0, k1));
                }
                __syncwarp(gmask);  // positions are rewritten by the group's next offspring
            }
            if (ok) {
                chi[(size_t)j * R4 + li] = c0;
                chi[(size_t)j * R4 + G + li] = c1;
            }
            // this lane's part of the phenotype sum, its heterozygous loci and
            // squares (no values, so zeros, past the population's end)
            int32_t part = sum8(c0, sum8(c1, 0));
            lane_het += differ8(c0, c1);
            squares8(c0, sq_hh, sq_hl, sq_ll);
            squares8(c1, sq_hh, sq_hl, sq_ll);
#pragma unroll
            for (int o = G / 2; o > 0; o >>= 1) part += __shfl_xor_sync(0xFFFFFFFFu, part, o);
            // (C) phenotype: the sum of all values, plus the environmental step
            const int32_t raw = part + s_envs[warp][bit[u]];
            // (D) survival
            const long long v = (long long)raw + (long long)bias;
            const uint32_t bin = v < 0 ? 0u : (uint32_t)min(v >> shift_bin, (long long)(kBins - 1));
            uint32_t thr = __ldg(&P->table[bin]);
            if (f != kCertain) thr = __umulhi(thr, f);
            const bool alive = (thr == kCertain) || (rz[u] < thr);
            if (ok) {
                mn = min(mn, raw);
                mx = max(mx, raw);
                if (alive) alive_bits |= 1u << bit[u];
                if (li == 0u) {  // per-offspring sums once per group
                    sum_raw += raw;
                    sum_raw2 += (unsigned long long)((long long)raw * (long long)raw);
                    if (alive) {
                        ++nsurv;
                        sum_raw_s += raw;
                        if (has_eco) cons += __ldg(&P->attack[bin]);
                    }
                }
            }
        }
    }
    const unsigned long long lane_allele = (unsigned long long)(65536LL * sq_hh + 512LL * sq_hl + (long long)sq_ll);
    alive_bits = __reduce_or_sync(0xFFFFFFFFu, alive_bits);
    const uint32_t w_surv = __reduce_add_sync(0xFFFFFFFFu, nsurv);
    if (lane == 0 && wbase < n) {
        sg.alive[wbase >> 5] = alive_bits;
        if (w_surv) atomicAdd(&bucket_now[wbase / kBucket], w_surv);
    }
    // statistics over the warp: the per-offspring sums sit in the group
    // leaders, the het and allele sums in every lane
    const uint32_t w_het = __reduce_add_sync(0xFFFFFFFFu, lane_het);
    const unsigned long long w_allele = warp_sum_u64(lane_allele);
    const long long w_raw = (long long)warp_sum_u64((unsigned long long)sum_raw);
    const long long w_raw_s = (long long)warp_sum_u64((unsigned long long)sum_raw_s);
    const unsigned long long w_raw2 = warp_sum_u64(sum_raw2), w_cons = warp_sum_u64(cons);
    const int w_mn = __reduce_min_sync(0xFFFFFFFFu, mn), w_mx = __reduce_max_sync(0xFFFFFFFFu, mx);
    if (lane == 0) {
        s_ll[0][warp] = w_raw;
        s_ll[1][warp] = w_raw_s;
        s_ull[0][warp] = w_raw2;
        s_ull[1][warp] = w_cons;
        s_ull[2][warp] = w_allele;
        s_ull[3][warp] = w_surv;
        s_u32[0][warp] = w_het;
        s_mm[0][warp] = w_mn;
        s_mm[1][warp] = w_mx;
    }
    __syncthreads();
    if (tid == 0) {
        long long a0 = 0, a1 = 0;
        unsigned long long b0 = 0, b1 = 0, al = 0, sv = 0, hz = 0;
        int m0 = INT_MAX, m1 = INT_MIN;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            a0 += s_ll[0][w];
            a1 += s_ll[1][w];
            b0 += s_ull[0][w];
            b1 += s_ull[1][w];
            al += s_ull[2][w];
            sv += s_ull[3][w];
            hz += s_u32[0][w];
            m0 = min(m0, s_mm[0][w]);
            m1 = max(m1, s_mm[1][w]);
        }
        if (sv | hz | (unsigned long long)(m1 != INT_MIN)) {
            StatAcc *acc = sg.acc + blockIdx.x % kAccCopies;
            atomicAdd(&acc->s, sv);
            atomicAdd(reinterpret_cast<unsigned long long *>(&acc->sum_raw), (unsigned long long)a0);
            atomicAdd(reinterpret_cast<unsigned long long *>(&acc->sum_raw_s), (unsigned long long)a1);
            atomicAdd(&acc->sum_raw2, b0);
            if (b1) atomicAdd(&acc->cons, b1);
            atomicAdd(&acc->het, hz);
            atomicAdd(&acc->allele, al);
            atomicMin(&acc->mn, m0);
            atomicMax(&acc->mx, m1);
        }
    }
}

// Continuous founders: value of copy q = h*L + l is effect[l] (decoded from the
// offset-binary planes) when the biallelic founder draw of q is below p0.
template <int C>
__global__ void k_founders_cont(const PopParams *__restrict__ P, uint32_t *__restrict__ geno,
                                uint32_t *__restrict__ surv, uint32_t n, uint32_t p0) {
    constexpr uint32_t L = 32u * C, W = C;  // W = L / 32 words of the planes
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int16_t *rec = reinterpret_cast<int16_t *>(geno + (size_t)i * L);
    for (uint32_t q4 = 0; q4 < 2u * L / 4u; ++q4) {
        const uint4 d = philox(make_uint4(i, 0u, P->rep, (kFounder << 24) | q4), P->key0, P->key1);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const uint32_t q = 4u * q4 + (uint32_t)c, l = q % L;
            int32_t e = P->e_min;
            for (uint32_t b = 0; b < P->nplanes; ++b) e += (int32_t)((P->planes[b * W + l / 32u] >> (l % 32u)) & 1u) << b;
            rec[q] = (int16_t)(lane_of(d, c) < p0 ? e : 0);
        }
    }
    surv[i] = i;
}

// ---------------------------------------- compaction kernel (Fig. 1E, 1F)
// One block per bucket of kBucket offspring.  Its first kBucketWords threads
// read the bucket's bitmap words and the survivor counts of all earlier
// buckets and scan the words' popcounts; then kCompactCopyThreads threads
// (8 warps) write every survivor's index, in offspring order, at its rank =
// (survivors of earlier buckets) + (survivors before it in the bucket).  In a
// population's first bucket an extra warp closes the generation meanwhile
// (finalize_warp).  The block that finishes the last bucket commits the new
// state.  Every load that does not depend on the population state is issued
// together with it (both parities of the bucket counts are summed; the state
// picks one).
__device__ __forceinline__ void compaction_barrier() {
    asm volatile("bar.sync 1, %0;" ::"n"(kCompactCopyThreads) : "memory");  // the compaction threads
}

__device__ __forceinline__ void compact_bucket(const Segment &sg, uint32_t b) {
    constexpr int NW = kBucketWords / 32;  // warps that scan the bitmap words
    constexpr int WPW = (int)(kBucketWords / (kCompactCopyThreads / 32));  // bitmap words per writing warp
    __shared__ uint32_t s_warp[NW];
    __shared__ uint32_t s_prev[NW];
    __shared__ uint32_t s_bits[kBucketWords], s_incl[kBucketWords];
    __shared__ uint32_t s_last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool closer = tid >= (int)kCompactCopyThreads;  // the generation-closing warp
    const bool scanner = tid < (int)kBucketWords;
    const uint32_t valid_words = (sg.n + 31u) >> 5;
    const uint32_t w = b * kBucketWords + (uint32_t)tid;
    const uint32_t bits = (scanner && w < valid_words) ? __ldcg(sg.alive + w) : 0u;
    uint32_t prev0 = 0, prev1 = 0;
    for (uint32_t i = (uint32_t)tid; scanner && i < b; i += kBucketWords) {
        prev0 += __ldcg(sg.bucket_sum + i);
        prev1 += __ldcg(sg.bucket_sum + sg.nbuckets + i);
    }
    const PopNow now = read_state(sg.state);
    if (!now.active) return;
    const uint32_t g = now.gen + 1u;
    const uint32_t first = b * kBucket;
    if (closer) {
        if (b == 0u) finalize_warp(sg, sg.prm, g, now.f);
        __threadfence();
    } else {
        if (scanner) {
            const uint32_t prev = __reduce_add_sync(0xFFFFFFFFu, (g & 1u) ? prev1 : prev0);
            uint32_t incl = __popc(bits);
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                if (lane >= o) incl += y;
            }
            s_bits[tid] = bits;
            s_incl[tid] = incl;
            if (lane == 31) s_warp[warp] = incl;
            if (lane == 0) s_prev[warp] = prev;
        }
        compaction_barrier();
        uint32_t before = 0;  // survivors of all earlier buckets
#pragma unroll
        for (int q = 0; q < NW; ++q) before += s_prev[q];
        uint32_t *__restrict__ sout = sg.surv[g & 1u];
        const uint32_t lt = (1u << lane) - 1u;
#pragma unroll
        for (int k = 0; k < WPW; ++k) {
            const int q = warp * WPW + k;  // bitmap word of the bucket
            const uint32_t word = s_bits[q];
            uint32_t r0 = before + s_incl[q] - __popc(word);
#pragma unroll
            for (int v = 0; v < NW; ++v) r0 += v < q / 32 ? s_warp[v] : 0u;
            if ((word >> lane) & 1u) sout[r0 + __popc(word & lt)] = first + (uint32_t)q * 32u + lane;
        }
    }
    // every block has read the state by now (its values fed the stores
    // above), and the closing warp of bucket 0 has published the next state
    __syncthreads();
    if (tid == 0) s_last = (atomicAdd(&sg.state->done, 1u) == sg.nbuckets - 1u) ? 1u : 0u;
    __syncthreads();
    if (s_last && tid == 0) {
        __threadfence();
        commit_state(sg.state, g);
    }
}

__global__ void __launch_bounds__(kCompactThreads, 3) k_compact(const __grid_constant__ GenArgs a) {
    griddep_release();  // the next generation's blocks may take this grid's place as its blocks finish
    griddep_wait();     // everything below reads the offspring kernel's results
    const uint32_t bkt = blockIdx.x;
    if (a.nsegs == 1u) {
        compact_bucket(a.one, bkt);
    } else {
        const Segment &sg = a.segs[__ldg(a.bucket_seg + bkt)];
        compact_bucket(sg, bkt - sg.bucket_begin);
    }
}

// ------------------------------- closing a generation formed without a barrier
// The generation that k_generations has formed just before (its number in
// state->done): a block lists the survivors of a.close_slots slots, and the extra
// warp of the first one writes the statistics record and the state meanwhile.
// Only that warp writes what other launches read of the state, so no block waits
// for another.  It is a chain of latencies, so every load is issued at once, for
// both parities of the generation (and all three accumulators), and its number
// picks one.  The blocks start as the previous kernel's leave; kCloseSmem bytes
// of shared memory keep them from crowding onto the first SMs that are free (N =
// 10^6: 45.7 us a call without, 41.1 with).
__device__ __forceinline__ void close_part(const SoloArgs &a, uint32_t part) {
    constexpr uint32_t NW = (kCloseThreads - 32u) / 32u;
    __shared__ uint32_t s_gen, s_sum[2][NW], s_own[2][NW], s_first[2][32u * NW];
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const bool close = part == 0u;
    const uint32_t slot0 = part * a.close_slots, slot1 = min(slot0 + a.close_slots, a.nslots);
    DevState *st = a.state;
    if (warp == NW) {
        if (!close) {
            __syncthreads();
            return;
        }
        const uint32_t g = ld_relaxed_u32(&st->done);
        double R = ld_relaxed_f64(&st->R);
        uint32_t f = ld_relaxed_u32(&st->f);
        const unsigned long long *acc = reinterpret_cast<const unsigned long long *>(a.acc) + lane;
        const unsigned long long x0 = __ldcg(acc), x1 = __ldcg(acc + 8u * kGenAccCopies), x2 = __ldcg(acc + 16u * kGenAccCopies);
        const unsigned long long sum = total_stats(g % 3u == 0u ? x0 : g % 3u == 1u ? x1 : x2, lane);
        const unsigned long long cons = __shfl_sync(0xFFFFFFFFu, sum, 3);
        if (lane == 0u && a.has_eco) {
            const double grown = a.eco_model == 1u
                                     ? resource_grown_bh(R, growth_rate(a.eco_r, a.eco_r_sd, g, a.rep, a.keys[0], a.keys[1]),
                                                         a.eco_K)
                                     : resource_grown(R, a.eco_r, a.eco_K);
            R = resource_eaten(grown, cons);
            f = factor_q32(R, a.eco_R_half);
        }
        __syncthreads();
        uint32_t S = 0;
#pragma unroll
        for (uint32_t i = 0; i < NW; ++i) S += s_sum[g & 1u][i];
        if (g != 0u) write_state(a, lane, g, sum, S, R, f);
        return;
    }
    // survivors of the slots before the block's (the first block: of all), and
    // the ranks of its own among those of the warp's 32 slots
    if (tid == 0u) s_gen = ld_relaxed_u32(&st->done);
    uint32_t sum0 = 0, sum1 = 0, own[2] = {0u, 0u};
    for (uint32_t i = tid; i < (close ? a.nslots : slot0); i += 32u * NW) {
        sum0 += __ldcg(a.counts[0] + i);
        sum1 += __ldcg(a.counts[1] + i);
    }
    if (slot0 + tid < slot1) {
        own[0] = __ldcg(a.counts[0] + slot0 + tid);
        own[1] = __ldcg(a.counts[1] + slot0 + tid);
    }
    uint32_t g = 0, before = 0;
    list_survivors(
        a, slot0, slot1, warp, NW, lane,
        [&] {
            sum0 = __reduce_add_sync(0xFFFFFFFFu, sum0);
            sum1 = __reduce_add_sync(0xFFFFFFFFu, sum1);
            uint32_t incl[2] = {own[0], own[1]};
#pragma unroll
            for (int o = 1; o < 32; o <<= 1)
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl[p], o);
                    if ((int)lane >= o) incl[p] += y;
                }
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                s_first[p][tid] = incl[p] - own[p];
                if (lane == 31u) {
                    s_sum[p][warp] = p ? sum1 : sum0;
                    s_own[p][warp] = incl[p];
                }
            }
            __syncthreads();
            g = s_gen;
            if (!close)
#pragma unroll
                for (uint32_t i = 0; i < NW; ++i) before += s_sum[g & 1u][i];
            return g != 0u;
        },
        [&](uint32_t slot) {
            uint32_t r = before + s_first[g & 1u][slot - slot0];
#pragma unroll
            for (uint32_t i = 0; i + 1u < NW; ++i) r += i < (slot - slot0) / 32u ? s_own[g & 1u][i] : 0u;
            return r;
        });
    if (close && g != 0u && a.locus_row[0]) {  // the counted row to its place; clear for the generation after next
        const uint32_t L = 32u * a.words;
        uint32_t *row = a.locus_row[g & 1u], *dst = a.locus_ring + (size_t)((g - 1u) % a.locus_cap) * L;
        for (uint32_t i = tid; i < L; i += 32u * NW) {
            dst[i] = __ldcg(row + i);
            row[i] = 0u;
        }
    }
}
__global__ void __launch_bounds__(kCloseThreads) k_close(const __grid_constant__ SoloArgs a) {
    griddep_release();
    griddep_wait();
    close_part(a, blockIdx.x);
}
// The same of the members of a batch.
__global__ void __launch_bounds__(kCloseThreads) k_close_members(const ClosePart *__restrict__ parts) {
    __shared__ SoloArgs s_args;
    const ClosePart part = parts[blockIdx.x];
    for (uint32_t i = threadIdx.x; i < sizeof(SoloArgs) / 4u; i += kCloseThreads)
        reinterpret_cast<uint32_t *>(&s_args)[i] = reinterpret_cast<const uint32_t *>(part.member)[i];
    griddep_release();
    griddep_wait();
    __syncthreads();
    close_part(s_args, part.part);
}

// ---------------------------------------------------------- founders
template <int W>
__global__ void k_founders(uint32_t *__restrict__ geno, uint32_t *__restrict__ surv, uint32_t n, uint32_t k0,
                           uint32_t k1, uint32_t rep, uint32_t p0) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    // allele copy q = h*L + l (L = 32W) lies in record word q/32 = h*W + l/32
#pragma unroll
    for (int hw = 0; hw < 2 * W; ++hw) {
        uint32_t word = 0;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const uint4 d = philox(make_uint4(i, 0u, rep, (kFounder << 24) | (uint32_t)(hw * 8 + c)), k0, k1);
            word |= (uint32_t)(d.x < p0) << (4 * c + 0);
            word |= (uint32_t)(d.y < p0) << (4 * c + 1);
            word |= (uint32_t)(d.z < p0) << (4 * c + 2);
            word |= (uint32_t)(d.w < p0) << (4 * c + 3);
        }
        geno[(size_t)i * (2 * W) + hw] = word;
    }
    surv[i] = i;
}

__global__ void k_iota(uint32_t *__restrict__ surv, uint32_t n) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) surv[i] = i;
}

// Phenotype bin of a record, its genetic value from the effect planes.
template <int W>
__device__ __forceinline__ uint32_t record_bin(const PopParams *__restrict__ P, const uint32_t (&rec)[2 * W]) {
    uint32_t total = 0, het = 0;
#pragma unroll
    for (int w = 0; w < W; ++w) {
        total += __popc(rec[w]) + __popc(rec[W + w]);
        het += __popc(rec[w] ^ rec[W + w]);
    }
    int32_t raw = P->e_min * (int32_t)total + P->d_min * (int32_t)het;
    for (uint32_t b = 0; b < P->nplanes; ++b) {
        int32_t cnt = 0;
#pragma unroll
        for (int w = 0; w < W; ++w) {
            const uint32_t pl = P->planes[b * W + w];
            cnt += __popc(pl & rec[w]) + __popc(pl & rec[W + w]);
        }
        raw += cnt << b;
    }
    for (uint32_t b = 0; b < P->ndplanes; ++b) {
        int32_t cnt = 0;
#pragma unroll
        for (int w = 0; w < W; ++w) cnt += __popc(P->dplanes[b * W + w] & (rec[w] ^ rec[W + w]));
        raw += cnt << b;
    }
    const long long v = (long long)raw + (long long)P->bias;
    return v < 0 ? 0u : (uint32_t)min(v >> P->shift, (long long)(kBins - 1));
}

// The last bitmap word of a population whose size is not a multiple of 32.
__global__ void k_mark_tail(uint32_t *word, uint32_t count) {
    if (threadIdx.x == 0) *word = (1u << count) - 1u;
}

// Bitmap of a survivor list (the bitmap cleared before).
__global__ void k_mark_alive(const uint32_t *__restrict__ surv, uint32_t S, uint32_t *__restrict__ alive) {
    const uint32_t r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r < S) atomicOr(alive + (surv[r] >> 5), 1u << (surv[r] & 31u));
}

// The slot layout of a generation (generations.cuh) from its full records and
// bitmap, one warp per slot; mate: the survivors' thresholds as mother and
// father, each bin from its record's genetic value.
template <int W>
__global__ void k_pack(const PopParams *__restrict__ P, const uint32_t *__restrict__ geno,
                       const uint32_t *__restrict__ alive, uint32_t n, uint32_t slot_len, uint32_t nslots,
                       uint32_t *__restrict__ packed, uint32_t *__restrict__ counts, uint2 *__restrict__ mate,
                       GenAcc *__restrict__ acc, unsigned long long *__restrict__ barrier) {
    const uint32_t gid = blockIdx.x * blockDim.x + threadIdx.x;
    if (gid < 3u * kGenAccCopies * 8u)
        reinterpret_cast<unsigned long long *>(acc)[gid] = (gid & 7u) == 6u ? kEmptyMinMax : 0ull;
    if (gid == 0u) *barrier = 0ull;
    const uint32_t lane = threadIdx.x & 31u, slot = gid >> 5;
    if (slot >= nslots) return;
    const uint32_t base = slot * slot_len * 32u;
    uint32_t held = 0;
    for (uint32_t gi = 0; gi < slot_len && base + 32u * gi < n; ++gi) {
        const uint32_t j = base + 32u * gi + lane, bits = alive[(base >> 5) + gi];
        const uint32_t at = base + held + __popc(bits & ((1u << lane) - 1u));
        held += __popc(bits);
        if (!((bits >> lane) & 1u)) continue;
        uint32_t rec[2 * W];
        load_record<W>(geno + (size_t)j * (2 * W), rec);
        store_record<W>(packed + (size_t)at * (2 * W), rec);
        if (mate) {
            const uint32_t bin = record_bin<W>(P, rec);
            mate[at] = make_uint2(P->weights->acc[0][bin], P->weights->acc[1][bin]);
        }
    }
    if (lane == 0u) counts[slot] = held;
}

__global__ void k_set_state(DevState *st, StatAcc *acc, uint32_t gen, uint32_t S, uint32_t f, double R,
                            int32_t status, uint32_t target) {
    if (threadIdx.x == 0) {
        st->target = target;
        st->gen = gen;
        st->S = S;
        st->f = f;
        st->status = status;
        st->R = R;
        st->done = 0;
    }
    if (threadIdx.x < (unsigned)kAccCopies) clear_acc(acc + threadIdx.x);
}

}  // namespace

bool supported_shape(uint32_t words, const Shape &s) {
    if (!(s.block == 128 || s.block == 256 || s.block == 512)) return false;
    if (s.lanes == 2) return words >= 4 && s.items == 1;
    if (s.lanes != 1) return false;
    return words <= 2 ? (s.items == 1 || s.items == 2) : s.items == 1;
}

GenKernel compact_kernel() { return &k_compact; }
const void *close_kernel() { return (const void *)&k_close; }
const void *close_members_kernel() { return (const void *)&k_close_members; }
int prepare_close() {
    return cudaFuncSetAttribute(close_kernel(), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCloseSmem) == cudaSuccess
               ? SPG_OK
               : SPG_ERR_CUDA;
}

template <int G>
GenKernel cont_instance(bool group) {
    return group ? &k_offspring_cont<G, kContInFlight, true> : &k_offspring_cont<G, kContInFlight, false>;
}

OffspringKernel continuous_kernel(uint32_t n_loci, bool group) {
    OffspringKernel k;
    switch (n_loci) {
        case 32: k.fn = cont_instance<4>(group); break;
        case 64: k.fn = cont_instance<8>(group); break;
        case 128: k.fn = cont_instance<16>(group); break;
        case 256: k.fn = cont_instance<32>(group); break;
        default: return OffspringKernel{};
    }
    k.tile = kBlock;
    return k;
}

int prepare_offspring(OffspringKernel &k) {
    if (!k.fn) return SPG_ERR_INVALID;
    const void *fn = reinterpret_cast<const void *>(k.fn);
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return SPG_ERR_CUDA;
    if (k.smem) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)k.smem);
    if (e != cudaSuccess) return SPG_ERR_CUDA;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kBlock, k.smem);
    if (e != cudaSuccess || per_sm <= 0) return SPG_ERR_CUDA;
    k.resident = (uint32_t)per_sm * (uint32_t)sms;
    return SPG_OK;
}

int launch_founders_cont(const PopParams *prm, uint32_t n_loci, uint32_t *geno, uint32_t *surv, uint32_t n,
                         uint32_t p0_q32, void *stream) {
    const dim3 grid((n + 127) / 128), block(128);
    cudaStream_t s = (cudaStream_t)stream;
    switch (n_loci) {
        case 32: k_founders_cont<1><<<grid, block, 0, s>>>(prm, geno, surv, n, p0_q32); break;
        case 64: k_founders_cont<2><<<grid, block, 0, s>>>(prm, geno, surv, n, p0_q32); break;
        case 128: k_founders_cont<4><<<grid, block, 0, s>>>(prm, geno, surv, n, p0_q32); break;
        case 256: k_founders_cont<8><<<grid, block, 0, s>>>(prm, geno, surv, n, p0_q32); break;
        default: return SPG_ERR_INVALID;
    }
    return cudaGetLastError() == cudaSuccess ? SPG_OK : SPG_ERR_CUDA;
}

int launch_founders(uint32_t words, uint32_t *geno, uint32_t *surv, uint32_t n, uint32_t key0, uint32_t key1,
                    uint32_t rep, uint32_t p0_q32, void *stream) {
    const dim3 grid((n + 127) / 128), block(128);
    cudaStream_t s = (cudaStream_t)stream;
    switch (words) {
        case 1: k_founders<1><<<grid, block, 0, s>>>(geno, surv, n, key0, key1, rep, p0_q32); break;
        case 2: k_founders<2><<<grid, block, 0, s>>>(geno, surv, n, key0, key1, rep, p0_q32); break;
        case 4: k_founders<4><<<grid, block, 0, s>>>(geno, surv, n, key0, key1, rep, p0_q32); break;
        case 8: k_founders<8><<<grid, block, 0, s>>>(geno, surv, n, key0, key1, rep, p0_q32); break;
        default: return SPG_ERR_INVALID;
    }
    return cudaGetLastError() == cudaSuccess ? SPG_OK : SPG_ERR_CUDA;
}

int launch_iota(uint32_t *surv, uint32_t n, void *stream) {
    k_iota<<<(n + 255) / 256, 256, 0, (cudaStream_t)stream>>>(surv, n);
    return cudaGetLastError() == cudaSuccess ? SPG_OK : SPG_ERR_CUDA;
}

int launch_pack(const PopParams *prm, uint32_t words, const uint32_t *geno, const uint32_t *surv, uint32_t S, uint32_t n,
                uint32_t slot_len, uint32_t nslots, uint32_t *alive, uint32_t *packed, uint32_t *counts, uint2 *mate,
                GenAcc *acc, unsigned long long *barrier, void *stream) {
    cudaStream_t s = (cudaStream_t)stream;
    const size_t words32 = ((size_t)n + 31) / 32;
    cudaError_t e = cudaMemsetAsync(alive, surv ? 0 : 0xFF, words32 * 4, s);
    if (e != cudaSuccess) return SPG_ERR_CUDA;
    if (surv && S) k_mark_alive<<<(S + 255) / 256, 256, 0, s>>>(surv, S, alive);
    if (!surv && (n & 31u)) k_mark_tail<<<1, 32, 0, s>>>(alive + words32 - 1, n & 31u);
    const dim3 grid((nslots + 7) / 8), block(256);
    switch (words) {
        case 1: k_pack<1><<<grid, block, 0, s>>>(prm, geno, alive, n, slot_len, nslots, packed, counts, mate, acc, barrier); break;
        case 2: k_pack<2><<<grid, block, 0, s>>>(prm, geno, alive, n, slot_len, nslots, packed, counts, mate, acc, barrier); break;
        case 4: k_pack<4><<<grid, block, 0, s>>>(prm, geno, alive, n, slot_len, nslots, packed, counts, mate, acc, barrier); break;
        case 8: k_pack<8><<<grid, block, 0, s>>>(prm, geno, alive, n, slot_len, nslots, packed, counts, mate, acc, barrier); break;
        default: return SPG_ERR_INVALID;
    }
    return cudaGetLastError() == cudaSuccess ? SPG_OK : SPG_ERR_CUDA;
}

SoloKernel solo_kernel_w1(bool linked, bool weighted, bool general);
SoloKernel solo_kernel_w2(bool linked, bool weighted, bool general);
SoloKernel solo_kernel_w4(bool linked, bool weighted, bool general);
SoloKernel solo_kernel_w8(bool linked, bool weighted, bool general);

SoloKernel solo_kernel(uint32_t words, bool linked, bool weighted, bool general) {
    switch (words) {
        case 1: return solo_kernel_w1(linked, weighted, general);
        case 2: return solo_kernel_w2(linked, weighted, general);
        case 4: return solo_kernel_w4(linked, weighted, general);
        case 8: return solo_kernel_w8(linked, weighted, general);
        default: return SoloKernel{};
    }
}

SoloKernel team_kernel_plain();
SoloKernel team_kernel_general();
SoloKernel team_kernel_linked();
SoloKernel team_kernel_weighted();
SoloKernel team_kernel_both();

SoloKernel team_kernel(uint32_t kind) {
    switch (kind) {
        case 0: return team_kernel_plain();
        case 1: return team_kernel_general();
        case 2: return team_kernel_linked();
        case 3: return team_kernel_weighted();
        default: return team_kernel_both();
    }
}

int prepare_solo(SoloKernel &k) {
    if (!k.fn) return SPG_ERR_INVALID;
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)k.smem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k.fn, (int)kSoloThreads, k.smem);
    if (e != cudaSuccess || per_sm <= 0) return SPG_ERR_CUDA;
    k.resident = (uint32_t)per_sm * (uint32_t)sms;
    return SPG_OK;
}

int launch_set_state(DevState *st, StatAcc *acc, uint32_t gen, uint32_t S, uint32_t f, double R, int32_t status,
                     uint32_t target, void *stream) {
    k_set_state<<<1, 32, 0, (cudaStream_t)stream>>>(st, acc, gen, S, f, R, status, target);
    return cudaGetLastError() == cudaSuccess ? SPG_OK : SPG_ERR_CUDA;
}

}  // namespace spg